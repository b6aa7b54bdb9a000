"""step_plan.h compiled for the host. The launches of a call's steps on a D2Q9 grid: never dearer by the rule's
own figures than single steps, for every number of steps of a call and not only for many, an even number
where the parity of the steps asks for one, and within the kernel's limits; the expected plans are those of the
measured times named beside them. The blocks of a single step: every cell of a plane in one lane, and 64-bit
addresses from 2^29 cells on.
"""
import ctypes
import subprocess
from pathlib import Path

import pytest

from paper_2407_12263_gb300 import inputs as I
from paper_2407_12263_gb300 import lbm

CSRC = Path(__file__).resolve().parent.parent / "paper_2407_12263_gb300" / "csrc"
SMS = 152


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(f'''#include "{CSRC}/step_plan.h"
extern "C" double plan(int nx, int ny, int fd, int n, int parity, int sms, int* out) {{
    const lbm::StepPlan p = lbm::plan_steps(nx, ny, fd, n, parity, sms);
    *out = p.parts;
    return p.cost;
}}
extern "C" void shape(int nx, int ny, int nz, int narrow, unsigned* out) {{
    const lbm::StepShape h = lbm::step_shape(nx, ny, nz, narrow);
    const unsigned v[] = {{h.block[0], h.block[1], h.grid[0], h.grid[1], h.grid[2], (unsigned)h.form, h.d.mul, (unsigned)h.d.shift}};
    for (int k = 0; k < 8; ++k) out[k] = v[k];
}}''')
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wall", "-Werror", "-o", d / "plan.so", d / "plan.cpp"], check=True)
    return ctypes.CDLL(str(d / "plan.so"))


@pytest.fixture(scope="module")
def plan(library):
    f = library.plan
    f.restype = ctypes.c_double
    out = ctypes.c_int()

    def call(nx, ny, fd, n, parity, sms=SMS):
        cost = f(nx, ny, fd, n, parity, sms, ctypes.byref(out))
        return out.value, cost
    return call


@pytest.fixture(scope="module")
def shape(library):
    def call(nx, ny, nz, narrow):
        out = (ctypes.c_uint * 8)()
        library.shape(nx, ny, nz, narrow, out)
        return dict(zip(("bx", "by", "gx", "gy", "gz", "form", "mul", "shift"), out))
    return call


WHOLE, PACKED, WIDE = 0, 1, 2


@pytest.mark.parametrize("ny", [3, 20, 129])
def test_step_blocks_cover_a_plane(shape, ny):
    for nx in list(range(3, 3000)) + [65535, 65537, 1 << 20, (1 << 20) + 1, 5000011, 16000001]:
        h = shape(nx, ny, 5, 0)
        assert h["bx"] * h["by"] == 128 and h["gz"] == 5
        if h["form"] == WHOLE:
            assert h["gx"] * h["bx"] >= nx > (h["gx"] - 1) * h["bx"] and h["gy"] * h["by"] >= ny > (h["gy"] - 1) * h["by"]
            assert h["gx"] * h["gy"] == -(-nx * ny // 128)
        else:
            assert h["form"] == PACKED and h["gy"] == 1 and h["gx"] * 128 >= nx * ny > (h["gx"] - 1) * 128
            # the row of a cell, at the ends of rows and of the plane and of the largest plane
            last = (1 << 31) - 1
            for i in (0, nx - 1, nx, 2 * nx - 1, nx * ny - 1, nx * ny, last // nx * nx - 1, last // nx * nx, last):
                assert (i * h["mul"] >> 32) >> h["shift"] == i // nx


@pytest.mark.parametrize("grid,narrow,form", [((512, 512, 2048), 1, WIDE), ((512, 512, 2047), 1, WHOLE), ((512, 512, 2048), 0, WHOLE),
                                              ((1000, 700, 766), 1, PACKED), ((1000, 700, 767), 1, WIDE), ((1000, 700, 767), 0, PACKED),
                                              ((1 << 29, 3, 1), 0, WHOLE), ((700000001, 3, 1), 0, PACKED)])
def test_step_form_around_2_to_the_29_cells(shape, grid, narrow, form):
    assert shape(*grid, narrow)["form"] == form
    assert narrow == 0 or (form == WIDE) == (grid[0] * grid[1] * grid[2] >= 1 << 29)


@pytest.mark.parametrize("fd", [0, 1])
@pytest.mark.parametrize("grid", [(3, 3), (40, 40), (64, 64), (97, 96), (128, 128), (184, 184), (200, 168), (216, 216), (256, 256), (304, 304),
                                  (16, 700), (700, 16), (3, 4000), (300, 40), (1200, 1200), (3, 700000000)])
def test_a_plan_is_never_dearer_than_single_steps(plan, grid, fd):
    for parity in (0, 1):
        for n in range(1, 70):
            parts, cost = plan(*grid, fd, n, parity)
            single = plan(*grid, fd, 1, 0)[1]
            assert cost <= n * single * (1 + 1e-12)
            if parts:
                most = -(-n // parts)
                tile = 16 - 2 * most * (2 if fd else 1)
                assert tile >= 4 and parts >= 1 and most >= 1
                assert not parity or (parts - n) % 2 == 0
            assert plan(*grid, fd, n, parity, 0)[0] == 0


@pytest.mark.parametrize("side,n,parity", [
    (64, 2, 1),     # two single steps of a captured call 3.1 us, two regions of a step each 4.4
    (128, 2, 1),    # 3.4 and 6.6
    (184, 2, 0),    # 4.0 and 4.96
    (200, 2, 0),    # 4.1 and 5.0
    (200, 4, 0),    # 8.2 and 9.9
    (184, 2, 1), (200, 4, 1)])
def test_short_calls_that_take_single_steps(plan, side, n, parity):
    assert plan(side, side, 0, n, parity)[0] == 0


# launches for 32 steps; 0 where four handles side by side are faster with single steps
@pytest.mark.parametrize("side,fd,parts", [(64, 0, 7), (96, 0, 8), (128, 0, 16), (184, 0, 0), (216, 0, 0),
                                           (64, 1, 16), (96, 1, 16), (128, 1, 16), (184, 1, 32), (216, 1, 0)])
def test_plans_leave_room_for_other_handles(plan, side, fd, parts):
    assert plan(side, side, fd, 32, 0)[0] == parts


@pytest.mark.gpu
@pytest.mark.parametrize("side,n", [(184, 2), (200, 2), (200, 4)])
def test_short_calls_launch_single_steps(side, n):
    grid = (side, side, 1)
    with lbm.Lattice(grid, 9) as g:
        g.init_phi(I.droplet_phi(grid, side / 4, 4.0))
        before = g.launch_count
        g.step(n)
        assert g.launch_count - before == n
