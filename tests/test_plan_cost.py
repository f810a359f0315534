"""What the host does for a box of many cells: a few runs of regions, not a table of them.  On the CPU (stand-in runtime)."""
import ctypes
import time

import pytest

import paper_1001_3764_gb300 as md
from fake_cudart import Fake, lattice, link


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return link(str(tmp_path_factory.mktemp("fake")))


def test_the_size_of_a_nearly_empty_box_is_planned_at_once(lib):
    """390 cells a side, 59 million, 6.6 million regions: their tables take seconds and 1.3 GB on the host."""
    s = Fake(lib, lattice(10, 150, 430.0))
    size, t = ctypes.c_size_t(), []
    for _ in range(3):
        t0 = time.perf_counter()
        assert lib.md_workspace_size(ctypes.byref(s.desc), ctypes.byref(size)) == md.MD_OK
        t.append(time.perf_counter() - t0)
    assert size.value > 59e6 * 8 and min(t) < 0.1


@pytest.mark.parametrize("boxes", [[3.875], [19.5], [4.5, 9.0, 3.375], [40.0]])
@pytest.mark.parametrize("region", [2, 3])
def test_the_blocks_are_as_many_as_the_rules_ask_for(lib, boxes, region):
    """Launch sizes of the list build and the task order: whole regions, rows or cells, as counted here one by one."""
    s = Fake(lib, [lattice(10, 150, L) for L in boxes], lj_region=region)
    assert s.create() == md.MD_OK
    lib.fake_reset()
    assert lib.md_rebin(s.h) == md.MD_OK
    grid = {n: lib.fake_grid(i) for i in range(lib.fake_ran()) for n in (b"k_cl_build", b"k_cl_rank") if n in lib.fake_kernel(i)}
    regions = []                        # (cells, rows) of each
    for L in boxes:
        M = int(L / 1.1)
        sides = [min(region, M - x) for x in range(0, M, region)]
        regions += [(sx * sy, sy) for _ in range(M) for sy in sides for sx in sides]
    cells, rows = (sum(r[k] for r in regions) for k in (0, 1))
    build = len(regions) if len(regions) >= 12 * 152 else rows if len(regions) >= 2 * 152 else cells
    assert grid[b"k_cl_build"] == build * (3 if cells <= 128 else 1)
    slots = (2 if region == 3 else 3) * 152     # tiles of 1.1 nm cells that two (three) blocks an SM hold
    if cells <= slots:
        lj = cells
    elif rows <= slots:
        lj = rows
    elif len(regions) <= slots:
        order = sorted(regions, reverse=True, key=lambda r: r[0])
        lj = min(152, len(order)) + sum(r[1] for r in order[152:])
    else:
        lj = len(regions)
    assert grid[b"k_cl_rank"] == lj
    s.close()
