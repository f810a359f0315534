"""What an early rebin (an atom beyond skin/2) costs: the launches of its group of steps, however long the block is.  On
the CPU, from the graphs that the host code makes on the stand-in runtime."""
import pytest

import paper_1001_3764_gb300 as md
from fake_cudart import Fake, lattice, link


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return link(str(tmp_path_factory.mktemp("fake")))


@pytest.mark.parametrize("rebin_every", [1, 10, 16, 17, 25, 50, 200])
@pytest.mark.parametrize("fields", [{}, dict(thermostat=md.MD_NOSE_HOOVER), dict(displacement=md.MD_DISP_ERROR)])
def test_no_group_is_longer_than_sixteen_steps(lib, rebin_every, fields):
    s = Fake(lib, lattice(10, 150, 3.875), rebin_every=rebin_every, **fields)
    lib.fake_reset()
    assert s.create() == md.MD_OK
    nodes = lib.fake_calls(b"cudaGraphAddNode")          # WHILE nodes of the two graphs of a block
    if s.desc.displacement == md.MD_DISP_ERROR:
        assert nodes == 0
    else:
        assert nodes % 2 == 0 and 16 * (nodes // 2) >= rebin_every
        assert rebin_every > 16 or nodes == 2
    # the block itself is the same launches whatever the groups
    assert lib.md_step(s.h, rebin_every) == md.MD_OK
    lib.fake_reset()
    assert lib.md_step(s.h, rebin_every) == md.MD_OK
    assert lib.fake_ran() == lib.md_launches_per_call(s.h, rebin_every) == 8 + 2 * rebin_every
    assert sum(b"k_cl_force" in lib.fake_kernel(i) for i in range(lib.fake_ran())) == rebin_every
    s.close()
