"""md_launches_per_call against the launches and memsets that the graphs hold, on the CPU (stand-in runtime)."""
import pytest

import paper_1001_3764_gb300 as md
from fake_cudart import Fake, lattice, link


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return link(str(tmp_path_factory.mktemp("fake")))


# 3 and 50 cells per side, 51 (more than 131,072 cells: a scan in two launches), and tiles for two LJ launches
@pytest.mark.parametrize("boxes,fields", [([3.875], {}), ([55.25], {}), ([56.5], {}), ([3.875], dict(displacement=md.MD_DISP_ERROR)),
                                          ([19.625] * 8 + [5.625], dict(skin=0.3))])
def test_launches_per_call_counts_what_runs(lib, boxes, fields):
    s = Fake(lib, [lattice(60 if len(boxes) > 1 else 10, 150, L) for L in boxes], rebin_every=5, **fields)
    assert s.create() == md.MD_OK
    assert lib.md_step(s.h, 5) == md.MD_OK      # the first block takes the bins of the creation
    for n in (5, 15, 3, 12, 0):
        lib.fake_reset()
        assert lib.md_step(s.h, n) == md.MD_OK
        assert lib.fake_ran() == lib.md_launches_per_call(s.h, n)
    s.close()
