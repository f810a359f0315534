"""md_autotune where the default block of the LJ kernel is one that no explicit lj_block names (768 threads, cells of
which one tile fills an SM): the default is a candidate.  On the CPU, with the stand-in runtime's times."""
import ctypes

import pytest

import paper_1001_3764_gb300 as md
from fake_cudart import Fake, lattice, link


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return link(str(tmp_path_factory.mktemp("fake")))


def tune(lib, s, cache=None):
    out = md.md_tuning()
    assert lib.md_autotune(ctypes.byref(s.desc), 1, cache, ctypes.byref(out)) == md.MD_OK
    return out


def lj_block(lib, s):
    assert s.create() == md.MD_OK
    lib.fake_reset()
    assert lib.md_step(s.h, 1) == md.MD_OK
    blocks = {lib.fake_block(i) for i in range(lib.fake_ran()) if b"k_cl_force" in lib.fake_kernel(i)}
    s.close()
    return blocks


@pytest.mark.parametrize("fast,want", [(768, 0), (384, 384), (256, 256)])
def test_the_default_block_is_tried_and_kept_where_it_is_fastest(lib, tmp_path, fast, want):
    """LJ launches of smaller blocks than `fast` take twice as long as others (so the first candidate at it wins)."""
    cache = str(tmp_path / "cache.txt").encode()
    make = lambda: Fake(lib, lattice(60, 150, 27.25), skin=0.3, rebin_every=10)
    assert lj_block(lib, make()) == {768}
    lib.fake_slow(b"k_cl_force", fast)
    s = make()
    t = tune(lib, s, cache)
    assert t.lj_block == s.desc.lj_block == want and t.from_cache == 0
    if fast == 768:
        assert lj_block(lib, s) == {768}
        again = make()
        t2 = tune(lib, again, cache)
        assert t2.from_cache == 1 and again.desc.lj_block == 0 and lj_block(lib, again) == {768}
    lib.fake_slow(b"", 0)


def test_a_default_of_named_size_is_reported_by_its_size(lib):
    s = Fake(lib, lattice(10, 150, 3.875))
    lib.fake_slow(b"k_cl_force", 384)
    assert tune(lib, s).lj_block == 384
    lib.fake_slow(b"", 0)
