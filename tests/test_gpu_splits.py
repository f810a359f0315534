"""How regions are split over blocks (whole, rows, single cells, parts of a cell's clusters) must not be seen in
any result: the same melt run alone and in a batch large enough to change the split gives the same bits."""
import numpy as np
import pytest

import chaingen
import oracle
import paper_1001_3764_gb300 as md

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    md.load()


@pytest.mark.parametrize("exact", [False, True])
def test_split_regions_give_the_bits_of_whole_ones(exact):
    """Alone: 3 (parts of cells), 6, 7 and 9 (cells, rows) cells per side.  Together: over 304 regions, whole."""
    melts = [chaingen.melt(n, seed=70 + k, T=300.0) for k, n in enumerate((10, 60, 120, 230, 230, 230, 200, 180))]
    kw = dict(precision=md.MD_MIXED, rebin_every=4, lj_pair_exact=exact)
    both = md.System(melts, **kw)
    f_both, e_both = both.forces(), both.energy()
    both.step(9)
    x_both, v_both, _ = both.state()
    off = 0
    for r, m in enumerate(melts):
        n = len(m["pos"])
        if r < 4:
            alone = md.System(m, **kw)
            assert np.array_equal(alone.forces(), f_both[off:off + n])
            e = alone.energy()[0]
            assert e == e_both[r]
            alone.step(9)
            x, v, _ = alone.state()
            assert np.array_equal(x, x_both[off:off + n]) and np.array_equal(v, v_both[off:off + n])
            alone.close()
        off += n
    both.close()


@pytest.mark.parametrize("L,n_chains", [(3.35, 8), (4.5, 20), (7.8, 105), (9.95, 216), (13.4, 520)])
def test_every_split_gives_the_oracle_forces(L, n_chains):
    """3 to 12 cells per side (whole regions behind rows at 12), dilute and dense, narrow regions at 4, 7 and 8."""
    m = chaingen.melt(n_chains, seed=80, L=L)
    s = md.System(m, precision=md.MD_MIXED)
    n = len(m["pos"])
    ref = oracle.System(oracle.chain_topology(m["sites"]), n_chains, m["L"], use_cells=n > 3000)
    f_orc, en, _ = ref.forces(np.array(m["pos"], np.float64))
    f = s.forces()
    # relative RMS of the FP32 pair and bonded arithmetic (the suite's force tolerance)
    assert np.linalg.norm(f - f_orc) <= 1e-5 * np.linalg.norm(f_orc)
    e = s.energy()[0]
    for k, idx in (("lj", 0), ("lj_shifted", 1), ("bond", 2), ("angle", 3), ("dihedral", 4)):
        assert abs(e[k] - en[idx]) <= 1e-5 * max(1.0, abs(en[idx]))
    s.close()


def test_large_tiles_of_an_uneven_box():
    """Cells of 1.31 nm (skin 0.3): in the batch (441 rows) the force kernel's tile is the one that fits an SM twice,
    3,776 atoms, and the dense parts (42 sites/nm^3 in 44 cells: 4,200 atoms) of the first replica go to the launch for
    large tiles.  Alone it is split into rows.  The bits are the same."""
    L0, L, sites = 7.0, 9.2, 8
    melts = []
    for seed, n, side in ((5, 1800, L0), (6, 3200, L), (7, 3200, L)):
        m = chaingen.melt(n, sites=sites, seed=seed, T=300.0, L=side)
        x = m["pos"].reshape(n, sites, 3).copy()
        d = np.diff(x, axis=1)
        x[:, 1:] = x[:, :1] + np.cumsum(d - side * np.round(d / side), axis=1)
        melts.append(dict(m, pos=np.mod(x.reshape(-1, 3) + (2.4, 2.4, 0.0), L), L=L))
    kw = dict(precision=md.MD_MIXED, skin=0.3, rebin_every=3)
    both, alone = md.System(melts, **kw), md.System(melts[0], **kw)
    n = len(melts[0]["pos"])
    for _ in range(2):
        assert np.array_equal(alone.forces(), both.forces()[:n])
        assert alone.energy()[0] == both.energy()[0]
        alone.step(4)
        both.step(4)
    assert np.array_equal(alone.state()[0], both.state()[0][:n])
    alone.close()
    both.close()
