"""RDF and chain observables of the CUDA path where their fast forms can go wrong."""
import numpy as np
import pytest

import chaingen
import paper_1001_3764_gb300 as md

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    md.load()


def _lattice_chains(sites, L, spacing, n_chains, seed):
    """Straight chains along x on a cubic lattice (exact in FP32), one row each, rows drawn at random:
    many pairs at distances that are exact multiples of the spacing."""
    per = int(round(L / spacing))
    rng = np.random.default_rng(seed)
    rows = rng.permutation(per * per)[:n_chains]
    x0 = rng.integers(0, per, n_chains)
    k = np.arange(sites)
    pos = np.empty((n_chains, sites, 3))
    pos[:, :, 0] = ((x0[:, None] + k[None]) % per) * spacing
    pos[:, :, 1] = (rows // per)[:, None] * spacing
    pos[:, :, 2] = (rows % per)[:, None] * spacing
    return dict(pos=pos.reshape(-1, 3), vel=np.zeros((n_chains * sites, 3)), L=L, n_chains=n_chains, sites=sites)


@pytest.mark.parametrize("precision", [md.MD_MIXED, md.MD_PLAIN_FP32])
@pytest.mark.parametrize("L,n_bins", [(3.5, 64), (4.5, 64), (3.5, 5000)])
def test_rdf_of_lattice_distances_on_bin_edges(precision, L, n_bins):
    """Distances that lie exactly on bin edges and on r_max, 3 and 4 cells per side, and bins narrower than the
    FP32 distance's error band allows to decide: the integer counts equal the FP64 definition's."""
    from oracle import observables as ob
    m = _lattice_chains(6, L, 0.25, 120, seed=3)
    s = md.System(m, precision=precision)
    _, _, counts = s.rdf(1.0, n_bins)
    _, _, want = ob.rdf(m["pos"], L, m["sites"], 1.0, n_bins)
    assert np.array_equal(counts[0], want)
    s.close()


@pytest.mark.parametrize("skin,L,n_chains", [(0.1, 4.375, 55), (0.4, 6.625, 192)])
@pytest.mark.parametrize("r_max", [0.35, 1.0])
def test_rdf_of_full_cells(skin, L, n_chains, r_max):
    """Cells of about 102 atoms at 3 a side (folded images) and 150 at 4 (home atoms in two stages, the second of few
    and odd numbers), with most of the candidates in reach and with few: counts equal to the FP64 definition's."""
    from oracle import observables as ob
    m = chaingen.melt(n_chains, sites=50, seed=23, T=300.0, L=L)
    s = md.System(m, skin=skin, lj_region=2)   # 3 x 3 cells of 150 atoms do not fit a tile
    _, _, counts = s.rdf(r_max, 200)
    _, _, want = ob.rdf(s.state()[0], L, 50, r_max, 200)
    assert np.array_equal(counts[0], want)
    s.close()


def test_rdf_from_a_positive_first_edge():
    """edges[0] > 0: nearer pairs are left out, and the first edge is inclusive."""
    import ctypes
    m = _lattice_chains(6, 3.5, 0.25, 120, seed=4)
    s = md.System(m)
    edges = np.linspace(0.5, 1.0, 33)
    counts = np.zeros(32, np.int64)
    rc = md.load().md_rdf(s.h, 32, edges.ctypes.data_as(ctypes.c_void_p), counts.ctypes.data_as(ctypes.c_void_p))
    assert rc == md.MD_OK
    x, n = m["pos"], len(m["pos"])
    d = x[:, None] - x[None]
    d -= 3.5 * np.round(d / 3.5)
    r = np.sqrt((d * d).sum(2))
    i, j = np.triu_indices(n, 1)
    keep = ~((i // 6 == j // 6) & (j - i <= 2))
    want, _ = np.histogram(r[i[keep], j[keep]], bins=edges)
    assert np.array_equal(counts, want)
    s.close()


@pytest.mark.parametrize("sites", [4, 31, 32, 33, 64, 65, 97])
def test_chain_observables_at_warp_remainders(sites):
    """Chain lengths around multiples of the 32 lanes a chain is walked with, several replicas."""
    from oracle import observables as ob
    n_chains = max(3, 1300 // sites)
    melts = [chaingen.melt(n_chains + k, sites, seed=60 + k, L=3.6) for k in range(3)]
    s = md.System(melts)
    got = s.observables()
    off = 0
    for r, m in enumerate(melts):
        xu, n = chaingen.unwrapped(m), m["n_chains"]
        assert np.allclose(got["r_ee"][off:off + n], ob.end_to_end(xu, sites), rtol=1e-12, atol=1e-12)
        assert np.allclose(got["rg2"][off:off + n], ob.radius_of_gyration_sq(xu, sites, m["masses"]), rtol=1e-10)
        phi = ob.dihedral_angles(xu, sites)
        near = np.sum(np.abs(np.abs(phi) - 120.0) < 1e-6)
        assert abs(got["trans_fraction"][r] - np.mean(np.abs(phi) > 120.0)) <= near / phi.size + 1e-15
        off += n
    s.close()
