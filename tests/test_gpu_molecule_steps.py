"""The step kernel of general molecules, over the sizes its blocks take: several molecules to one, 128 threads and more."""
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


@pytest.mark.parametrize("sites,n_chains,thermostat",
                         [(4, 331, md.MD_NVE), (7, 190, md.MD_NOSE_HOOVER), (64, 21, md.MD_VRESCALE), (65, 20, md.MD_NVE),
                          (128, 11, md.MD_NOSE_HOOVER), (129, 11, md.MD_VRESCALE), (1000, 2, md.MD_NVE),
                          (1022, 2, md.MD_NOSE_HOOVER)])
def test_chains_as_bond_graphs_step_like_chains(sites, n_chains, thermostat):
    """The same chains by their bond graph and by the chain kernels.  Forces agree to the relative error of the FP32
    terms (1e-5, the suite's), so after n steps v may differ by n dt |F| / m of that and x by n dt of v's difference."""
    m = chaingen.melt(n_chains, sites=sites, seed=100 + sites, T=300.0)
    bonds = np.array([(k, k + 1) for k in range(sites - 1)], np.int32)
    types = np.zeros(sites, np.int32)
    types[[0, -1]] = 1
    kw = dict(precision=md.MD_MIXED, thermostat=thermostat, rebin_every=4)
    if thermostat != md.MD_NVE:
        kw["T_target"] = 300.0
    a, b = md.System(m, **kw), md.System(m, topology=(bonds, types), **kw)
    n, dt = 6, 0.001
    scale = np.linalg.norm(a.forces()) * dt / 14.0
    a.step(n)
    b.step(n)
    (xa, va, ia), (xb, vb, ib) = a.state(), b.state()
    fa, fb = a.forces(), b.forces()
    assert np.linalg.norm(fa - fb) <= 1e-5 * np.linalg.norm(fa)
    assert np.linalg.norm(va - vb) <= 1e-5 * n * scale
    dx = (xa - xb) + m["L"] * (np.asarray(ia) - np.asarray(ib))
    assert np.linalg.norm(dx) <= 1e-5 * n * scale * n * dt
    a.close()
    b.close()
