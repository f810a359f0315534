"""The adjoint's cell order over its radix passes: two up to 262,144 cells (64 a side), three above, with the last pass's
places found by its blocks (up to 8,192 atoms) and by a launch of their own."""
import numpy as np
import pytest

import chaingen
import oracle
import paper_1001_3764_gb300 as md

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_chains", [12, 60])
@pytest.mark.parametrize("L", [64.5, 65.5, 131.5])
def test_gradient_and_means_in_boxes_of_many_cells(n_chains, L):
    """One energy gradient and a three-step trajectory against the oracle, with the tolerances of the suite's small boxes."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    m = chaingen.melt(n_chains, seed=77, L=L, T=300.0)
    x = chaingen.unwrapped(m)
    ref = oracle.System(oracle.chain_topology(150), n_chains, m["L"], use_cells=True)
    f, en, _ = ref.forces(x)
    a = md.Adjoint(m, n_steps=3, checkpoint_every=2)
    d = np.random.default_rng(1).standard_normal(x.shape)
    g, h, _, _ = a.tangent(x, d)
    assert np.abs(g + f).max() <= 1e-10 * np.abs(f).max()
    e = a.energy()
    assert e["U"] == pytest.approx(en[1] + en[2] + en[3] + en[4], rel=1e-11)
    step = 1e-6
    fd = -(ref.forces(x + step * d)[0] - ref.forces(x - step * d)[0]) / (2 * step)
    assert np.linalg.norm(h - fd) < 1e-6 * np.linalg.norm(fd)
    assert a.forward() == pytest.approx(ref.traj_means(x, m["vel"], 0.001, 3), rel=1e-9)
    a.close()


def test_pairs_just_inside_the_cutoff_are_found_in_boxes_of_hundreds_of_nm():
    """Dimers whose first sites lie 2e-6 nm inside r_c of another's, over a box of 1,800 nm and across its faces: an FP32
    coordinate there is known to 6e-5 nm.  Each such site feels the truncated force of its one pair."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    rng = np.random.default_rng(5)
    L, rc, n = 1800.0, 1.0, 4000
    p = md.default_params()
    a = rng.uniform(0.0, L, (n, 3))
    a[::4, 0] = rng.uniform(-0.5, 0.5, n // 4)          # pairs across a face
    u = rng.standard_normal((n, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    b = a + (rc - 2e-6) * u
    x = np.empty((2 * n, 2, 3))
    x[0::2, 0], x[1::2, 0] = a, b
    x[0::2, 1], x[1::2, 1] = a - p["b0"] * u, b + p["b0"] * u     # the second sites point away: out of range
    x = x.reshape(-1, 3)
    m = dict(pos=x, vel=np.zeros_like(x), L=L, n_chains=2 * n, sites=2)
    adj = md.Adjoint(m, n_steps=0, rc=rc, params=dict(p, kb=0.0))
    g, _, _, _ = adj.tangent(x, np.zeros_like(x))
    adj.close()
    d = b - a
    r = np.linalg.norm(d, axis=1)
    eps, sig = p["eps"][1], p["sigma"][1]               # all sites are chain ends
    dEdr = 4 * eps * (6 * sig ** 6 / r ** 7 - 12 * sig ** 12 / r ** 13)
    want = -(dEdr / r)[:, None] * d                      # on a; r itself is rounded by 2^-53 L / r_c in x
    got = g.reshape(-1, 2, 3)
    assert np.abs(got[0::2, 0] - want).max() <= 1e-9 * np.abs(want).max()
    assert np.abs(got[1::2, 0] + want).max() <= 1e-9 * np.abs(want).max()
    assert np.abs(got[:, 1]).max() == 0.0
