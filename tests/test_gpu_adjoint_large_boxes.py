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
