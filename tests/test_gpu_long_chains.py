"""Chains of 257 to 513 sites with a thermostat: the step kernel's 512-thread block and its neighbours."""
import numpy as np
import pytest

import chaingen
import oracle
import paper_1001_3764_gb300 as md

pytestmark = pytest.mark.gpu

TOL = {md.MD_MIXED: 1e-5, md.MD_PLAIN_FP32: 2e-4}   # nm, the suite's for 50 steps of these ensembles


@pytest.mark.parametrize("precision", [md.MD_MIXED, md.MD_PLAIN_FP32])
@pytest.mark.parametrize("thermostat", [md.MD_VRESCALE, md.MD_NOSE_HOOVER])
@pytest.mark.parametrize("sites", [257, 352, 353, 384, 480, 481, 512, 513])
def test_thermostatted_long_chains_follow_the_oracle(sites, thermostat, precision):
    """14 steps (a block, and a remainder with its own graph) from 450 K towards 300 K, against the oracle's run."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    m = chaingen.melt(5, sites=sites, seed=300 + sites, T=450.0, L=4.375)
    s = md.System(m, precision=precision, thermostat=thermostat, T_target=300.0, tau_t=0.1)
    x0, v0, _ = s.state()
    s.step(14)
    x, _, img = s.state()
    s.close()
    ref = oracle.System(oracle.chain_topology(sites), 5, m["L"])
    if thermostat == md.MD_NOSE_HOOVER:
        xo, *_ = ref.run_nh(x0, v0, 0.001, 14, T0=300.0, tau=0.1, sample_every=0)
    else:
        xo, *_ = ref.run(x0, v0, 0.001, 14, thermostat=True, T0=300.0, tau=0.1, sample_every=0)
    d = x + img * m["L"] - xo
    d -= m["L"] * np.round(d / m["L"])
    assert np.abs(d).max() < TOL[precision]
    moved = x + img * m["L"] - x0
    assert np.sqrt(np.mean(moved ** 2)) > 10 * TOL[precision]
