"""Boxes with far more cells than atoms: blocks without atoms do nothing, and leave nothing of an earlier state."""
import numpy as np
import pytest

import chaingen
import oracle
import paper_1001_3764_gb300 as md

pytestmark = pytest.mark.gpu


# 7, 16 and 48 cells a side for 600 atoms (the last: cells ordered 32 to a block); regions of 3 and 2 cells, and the fixed grid
@pytest.mark.parametrize("L", [8.0, 18.0, 53.0])
@pytest.mark.parametrize("fields", [{}, dict(lj_region=2), dict(schedule=md.MD_SCHED_PERSISTENT), dict(precision=md.MD_PLAIN_FP32)])
def test_sparse_boxes_match_the_oracle_wherever_the_atoms_are(L, fields):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    m = chaingen.melt(4, seed=91, L=L, T=300.0)
    s = md.System(m, **fields)
    ref = oracle.System(oracle.chain_topology(150), 4, m["L"], use_cells=False)
    for shift in (0.0, 2.5, 0.4 * L):        # cells that held atoms are empty afterwards
        x = np.mod(m["pos"] + shift, m["L"])
        s.set_state(x, m["vel"])
        x, v, _ = s.state()
        f, en, _ = ref.forces(x)
        assert np.linalg.norm(s.forces() - f) <= 1e-5 * np.linalg.norm(f)
        e = s.energy()[0]
        for k, want in (("lj", en[0]), ("lj_shifted", en[1]), ("bond", en[2]), ("angle", en[3]), ("dihedral", en[4])):
            assert e[k] == pytest.approx(want, rel=1e-5, abs=1e-5 * abs(en[1])), k
        perm = s.bins()[2]
        assert np.array_equal(np.sort(perm), np.arange(600))
    s.step(12)
    xs, _, img = s.state()
    xo, *_ = ref.run(x, v, 0.001, 12, sample_every=0)
    d = xs + img * m["L"] - xo
    d -= m["L"] * np.round(d / m["L"])
    assert np.abs(d).max() < (2e-4 if fields.get("precision") == md.MD_PLAIN_FP32 else 1e-5)   # the suite's
    s.close()
