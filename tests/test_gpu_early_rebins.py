"""Early rebins (an atom beyond skin/2 before the block's end) at every place they can come: each drift of a block, the
opening one among them, group ends, remainders, thermostats, general molecules, two LJ launches a step."""
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


def follows(a, b, n, dt=0.001):
    """Both after n steps from one state.  Forces agree to the relative error of the FP32 terms (1e-5, the suite's), so v
    may differ by n dt |F| / m of that and x by n dt of v's difference."""
    scale = np.linalg.norm(a.forces()) * dt / 14.0
    a.step(n)
    b.step(n)
    (xa, va, ia), (xb, vb, ib) = a.state(), b.state()
    L = np.repeat([m["L"] for m in a.melts], [len(m["pos"]) for m in a.melts])[:, None]
    assert np.linalg.norm(va - vb) <= 1e-5 * n * scale
    assert np.linalg.norm((xa - xb) + L * (np.asarray(ia) - np.asarray(ib))) <= 1e-5 * n * scale * n * dt


# skin 0.0004: every drift reports; 0.004: about every second; 0.02: a few a block
@pytest.mark.parametrize("skin", [0.0004, 0.004, 0.02])
@pytest.mark.parametrize("thermostat", [md.MD_NVE, md.MD_VRESCALE, md.MD_NOSE_HOOVER])
@pytest.mark.parametrize("kind,rebin_every,n", [("chains", 7, 18), ("chains", 25, 34), ("molecules", 17, 24)])
def test_runs_with_early_rebins_follow_those_without(kind, rebin_every, n, thermostat, skin):
    m = chaingen.melt(10, seed=1, L=3.75, T=300.0)
    kw = dict(thermostat=thermostat)
    if thermostat != md.MD_NVE:
        kw["T_target"] = 350.0
    if kind == "molecules":
        kw["topology"] = (np.array([(k, k + 1) for k in range(149)], np.int32), np.array([1] + [0] * 148 + [1], np.int32))
    a = md.System(m, skin=skin, rebin_every=rebin_every, **kw)
    b = md.System(m, skin=0.2, rebin_every=5, **kw)
    follows(a, b, n)
    assert a.early_rebins() > 0 and b.early_rebins() == 0
    if skin == 0.0004:
        # every drift of the run
        assert a.early_rebins() == n
    a.close()
    b.close()


@pytest.mark.parametrize("thermostat", [md.MD_NVE, md.MD_NOSE_HOOVER])
def test_early_rebins_with_two_lj_launches_a_step(thermostat):
    """Eight sparse replicas and a dense one whose cells are larger: its tiles are left to a second LJ launch."""
    melts = [chaingen.melt(60, seed=400 + k, L=19.625, T=300.0) for k in range(8)] + [chaingen.melt(40, seed=420, L=5.625, T=300.0)]
    kw = dict(rc=1.3, thermostat=thermostat)
    if thermostat != md.MD_NVE:
        kw["T_target"] = 350.0
    a = md.System(melts, skin=0.004, rebin_every=12, **kw)
    b = md.System(melts, skin=0.1, rebin_every=5, **kw)
    assert md.md_launches_per_call(a.h, 12) == 8 + 3 * 12
    follows(a, b, 15)
    assert a.early_rebins() > 0 and b.early_rebins() == 0
    a.close()
    b.close()


@pytest.mark.parametrize("skin", [0.1, 0.004])
@pytest.mark.parametrize("thermostat", [md.MD_VRESCALE, md.MD_NOSE_HOOVER])
def test_the_schedules_give_the_same_bits_with_a_thermostat(thermostat, skin):
    """The thermostat's blocks come before the LJ kernel's, whichever way these get their items."""
    melts = [chaingen.melt(c, seed=30 + c, T=300.0) for c in (10, 25)]
    kw = dict(thermostat=thermostat, T_target=[300.0, 400.0], skin=skin, rebin_every=8)
    a = md.System(melts, schedule=md.MD_SCHED_GRID, **kw)
    b = md.System(melts, schedule=md.MD_SCHED_PERSISTENT, **kw)
    for s in (a, b):
        s.step(21)
    for p, q in zip(a.state(), b.state()):
        assert np.array_equal(p, q)
    a.close()
    b.close()
