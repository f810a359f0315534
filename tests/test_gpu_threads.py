"""Systems of several threads at once: created, stepped (blocks and remainders, whose graphs are captured on first use),
read out and closed, with histograms of different sizes; the same bits as one after another."""
import threading

import numpy as np
import pytest

import chaingen
import paper_1001_3764_gb300 as md

pytestmark = pytest.mark.gpu

KINDS = [dict(), dict(precision=md.MD_PLAIN_FP32, thermostat=md.MD_NOSE_HOOVER, T_target=300.0),
         dict(thermostat=md.MD_VRESCALE, T_target=350.0, skin=0.004), dict(schedule=md.MD_SCHED_PERSISTENT, rebin_every=25)]


def work(k):
    m = chaingen.melt(10 + k, seed=5 + k, L=4.0, T=300.0)
    out = []
    for _ in range(2):
        s = md.System(m, **KINDS[k])
        for j in range(4):
            s.step(7 + j)
            out += [[s.energy()[0][q] for q in ("lj", "bond", "kinetic")], s.rdf(0.9, (50, 9500, 16384, 12000)[(j + k) % 4])[2]]
        out += list(s.state())
        s.close()
    return np.concatenate([np.asarray(a, np.float64).ravel() for a in out])


def test_threads_get_the_bits_of_one_thread():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    md.load()
    want = [work(k) for k in range(len(KINDS))]
    got, errors = [None] * len(KINDS), []

    def run(k):
        try:
            got[k] = work(k)
        except Exception as e:
            errors.append((k, e))

    threads = [threading.Thread(target=run, args=(k,)) for k in range(len(KINDS))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for a, b in zip(want, got):
        assert np.array_equal(a, b)
