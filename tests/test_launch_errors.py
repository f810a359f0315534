"""A launch or graph call that the runtime refuses fails the call that made it, and that call alone.  On the CPU: the
library's host code on a stand-in runtime whose nth launch, memset or graph call fails."""
import ctypes

import numpy as np
import pytest

import paper_1001_3764_gb300 as md
from fake_cudart import Fake, lattice, link

GRAPH_CALLS = ["cudaStreamBeginCapture", "cudaStreamGetCaptureInfo", "cudaGraphConditionalHandleCreate", "cudaGraphAddNode",
               "cudaStreamUpdateCaptureDependencies", "cudaStreamBeginCaptureToGraph", "cudaStreamEndCapture",
               "cudaGraphInstantiate", "cudaGraphLaunch",
               "invalidated"]    # the capture is found invalidated by another thread's call: no graph to add to


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return link(str(tmp_path_factory.mktemp("fake")))


def calls(lib, s):
    """every call that launches something, by name"""
    n = s.n
    out = [np.zeros(3 * n) for _ in range(2)] + [np.zeros(3 * n, np.int32)]
    p = [a.ctypes.data for a in out]
    edges, counts = np.linspace(0.0, 0.9, 11), np.zeros(10 * s.replicas, np.int64)
    energy, params = (md.md_energy_t * s.replicas)(), s.desc.params
    table = dict(step=lambda: lib.md_step(s.h, 10), remainder=lambda: lib.md_step(s.h, 7),
                 energy=lambda: lib.md_energy(s.h, energy), forces=lambda: lib.md_forces(s.h, p[0]),
                 set_state=lambda: lib.md_set_state(s.h, s.desc.pos, s.desc.vel),
                 get_state=lambda: lib.md_get_state(s.h, *p), rebin=lambda: lib.md_rebin(s.h),
                 set_params=lambda: lib.md_set_params(s.h, ctypes.byref(params)))
    if not s.desc.topology:
        table.update(rdf=lambda: lib.md_rdf(s.h, 10, edges.ctypes.data, counts.ctypes.data),
                     observables=lambda: lib.md_observables(s.h, p[0], None, None))
    s.out, s.keep = out, s.keep + out + [edges, counts]
    return table


SYSTEMS = dict(chains=dict(thermostat=md.MD_NOSE_HOOVER), molecules=dict(topology=([(k, k + 1) for k in range(29)], [0] * 30)),
               large_tiles=dict(skin=0.3))


def system(lib, kind):
    if kind == "large_tiles":   # two LJ launches a step
        melts = [lattice(60, 150, 19.625)] * 8 + [lattice(60, 150, 5.625)]
    else:
        melts = lattice(20, 30, 3.875)
    return Fake(lib, melts, **SYSTEMS[kind])


@pytest.mark.parametrize("kind", list(SYSTEMS))
def test_every_refused_launch_fails_its_call(lib, kind):
    lib.fake_reset()
    s = system(lib, kind)
    assert s.create() == md.MD_OK
    n_create = {w: lib.fake_calls(w.encode()) for w in ["launch", "memset"] + GRAPH_CALLS}
    table = calls(lib, s)
    for name, call in table.items():
        lib.fake_reset()
        assert call() == md.MD_OK, name
    for name in table:
        fresh = system(lib, kind)      # a remainder's graph is captured on its first use
        lib.fake_reset()
        assert fresh.create() == md.MD_OK
        fresh_table = calls(lib, fresh)
        lib.fake_reset()
        assert fresh_table[name]() == md.MD_OK
        seen = {w: lib.fake_calls(w.encode()) for w in ["launch", "memset"] + GRAPH_CALLS}
        fresh.close()
        for what, n in seen.items():
            for k in sorted({1, 2, n // 2, n - 1, n} & set(range(1, n + 1))):
                fresh = system(lib, kind)
                lib.fake_reset()
                assert fresh.create() == md.MD_OK
                call = calls(lib, fresh)[name]
                lib.fake_fail(what.encode(), k)
                assert call() == md.MD_ECUDA, (name, what, k)
                assert lib.fake_open_captures() == 0 and lib.fake_null_graphs() == 0
                lib.fake_fail(b"", 0)
                assert lib.md_get_state(s.h, *[a.ctypes.data for a in s.out]) == md.MD_OK   # another system's call
                assert lib.md_step(fresh.h, 13) == md.MD_OK, (name, what, k)   # graphs that a failed capture left out are made
                assert call() == md.MD_OK, (name, what, k)
                fresh.close()
    for what, n in n_create.items():
        for k in sorted({1, 2, n // 3, n // 2, n - 1, n} & set(range(1, n + 1))):
            fresh = system(lib, kind)
            lib.fake_fail(what.encode(), k)
            assert fresh.create() == md.MD_ECUDA and not fresh.h, (what, k)
            assert lib.fake_open_captures() == 0 and lib.fake_null_graphs() == 0
            lib.fake_fail(b"", 0)
            assert lib.md_rebin(s.h) == md.MD_OK
    s.close()
