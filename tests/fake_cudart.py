"""The library's objects linked with a stand-in for the CUDA runtime (fake_cudart.cpp): its host code on the CPU."""
import ctypes
import os
import subprocess

import numpy as np

import paper_1001_3764_gb300 as md
from paper_1001_3764_gb300 import build as cuda_build

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA = os.path.dirname(os.path.dirname(cuda_build.NVCC))


def link(folder):
    """CDLL of the library on the stand-in runtime, built in `folder`."""
    objs = [os.path.join(cuda_build.BUILD, os.path.basename(s)[:-3] + ".o") for s in cuda_build._sources()]
    cuda_build.build(force=not all(map(os.path.exists, objs)))
    out = os.path.join(folder, "libfake.so")
    subprocess.run(["g++", "-O1", "-fPIC", "-shared", "-I" + os.path.join(CUDA, "include"), "-Wl,-Bsymbolic", "-o", out,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs], check=True)
    lib = ctypes.CDLL(out)
    lib.md_launches_per_call.restype = ctypes.c_int64
    lib.md_launches_per_call.argtypes = [ctypes.c_void_p, ctypes.c_int64]
    lib.fake_kernel.restype = ctypes.c_char_p
    lib.fake_smem.restype = lib.fake_opt_in.restype = ctypes.c_longlong
    lib.md_last_error.restype = ctypes.c_char_p
    for f in ("md_step", "md_step_async"):
        getattr(lib, f).argtypes = [ctypes.c_void_p, ctypes.c_int64]
    for f in ("md_sync", "md_rebin", "md_destroy", "md_last_error"):
        getattr(lib, f).argtypes = [ctypes.c_void_p]
    for f, n in (("md_create", 1), ("md_energy", 1), ("md_forces", 1), ("md_set_params", 1), ("md_set_state", 2),
                 ("md_get_state", 3), ("md_observables", 3)):
        getattr(lib, f).argtypes = [ctypes.c_void_p] * (n + 1)
    lib.md_rdf.argtypes = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_void_p, ctypes.c_void_p]
    return lib


class Fake:
    """A system's descriptor and handle on the stand-in runtime."""

    def __init__(self, lib, melts, precision=md.MD_MIXED, thermostat=md.MD_NVE, rebin_every=10, skin=0.1, topology=None,
                 **fields):
        melts = [melts] if isinstance(melts, dict) else melts
        self.lib, self.h = lib, ctypes.c_void_p()
        arrays = [np.array([m["n_chains"] for m in melts], np.int32), np.array([m["L"] for m in melts], np.float64),
                  np.concatenate([m["pos"] for m in melts]).astype(np.float64),
                  np.concatenate([m["vel"] for m in melts]).astype(np.float64), np.full(len(melts), 300.0)]
        d = self.desc = md.md_desc()
        d.n_replicas, d.sites_per_chain = len(melts), melts[0]["sites"]
        d.n_chains, d.box, d.pos, d.vel, d.T_target = (a.ctypes.data_as(ctypes.c_void_p) for a in arrays)
        d.params = md.make_params(md.default_params())
        d.dt, d.rc, d.skin, d.tau_t = 0.001, 1.0, skin, 0.1
        d.rebin_every, d.precision, d.thermostat = rebin_every, precision, thermostat
        if topology is not None:
            bonds, types = (np.ascontiguousarray(a, np.int32) for a in topology)
            t = md.md_topology(len(types), len(bonds), bonds.ctypes.data, types.ctypes.data)
            d.topology = ctypes.cast(ctypes.pointer(t), ctypes.c_void_p)
            arrays += [bonds, types, t]
        for k, v in fields.items():
            setattr(d, k, v)
        self.keep, self.n, self.replicas = arrays, len(arrays[2]), len(melts)

    def create(self):
        return self.lib.md_create(ctypes.byref(self.desc), ctypes.byref(self.h))

    def close(self):
        if self.h:
            self.lib.md_destroy(self.h)
        self.h = ctypes.c_void_p()


def lattice(n_chains, sites, L):
    """A melt-format dict for host tests: no kernel runs, so only sizes and the box matter."""
    x = np.mod(np.arange(3 * n_chains * sites, dtype=np.float64).reshape(-1, 3) * 0.0371, L)
    return dict(pos=x, vel=np.zeros_like(x), L=L, n_chains=n_chains, sites=sites)
