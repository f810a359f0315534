"""Shared memory of the step and histogram kernels: what each launch asks for beside its static arrays against the
48 KB limit or the kernel's opt-in, over the chain lengths at the edges of the block sizes and the numbers of bins.
On the CPU: the host code runs on a stand-in runtime, the static bytes are the compiler's."""
import os
import re
import subprocess

import numpy as np
import pytest

import paper_1001_3764_gb300 as md
from fake_cudart import Fake, lattice, link
from paper_1001_3764_gb300 import build as cuda_build

LIMIT, SM_LIMIT = 48 * 1024, 227 * 1024


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return link(str(tmp_path_factory.mktemp("fake")))


@pytest.fixture(scope="module")
def static_bytes(tmp_path_factory):
    """static shared memory of every kernel of two sources, by its name in the object file"""
    out, found = str(tmp_path_factory.mktemp("ptxas")), {}
    for source in ("k_step.cu", "k_observe.cu"):
        r = subprocess.run([cuda_build.NVCC, *cuda_build.ARCH, *cuda_build.FLAGS, "-Xptxas", "-v", "-c",
                            os.path.join(cuda_build.CSRC, source), "-o", os.path.join(out, source + ".o")],
                           capture_output=True, text=True, check=True)
        for name, used in re.findall(r"entry function '(\w+)'.*?Used ([^\n]*)", r.stderr, re.S):
            smem = re.search(r"(\d+) bytes smem", used)
            found[name] = int(smem.group(1)) if smem else 0
    assert len(found) >= 40
    return found


@pytest.mark.parametrize("precision", [md.MD_MIXED, md.MD_PLAIN_FP32])
@pytest.mark.parametrize("thermostat", [md.MD_NVE, md.MD_VRESCALE, md.MD_NOSE_HOOVER])
def test_chain_step_launches_fit(lib, static_bytes, precision, thermostat):
    for sites in (4, 150, 256, 257, 352, 353, 384, 480, 481, 512, 513, 1022):
        check(lib, static_bytes, Fake(lib, lattice(3, sites, 6.0), precision=precision, thermostat=thermostat))


@pytest.mark.parametrize("thermostat", [md.MD_NVE, md.MD_VRESCALE, md.MD_NOSE_HOOVER])
def test_molecule_step_launches_fit(lib, static_bytes, thermostat):
    for sites in (4, 128, 129, 1022):
        topology = ([(k, k + 1) for k in range(sites - 1)], [0] * sites)
        check(lib, static_bytes, Fake(lib, lattice(3, sites, 6.0), topology=topology, thermostat=thermostat))


def fits(lib, static_bytes, name, dynamic):
    total, opt_in = static_bytes[name.decode()] + dynamic, lib.fake_opt_in(name)
    assert total <= LIMIT or (dynamic <= opt_in and total <= SM_LIMIT), (name, total, opt_in)


def check(lib, static_bytes, s):
    assert s.create() == md.MD_OK, lib.md_last_error(None)
    lib.fake_reset()
    assert lib.md_step(s.h, 13) == md.MD_OK
    steps = [(lib.fake_kernel(i), lib.fake_smem(i)) for i in range(lib.fake_ran()) if b"k_step" in lib.fake_kernel(i)]
    assert len(steps) == 13          # one update after every LJ launch
    for name, dynamic in steps:
        fits(lib, static_bytes, name, dynamic)
    s.close()


@pytest.mark.parametrize("precision", [md.MD_MIXED, md.MD_PLAIN_FP32])
def test_histogram_launches_fit_whatever_was_asked_before(lib, static_bytes, precision):
    """Fewer bins after more: the opt-in that another thread's larger histogram counts on stays."""
    s = Fake(lib, lattice(3, 150, 6.0), precision=precision)
    assert s.create() == md.MD_OK
    largest = {}
    for bins in (1, 9000, 9001, 16384, 9001, 12000, 200):
        edges, counts = np.linspace(0.0, 0.9, bins + 1), np.zeros(bins, np.int64)
        lib.fake_reset()
        assert lib.md_rdf(s.h, bins, edges.ctypes.data, counts.ctypes.data) == md.MD_OK
        (name, dynamic), = [(lib.fake_kernel(i), lib.fake_smem(i)) for i in range(lib.fake_ran()) if b"k_rdf" in lib.fake_kernel(i)]
        largest[name] = max(largest.get(name, 0), dynamic)
        for asked in (dynamic, largest[name]):
            fits(lib, static_bytes, name, asked)
    s.close()
