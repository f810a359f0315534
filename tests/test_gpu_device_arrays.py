"""The caller's arrays on the device, used where they lie, against host arrays, which are copied: the same numbers."""
import ctypes

import numpy as np
import pytest

import chaingen
import paper_1001_3764_gb300 as md

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [md.MD_MIXED, md.MD_PLAIN_FP32])
@pytest.mark.parametrize("shift", [0, 4, 8])   # bytes off the allocation's alignment: 4 cannot be used in place
def test_device_arrays_give_the_numbers_of_host_arrays(precision, shift):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    m = chaingen.melt(11, seed=61, T=300.0)
    n = 3 * len(m["pos"])
    s = md.System(m, precision=precision)
    lib, room = md.load(), 64
    s.step(3)
    x, v, im = s.state()
    f = s.forces()
    buf = torch.full((4, n * 8 + room), 0xAB, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    px, pv, pi, pf = (ctypes.c_void_p(buf[k].data_ptr() + shift) for k in range(4))
    assert lib.md_get_state(s.h, px, pv, pi) == 0
    assert lib.md_forces(s.h, pf) == 0
    host = buf.cpu().numpy()
    for k, (want, size) in enumerate([(x, 8), (v, 8), (im, 4), (f, 8)]):
        got = host[k, shift:shift + n * size].view(np.float64 if size == 8 else np.int32)
        assert np.array_equal(got, np.asarray(want).ravel())
        assert (host[k, :shift] == 0xAB).all() and (host[k, shift + n * size:] == 0xAB).all()   # nothing beside it
    # one output alone, and the state set from the device
    buf[0].fill_(0)
    torch.cuda.synchronize()
    assert lib.md_get_state(s.h, px, None, None) == 0
    assert np.array_equal(buf[0].cpu().numpy()[shift:shift + 8 * n].view(np.float64), x.ravel())
    s.set_state(x, v)
    want = s.forces()
    s.step(1)
    assert lib.md_set_state(s.h, px, pv) == 0
    assert np.array_equal(s.forces(), want)
    s.close()
