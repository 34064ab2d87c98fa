"""A batch over densities in the caller's device buffers.

Bound: fp64 sums in another order, 1e-13 of the largest component."""
import ctypes

import numpy as np
import pytest

from paper_2407_16586_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tg():
    from paper_2407_16586_gb300 import build
    build.build()
    import paper_2407_16586_gb300 as m
    return m


def test_batch_reads_device_densities_at_every_run(tg):
    """A batch created with device_ptrs reads the caller's buffers when it runs:
    after their contents change, a run gives the gradient of the new ones."""
    torch = pytest.importorskip("torch")
    s = synth.molecule(20, 1, 2)
    b = tg.Basis(s)
    opt = tg.tg_options_default()
    opt.screen_tol, opt.device_ptrs = 0.0, 1
    opt.stream = torch.cuda.current_stream().cuda_stream
    n = len(s["pairs"])
    mats = [[torch.from_numpy(np.array(m)).cuda() for m in p[:2]] for p in s["pairs"]]
    arr = (tg.tg_pair * n)(*[tg.tg_pair(x.data_ptr(), y.data_ptr(), *p[2:]) for (x, y), p in zip(mats, s["pairs"])])
    pp = (ctypes.POINTER(tg.tg_pair) * 1)(ctypes.cast(arr, ctypes.POINTER(tg.tg_pair)))
    h = ctypes.c_void_p()
    assert tg.lib().tg_batch_create(1, (ctypes.c_void_p * 1)(b.h), (ctypes.c_int * 1)(n), pp, ctypes.byref(opt),
                                    ctypes.byref(h)) == tg.TG_OK
    try:
        for f in (1.0, -0.7):
            now = []
            for (x, y), p in zip(mats, s["pairs"]):
                x.copy_(f * x + 0.1 * x.roll(1, 0))
                y.copy_(y.roll(1, 1))
                now.append((x.clone(), y.clone(), *p[2:]))
            out = torch.zeros((s["natom"], 3), dtype=torch.float64, device="cuda")
            assert tg.lib().tg_batch_run(h, (ctypes.c_void_p * 1)(out.data_ptr()), ctypes.byref(opt), None) == tg.TG_OK
            ref = tg.Basis(s).grad2e(now, screen_tol=0.0)[0]
            assert (out - ref).abs().max() <= 1e-13 * ref.abs().max()
    finally:
        tg.lib().tg_batch_destroy(h)
