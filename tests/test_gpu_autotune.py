"""The autotuner's choices against the automatic ones, by per-class kernel times
(CUDA events, one list after the other)."""
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


def test_tuned_fp64_classes_are_no_slower(tg):
    """(ss|ss), (ps|ss) and (ds|ss) of the 32-atom workload in fp64, whose lists
    are many times longer than what the tuner times (chosen from a sample of it,
    (ss|ss) took 1.33 times as long).  Two runs of these lists differ by 1 %; the
    best of five may be 20 % apart, which leaves room for other users of the
    machine."""
    s = synth.config(1)
    kw = dict(class_mask=1 | 1 << 1 | 1 << 6, timing=True)
    plain, tuned = tg.Basis(s), tg.Basis(s)
    g = plain.grad2e(s["pairs"], **kw)[0]
    h = tuned.grad2e(s["pairs"], autotune=1, **kw)[0]
    assert np.abs(h - g).max() <= 1e-11
    ms = np.array([[b.grad2e(s["pairs"], autotune=a, **kw)[1]["class_ms"] for b, a in ((plain, 0), (tuned, 1))]
                   for _ in range(5)]).min(0)
    for qc in (0, 1, 6):
        assert ms[1, qc] <= 1.2 * ms[0, qc], (qc, ms[:, qc])
