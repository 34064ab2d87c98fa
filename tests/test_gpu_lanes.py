"""The lane kernels at the sizes where their splits change: one and many
primitives per shell (blocks of bra primitive pairs, partly filled passes,
groups of ket pairs with different counts), a molecule whose gradient no
longer fits beside the kernels' arrays, two handles at work on two streams,
and the tile features of the device planner against those of the samples.

Tolerance: fp64 throughout; the gradient agrees with the oracle to 1e-12 of
the largest component plus 1e-11 (rounding of sums of up to 10^6 fp64 terms of
that size; the oracle's own evaluation is good to 1e-13)."""
import numpy as np
import pytest

import oracle
from paper_2407_16586_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tg():
    from paper_2407_16586_gb300 import build
    build.build()
    import paper_2407_16586_gb300 as m
    return m


def _system(shells, natom=3, seed=5):
    """shells: (atom, l, primitives); atoms on a bent line, 1.7 bohr apart, and
    two random density pairs with both operators."""
    rng = np.random.default_rng(seed)
    xyz = np.zeros((natom, 3))
    xyz[:3] = [[0.0, 0.1, -0.2], [1.6, 0.4, 0.3], [-0.5, 1.5, 0.9]]
    xyz[3:] = 50.0 + np.arange(3 * (natom - 3)).reshape(-1, 3)
    ex = [np.sort(np.exp(rng.uniform(np.log(0.2), np.log(60.0), k)))[::-1] for _a, _l, k in shells]
    s = dict(natom=natom, xyz=xyz, shell_atom=np.array([a for a, _l, _k in shells], np.int32),
             shell_l=np.array([l for _a, l, _k in shells], np.int32),
             shell_nprim=np.array([k for _a, _l, k in shells], np.int32),
             exps=np.concatenate(ex), coefs=np.concatenate([rng.uniform(0.2, 1.0, len(e)) for e in ex]))
    n = s["nbf"] = synth.nbf_of(s["shell_l"])
    m = [rng.normal(size=(n, n)) / n for _ in range(3)]
    s["pairs"] = [(m[0], m[1], 1.0, -0.3, -0.7, 0.35), (m[2], m[2], 0.5, 0.2, 0.0, 0.0)]
    return s


SHAPES = {
    # every shell one primitive: one primitive quartet per contracted quartet
    "one": [(0, 0, 1), (0, 1, 1), (0, 2, 1), (1, 0, 1), (1, 1, 1), (1, 2, 1), (2, 0, 1), (2, 1, 1), (2, 2, 1)],
    # pair counts at and next to the 32 lanes: 2 x 16 = 32, 3 x 11 = 33
    "near32": [(0, 0, 16), (1, 0, 2), (1, 1, 11), (2, 1, 3), (2, 2, 2), (0, 2, 1)],
    # the largest contraction a shell may have beside single primitives
    "deep": [(0, 1, 16), (1, 2, 5), (2, 0, 16), (2, 1, 1)],
    # many pairs of one class with different counts: groups of ket pairs
    "uneven": [(a, l, k) for a in range(3) for l, k in ((0, 1), (0, 4), (0, 7), (1, 2), (1, 5))],
}


@pytest.mark.parametrize("name", SHAPES)
@pytest.mark.parametrize("tau", [0.0, 1e-8])
def test_contraction_shapes(tg, name, tau):
    s = _system(SHAPES[name])
    ref, _, nq = oracle.grad2e(s, tau=tau)
    g, st = tg.Basis(s).grad2e(s["pairs"], screen_tol=tau)
    assert st["quartets"] == nq
    assert np.abs(g - ref).max() <= 1e-12 * np.abs(ref).max() + 1e-11, np.abs(g - ref).max()


@pytest.mark.parametrize("natom", [3, 1200, 9000])
def test_gradient_beside_or_beyond_shared_memory(tg, natom):
    """The atoms past the third carry no shells: the result is the small
    molecule's, while the gradient array grows from 72 B to 216 KB."""
    s = _system(SHAPES["one"], natom=natom)
    ref = tg.Basis(_system(SHAPES["one"])).grad2e(s["pairs"], screen_tol=0.0)[0]
    b = tg.Basis(s)
    for precision in (tg.TG_FP64, tg.TG_FP32):
        g = b.grad2e(s["pairs"], screen_tol=0.0, precision=precision)[0]
        tol = 1e-13 if precision == tg.TG_FP64 else 6e-6
        assert np.abs(g[:3] - ref).max() <= tol * np.abs(ref).max()
        assert not g[3:].any()


def test_two_handles_on_two_streams(tg):
    """Each handle's launches spread over streams of its own; calls from two
    threads on two caller streams give what each gives alone, bit for bit."""
    import threading
    import torch
    systems = [_system(SHAPES["uneven"], seed=5), _system(SHAPES["near32"], seed=6)]
    bases = [tg.Basis(s) for s in systems]
    alone = [b.grad2e(s["pairs"])[0] for b, s in zip(bases, systems)]
    streams = [torch.cuda.Stream() for _ in systems]
    got = [[], []]

    def work(i):
        for _ in range(5):
            got[i].append(bases[i].grad2e(systems[i]["pairs"], stream=streams[i].cuda_stream)[0])
    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i in range(2):
        assert len(got[i]) == 5
        for g in got[i]:
            assert np.array_equal(g, alone[i])


@pytest.mark.parametrize("size", [(5, 2, 0), (14, 3, 3), (12, 5, 7)])
def test_planner_features_route_as_the_sampled_ones(tg, size):
    """The device planner's tile features come from tables, those of
    tile_samples from the tiles' pairs.  All tiles go to fp32 exactly when the
    squared upper edges of their routing bins (8 per octave) sum to at most
    mixed_tol^2, so the threshold computed from the sampled features has to
    switch the planner's route (ragged tiles and tiles of one class with itself
    among them)."""
    import os
    router = tg.Router(path=os.path.join(os.path.dirname(tg.__file__), "data", "router.bin"))
    s = synth.molecule(*size)
    b = tg.Basis(s)
    X = b.tile_samples(s["pairs"], stride=1, cap=2000000)[0]
    _, _, _, (margin, eps_rel, _) = router.get()
    e = float(eps_rel) * 10.0 ** (router.predict(X).astype(np.float64) + float(margin))
    upper = 2.0 ** ((np.floor(np.log2(e) * 8.0) + 1.0) / 8.0)
    tol = float(np.sqrt(np.sum(upper ** 2)))
    for f, all32 in ((1.0 + 1e-6, True), (1.0 - 1e-6, False)):
        st = b.grad2e(s["pairs"], precision=tg.TG_MIXED_LEARNED, router=router, mixed_tol=tol * f)[1]
        assert st["tiles"] == len(X)
        assert (st["fp32_quartets"] == st["quartets"]) == all32
