"""Calls at the limits of what is shared or scarce: molecules whose gradient
just fits or no longer fits beside a kernel's arrays, kernel attributes
while two threads work on molecules of different sizes, device memory too short
for the router's tables or for all sets of partial-gradient slabs, and omega so
large that its square is infinite.

Bounds: the same sums in the same order are bitwise equal; fp64 sums in
another order agree to 1e-13 of the largest component (a few hundred partial
sums of that size); the fp32 route to 6e-6 of it, as elsewhere."""
import os
import threading

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


def _system(shells, xyz, seed=5):
    """shells: (atom, l, primitives); two random density pairs with both operators."""
    rng = np.random.default_rng(seed)
    ex = [np.sort(np.exp(rng.uniform(np.log(0.2), np.log(60.0), k)))[::-1] for _a, _l, k in shells]
    s = dict(natom=len(xyz), xyz=np.asarray(xyz, float), shell_atom=np.array([a for a, _l, _k in shells], np.int32),
             shell_l=np.array([l for _a, l, _k in shells], np.int32),
             shell_nprim=np.array([k for _a, _l, k in shells], np.int32),
             exps=np.concatenate(ex), coefs=np.concatenate([rng.uniform(0.2, 1.0, len(e)) for e in ex]))
    n = s["nbf"] = synth.nbf_of(s["shell_l"])
    m = [rng.normal(size=(n, n)) / n for _ in range(3)]
    s["pairs"] = [(m[0], m[1], 1.0, -0.3, -0.7, 0.35), (m[2], m[2], 0.5, 0.2, 0.0, 0.0)]
    return s


def _padded(natom):
    """Three atoms with s, p and d shells; the others carry none."""
    xyz = np.zeros((natom, 3))
    xyz[:3] = [[0.0, 0.1, -0.2], [1.6, 0.4, 0.3], [-0.5, 1.5, 0.9]]
    xyz[3:] = 50.0 + np.arange(3 * (natom - 3)).reshape(-1, 3)
    return _system([(a, l, 1) for a in range(3) for l in range(3)], xyz)


@pytest.mark.parametrize("natom", [4746, 4747, 5500, 6173, 6174])
def test_fp32_gradient_at_the_shared_memory_limit(tg, natom):
    """From 4747 to 6173 atoms the gradient (111 to 145 KB) fits in a CTA's shared
    memory, but not beside the arrays of (dd|pp) as well."""
    ref = tg.Basis(_padded(3)).grad2e(_padded(3)["pairs"], screen_tol=0.0)[0]
    s = _padded(natom)
    g = tg.Basis(s).grad2e(s["pairs"], screen_tol=0.0, precision=tg.TG_FP32)[0]
    assert np.abs(g[:3] - ref).max() <= 6e-6 * np.abs(ref).max()
    assert not g[3:].any()


def test_two_threads_on_molecules_of_different_sizes(tg):
    """A kernel's shared-memory limit is common to all threads of the process;
    a launch for 1200 atoms needs more of it than one for three."""
    systems = [_padded(3), _padded(1200)]
    bases = [tg.Basis(s) for s in systems]
    kw = dict(screen_tol=0.0)
    alone = [[b.grad2e(s["pairs"], precision=p, **kw)[0] for p in (tg.TG_FP64, tg.TG_FP32)]
             for b, s in zip(bases, systems)]
    got, errors = [[], []], []

    def work(i):
        try:
            for _ in range(100):
                got[i].append([bases[i].grad2e(systems[i]["pairs"], precision=p, **kw)[0]
                               for p in (tg.TG_FP64, tg.TG_FP32)])
        except tg.TGError as e:
            errors.append(e)
    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i in range(2):
        for g in got[i]:
            assert np.array_equal(g[0], alone[i][0]) and np.array_equal(g[1], alone[i][1])


def test_learned_route_without_room_for_its_tables(tg, monkeypatch):
    """Where the router's feature tables do not fit, the tiles gather their
    features themselves: the same route and the same gradient, bit for bit."""
    natom = 100
    xyz = np.zeros((natom, 3))
    xyz[:, 0] = 30.0 * np.arange(natom)  # pairs on one atom only: few tiles, many shells
    s = _system([(a, l, k) for a in range(natom) for l, k in ((0, 2), (0, 1), (1, 1))], xyz)
    router = tg.Router(path=os.path.join(os.path.dirname(tg.__file__), "data", "router.bin"))
    kw = dict(precision=tg.TG_MIXED_LEARNED, router=router)
    ample, tight = tg.Basis(s), tg.Basis(s)
    st = tight.grad2e(s["pairs"])[1]  # the other work areas have their sizes after this
    # 124 B a tile without tables; with them 108 B and 8 nshell a bra tile of 16 pairs
    limit = 124 * st["tiles"] + 8192
    assert 108 * st["tiles"] + 8 * len(s["shell_l"]) * (st["pairs"] // 16) > limit
    mixed = 0
    for tol in (1e-5, 1e-6, 1e-7, 1e-8, 1e-9, 1e-10):
        g, sa = ample.grad2e(s["pairs"], mixed_tol=tol, **kw)
        monkeypatch.setenv("TDGRAD_FAIL_ALLOC", str(limit))
        h, sb = tight.grad2e(s["pairs"], mixed_tol=tol, **kw)
        monkeypatch.delenv("TDGRAD_FAIL_ALLOC")
        assert sb["launches"] < sa["launches"]  # the tables take launches of their own
        assert sb["fp32_quartets"] == sa["fp32_quartets"]
        assert np.array_equal(g, h)
        mixed += 0 < sa["fp32_quartets"] < sa["quartets"]
    assert mixed


def test_gradient_without_room_for_all_slabs(tg, monkeypatch):
    """9000 atoms: one set of slabs, 4 an SM, takes 131 MB on 152 SMs, six sets of
    8 an SM 1.6 GB.  With 200 MB to be had the call works on the smaller set."""
    ref = tg.Basis(_padded(3)).grad2e(_padded(3)["pairs"], screen_tol=0.0)[0]
    s = _padded(9000)
    b = tg.Basis(s)
    monkeypatch.setenv("TDGRAD_FAIL_ALLOC", str(200 << 20))
    g = b.grad2e(s["pairs"], screen_tol=0.0)[0]
    assert np.abs(g[:3] - ref).max() <= 1e-13 * np.abs(ref).max()
    assert not g[3:].any()
    timed = b.grad2e(s["pairs"], screen_tol=0.0, timing=True)[0]
    assert np.abs(timed[:3] - ref).max() <= 1e-13 * np.abs(ref).max()


def test_batch_without_room_for_all_slabs(tg, monkeypatch):
    """The same for a batch of two such molecules (262 MB against 3.2 GB); its
    molecules' own work areas hold no slabs."""
    ref = tg.Basis(_padded(3)).grad2e(_padded(3)["pairs"], screen_tol=0.0)[0]
    monkeypatch.setenv("TDGRAD_FAIL_ALLOC", str(300 << 20))
    batch = tg.Batch([_padded(9000), _padded(9000)], screen_tol=0.0)
    for _ in range(2):
        for g in batch.run()[0]:
            assert np.abs(g[:3] - ref).max() <= 1e-13 * np.abs(ref).max()
            assert not g[3:].any()


def test_omega_whose_square_overflows(tg):
    """erf(omega r)/r is 1/r to the last bit long before omega^2 leaves the
    range of fp64 (1e154) or fp32 (1e19): the result is that of omega = inf."""
    s = _padded(3)
    b = tg.Basis(s)

    def grad(om, precision):
        return b.grad2e([(*p[:5], om) for p in s["pairs"]], screen_tol=0.0, precision=precision)[0]

    def fock(om):
        return b.fock2e([(s["pairs"][0][0], 1.0, -0.3, -0.7, om)])[0]
    for precision, tol in ((tg.TG_FP64, 1e-13), (tg.TG_FP32, 0.0)):
        inf = grad(np.inf, precision)
        assert np.isfinite(inf).all()
        for om in (1e25, 1e160):
            assert np.abs(grad(om, precision) - inf).max() <= tol * np.abs(inf).max(), om
    assert np.abs(fock(1e160) - fock(np.inf)).max() <= 1e-13 * np.abs(fock(np.inf)).max()
