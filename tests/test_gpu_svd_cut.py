"""The SVD of a truncation: directions below the cut are not told apart, which may change neither the
rank that the truncation finds nor what it keeps -- also for a cut that discards all but one direction.

Against LAPACK.  Tolerances: a rounding unit of the precision (FP32 6e-8, FP64 1.1e-16, double-float
3.6e-15) times 10^3 terms per entry, TOL; the kept subspace is perturbed by that over its gap to the rest."""
import numpy as np
import pytest

from oracle import mps_tjm as O1
from paper_2501_17913_gb300 import inputs as I
from paper_2501_17913_gb300 import tjm

from gpu_common import lib_ready

pytestmark = pytest.mark.gpu

TOL = {0: 6e-5, 1: 1.1e-13, 2: 3.6e-12}


def _rand(rng, m, n):
    return rng.standard_normal((m, n)) + 1j * rng.standard_normal((m, n))


def _rank(s, cut):
    """Smallest r >= 1 whose tail of squares is at most cut of their sum."""
    tail = np.append(np.cumsum((s ** 2)[::-1])[::-1][1:], 0.0)
    return 1 + int(np.argmax(tail <= cut * np.sum(s ** 2)))


@pytest.mark.parametrize("dp", [0, 1, 2])
@pytest.mark.parametrize("m,n", [(2, 2), (8, 4), (6, 12), (7, 7), (8, 16), (13, 12), (24, 24), (128, 33), (64, 128)])
@pytest.mark.parametrize("cut", [1e-10, 1e-4, 0.3, 0.99, 1.5, "all"])
def test_truncation_keeps_what_it_kept_without_the_cut(m, n, dp, cut):
    lib_ready()
    k = min(m, n)
    cut = 4.0 * k * k if cut == "all" else cut
    rng = np.random.default_rng(100 * m + n)
    qa, qb = np.linalg.qr(_rand(rng, m, k))[0], np.linalg.qr(_rand(rng, n, k))[0]
    big = (k + 1) // 2
    mats = [_rand(rng, m, n)]
    for level in (0.5, 2.0):           # the rest of the directions just below and just above the cut
        s = np.ones(k)
        s[:big] = np.linspace(1.0, 0.5, big)
        s[big:] = np.sqrt(min(level * cut / k ** 2, 0.05 / k) * np.sum(s[:big] ** 2))
        mats.append((qa * s) @ qb.conj().T)
    for A in mats:
        u, s, vh = np.linalg.svd(A, full_matrices=False)
        r = _rank(s, cut)
        U, S, V = tjm.selftest_svd(A, dp, cut=cut)
        assert _rank(S, cut) == r
        assert np.abs(S[:r] - s[:r]).max() <= TOL[dp] * s[0]
        assert abs(np.sum(S ** 2) - np.sum(s ** 2)) <= TOL[dp] * np.sum(s ** 2)
        gap = s[r - 1] - (s[r] if r < k else 0.0)
        for got, ref in ((U, u), (V, vh.conj().T)):
            g, f = got[:, :r], ref[:, :r]
            assert np.linalg.norm(g.conj().T @ g - np.eye(r), 2) <= 10 * TOL[dp]
            assert np.linalg.norm(g @ g.conj().T - f @ f.conj().T, 2) <= (10 + 4 * s[0] / gap) * TOL[dp]


def test_negative_cut_is_refused():
    lib_ready()
    with pytest.raises(tjm.TJMError):
        tjm.selftest_svd(np.eye(2), 1, cut=-1.0)


@pytest.mark.parametrize("eps", [0.3, 1.0, 20.0])
@pytest.mark.parametrize("prec,tol", [(tjm.PREC_FP64, 1e-10), (tjm.PREC_FP32_DF64, 1e-4), (tjm.PREC_FP32_DEC32, 1e-4)])
def test_run_that_keeps_one_direction_per_bond(eps, prec, tol):
    """Whole trajectories against the oracle, at the tolerances of the other parity tests."""
    lib_ready()
    L, n, dt = 6, 4, 0.3
    W, jumps, obs = I.xxx_mpo(L, 1.0, 0.5), I.noise(L, 0.1, 0.1), I.z_observables(L)
    ctx = tjm.Context(W, jumps, dt, 8, eps, precision=prec)
    pt = ctx.result(ctx.run(np.array(I.neel(L)), 4, 3, obs, [dt * j for j in range(n + 1)]))[2]
    ctx.close()
    prob = O1.Problem(W, jumps, dt, 8, eps)
    compared = 0
    for t in range(4):
        v, st = O1.run_trajectory(prob, O1.product_mps(I.neel(L)), t, 3, obs, n, list(range(n + 1)))
        if min(st['min_margin1'], st['min_margin2']) < 1e-5:
            continue
        assert np.abs(pt[t] - v).max() < tol, t
        compared += 1
    assert compared >= 2
