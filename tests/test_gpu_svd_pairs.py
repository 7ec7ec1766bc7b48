"""Matrices of one and two columns, where one rotation is the whole SVD, in FP64 (angles from its own
roots) and in the other precisions (angles from FP32 words).

Tolerance: 8 roundings on the way of an entry (product, rotation of four terms, norm, division) times
sqrt(m) for the sums of m terms, in units of the precision."""
import numpy as np
import pytest

from paper_2501_17913_gb300 import tjm

from gpu_common import lib_ready

pytestmark = pytest.mark.gpu

UNIT = {0: 1.2e-7, 1: 2.2e-16, 2: 7.2e-15}


def _pairs(rng, m):
    x = rng.standard_normal(m) + 1j * rng.standard_normal(m)
    y = rng.standard_normal(m) + 1j * rng.standard_normal(m)
    z = y - x * (x.conj() @ y) / (x.conj() @ x)
    yield np.stack([x, y], 1)
    yield np.stack([x, 1e-3 * y], 1)
    yield np.stack([1e-3j * x, y], 1)
    yield np.stack([x, 1j * x + 0.1 * y], 1)                                   # nearly parallel
    yield np.stack([x + z, x - z * np.linalg.norm(x) / np.linalg.norm(z)], 1)
    yield np.stack([x, z * np.linalg.norm(x) / max(np.linalg.norm(z), 1e-30)], 1) if m > 1 else np.stack([x, y], 1)
    yield np.stack([x, 0 * y], 1)


@pytest.mark.parametrize("dp", [0, 1, 2])
@pytest.mark.parametrize("m", [2, 3, 8, 33, 64, 128])
def test_two_columns(m, dp):
    lib_ready()
    rng = np.random.default_rng(m)
    tol = 8 * np.sqrt(m) * UNIT[dp]
    for A in _pairs(rng, m):
        for B in (A, A.T.copy()):
            ref = np.linalg.svd(B, compute_uv=False)
            U, S, V = tjm.selftest_svd(B, dp)
            assert np.abs(S - ref).max() <= tol * ref[0]
            assert np.abs(V.conj().T @ V - np.eye(2)).max() <= tol
            assert np.abs((U * S) @ V.conj().T - B).max() <= tol * ref[0]
            # a left vector of a small value is a difference of columns over that value
            assert np.abs(U.conj().T @ U - np.eye(2)).max() <= tol * max(1.0, ref[0] / max(ref[1], 1e-3 * ref[0]))


@pytest.mark.parametrize("dp", [0, 1, 2])
@pytest.mark.parametrize("m", [1, 2, 7, 128])
def test_one_column(m, dp):
    lib_ready()
    rng = np.random.default_rng(m)
    A = (rng.standard_normal((m, 1)) + 1j * rng.standard_normal((m, 1))) * 3.0
    tol = 8 * np.sqrt(m) * UNIT[dp]
    for B in (A, A.T.copy()):
        U, S, V = tjm.selftest_svd(B, dp)
        assert abs(S[0] - np.linalg.norm(A)) <= tol * np.linalg.norm(A)
        assert np.abs((U * S) @ V.conj().T - B).max() <= tol * np.linalg.norm(A)
        assert abs(np.linalg.norm(U) - 1) <= tol and abs(np.linalg.norm(V) - 1) <= tol
