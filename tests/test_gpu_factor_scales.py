"""QR and SVD of matrices near the ends of the FP32 exponent range (FP32 and double-float), where squared
norms of columns are finite but little else is.

Tolerances: a rounding unit of the precision (FP32 6e-8, FP64 1.1e-16, double-float 3.6e-15) times 10^3
terms per entry, relative to the matrix.  A double-float reflector has the factor 1 / v^H v, whose low word
is below the exponent range where v^H v is above 1e30: its QR is good to FP32 rounding there."""
import numpy as np
import pytest

from paper_2501_17913_gb300 import tjm

from gpu_common import lib_ready

pytestmark = pytest.mark.gpu

TOL = {0: 6e-5, 1: 1.1e-13, 2: 3.6e-12}


def _rand(rng, m, n):
    return rng.standard_normal((m, n)) + 1j * rng.standard_normal((m, n))


@pytest.mark.parametrize("dp", [0, 1, 2])
@pytest.mark.parametrize("m,n,size", [(64, 48, 5e17), (48, 64, 5e17), (128, 128, 3e17), (130, 60, 3e17), (8, 6, 2e18),
                                      (64, 48, 1e-12)])
def test_factorizations_of_large_and_small_matrices(m, n, size, dp):
    """The sum of all squares is above the FP32 range, that of any column (also a rotated one) below."""
    lib_ready()
    rng = np.random.default_rng(m + n)
    k = min(m, n)
    A = _rand(rng, m, n)
    ref = np.linalg.svd(A, compute_uv=False)
    U, S, V = tjm.selftest_svd(A * size, dp)
    assert np.abs(S / size - ref).max() <= TOL[dp] * ref[0]
    assert np.abs(U.conj().T @ U - np.eye(k)).max() <= 10 * TOL[dp]
    assert np.abs((U * (S / size)) @ V.conj().T - A).max() <= TOL[dp] * ref[0]
    Q, R = tjm.selftest_qr(A * size, dp)
    tol = TOL[0] if dp == 2 and size > 1e15 else TOL[dp]
    assert np.abs(Q.conj().T @ Q - np.eye(k)).max() <= 10 * tol
    assert np.abs(Q @ (R / size) - A).max() <= tol * ref[0]
    assert np.abs(np.tril(R, -1)).max() == 0.0


# largest squared norms just below the last binade of the range that holds them (dp 0 and 2: FP32, 2^127 = 1.7e38; dp 1:
# FP64, 2^1023 = 9.0e307) and in it
TOP = {0: [1.2e19, 1.35e19, 1.7e19], 1: [8e153, 1.0e154, 1.2e154], 2: [1.2e19, 1.35e19, 1.7e19]}


@pytest.mark.parametrize("dp", [0, 1, 2])
@pytest.mark.parametrize("m", [2, 20])
def test_rotations_at_the_top_of_the_exponent_range(m, dp):
    lib_ready()
    rng = np.random.default_rng(m)
    for size in TOP[dp]:
        A = 1e-3 * _rand(rng, m, 2)
        A[0], A[1] = [1.0, 0.1j], [0.0, 0.3]
        ref = np.linalg.svd(A, compute_uv=False)
        U, S, V = tjm.selftest_svd(A * size, dp)
        assert np.abs(S / size - ref).max() <= TOL[dp] * ref[0]
        assert np.abs((U * (S / size)) @ V.conj().T - A).max() <= TOL[dp] * ref[0]
        assert np.abs(U.conj().T @ U - np.eye(2)).max() <= 10 * TOL[dp]


@pytest.mark.parametrize("size", [1e-18, 1e-19])
def test_rotations_at_the_bottom_of_the_exponent_range(size):
    """Squared norms of 1e-36 and 1e-38 (the second below the normal range, with 20 bits left)."""
    lib_ready()
    A = np.array([[1.0, 0.1j], [0.0, 0.3]])
    ref = np.linalg.svd(A, compute_uv=False)
    U, S, V = tjm.selftest_svd(A * size, 0)
    assert np.abs(S / size - ref).max() <= (TOL[0] if size > 5e-19 else 1e-3) * ref[0]
    assert np.abs(V.conj().T @ V - np.eye(2)).max() <= 10 * TOL[0]
