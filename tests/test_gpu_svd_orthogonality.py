"""Orthogonality and reconstruction of the SVD at working precision, at bounds narrow enough to notice that a
step which restores them is missing.

With u the rounding unit (FP32 6e-8, FP64 1.1e-16, double-float 3.6e-15):
* FP32 factors leave a Gram-Schmidt pass: eight roundings (a norm as a tree of sums, its root, the scaling,
  twice) = 8 u, against 8e-7 or more of columns that are only converged to the iteration's own tolerance;
* V of the others is a product of Householder reflectors and rotations, each unitary to a few u, over the columns' m
  entries: 16 sqrt(m) u, against 1e-13 where rotations are unitary to first order in their FP32 angles only;
* U of the others is divided out of columns that the iteration leaves once their cosine is below m times its eps (FP64
  2^-52 = 2 u, double-float 2^-46 = 4 u): that, and V's;
* reconstruction: 32 sqrt(m) u of the matrix."""
import numpy as np
import pytest

from paper_2501_17913_gb300 import tjm

from gpu_common import lib_ready

pytestmark = pytest.mark.gpu

U32, U64, UDF = 6.0e-8, 1.1e-16, 3.6e-15
STOP = {1: 2.0 ** -52, 2: 2.0 ** -46}


def _rand(rng, m, n):
    return rng.standard_normal((m, n)) + 1j * rng.standard_normal((m, n))


def _defect(x):
    return np.abs(x.conj().T @ x - np.eye(x.shape[1])).max()


@pytest.mark.parametrize("dp,u", [(0, U32), (1, U64), (2, UDF)])
@pytest.mark.parametrize("m,n", [(3, 2), (8, 8), (12, 12), (16, 9), (32, 31), (33, 17), (64, 64), (96, 48), (128, 64), (128, 127)])
def test_factors_to_working_precision(m, n, dp, u):
    lib_ready()
    rng = np.random.default_rng(1000 * m + n)
    full = _rand(rng, m, n)
    qa, qb = np.linalg.qr(_rand(rng, m, n))[0], np.linalg.qr(_rand(rng, n, n))[0]
    for A in (full, (qa * np.linspace(1.0, 0.01, n)) @ qb.conj().T):
        U, S, V = tjm.selftest_svd(A, dp)
        if dp == 0:
            assert _defect(U) <= 8 * u and _defect(V) <= 8 * u
        else:
            assert _defect(V) <= 16 * np.sqrt(m) * u
            assert _defect(U) <= m * STOP[dp] + 16 * np.sqrt(m) * u
        top = np.linalg.norm(A, 2)
        assert np.abs((U * S) @ V.conj().T - A).max() <= 32 * np.sqrt(m) * u * top
        assert np.abs(S - np.linalg.svd(A, compute_uv=False)).max() <= 32 * np.sqrt(m) * u * top
