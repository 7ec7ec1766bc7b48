"""The SVD's work counter: what the iteration did, in complex multiply-adds (8 real flops).

Matrices whose iteration is known: orthogonal columns (one sweep that forms every product and rotates
nothing), two columns in FP64 (one rotation), columns below the cut (no product)."""
import numpy as np
import pytest

from paper_2501_17913_gb300 import tjm

from gpu_common import lib_ready

pytestmark = pytest.mark.gpu


def _cmacs(A, dp, cut=0.0):
    lib_ready()
    fl = []
    tjm.selftest_svd(A, dp, cut=cut, flops=fl)
    return fl[0] / 8


def _diag(m, values):
    A = np.zeros((m, len(values)), complex)
    np.fill_diagonal(A, values)
    return A


def _idle_sweep(m, n, pairs=None):
    return (n * (n - 1) // 2 if pairs is None else pairs) * m + m * n // 2      # products, norms


@pytest.mark.parametrize("dp", [0, 1, 2])
def test_orthogonal_columns(dp):
    m, n = 6, 4
    gram_schmidt = m * n * n + n ** 3 if dp == 0 else 0
    for A in (_diag(m, [4, 3, 2, 1]), _diag(m, [4, 3, 2, 1]).T.copy()):
        assert _cmacs(A, dp) == _idle_sweep(m, n) + gram_schmidt
    assert _cmacs(_diag(5, [2]), dp) == (5 + 1 if dp == 0 else 0)


@pytest.mark.parametrize("m", [2, 40])
def test_two_columns_in_fp64_take_one_rotation(m):
    rng = np.random.default_rng(m)
    A = rng.standard_normal((m, 2)) + 1j * rng.standard_normal((m, 2))
    assert _cmacs(A, 1) == 2 * _idle_sweep(m, 2) + 2 * (m + 2)


@pytest.mark.parametrize("dp", [1, 2])
def test_pairs_below_the_cut_are_not_counted(dp):
    m, A = 6, _diag(6, [1, 1e-6, 1e-6, 1e-6])
    assert _cmacs(A, dp, cut=1e-8) == _idle_sweep(m, 4, pairs=3)
    assert _cmacs(A, dp, cut=1e-14) == _idle_sweep(m, 4)


@pytest.mark.parametrize("dp", [1, 2])
def test_the_fp32_start_is_counted(dp):
    m, n = 16, 12
    start = _idle_sweep(n, n) + (6 * m - 2 * n) * n * n // 3 + 8 * n ** 3 // 3 + m * n * n
    assert _cmacs(_diag(m, np.linspace(2, 1, n)), dp) == start + _idle_sweep(m, n)
