"""Left-environment updates whose last product has more columns (MPO bond times right bond) than the CTA
has threads, the widest among them, in FP64 and FP32.

Against the oracle's contraction, element by element within the tolerances of the other contraction tests."""
import numpy as np
import pytest

from oracle import mps_tjm as O1
from paper_2501_17913_gb300 import tjm

from gpu_common import lib_ready

pytestmark = pytest.mark.gpu


def _rand(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) / np.sqrt(2)


@pytest.mark.parametrize("prec,tol", [(tjm.PREC_FP64, 1e-12), (tjm.PREC_FP32, 1e-5)])
@pytest.mark.parametrize("chl,chr_,D", [(1, 33, 8), (3, 32, 8), (2, 43, 6), (5, 64, 4), (4, 52, 5), (7, 64, 5), (2, 64, 8)])
def test_wide_left_environment(chl, chr_, D, prec, tol):
    lib_ready()
    rng = np.random.default_rng(10 * chr_ + D)
    W = _rand(rng, 3, D, 2, 2)
    Lenv, A = _rand(rng, chl, 3, chl), _rand(rng, chl, 2, chr_)
    got = tjm.selftest_contract(3, prec, Lenv, np.zeros((1, 1, 1)), A, W1=W, tensor_cores=False)
    ref, mag = O1.env_left_update(Lenv, A, W), O1.env_left_update(abs(Lenv), abs(A), abs(W))
    assert (np.abs(got - ref) <= tol * mag).all()
