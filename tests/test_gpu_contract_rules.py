"""The tiled FP32 products under both tile rules: 64 x 64 tiles, and 32 x 32 tiles where an output side is at most 32.

Element by element against the oracle's contractions, with the tolerance of the other contraction tests, at sizes
whose products are tiled (more than 8192 multiply-adds): one row or column over or short of a tile, last slices of
1 to 16 terms, each operand contiguous either way (left environments read their site transposed, right ones
multiply by a transposed site)."""
import numpy as np
import pytest

from oracle import mps_tjm as O1
from paper_2501_17913_gb300 import tjm

from gpu_common import lib_ready

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _rand(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) / np.sqrt(2)


@pytest.mark.parametrize("rule", [0, 1])
@pytest.mark.parametrize("chl,chr_,D", [(16, 17, 5), (31, 31, 5), (32, 32, 3), (33, 32, 4), (32, 33, 5), (64, 16, 5), (17, 64, 5),
                                        (64, 31, 8), (25, 60, 8), (64, 64, 5)])
def test_contractions_under_both_tile_rules(chl, chr_, D, rule):
    lib_ready()
    rng = np.random.default_rng(100 * chl + chr_)
    W, W2 = _rand(rng, D, D, 2, 2), _rand(rng, D, D, 2, 2)
    Lenv, Renv = _rand(rng, chl, D, chl), _rand(rng, D, chr_, chr_)
    C, M, th = _rand(rng, chl, chr_), _rand(rng, chl, 2, chr_), _rand(rng, chl, 2, 2, chr_)
    none = np.zeros((1, 1, 1))
    for kind, kw, f, args in [
        (0, dict(Lenv=Lenv, Renv=Renv, x=C), O1.heff0, (Lenv, Renv, C)),
        (1, dict(Lenv=Lenv, Renv=Renv, x=M, W1=W), O1.heff1, (Lenv, W, Renv, M)),
        (2, dict(Lenv=Lenv, Renv=Renv, x=th, W1=W, W2=W2), O1.heff2, (Lenv, W, W2, Renv, th)),
        (3, dict(Lenv=Lenv, Renv=none, x=M, W1=W), O1.env_left_update, (Lenv, M, W)),
        (4, dict(Lenv=none, Renv=Renv, x=M, W1=W), O1.env_right_update, (Renv, M, W)),
    ]:
        got = tjm.selftest_contract(kind, tjm.PREC_FP32, tensor_cores=False, tile_rule=rule, **kw)
        ref, mag = f(*args), f(*[abs(a) for a in args])
        assert (np.abs(got - ref) <= TOL * mag).all(), (kind, float((np.abs(got - ref) / mag).max()))


def test_unknown_tile_rule_is_refused():
    lib_ready()
    with pytest.raises(tjm.TJMError):
        tjm.selftest_contract(0, tjm.PREC_FP32, np.zeros((2, 2, 2)), np.zeros((2, 2, 2)), np.zeros((2, 2)), tile_rule=2)
