"""All-FP32 runs (FP32 factorizations) in exact mode against state vectors in 64 bits, averaged over seeds
because a single run's rounding error varies by 15 %.

The bound is the error measured on 200 seeds with correctly rounded rotations throughout, 4.9e-7 (standard
error 0.06e-7); with rotations from approximate roots it was 5.1e-7 to 5.3e-7, with a correctly rounded cosine
and phase alone 4.3e-7."""
import importlib.util
import os

import numpy as np
import pytest

from gpu_common import lib_ready

pytestmark = pytest.mark.gpu


def test_mean_error_of_all_fp32_runs():
    lib_ready()
    path = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "perf", "cases.py")
    spec = importlib.util.spec_from_file_location("perf_cases", path)
    cases = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(cases)
    c = cases.case("", L=8, chi=32, n_traj=152, steps=3, prec="f32dec32", start="neel", exact=True)
    err = []
    for seed in range(201, 241):
        (got,), (ref,) = cases.run(cases.prepare(c, seed)), cases.exact(c, seed)
        keys = [k for k in ref if ref[k] is not None]
        err.append(np.sqrt(sum(((got[k].astype(np.float64) - ref[k]) ** 2).sum() for k in keys)
                           / sum((ref[k] ** 2).sum() for k in keys)))
    assert np.mean(err) <= 4.9e-7, np.mean(err)
