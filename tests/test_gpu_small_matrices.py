"""The one-cluster-per-matrix Newton-Schulz kernel (shorter side <= 64): padded and exact block sizes, one to eight blocks per
matrix, both orientations, more matrices than blocks fit, the longest rows it takes."""
import pytest

import paper_2605_26842_b200 as pkg
from tests.parity_util import TOL_O_FP32, TOL_O_MAX_FP32, TOL_STATE, TOL_W, run_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,T", [((1, 1, 300), 5), ((1, 5, 3), 5), ((2, 32, 127), 5), ((1, 32, 128), 5), ((3, 33, 129), 5),
                                     ((1, 1025, 32), 5), ((40, 8, 1024), 3), ((200, 24, 135), 2), ((1, 64, 4095), 2), ((1, 4096, 63), 2),
                                     ((2, 64, 65), 1), ((1, 17, 1030), 6)])
def test_small_matrices(shape, T):
    hp = pkg.default_hparams(ns_steps=T, ns_precision=1)
    errs = run_case([shape], steps=2, hp=hp, seed=17, sample={0: sorted({0, shape[0] // 2, shape[0] - 1})})
    assert errs["M"] <= TOL_STATE, errs
    assert errs["O"] <= TOL_O_FP32 and errs["O_max"] <= TOL_O_MAX_FP32 and errs["dW"] <= TOL_W, errs
    assert errs["launches"] == 3, errs          # prologue, iteration, update
