"""The fp32 products (sizes the tensor-core path does not take, and the validation mode): remainders of the 64 x 64 tile and of the
64-wide k-slab, one tile and many, both orientations, stacks."""
import pytest

import paper_2605_26842_b200 as pkg
from tests.parity_util import TOL_O_FP32, TOL_O_MAX_FP32, TOL_STATE, TOL_W, run_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 65, 65), (1, 67, 4001), (2, 127, 129), (1, 128, 192), (3, 193, 95), (1, 257, 321), (1, 511, 130), (1, 1001, 71)])
def test_fp32_products(shape):
    errs = run_case([shape], steps=2, seed=61, hp=pkg.default_hparams(ns_precision=1))
    assert errs["M"] <= TOL_STATE, errs
    assert errs["O"] <= TOL_O_FP32 and errs["O_max"] <= TOL_O_MAX_FP32 and errs["dW"] <= TOL_W, errs
