"""The first two Newton-Schulz iterations taken together on the short side: sets wide and numerous enough for the rule that
selects it (tile work of the pair at most 0.8 of two plain iterations, at least 150 tiles per product), with ragged tiles, both
orientations, and iteration counts around the smallest that takes it."""
import pytest

import paper_2605_26842_b200 as pkg
from tests.parity_util import TOL_O_BF16, TOL_O_MAX_BF16, TOL_STATE, TOL_W, run_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,T", [((150, 136, 776), 5), ((50, 264, 1048), 5), ((50, 1048, 264), 5), ((25, 520, 2056), 5),
                                     ((50, 264, 1048), 3), ((50, 264, 1048), 4), ((50, 1048, 264), 7), ((49, 264, 1048), 5)])
def test_first_two_iterations_together(shape, T):
    """Against the oracle, to the tolerances of the plain iteration (its error is the same bf16 storage of A, B' and X)."""
    errs = run_case([shape], steps=2, seed=41, hp=pkg.default_hparams(ns_steps=T), sample={0: [0, shape[0] // 2, shape[0] - 1]})
    assert errs["M"] <= TOL_STATE, errs
    assert errs["O"] <= TOL_O_BF16 and errs["O_max"] <= TOL_O_MAX_BF16 and errs["dW"] <= TOL_W, errs
