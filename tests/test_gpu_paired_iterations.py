"""The first two Newton-Schulz iterations taken together on the short side: shapes wide enough for the rule that selects it (tile
work of the pair at most 0.8 of two plain iterations), with ragged tiles, both orientations, one matrix and many, and iteration
counts around the smallest that takes it."""
import pytest
import torch

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


def bf16_iterations(M, coefficients, T):
    """Eq. newton_schulz with A, b A + c A^2 + a I and X stored in bfloat16 and every sum in fp32, one iteration after the other."""
    a, b, c = coefficients

    def stored(x):
        return x.to(torch.bfloat16).float()
    X, scale = stored(M), 1.0 / M.norm()
    for _ in range(T):
        A = stored(X @ X.T * scale * scale)
        B = b * A + c * (A @ A)
        B.diagonal().add_(a)
        X, scale = stored(stored(B) @ X * scale), 1.0
    return X


@pytest.mark.parametrize("coefficients", [(3.4445, -4.7750, 2.0315), (4.0848, -6.8946, 2.9270), (3.6, -5.2, 2.3), (1.5, -0.5, 0.0)])
def test_no_further_from_64_bits_than_plain_iterations(coefficients):
    """Whatever the coefficients, O is as close to the iteration in 64 bits as a plain bfloat16 iteration leaves it, on rows whose
    scales differ by a factor of ten and on a condition number of 100 (the first four matrices of each kind, their mean error).
    The fifth on top is for the draw: errors of single matrices scatter by about a tenth."""
    dev = torch.device("cuda", 0)
    gen = torch.Generator(device=dev).manual_seed(43)
    n, s, l = 50, 264, 1048
    G = torch.randn(n, s, l, generator=gen, device=dev)
    G[:4] *= 10 ** -torch.rand(4, s, 1, generator=gen, device=dev)
    for i in range(4, 8):
        U, _, V = torch.linalg.svd(G[i].double(), full_matrices=False)
        G[i] = (U * torch.logspace(0, -2, s, device=dev, dtype=torch.float64) @ V).float()
    hp = pkg.default_hparams(accel_alpha=0.0, ns_a=coefficients[0], ns_b=coefficients[1], ns_c=coefficients[2])
    p, o = [torch.zeros(n, s, l, device=dev)], [torch.zeros(n, s, l, device=dev)]
    opt = pkg.MonaOptimizer(p)
    opt.step_ex(hp, p, [G], o, 7)
    assert opt.poll_status()[0] == 0
    M = opt.state_views(0)[0]
    for first in (0, 4):
        errs = [0.0, 0.0]
        for i in range(first, first + 4):
            X = M[i].double() / M[i].double().norm()
            for _ in range(hp.ns_steps):
                A = X @ X.T
                X = coefficients[0] * X + coefficients[1] * (A @ X) + coefficients[2] * (A @ (A @ X))
            for k, got in enumerate((o[0][i], bf16_iterations(M[i], coefficients, hp.ns_steps))):
                errs[k] += float((got.double() - X).norm() / X.norm()) / 4
        assert errs[0] <= 1.2 * errs[1], (first, errs)
    opt.close()


@pytest.mark.parametrize("shape,T,coefficient,paired", [((50, 264, 1048), 5, 3.4445, True), ((1, 264, 1048), 5, 3.4445, True), ((2, 1048, 264), 4, 3.4445, True),
                                                        ((50, 264, 1048), 3, 3.4445, False), ((50, 264, 1048), 5, 3.4446, False),
                                                        ((50, 264, 520), 5, 3.4445, False), ((1, 256, 768), 7, 3.4445, True)])
def test_which_launches_take_the_pair(shape, T, coefficient, paired):
    """Plain iterations all execute the same number of flops; the pair executes fewer than two of them."""
    dev = torch.device("cuda", 0)
    p, g = [torch.zeros(shape, device=dev)], [torch.full(shape, 1e-3, device=dev)]
    opt = pkg.MonaOptimizer(p)
    flops = []
    for steps in (1, T):
        opt.step(pkg.default_hparams(ns_steps=steps, ns_a=coefficient), p, g)
        flops.append(opt.last_ns_flops()[0])
    assert opt.poll_status()[0] == 0
    opt.close()
    assert (flops[1] < 0.999 * T * flops[0]) == paired and flops[1] <= 1.001 * T * flops[0], flops
