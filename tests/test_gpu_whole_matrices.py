"""Launches in which an SM pair owns whole matrices (shorter side of one tile): counts around a round of two matrices per pair, edges of
tiles in both directions, iterations taken together, more iterations than one launch holds.  The same matrices in a handle too small
for that form give the same bits, with and without a copy of O."""
import pytest
import torch

import paper_2605_26842_b200 as pkg
from paper_2605_26842_b200.binding import FORM_WHOLE_MATRICES, describe_step

pytestmark = pytest.mark.gpu


def two_steps(W0, G, hp, want_o):
    p = [W0.clone()]
    opt = pkg.MonaOptimizer(p, grad_dtype=G[0].dtype)
    o = [torch.zeros_like(W0)] if want_o else None
    for g in G:
        opt.step_ex(hp, p, [g], o, 7)
    assert opt.poll_status()[0] == 0
    out = [p[0].clone(), opt.state_views(0)[0].clone()] + (o or [])
    opt.close()
    return out


@pytest.mark.parametrize("shape,T", [((8, 64, 64), 5), ((9, 256, 256), 5), ((75, 136, 200), 7), ((148, 256, 264), 5), ((148, 72, 648), 4),
                                     ((296, 520, 256), 7), ((297, 248, 1032), 5), ((370, 1288, 128), 1),
                                     ((222, 248, 768), 7), ((370, 712, 136), 7), ((149, 128, 120), 5), ((297, 64, 128), 7), ((370, 256, 264), 5)])
@pytest.mark.parametrize("want_o", [False, True])
def test_whole_matrices_give_the_bits_of_single_ones(shape, T, want_o):
    dev = torch.device("cuda", 0)
    gen = torch.Generator(device=dev).manual_seed(17)
    W0 = torch.randn(shape, generator=gen, device=dev) * 0.02
    G = [torch.randn(shape, generator=gen, device=dev) * 1e-3 for _ in range(2)]
    hp = pkg.default_hparams(ns_steps=T)
    if shape not in ((296, 520, 256), (297, 248, 1032), (370, 1288, 128)):      # counts at which these spread their products
        assert describe_step([pkg.MatrixDesc(shape[1], shape[2], shape[0], 0, 0, 0)], hp)[0].form == FORM_WHOLE_MATRICES
    whole = two_steps(W0, G, hp, want_o)
    for lo, hi in ((0, 2), (shape[0] // 2, shape[0] // 2 + 1), (shape[0] - 1, shape[0])):
        part = two_steps(W0[lo:hi], [g[lo:hi].clone() for g in G], hp, want_o)
        for x, y in zip(whole, part):
            assert torch.equal(x[lo:hi], y), (lo, hi)
