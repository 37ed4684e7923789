"""What a step does to a matrix follows from the matrix, the options and the arguments of the call, never from how many others of
its shape the handle holds, how they are cut into chunks or what runs beside them: a set in one handle and the same set in
several give the same bits.  The sizes lie on both sides of every rule that looks at counts (tile widths, the claim gate, slab
lengths, chunks) and inside every path."""
import pytest
import torch

import paper_2605_26842_b200 as pkg

pytestmark = pytest.mark.gpu


def two_steps(W0, G, grad_dtype, state_dtype, hp, beside=()):
    """Parameters, O and momentum after two steps of one stack, with `beside` further (zero) stacks in the same handle."""
    dev = torch.device("cuda", 0)
    p = [W0.clone()] + [torch.zeros(s, device=dev) for s in beside]
    opt = pkg.MonaOptimizer(p, grad_dtype=grad_dtype, state_dtype=state_dtype)
    o = [torch.zeros_like(t) for t in p]
    for g in G:
        opt.step_ex(hp, p, [g] + [torch.zeros(s, device=dev, dtype=grad_dtype) for s in beside], o, 7)
    assert opt.poll_status()[0] == 0
    out = p[0].clone(), o[0].clone(), opt.state_views(0)[0].clone()
    opt.close()
    return out


@pytest.mark.parametrize("shape,cuts,grad,state", [
    ((50, 264, 1048), (1, 20, 50), torch.float32, torch.float32),        # two iterations taken together, one tile row and a bit
    ((20, 2056, 520), (3, 20), torch.bfloat16, pkg.MONA_STATE_COMBINED),
    ((40, 256, 512), (1, 2, 17, 40), torch.float32, torch.float32),      # slabs of one trip to slabs of sixteen
    ((300, 136, 264), (1, 150, 300), torch.bfloat16, torch.bfloat16),
    ((9, 1032, 1160), (1, 4, 9), torch.float32, torch.float32),
    ((100, 32, 1024), (1, 37, 64, 100), torch.float32, torch.float32),   # one block cluster per matrix
    ((300, 520, 24), (2, 300), torch.float32, torch.bfloat16),
    ((150, 63, 1000), (1, 20, 150), torch.float32, torch.float32),
    ((23, 257, 1001), (1, 8, 23), torch.bfloat16, torch.float32),        # fp32 products, scalar elementwise passes
])
def test_a_part_of_a_set_gives_the_bits_of_the_whole(shape, cuts, grad, state):
    dev = torch.device("cuda", 0)
    gen = torch.Generator(device=dev).manual_seed(91)
    W0 = torch.randn(shape, generator=gen, device=dev) * 0.02
    G = [(torch.randn(shape, generator=gen, device=dev) * 1e-3).to(grad) for _ in range(2)]
    hp = pkg.default_hparams()
    whole = two_steps(W0, G, grad, state, hp)
    for lo, hi in zip((0,) + cuts, cuts):
        part = two_steps(W0[lo:hi], [g[lo:hi].clone() for g in G], grad, state, hp)
        for x, y in zip(whole, part):
            assert torch.equal(x[lo:hi], y), (lo, hi)
    beside = [(1, 512, 512), (3,) + shape[1:], (1, 32, 512), (200, 256, 256)]
    lo, hi = 0, cuts[0]
    for x, y in zip(whole, two_steps(W0[lo:hi], [g[lo:hi].clone() for g in G], grad, state, hp, beside)):
        assert torch.equal(x[lo:hi], y)


@pytest.mark.parametrize("shape", [(40, 256, 512), (3, 768, 2048), (2, 2056, 2048), (5, 33, 17)])
def test_prologue_noalloc_gives_the_norm_of_a_stack(shape):
    """With T = 0 the step's O is M * inv, one fp32 product per element."""
    dev = torch.device("cuda", 0)
    gen = torch.Generator(device=dev).manual_seed(92)
    G = torch.randn(shape, generator=gen, device=dev) * 1e-3
    hp = pkg.default_hparams(ns_steps=0)
    p = [torch.zeros(shape, device=dev)]
    o = [torch.zeros(shape, device=dev)]
    opt = pkg.MonaOptimizer(p)
    opt.step_ex(hp, p, [G], o, 7)
    for b in range(shape[0]):
        M, A, Gp = (torch.zeros(shape[1:], device=dev) for _ in range(3))
        inv = torch.zeros(1, device=dev)
        g = torch.empty(shape[1:], device=dev).copy_(G[b])
        pkg.prologue_noalloc(g, M, A, Gp, inv, hp)
        assert torch.equal(M, opt.state_views(0)[0][b])
        assert torch.equal(M * inv, o[0][b])
    opt.close()
