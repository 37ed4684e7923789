"""Newton-Schulz launches of few tiles per product: narrow (256 x 128) tiles, the claim gate, several buckets side by side on
streams and SM pairs of their own.  Sizes around the edges of a narrow tile (a last tile of 8 to 128 columns, or none), one and many
tile rows, both orientations; more buckets than there are slots; results must not depend on the overlap."""
import pytest
import torch

import paper_2605_26842_b200 as pkg
from paper_2605_26842_b200.binding import FORM_FEW_TILES, FORM_MANY_TILES, FORM_WHOLE_MATRICES, describe_step
from tests.parity_util import TOL_O_BF16, TOL_O_MAX_BF16, TOL_STATE, TOL_W, run_case

pytestmark = pytest.mark.gpu


def check(errs):
    assert errs["M"] <= TOL_STATE, errs
    assert errs["O"] <= TOL_O_BF16 and errs["O_max"] <= TOL_O_MAX_BF16 and errs["dW"] <= TOL_W, errs


@pytest.mark.parametrize("shape", [(1, 64, 64), (1, 120, 136), (1, 128, 512), (1, 136, 128), (1, 256, 264), (1, 264, 376), (1, 392, 384),
                                   (2, 520, 648), (1, 1032, 1160), (30, 256, 256), (40, 128, 384)])
def test_one_bucket(shape):
    check(run_case([shape], steps=2, seed=51, sample={0: sorted({0, shape[0] - 1})}))


def test_more_buckets_than_slots():
    shapes = [(1, 256, 512), (1, 512, 256), (2, 384, 640), (1, 72, 200), (1, 1000, 136), (3, 192, 320), (1, 32, 512), (1, 33, 17)]
    check(run_case(shapes, steps=3, seed=52))


@pytest.mark.parametrize("large,form", [((400, 256, 256), FORM_WHOLE_MATRICES), ((120, 264, 264), FORM_MANY_TILES)])
def test_small_buckets_beside_a_large_one_match_a_single_stream(large, form):
    """Parameters and state agree bit for bit (a tile of any width accumulates over k in the same order), also in validation mode,
    whose chunks are smaller than a bucket."""
    dev = torch.device("cuda", 0)
    gen = torch.Generator().manual_seed(53)
    shapes = [large, (2, 264, 520), (1, 520, 264), (2, 32, 256)]
    launches = describe_step([pkg.MatrixDesc(r, c, b, 0, 0, 0) for b, r, c in shapes], options=pkg.default_options(chunk_budget_bytes=64 << 20))
    assert next(g for g in launches if (g.rows, g.cols) == large[1:]).form == form and any(g.form == FORM_FEW_TILES for g in launches)
    W0 = [torch.randn(s, generator=gen) * 0.02 for s in shapes]
    G = [[torch.randn(s, generator=gen) * 1e-3 for s in shapes] for _ in range(2)]
    for precision in (0, 1):
        def run(overlap):
            p = [w.clone().to(dev) for w in W0]
            opt = pkg.MonaOptimizer(p, options=pkg.default_options(chunk_overlap=overlap, chunk_budget_bytes=64 << 20))
            hp = pkg.default_hparams(ns_precision=precision)
            for k in range(2):
                opt.step(hp, p, [g.to(dev) for g in G[k]])
            assert opt.poll_status()[0] == 0
            out = [t.clone() for t in p] + [opt.state.clone()]
            opt.close()
            return out
        for x, y in zip(run(1), run(0)):
            assert torch.equal(x, y)


def test_repeated_steps_agree_bit_for_bit():
    """The operands that the epilogue and the copies of a phase read were written by other blocks moments before."""
    dev = torch.device("cuda", 0)
    gen = torch.Generator().manual_seed(54)
    shapes = [(1, 256, 512), (2, 512, 264), (1, 776, 520), (3, 136, 200)]
    W0 = [(torch.randn(s, generator=gen) * 0.02).to(dev) for s in shapes]
    G = [(torch.randn(s, generator=gen) * 1e-3).to(dev) for s in shapes]
    p = [w.clone() for w in W0]
    opt = pkg.MonaOptimizer(p)
    hp = pkg.default_hparams()
    first = None
    for _ in range(100):
        opt.state.zero_()
        for w, w0 in zip(p, W0):
            w.copy_(w0)
        opt.step(hp, p, G)
        if first is None:
            first = [w.clone() for w in p]
        for x, y in zip(p, first):
            assert torch.equal(x, y)
    assert opt.poll_status()[0] == 0
    opt.close()


@pytest.mark.parametrize("shape,form", [((1, 256, 512), FORM_FEW_TILES), ((2, 136, 200), FORM_FEW_TILES), ((1, 1032, 1160), FORM_FEW_TILES), ((400, 256, 256), None),
                                        ((100, 520, 648), FORM_MANY_TILES), ((20, 256, 256), FORM_WHOLE_MATRICES), ((148, 248, 1016), FORM_WHOLE_MATRICES)])
def test_waits_that_cannot_end_time_out_in_every_form_of_the_launch(shape, form):
    """Few tiles (early publication, claim gate, narrow tiles; one pair and several), many, and whole matrices (with and without tensors
    of the lanes' own): the launch reports the time-out, leaves, and the next step on the same handle gives the bits that it
    gives on a fresh one."""
    assert form is None or describe_step([pkg.MatrixDesc(shape[1], shape[2], shape[0], 0, 0, 0)])[0].form == form
    dev = torch.device("cuda", 0)
    gen = torch.Generator().manual_seed(55)
    W0 = (torch.randn(shape, generator=gen) * 0.02).to(dev)
    G = (torch.randn(shape, generator=gen) * 1e-3).to(dev)
    out = []
    for selftest in (False, True):
        p = [W0.clone()]
        opt = pkg.MonaOptimizer(p)
        if selftest:
            opt.selftest_timeout()
            assert pkg.STATUS_NAMES[opt.poll_status()[0]] == "MONA_ERR_TIMEOUT"
        opt.step(pkg.default_hparams(), p, [G])
        assert opt.poll_status()[0] == 0
        opt.close()
        out.append(p[0])
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("shape,columns", [((1, 256, 264), 384), ((1, 136, 136), 256), ((400, 256, 264), 512)])
def test_which_launches_take_narrow_tiles(shape, columns):
    """Executed flops of one iteration: the two symmetric products of one 256-row tile (two narrow tiles or one whole one, less where
    the second narrow tile has no columns) and B' X over `columns` columns, with the inner dimension padded to 64."""
    dev = torch.device("cuda", 0)
    p, g = [torch.zeros(shape, device=dev)], [torch.full(shape, 1e-3, device=dev)]
    opt = pkg.MonaOptimizer(p)
    opt.step(pkg.default_hparams(ns_steps=1), p, g)
    assert opt.poll_status()[0] == 0
    executed = opt.last_ns_flops()[0]
    opt.close()
    s, l = min(shape[1:]), max(shape[1:])
    ks, kl = -(-s // 64) * 64, -(-l // 64) * 64
    assert executed == shape[0] * 2.0 * 256 * (256 * kl + 256 * ks + columns * ks), executed
