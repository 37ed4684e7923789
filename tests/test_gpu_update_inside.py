"""The parameter update inside the last product of a step gives the bits of the separate pass, which runs where O is asked for: tiles
cut in both directions, wide, plain and narrow, parameters off a 32-byte boundary, a second launch, every form of the launch."""
import pytest
import torch

import paper_2605_26842_b200 as pkg
from paper_2605_26842_b200.binding import FORM_FEW_TILES, FORM_MANY_TILES, FORM_WHOLE_MATRICES, describe_step

pytestmark = pytest.mark.gpu


# form of the last launch and columns of its update's work items, by the shapes below
KINDS = {(20, 520, 648): (FORM_MANY_TILES, 512), (10, 1032, 1000): (FORM_FEW_TILES, 512), (80, 520, 648): (FORM_MANY_TILES, 256), (1, 264, 776): (FORM_FEW_TILES, 128),
         (148, 248, 1016): (FORM_WHOLE_MATRICES, 256), (100, 200, 72): (FORM_WHOLE_MATRICES, 256), (222, 712, 136): (FORM_WHOLE_MATRICES, 256)}


@pytest.mark.parametrize("shape,T", [((20, 520, 648), 5), ((10, 1032, 1000), 5), ((148, 248, 1016), 5), ((100, 200, 72), 7), ((222, 712, 136), 5), ((1, 64, 72), 5), ((1, 256, 512), 5), ((1, 264, 776), 7), ((2, 1032, 392), 1), ((80, 520, 648), 5),
                                     ((80, 648, 520), 4), ((90, 264, 1160), 5), ((16, 128, 136), 5), ((150, 248, 520), 5), ((150, 520, 248), 6)])
def test_update_inside_the_last_product(shape, T):
    dev = torch.device("cuda", 0)
    gen = torch.Generator(device=dev).manual_seed(23)
    n = shape[0] * shape[1] * shape[2]
    hp = pkg.default_hparams(ns_steps=T)
    if shape in KINDS:
        last = describe_step([pkg.MatrixDesc(shape[1], shape[2], shape[0], 0, 0, 0)], hp)[-1]
        assert (last.form, last.update_columns) == KINDS[shape]
    W0 = torch.randn(n, generator=gen, device=dev) * 0.02
    G = [torch.randn(shape, generator=gen, device=dev) * 1e-3 for _ in range(2)]
    out = []
    for want_o in (False, True):
        buf = torch.full((n + 8,), 7.0, device=dev)
        p = buf[4:4 + n].view(shape)                     # 16 bytes into a line, guarded on both sides
        p.copy_(W0.view(shape))
        opt = pkg.MonaOptimizer([p])
        o = [torch.zeros(shape, device=dev)] if want_o else None
        for g in G:
            opt.step_ex(hp, [p], [g], o, 7)
        launches = opt.last_launch_count()
        assert opt.poll_status()[0] == 0
        opt.close()
        assert torch.all(buf[:4] == 7.0) and torch.all(buf[4 + n:] == 7.0)
        out.append((buf, launches))
    assert torch.equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1] - 1


@pytest.mark.parametrize("shapes", [[(1, 256, 512)], [(100, 520, 648), (2, 264, 520), (1, 33, 17)], [(148, 248, 1016)]])
def test_newton_schulz_and_update_without_the_prologue(shapes):
    """The phases behind the prologue in a call of their own (as the benchmark times them) are the kernels of a whole step: the same bits,
    and one launch more, which writes the parameters' addresses, for every chunk whose last product updates the parameters."""
    dev = torch.device("cuda", 0)
    gen = torch.Generator(device=dev).manual_seed(29)
    W0 = [torch.randn(s, generator=gen, device=dev) * 0.02 for s in shapes]
    G = [torch.randn(s, generator=gen, device=dev) * 1e-3 for s in shapes]
    hp = pkg.default_hparams()
    out = []
    for masks in ((7,), (1, 6)):
        p = [w.clone() for w in W0]
        opt = pkg.MonaOptimizer(p)
        for mask in masks:
            opt.step_ex(hp, p, G, None, mask)
            out.append(opt.last_launch_count())
        assert opt.poll_status()[0] == 0
        out.append(p + [opt.state.clone()])
        inside = sum(g.update_columns > 0 for g in describe_step(opt.descs, hp))
        opt.close()
    whole, whole_out, prologue, rest, parts_out = out
    assert rest == whole - prologue + inside
    for x, y in zip(whole_out, parts_out):
        assert torch.equal(x, y)
