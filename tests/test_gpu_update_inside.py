"""The parameter update inside the last product of a step gives the bits of the separate pass, which runs where O is asked for: tiles
cut in both directions, wide, plain and narrow, parameters off a 32-byte boundary, a second launch, every form of the launch."""
import pytest
import torch

import paper_2605_26842_b200 as pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,T", [((1, 64, 72), 5), ((1, 256, 512), 5), ((1, 264, 776), 7), ((2, 1032, 392), 1), ((80, 520, 648), 5),
                                     ((80, 648, 520), 4), ((90, 264, 1160), 5), ((16, 128, 136), 5), ((150, 248, 520), 5), ((150, 520, 248), 6)])
def test_update_inside_the_last_product(shape, T):
    dev = torch.device("cuda", 0)
    gen = torch.Generator(device=dev).manual_seed(23)
    n = shape[0] * shape[1] * shape[2]
    hp = pkg.default_hparams(ns_steps=T)
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
