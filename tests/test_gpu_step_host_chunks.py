"""mona_step_host cuts a set into chunks of its own (8 MiB of parameters at least): chunks that span descriptors and end inside one, a
stack with padding between its matrices, sets below and above the smallest chunk.  Everything must equal mona_step bit for bit."""
import pytest
import torch

import paper_2605_26842_b200 as pkg
from tests.parity_util import _init_from_descs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes,pad", [([(1, 64, 128)], 0), ([(7, 512, 520), (13, 512, 520), (3, 520, 512), (1, 33, 1001), (1, 32, 256)], 0),
                                        ([(9, 512, 512), (2, 512, 512)], 64), ([(100, 32, 1024), (1, 256, 512)], 0)])
def test_step_host_equals_step(shapes, pad):
    dev = torch.device("cuda", 0)
    gen = torch.Generator().manual_seed(71)
    descs = [pkg.MatrixDesc(r, c, b, r * c + pad, 0, 0) for b, r, c in shapes]
    sizes = [(b - 1) * (r * c + pad) + r * c for b, r, c in shapes]
    W0 = [torch.randn(n, generator=gen) * 0.02 for n in sizes]
    G = [[torch.randn(n, generator=gen) * 1e-3 for n in sizes] for _ in range(2)]
    hp = pkg.default_hparams()

    def run(host):
        p = [w.clone().to(dev) for w in W0]
        opt = pkg.MonaOptimizer.__new__(pkg.MonaOptimizer)
        _init_from_descs(opt, descs, dev, None)
        for k in range(2):
            if host:
                g_host = [g.clone().pin_memory() for g in G[k]]
                p_host = [torch.full((n,), 5.0).pin_memory() for n in sizes]
                opt.step_host(hp, p, [torch.zeros(n, device=dev) for n in sizes], g_host, p_host)
                torch.cuda.synchronize()
                for a, b in zip(p_host, p):
                    assert torch.equal(a, b.cpu())
            else:
                opt.step(hp, p, [g.to(dev) for g in G[k]])
        assert opt.poll_status()[0] == 0
        out = [t.clone() for t in p] + [opt.state.clone()]
        opt.close()
        return out
    for x, y in zip(run(False), run(True)):
        assert torch.equal(x, y)
