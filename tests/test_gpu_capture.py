"""A step captured into a CUDA graph and replayed gives the bits of a step that is launched: launches that start early, several
streams, the fp32 chain, the update inside the last product."""
import pytest
import torch

import paper_2605_26842_b200 as pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes", [[(1, 256, 512)], [(1, 257, 129), (2, 32, 256), (3, 136, 264), (1, 520, 264)], [(160, 256, 264), (9, 128, 128)],
                                    [(40, 1032, 1160), (1, 33, 17)]])
def test_a_captured_step_gives_the_bits_of_a_launched_one(shapes):
    dev = torch.device("cuda", 0)
    gen = torch.Generator(device=dev).manual_seed(31)
    W0 = [torch.randn(s, generator=gen, device=dev) * 0.02 for s in shapes]
    G = [torch.randn(s, generator=gen, device=dev) * 1e-3 for s in shapes]
    hp = pkg.default_hparams()
    out = []
    for captured in (False, True):
        p = [w.clone() for w in W0]
        opt = pkg.MonaOptimizer(p)
        opt.step(hp, p, G)
        if captured:
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                opt.step(hp, p, G)
            for _ in range(2):
                graph.replay()
        else:
            for _ in range(2):
                opt.step(hp, p, G)
        assert opt.poll_status()[0] == 0
        out.append(p + [opt.state.clone()])
        opt.close()
    for x, y in zip(*out):
        assert torch.equal(x, y)
