"""Performance cases of the MONA step: parameter sets a training job hands to the library, one optimizer step each.

A case is a dict of plain values:
  shapes     space-separated matrices "rows x cols" or stacks of them "batch * rows x cols", one descriptor each
  grad       gradient type, "f32" or "bf16"
  state      storage of A and G_prev: "f32" (Algorithm 1), "bf16" (MONA-Lite) or "combined" (the single buffer Z)
  algorithm  "mona" or "muon"
  precision  "bf16" (tensor cores) or "f32" (validation mode)
  host       True: gradients arrive in, and parameters return to, pinned host memory (mona_step_host)
  ns_steps   Newton-Schulz iterations T
"""
from __future__ import annotations

import math

import torch

import paper_2605_26842_b200 as pkg

SIGMA = 1e-3            # gradient scale, as in the synthetic workloads
RHO = 0.9               # lag-1 correlation of consecutive gradients


def _case(name, shapes, grad="f32", state="f32", algorithm="mona", precision="bf16", host=False, ns_steps=5):
    c = {"shapes": " ".join(shapes), "grad": grad, "state": state, "algorithm": algorithm, "precision": precision,
         "host": host, "ns_steps": ns_steps}
    return dict(c, name=name) if name else c


def _dense_layer(d, ff):
    return [f"{d}x{d}"] * 4 + [f"{ff}x{d}"] * 2 + [f"{d}x{ff}"]


def _expert_layer(width, hidden, experts):
    return [f"{experts}*{width}x{hidden}"] * 2 + [f"{experts}*{hidden}x{width}"]


def listed():
    return [
        # the smallest call: one weight, nothing but launches and the chain of fifteen dependent products
        _case("single_256x512", ["256x512"]),
        # a toy model of a few stacked experts, attention and a router: several shape buckets, each far too small for the GPU
        _case("small_mixed_set", ["4*256x512", "4*512x256", "512x512", "32x512"], grad="bf16"),
        # one transformer block, stepped on its own (a pipeline stage, or a step taken as a layer's gradient arrives)
        _case("dense_block_1024", _dense_layer(1024, 2816), grad="bf16"),
        # the dense benchmark configuration: twelve transformer blocks in one call
        _case("dense_blocks_12L", _dense_layer(1024, 2816) * 12),
        # a shard of a ~1B MoE: four layers of 512x1024 experts, attention, and routers on the fp32 small-matrix path
        _case("moe_1b_4L", (_expert_layer(512, 1024, 32) + ["1024x1024"] * 4 + ["32x1024"]) * 4),
        # a shard of the headline ~7B MoE: three layers of 768x2048 experts, 2048x2048 attention and the shared expert
        _case("moe_7b_3L", (_expert_layer(768, 2048, 64) + ["2048x2048"] * 4 + ["1536x2048"]) * 3),
        # a large-MoE shard, one layer with half of its 128 experts, bf16 gradients: the largest matrices of the benchmark
        _case("moe_shard_64E", _expert_layer(1024, 4096, 64) + ["4096x4096"] * 4, grad="bf16"),
        # 256x768 experts, thousands of one-tile matrices, with bf16 gradients and MONA-Lite storage
        _case("experts_256x768_lite", _expert_layer(256, 768, 128) * 4, grad="bf16", state="bf16"),
        # 1024x1536 experts with the single-buffer acceleration state
        _case("experts_1024x1536_combined", _expert_layer(1024, 1536, 64), state="combined"),
        # plain Muon (the baseline algorithm) on dense blocks whose sides are multiples of 8 but of no tile size
        _case("ragged_dense_muon", _dense_layer(1160, 3096) * 4, algorithm="muon"),
        # sides that are not multiples of 8 (odd vocabularies, heads, adapters): the step runs in fp32
        _case("odd_sizes", ["2*1023x511", "257x1025", "1001x1500", "10x768", "33x17"]),
        # gradients produced in host memory (offloaded accumulation): one ~1B-MoE layer through the host-to-host call
        _case("host_moe_1b_1L", _expert_layer(512, 1024, 32) + ["1024x1024"] * 4 + ["32x1024"], host=True),
    ]


def _log_int(rng, lo, hi, multiple=1):
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / multiple)) * multiple
    return max(lo, min(hi, v))


def _options(rng):
    return {"grad": rng.choice(["f32", "bf16"]), "state": rng.choice(["f32", "f32", "bf16", "combined"]),
            "algorithm": rng.choice(["mona", "mona", "mona", "muon"])}


def draw(rng):
    kind = rng.choice(["few", "dense", "experts", "experts", "ragged", "odd", "host"])
    step = rng.choice([8, 8, 64, 128])
    if kind == "few":           # a handful of single matrices, down to one
        shapes = [f"{_log_int(rng, 64, 2048, 8)}x{_log_int(rng, 64, 2048, 8)}" for _ in range(rng.randint(1, 6))]
        if rng.random() < 0.3:
            shapes.append(f"{rng.choice([8, 16, 32])}x{_log_int(rng, 64, 1024, 8)}")
        return _bounded(shapes, dict(_options(rng)))
    if kind == "dense":         # transformer blocks
        d = _log_int(rng, 256, 2048, 64)
        return _bounded(_dense_layer(d, int(d * rng.choice([2.0, 2.75, 4.0])) // 8 * 8) * _log_int(rng, 1, 12), _options(rng))
    if kind == "experts":       # stacked experts with attention and routers
        hidden = _log_int(rng, 256, 4096, max(step, 64))
        width = max(64, int(hidden * rng.choice([0.25, 1 / 3, 0.375, 0.5, 2 / 3])) // step * step)
        layer = _expert_layer(width, hidden, _log_int(rng, 4, 128)) + [f"{hidden}x{hidden}"] * 4
        if hidden <= 1024 and rng.random() < 0.5:
            layer.append(f"32x{hidden}")
        return _bounded(layer * _log_int(rng, 1, 4), _options(rng))
    if kind == "ragged":        # multiples of 8 that no tile size divides
        d = _log_int(rng, 200, 1800, 8) // 16 * 16 + 8
        return _bounded(_dense_layer(d, int(d * rng.uniform(1.5, 4.0)) // 16 * 16 + 8) * _log_int(rng, 1, 6), _options(rng))
    if kind == "odd":           # sides that are not multiples of 8, in the default mode or in the fp32 mode
        shapes = [f"{_log_int(rng, 1, 2)}*{_log_int(rng, 10, 1500)}x{_log_int(rng, 10, 1500)}" for _ in range(rng.randint(1, 5))]
        return _bounded(shapes, dict(_options(rng), precision="f32"))
    hidden = _log_int(rng, 256, 1024, 64)
    return _bounded(_expert_layer(max(64, hidden // 2), hidden, _log_int(rng, 2, 32)) + [f"{hidden}x{hidden}"] * 4, dict(grad=rng.choice(["f32", "bf16"]), host=True))


def _bounded(shapes, options):
    """The case, cut to fewer descriptors and smaller stacks until it costs no more than the largest listed one."""
    while True:
        c = _case(None, shapes, **options)
        w = work(c)
        if w["flops"] <= 1.1e13 and w["bytes"] <= 3e10:
            return c
        if len(shapes) > 7:
            shapes = shapes[: (len(shapes) + 1) // 2]
        else:
            shapes = [f"{max(1, b // 2)}*{r}x{n}" for b, r, n in _parse(c)]


def _parse(case):
    out = []
    for item in case["shapes"].split():
        batch, _, shape = item.rpartition("*")
        rows, cols = shape.split("x")
        out.append((int(batch or 1), int(rows), int(cols)))
    return out


def _dtypes(case):
    grad = torch.bfloat16 if case["grad"] == "bf16" else torch.float32
    state = {"f32": torch.float32, "bf16": torch.bfloat16, "combined": pkg.MONA_STATE_COMBINED}[case["state"]]
    return grad, state


def prepare(case, seed):
    """Parameters, this step's gradients, and an optimizer in the middle of training: momentum with a few strong
    directions over noise whose rows differ in scale by a factor of ten, G_prev correlated with the new gradient."""
    grad_dtype, state_dtype = _dtypes(case)
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)

    def normal(shape, std):
        return torch.empty(shape, device=dev).normal_(0.0, std, generator=gen)

    shapes = _parse(case)
    # master weights in one flat buffer, as trainers keep them; every matrix starts on a 256-byte boundary
    starts = [0]
    for b, r, c in shapes:
        starts.append(starts[-1] + -(-b * r * c // 64) * 64)
    weights = normal((starts[-1],), 0.02)
    params = [weights[at:at + b * r * c].view(b, r, c) for at, (b, r, c) in zip(starts, shapes)]
    opt = pkg.MonaOptimizer(params, grad_dtype=grad_dtype, state_dtype=state_dtype)
    hp = pkg.default_hparams(ns_steps=case["ns_steps"], ns_precision=1 if case["precision"] == "f32" else 0,
                             algorithm=1 if case["algorithm"] == "muon" else 0)
    grads = []
    for i, (b, r, c) in enumerate(shapes):
        m, a, gp = opt.state_views(i)
        strength = (5 * SIGMA * (math.sqrt(r) + math.sqrt(c))) * 0.6 ** torch.arange(4, device=dev)
        torch.baddbmm(normal((b, r, c), 3 * SIGMA).mul_(10 ** -torch.rand((b, r, 1), device=dev, generator=gen)),
                      normal((b, r, 4), r ** -0.5) * strength, normal((b, 4, c), c ** -0.5), out=m)
        prev = normal((b, r, c), SIGMA)
        g = prev.mul(RHO).add_(normal((b, r, c), SIGMA), alpha=math.sqrt(1 - RHO * RHO))
        if case["algorithm"] != "muon":
            a.copy_(normal((b, r, c), (1 - hp.accel_beta) * SIGMA))
            if gp is not None:
                gp.copy_(prev)
            else:
                a.mul_(hp.accel_beta).sub_(prev, alpha=1 - hp.accel_beta)
        grads.append(g.to(grad_dtype))
        del prev, g
    # what a step updates: the flat weights, and M, A, G_prev of each shape (the state of equal shapes is contiguous)
    outputs = [weights]
    for shape in dict.fromkeys((r, c) for _, r, c in shapes):
        same = [i for i, (_, r, c) in enumerate(shapes) if (r, c) == shape]
        n = sum(params[i].numel() for i in same)
        for view in opt.state_views(same[0])[:1 if case["algorithm"] == "muon" else 3]:
            if view is not None:
                at = view.data_ptr() - opt.state.data_ptr()
                outputs.append(opt.state[at:at + n * view.element_size()].view(view.dtype).view(-1, *shape))
    state = {"opt": opt, "hp": hp, "params": params, "grads": grads, "outputs": outputs}
    if case["host"]:
        state["grads_host"] = [torch.empty(g.shape, dtype=g.dtype, pin_memory=True).copy_(g) for g in grads]
        state["params_host"] = [torch.empty(p.shape, dtype=p.dtype, pin_memory=True) for p in params]
    return state


def run(state):
    """One optimizer step; its outputs are the updated parameters and the updated optimizer state."""
    opt, hp, params, grads = state["opt"], state["hp"], state["params"], state["grads"]
    if "grads_host" in state:
        opt.step_host(hp, params, grads, state["grads_host"], state["params_host"])
        return state["outputs"] + state["params_host"]
    opt.step(hp, params, grads)
    return state["outputs"]


def work(case):
    """Bytes: the gradient read; parameter, momentum and acceleration state read and written.  Flops: per iteration and matrix
    with sides s <= l, the two symmetric products counted once per pair of entries and X' = B' X: 3 s^2 l + s^3."""
    nbytes = flops = 0
    for b, r, c in _parse(case):
        s, l = min(r, c), max(r, c)
        aux = 0 if case["algorithm"] == "muon" else {"f32": 16, "bf16": 8, "combined": 8}[case["state"]]
        nbytes += b * r * c * ((2 if case["grad"] == "bf16" else 4) + 8 + 8 + aux)
        flops += case["ns_steps"] * b * (3 * s * s * l + s ** 3)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Against the step in 64 bits the parameters, about 1 % of whose norm is the bf16 update, were off by 0.8-1.1e-4 (largest
    element 1.7e-3 rms); on the fp32 path everything by 3-5e-8 (4e-7, 1.1e-6 behind a rounded A).  With bf16 storage an element
    of A whose value lies near a tie may round the other way: one bf16 step, 2^-7 of it at most, on a small share of them."""
    fp32 = case["precision"] == "f32" or all(min(r, c) < 64 or r % 8 or c % 8 for _, r, c in _parse(case))
    if case["state"] == "bf16" and case["algorithm"] != "muon":
        return {"rel": 4e-4, "max": 1e-2}
    return {"rel": 3e-7, "max": 4e-6} if fp32 else {"rel": 4e-4, "max": 7e-3}
