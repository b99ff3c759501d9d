"""The calls that a program using this package makes, over the sizes it makes them at.

Three kinds of work:

* "linear": a clustered layer's projections at run time, from fp16 activations to fp32 outputs (input transformation,
  table lookup, accumulation), one token to a 2048-token prompt.  `path` says how the program calls the package:
  "fused" (one call from x to y per group of projections), "two_call" (quantise, then look up; the levels stay in the
  program's hands) or "host" (pinned host buffers in and out).  `layer` says which projections: "one" matrix N x K, a
  decoder "layer" (q, k, v, o: hidden x hidden, gate, up: ffn x hidden, down: hidden x ffn) whose inputs are all known,
  as a benchmark of the layer runs it, or the "mlp" alone in the order a model runs it: gate and up on one input, then
  down.
* "reclassify", "dbci", "smoothing": what the offline clustering of a layer calls between training rounds, at its
  start, and before it.

Weights are N(0, 0.02) smoothed per input channel and clustered to per-row quantile centroids; activations are N(0, 1)
with one channel in a hundred fifty times larger.
"""
import math

import torch

import paper_2506_12038_b200 as lcd


def linear(name, path, layer, bits, M, *, N=0, K=0, hidden=0, ffn=0, C=0, act_bits=4):
    return dict(name=name, kind="linear", path=path, layer=layer, bits=bits, C=C or 1 << bits, act_bits=act_bits, M=M,
                N=N, K=K, hidden=hidden, ffn=ffn)


def listed():
    return [
        # the smallest call: one 3-bit projection of a 7B-sized model for one token
        linear("one-4096-3bit-m1", "two_call", "one", 3, 1, N=4096, K=4096),
        # single-stream decode, all seven projections of a LLaMA-7B-shaped layer in one call
        linear("layer-7b-2bit-m1", "fused", "layer", 2, 1, hidden=4096, ffn=11008),
        # single-stream decode of a LLaMA-70B-shaped MLP: gate and up, then down
        linear("mlp-70b-2bit-m1", "fused", "mlp", 2, 1, hidden=8192, ffn=28672),
        # batched decode, sixteen sequences
        linear("layer-7b-3bit-m16", "two_call", "layer", 3, 16, hidden=4096, ffn=11008),
        # ten centroids per row (4-bit indices) and 8-bit activation levels, a few sequences
        linear("layer-7b-c10-act8-m4", "two_call", "layer", 4, 4, hidden=4096, ffn=11008, C=10, act_bits=8),
        # decode batch or speculative tokens beyond sixteen: the down projection
        linear("down-7b-2bit-m48", "two_call", "one", 2, 48, N=4096, K=11008),
        # a ragged prompt on a matrix whose sides are no multiple of anything
        linear("ragged-3bit-m333", "two_call", "one", 3, 333, N=5003, K=5001),
        # prompt processing of a LLaMA-13B-shaped layer
        linear("layer-13b-2bit-m2048", "fused", "layer", 2, 2048, hidden=5120, ffn=13824),
        # decode for a program that keeps its activations on the host
        linear("host-7b-2bit-m1", "host", "layer", 2, 1, hidden=4096, ffn=11008),
        # weights moved between clusters after a round of updates
        dict(name="reclassify-4096-c4", kind="reclassify", N=4096, K=4096, C=4),
        # initial centroids of a layer's weights
        dict(name="dbci-4096x11008", kind="dbci", n=4096 * 11008),
        # smoothing strength of a projection from 128 calibration tokens
        dict(name="smoothing-4096-t128", kind="smoothing", T=128, K=4096, G=21),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _side(rng, lo, hi):
    """A matrix side: a multiple of 256, of 64, or any number."""
    step = rng.choice((256, 64, 1))
    return max(lo, _log(rng, lo, hi) // step * step)


def draw(rng):
    pick = rng.random()
    if pick < 0.10:
        return dict(kind="reclassify", N=_side(rng, 512, 8192), K=_side(rng, 512, 8192), C=rng.choice((2, 4, 8, 10, 16)))
    if pick < 0.18:
        return dict(kind="dbci", n=_log(rng, 1 << 18, 45_000_000))
    if pick < 0.25:
        return dict(kind="smoothing", T=_log(rng, 32, 512), K=_side(rng, 1024, 14336), G=rng.randint(5, 33))
    bits = rng.choice((2, 2, 3, 4))
    C = {2: 4, 3: 8, 4: rng.choice((10, 16))}[bits]
    sizes = dict(N=0, K=0, hidden=0, ffn=0)
    if pick < 0.35:       # one matrix, few tokens
        path, layer, M = "two_call", "one", rng.choice((1, 1, _log(rng, 2, 16)))
        sizes.update(N=_side(rng, 512, 14336), K=_side(rng, 512, 14336))
    elif pick < 0.65:     # a group of projections, few tokens
        layer = rng.choice(("layer", "mlp"))
        M = rng.choice((1, 1, _log(rng, 2, 16)))
        path = rng.choice(("fused", "fused", "host")) if M == 1 else rng.choice(("two_call", "two_call", "host"))
        hidden = _side(rng, 1024, 5120 if layer == "layer" else 8192)
        sizes.update(hidden=hidden, ffn=int(hidden * rng.uniform(2.6, 3.5)) // 32 * 32)
    elif pick < 0.85:     # one matrix, a larger batch or a short prompt
        path, layer, M = "two_call", "one", _log(rng, 17, 1024)
        sizes.update(N=_side(rng, 1024, 14336), K=_side(rng, 1024, 14336))
    else:                 # a prompt through a layer
        path, layer, M = "fused", rng.choice(("layer", "mlp")), _log(rng, 64, 2048)
        hidden = _side(rng, 1024, 5120)
        sizes.update(hidden=hidden, ffn=int(hidden * rng.uniform(2.6, 2.7)) // 32 * 32)
    act_bits = rng.choice((4, 4, 8)) if path == "two_call" else 4
    return dict(kind="linear", path=path, layer=layer, bits=bits, C=C, act_bits=act_bits, M=M, **sizes)


# ------------------------------------------------------------------------------------------------- the inputs
def _groups(case):
    """The calls of a pass: a list of calls, a call being a list of (input number, N, K)."""
    h, f = case["hidden"], case["ffn"]
    if case["layer"] == "one":
        return [[(0, case["N"], case["K"])]]
    if case["layer"] == "mlp":
        return [[(0, f, h), (0, f, h)], [(1, h, f)]]
    return [[(0, h, h), (0, h, h), (0, h, h), (1, h, h), (2, f, h), (2, f, h), (3, h, f)]]


def _inputs(case):
    """The length of every input of a pass."""
    return {i: K for call in _groups(case) for i, _, K in call}


def _activations(g, M, K, outliers, scale=50.0):
    x = torch.randn(M, K, generator=g, device="cuda")
    x[:, outliers] *= scale
    return x.half()


def _weights(g, N, K, smooth, bits, C):
    """One clustered matrix as the program loads it: per-row quantile centroids, every weight at its nearest."""
    w = torch.randn(N, K, generator=g, device="cuda").mul_(0.02).mul_(smooth)
    centroids = torch.empty(N, C, dtype=torch.float16, device="cuda")
    idx = torch.empty(N, K, dtype=torch.uint8, device="cuda")
    at = ((torch.arange(C, device="cuda") + 0.5) / C * K).long()
    for lo in range(0, N, 4096):
        part = w[lo:lo + 4096]
        c = part.sort(dim=1).values[:, at].half()
        centroids[lo:lo + 4096] = c
        mid = (c[:, 1:].float() + c[:, :-1].float()) / 2
        idx[lo:lo + 4096] = torch.searchsorted(mid.contiguous(), part.contiguous()).to(torch.uint8)
    return lcd.PackedWeights(lcd.pack_weights(idx.cpu().numpy(), centroids.cpu().numpy(), bits, C))


def _prepare_linear(case, g):
    M, bits = case["M"], case["bits"]
    xs, smooth = {}, {}
    for i, K in _inputs(case).items():
        outliers = torch.randperm(K, generator=g, device="cuda")[: -(-K // 100)]
        xs[i] = _activations(g, M, K, outliers)
        calibration = _activations(g, 128, K, outliers).float().abs().amax(0)
        smooth[i] = (calibration / 0.08).sqrt().clamp(1e-5, 1e5)
    inv = {i: (1.0 / s).contiguous() for i, s in smooth.items()}
    calls = [[(i, _weights(g, N, K, smooth[i], bits, case["C"])) for i, N, K in call] for call in _groups(case)]
    if case["path"] == "host":
        batches = [lcd.HostBatch([(w, inv[i], M) for i, w in call]) for call in calls]
        for batch, call in zip(batches, calls):
            for j, (i, _) in enumerate(call):
                batch.x_view(j).copy_(xs[i])
            batch.capture()
        return dict(kind="host", batches=batches, inv=inv)
    ys = [[torch.empty(M, w.N, device="cuda") for _, w in call] for call in calls]
    if case["path"] == "fused":
        batches = [lcd.FusedBatch([(w, xs[i], inv[i], y) for (i, w), y in zip(call, out)]) for call, out in zip(calls, ys)]
        return dict(kind="fused", batches=batches, ys=ys)
    state = dict(kind="two_call", xs=xs, inv=inv, ys=ys, act_bits=case["act_bits"], calls=calls, idx={}, scale={})
    for i, K in _inputs(case).items():
        K_pad = -(-K // 256) * 256
        state["idx"][i] = (torch.empty(M, K_pad, dtype=torch.int8, device="cuda") if case["act_bits"] == 8 else
                           torch.empty(M, K_pad // 2, dtype=torch.uint8, device="cuda"))
        state["scale"][i] = torch.empty(M, device="cuda")
    if case["layer"] == "one":
        w = calls[0][0][1]
        state["workspace"] = torch.zeros(max(256, lcd.lut_linear_workspace_bytes(w, M)), dtype=torch.uint8, device="cuda")
        return state
    state["kind"] = "two_call_groups"
    state["batches"] = []
    for call, out in zip(calls, ys):
        mine = sorted({i for i, _ in call})
        quantise = lcd.ActBatch([(xs[i], inv[i], state["idx"][i], state["scale"][i]) for i in mine])
        look_up = lcd.LinearBatch([(w, state["idx"][i], state["scale"][i], y) for (i, w), y in zip(call, out)])
        state["batches"].append((quantise, look_up))
    return state


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if case["kind"] == "linear":
        return _prepare_linear(case, g)
    if case["kind"] == "reclassify":
        N, K, C = case["N"], case["K"], case["C"]
        centroids = torch.randn(N, C, generator=g, device="cuda").mul_(0.02).sort(dim=1).values.half()
        idx = torch.randint(0, C, (N, K), generator=g, device="cuda", dtype=torch.uint8)
        update = torch.randn(N, K, generator=g, device="cuda").mul_(0.004)
        out = (torch.empty_like(idx), torch.empty(N, C, dtype=torch.float64, device="cuda"),
               torch.empty(N, C, dtype=torch.int32, device="cuda"))
        return dict(kind="reclassify", args=(idx, centroids, update), out=out)
    if case["kind"] == "dbci":
        w = torch.randn(case["n"], generator=g, device="cuda").mul_(0.02)
        w[torch.randint(0, case["n"], (16,), generator=g, device="cuda")] *= 3      # a few weights far out
        return dict(kind="dbci", weights=w)
    K = case["K"]
    x = _activations(g, case["T"], K, torch.randperm(K, generator=g, device="cuda")[: -(-K // 100)])
    wmax = torch.rand(K, generator=g, device="cuda").mul_(0.03).add_(0.06)
    return dict(kind="smoothing", x=x, wmax=wmax, alphas=[i / (case["G"] - 1) for i in range(case["G"])])


# ------------------------------------------------------------------------------------------------- one pass
def run(state):
    kind = state["kind"]
    if kind == "fused":
        for batch in state["batches"]:
            batch.run()
        return state["ys"]
    if kind == "host":
        for batch in state["batches"]:
            batch.run()
        torch.cuda.current_stream().synchronize()      # the outputs are read on the host
        return [batch.y_view(j) for batch in state["batches"] for j in range(batch.count)]
    if kind == "two_call_groups":
        for quantise, look_up in state["batches"]:
            quantise.run()
            look_up.run()
        return [state["ys"], state["idx"], state["scale"]]
    if kind == "two_call":
        idx, scale = state["idx"][0], state["scale"][0]
        lcd.smooth_quantize_act(state["xs"][0], state["inv"][0], act_idx=idx, act_scale=scale, act_bits=state["act_bits"])
        lcd.lut_linear(state["calls"][0][0][1], idx, scale, y=state["ys"][0][0], workspace=state["workspace"])
        return [state["ys"], idx, scale]
    if kind == "reclassify":
        return lcd.reclassify(*state["args"], out=state["out"])
    if kind == "dbci":
        return lcd.dbci(state["weights"])
    return lcd.smoothing_search(state["x"], state["wmax"], state["alphas"])


def work(case):
    if case["kind"] == "reclassify":
        weights = case["N"] * case["K"]
        return {"bytes": 6 * weights + 14 * case["N"] * case["C"], "flops": 4 * weights}
    if case["kind"] == "dbci":
        return {"bytes": 12 * case["n"], "flops": 0}       # weights in, sorted weights and labels out
    if case["kind"] == "smoothing":
        return {"bytes": 2 * case["T"] * case["K"] + 8 * case["K"], "flops": 8 * case["T"] * case["K"] * case["G"]}
    M, moved, flops = case["M"], 0, 0
    for call in _groups(case):
        for _, N, K in call:
            moved += N * K * case["bits"] // 8 + 2 * N * case["C"] + 4 * M * N
            flops += 2 * M * N * K
    for K in _inputs(case).values():
        moved += 2 * M * K + 4 * K
        if case["path"] == "two_call":
            moved += M * K * case["act_bits"] // 8 + 4 * M
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    """About four times the distance from the same pass in 64 bits (2-norm: 3e-7 for the layers, 3e-16 for the sums of a
    reclassification, 9e-9 for the errors of a smoothing search, whose factors are fp32)."""
    if case["kind"] == "dbci":
        return "exact"
    if case["kind"] == "reclassify":
        return {"rel": 1e-14, "max": 4e-13, "differ": 0.0}
    if case["kind"] == "smoothing":
        return {"rel": 1e-6, "max": 1e-5, "differ": 0.0}
    return {"rel": 2e-6, "max": 2e-4, "differ": 0.0}
