"""Measured cases of the hybrid attention layer: the calls that training, prefill and the one-time installation of
frozen heads make through the public entry points (`paper_2609_34650_b200.Context`).

`op` says which part of a program a case is:

  update     forward and backward of one layer (a training update's share), pattern installed beforehand
  prefill    forward of one layer (inference; square causal attention, no cache)
  trainable  an update in which the patterns stay trainable: normalisers refreshed, forward, backward, pattern gradients
  calibrate  the calibration pass of one layer: forwards of all-ordinary heads in two batches, their attention
             statistics, and the mean map and scores at the end
  fit        compact patterns fitted to mean attention maps: target marginals, then 400 Adam steps

A state owns one `Context`, as a layer of a model does: a context holds the tables of one layer's patterns.
"""
import math

import numpy as np
import torch

import paper_2609_34650_b200 as saf

FIT_STEPS, FIT_LR, FIT_FLOOR = 400, 0.05, 1e-9      # the paper's optimiser settings


# --------------------------------------------------------------------------------------------------- the cases
def _layer(op, B, H, T, D, frozen, kv_group=1, slope=-0.01, grads="fp32", out="bf16", packed=False, layout="bthd"):
    return {"op": op, "B": B, "H": H, "T": T, "D": D, "frozen": frozen, "kv_group": kv_group, "slope": slope,
            "grads": grads, "out": out, "packed": packed, "layout": layout}


def listed():
    return [
        # the smallest test configuration: latency of a forward and a backward call
        dict(_layer("update", 1, 4, 256, 64, 1, slope=-0.05, layout="bhtd"), name="update-tiny"),
        # one user's short prompt on a grouped-query layer; launches and latency count
        dict(_layer("prefill", 1, 32, 333, 128, 10, kv_group=4), name="prefill-short-gqa"),
        # a small batch of unequal size on packed projections: bf16 gradients, half the heads frozen
        dict(_layer("update", 3, 12, 1537, 64, 6, grads="bf16", packed=True), name="update-ragged-packed"),
        # the 124M layer's update (12 heads x 64, 4K context, micro-batch 8, 25 % frozen)
        dict(_layer("update", 8, 12, 4096, 64, 3, slope=-0.05, layout="bhtd"), name="update-124m-4k"),
        # the 1B/8K layer's update
        dict(_layer("update", 4, 32, 8192, 64, 8), name="update-1b-8k"),
        # the layer of the paper's 1B model (16 heads x 96, 8K context, batch 2 per rank), bf16 gradients
        dict(_layer("update", 2, 16, 8192, 96, 4, grads="bf16"), name="update-d96-8k"),
        # the 124M layer's update at head dimension 128
        dict(_layer("update", 8, 12, 4096, 128, 3, slope=-0.05), name="update-d128-4k"),
        # batched prefill on grouped-query heads (32 query heads on 8 shared ones)
        dict(_layer("prefill", 4, 32, 4096, 128, 10, kv_group=4), name="prefill-gqa-4k"),
        # long-context prefill of one sequence
        dict(_layer("prefill", 1, 32, 32768, 128, 8, slope=-0.002, layout="bhtd"), name="prefill-32k"),
        # the pattern-control variant of an update: patterns trainable, fp32 output
        dict(_layer("trainable", 4, 12, 2048, 64, 6, out="fp32"), name="trainable-2k"),
        # calibration of one layer on 2 x 4 sequences
        {"op": "calibrate", "B": 4, "H": 12, "T": 2048, "D": 64, "kv_group": 1, "layout": "bthd", "name": "calibrate-2k"},
        # fit of the 124M model's 25 % set (36 heads)
        {"op": "fit", "heads": 36, "T": 4096, "name": "fit-36-heads-4k"},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same ranges: mostly updates and prefills, sizes spread over their logarithm."""
    op = rng.choice(["update"] * 5 + ["prefill"] * 3 + ["trainable", "calibrate", "fit"])
    if op == "fit":
        return {"op": op, "heads": rng.randint(1, 36), "T": _log_uniform(rng, 100, 4096)}
    H = rng.choice([4, 8, 12, 16, 32])
    D = rng.choice([64, 64, 96, 128, 128])
    layout = rng.choice(["bthd", "bhtd"])
    if op == "calibrate":
        return {"op": op, "B": rng.randint(2, 8), "H": H, "T": _log_uniform(rng, 100, 4096), "D": D,
                "kv_group": rng.choice([1, 1, 4]), "layout": layout}
    top = {"update": 8192, "prefill": 32768, "trainable": 4096}[op]
    T = _log_uniform(rng, {"update": 128, "prefill": 16, "trainable": 256}[op], top)
    if rng.random() < 0.4:
        T = min(top, -(-T // 128) * 128)                              # contexts are often round
    # batches up to the token count of the listed layers
    B = _log_uniform(rng, 1, max(1, min(32, 32768 // T)))
    kv_group = rng.choice([1, 1, 4])
    packed = kv_group == 1 and rng.random() < 0.3
    frozen = min(H, int(round(H * rng.choice([0.0, 0.25, 0.25, 0.5, 0.75, 1.0]))))
    if op == "trainable" and frozen == 0:
        frozen = H // 4
    if frozen == H:
        packed = False                                                # packed: at least one head has a query slot
    return _layer(op, B, H, T, D, frozen, kv_group, slope=rng.choice([-0.05, -0.01, -0.002]),
                  grads=rng.choice(["fp32", "bf16"]), out="fp32" if rng.random() < 0.2 else "bf16", packed=packed,
                  layout=layout)


# --------------------------------------------------------------------------------------------------- inputs
def _normal(gen, B, H, T, D, layout):
    """bf16 N(0,1) tensor seen as [B,H,T,D]; "bthd" is how projections leave it in memory."""
    if layout == "bthd":
        return torch.randn((B, T, H, D), generator=gen, device="cuda", dtype=torch.bfloat16).transpose(1, 2)
    return torch.randn((B, H, T, D), generator=gen, device="cuda", dtype=torch.bfloat16)


def _patterns(gen, mask, T, slope):
    """Structured-random alpha, decaying rho (rows of ordinary heads zero)."""
    H = mask.size
    a = torch.randn((H, T), generator=gen, device="cuda")
    r = slope * torch.arange(T, device="cuda", dtype=torch.float32) + 0.1 * torch.randn((H, T), generator=gen, device="cuda")
    keep = torch.from_numpy(mask.astype(np.float32)).cuda()[:, None]
    return a * keep, r * keep


def _prepare_layer(case, gen):
    B, H, T, D, g = case["B"], case["H"], case["T"], case["D"], case["kv_group"]
    layout, packed = case["layout"], case["packed"]
    order = torch.randperm(H, generator=gen, device="cuda").cpu().numpy()
    mask = np.zeros(H, dtype=np.uint8)
    mask[order[:case["frozen"]]] = 1
    nq = H - case["frozen"] if packed else H
    s = {"op": case["op"], "mask": mask, "ctx": saf.Context(torch.cuda.current_device())}
    s["Q"] = _normal(gen, B, nq, T, D, layout)
    s["K"] = _normal(gen, B, nq if packed else H // g, T, D, layout)
    s["V"] = _normal(gen, B, H // g, T, D, layout)
    s["alpha"], s["rho"] = _patterns(gen, mask, T, case["slope"])
    s["logZ"] = torch.zeros_like(s["alpha"])
    dO = _normal(gen, B, H, T, D, layout)
    s["O"] = torch.empty_like(dO, dtype=torch.float32 if case["out"] == "fp32" else torch.bfloat16)
    s["LSE"] = torch.empty((B, H, T), device="cuda")
    if case["op"] != "prefill":
        s["dO"] = dO
        gd = torch.float32 if case["grads"] == "fp32" else torch.bfloat16
        s["dQ"], s["dK"], s["dV"] = (torch.empty(t.shape, device="cuda", dtype=gd) for t in (s["Q"], s["K"], s["V"]))
    if case["op"] == "trainable":
        s["dalpha"], s["drho"] = torch.empty_like(s["alpha"]), torch.empty_like(s["rho"])
    s["prob"] = saf.make_problem(s["Q"], T, grad_dtype=saf.SAF_F32 if case["grads"] == "fp32" else saf.SAF_BF16,
                                 k_like=s["K"], v_like=s["V"], o_like=s["O"], kv_group=g, packed_qk=packed, H=H,
                                 o_dtype=saf.SAF_F32 if case["out"] == "fp32" else saf.SAF_BF16)
    if case["op"] != "trainable" and case["frozen"]:
        s["ctx"].saf_pattern_prepare(mask, s["alpha"], s["rho"], s["logZ"])       # installed once per layer
    return s


def _prepare_calibrate(case, gen):
    B, H, T, D, g = case["B"], case["H"], case["T"], case["D"], case["kv_group"]
    s = {"op": "calibrate", "ctx": saf.Context(torch.cuda.current_device()), "mask": np.zeros(H, dtype=np.uint8)}
    s["batches"] = [tuple(_normal(gen, B, h, T, D, case["layout"]) for h in (H, H // g, H // g)) for _ in range(2)]
    q, k, v = s["batches"][0]
    s["O"], s["LSE"] = torch.empty_like(q), torch.empty((B, H, T), device="cuda")
    s["prob"] = saf.make_problem(q, T, k_like=k, v_like=v, o_like=s["O"], kv_group=g, H=H)
    s["mean"] = torch.zeros((H, T, T), device="cuda")
    s["sumsq"], s["plogp"], s["s_var"], s["s_kl"] = (torch.zeros(H, device="cuda", dtype=torch.float64) for _ in range(4))
    s["size"] = (H, T, 2 * B)
    return s


def _prepare_fit(case, gen):
    """Stand-ins for calibrated mean attention maps: power-law decay in distance, an attention sink on key 0, per-key
    factors and log-normal noise, rows summing to one (the recipe of saf_inputs.mean_attention_maps, on the GPU)."""
    Hf, T = case["heads"], case["T"]
    s = {"op": "fit", "ctx": saf.Context(torch.cuda.current_device()), "size": (Hf, T)}
    maps = torch.empty((Hf, T, T), device="cuda")
    u = torch.rand((Hf, 2), generator=gen, device="cuda").tolist()
    i = torch.arange(T, device="cuda")
    dist = (i[:, None] - i[None, :]).float()
    log_dist = torch.log1p(dist.clamp_min(0.0))
    for h in range(Hf):
        power, sink = 1.0 + 2.0 * u[h][0], 0.5 * u[h][1]
        w = torch.randn((T, T), generator=gen, device="cuda").mul_(0.3)
        w.add_(log_dist, alpha=-power).add_(0.5 * torch.randn((1, T), generator=gen, device="cuda"))
        w.exp_().masked_fill_(dist < 0, 0.0)
        w.mul_((1.0 - sink) / w.sum(dim=1, keepdim=True))
        w[:, 0] += sink
        maps[h] = w
    s["maps"] = maps
    s["eta_abs"], s["eta_rel"] = (torch.empty((Hf, T), device="cuda", dtype=torch.float64) for _ in range(2))
    s["plogp"], s["loss"], s["kl"] = (torch.empty(Hf, device="cuda", dtype=torch.float64) for _ in range(3))
    s["alpha"], s["rho"], s["logZ"] = (torch.empty((Hf, T), device="cuda") for _ in range(3))
    return s


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    if case["op"] == "fit":
        return _prepare_fit(case, gen)
    if case["op"] == "calibrate":
        return _prepare_calibrate(case, gen)
    return _prepare_layer(case, gen)


# --------------------------------------------------------------------------------------------------- one pass
def run(state):
    s, ctx = state, state["ctx"]
    if s["op"] == "fit":
        Hf, T = s["size"]
        ctx.saf_fit_marginals(Hf, T, s["maps"], FIT_FLOOR, s["eta_abs"], s["eta_rel"], s["plogp"])
        ctx.saf_fit_compact(Hf, T, s["eta_abs"], s["eta_rel"], s["plogp"], FIT_STEPS, FIT_LR, s["alpha"], s["rho"],
                            s["logZ"], T, s["loss"], s["kl"])
        return {k: s[k] for k in ("eta_abs", "eta_rel", "plogp", "alpha", "rho", "logZ", "loss", "kl")}
    if s["op"] == "calibrate":
        H, T, n = s["size"]
        for k, (q, key, v) in enumerate(s["batches"]):
            ctx.saf_hybrid_attn_fwd(s["prob"], q, key, v, s["mask"], None, None, None, s["O"], s["LSE"])
            ctx.saf_calib_accumulate(s["prob"], q, key, s["LSE"], s["mean"], s["sumsq"], s["plogp"], k > 0)
        ctx.saf_calib_finalize(H, T, n, s["mean"], s["sumsq"], s["plogp"], s["s_var"], s["s_kl"])
        return {k: s[k] for k in ("mean", "s_var", "s_kl", "LSE")}
    if s["op"] == "trainable":
        ctx.saf_pattern_prepare(s["mask"], s["alpha"], s["rho"], s["logZ"])
    args = (s["mask"], s["alpha"], s["rho"], s["logZ"])
    ctx.saf_hybrid_attn_fwd(s["prob"], s["Q"], s["K"], s["V"], *args, s["O"], s["LSE"])
    out = ["O", "LSE"]
    if s["op"] != "prefill":
        ctx.saf_hybrid_attn_bwd(s["prob"], s["Q"], s["K"], s["V"], s["O"], s["dO"], s["LSE"], *args, s["dQ"], s["dK"], s["dV"])
        out += ["dQ", "dK", "dV"]
    if s["op"] == "trainable":
        ctx.saf_pattern_grad(s["prob"], s["V"], s["O"], s["dO"], *args, s["dalpha"], s["drho"])
        out += ["logZ", "dalpha", "drho"]
    return {k: s[k] for k in out}


# --------------------------------------------------------------------------------------------------- work, tolerance
def work(case):
    T = case["T"]
    pairs = T * (T + 1) // 2
    if case["op"] == "fit":
        # per step and pair one multiply-add for the normaliser and one for each of the two marginals
        return {"bytes": 4 * case["heads"] * pairs + 60 * case["heads"] * T, "flops": 6 * case["heads"] * pairs * FIT_STEPS}
    B, H, D, g = case["B"], case["H"], case["D"], case["kv_group"]
    if case["op"] == "calibrate":
        io = 2 * B * T * D * 2 * (2 * H + 2 * H // g) + 2 * 4 * B * H * T
        # scores and P V of the forward, and nothing of the statistics that the forward's scores do not give
        return {"bytes": io + 4 * H * pairs, "flops": 2 * B * H * 2 * 2 * D * pairs}
    hf = case["frozen"]
    ho = H - hf
    unit = 2 * D * pairs * B
    q, kv = B * ho * T * D, B * (H // g) * T * D                       # elements of the ordinary heads' Q, of V
    k = q if g == 1 else kv if ho else 0
    o, lse = B * H * T * D, 4 * B * H * T
    ob, gb = (4 if case["out"] == "fp32" else 2), (4 if case["grads"] == "fp32" else 2)
    bytes_ = 2 * (q + k + kv) + ob * o + lse + 12 * hf * T
    flops = unit * (2 * ho + hf)
    if case["op"] != "prefill":
        nq = q if case["packed"] else o
        nk = k if case["packed"] else kv
        bytes_ += 2 * (q + k + kv) + (ob * q + 2 * o) + lse + gb * (nq + nk + kv) + 12 * hf * T
        flops += unit * (5 * ho + hf)
    if case["op"] == "trainable":
        fo = B * hf * T * D
        bytes_ += 2 * kv + (ob + 2) * fo + 20 * hf * T
        flops += unit * hf + 4 * hf * pairs                            # dO V^T once more, normalisers
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    # About four times what these calls differ by from dense fp64 evaluations (T <= 4096).
    if case["op"] == "fit":            # after 400 Adam steps: logZ 1.3e-4, alpha 8e-5, elements 1.9e-3
        return {"rel": 5e-4, "max": 8e-3}
    if case["op"] == "calibrate":      # fp32 maps 1.6e-7, scores (differences of sums) 2.4e-6
        return {"rel": 1e-5}
    # bf16 tiles: outputs 2e-3, bf16 gradients 2.5e-3; single elements up to 0.19 of a tensor's rms
    return {"rel": 1e-2, "max": 0.7}
