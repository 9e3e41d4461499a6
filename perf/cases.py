"""Timing cases of the masked gated-MLP library: what a policy that serves an action expert calls, and at which sizes.

A case is one pass through the public entry points on inputs that live where such a program holds them: packed weights,
lists and activations on the device, except for the host-to-host step.  Sizes follow the repository's workloads (the
1024/4096 and 2048/16384 experts of 18 layers, chunks of 32 and 51 action tokens, the Context Cache layer with 768
visual rows) and, in draw(), the ragged sizes around them.
"""
from __future__ import annotations

import math

import torch

import paper_2609_19104_b200 as rm


# ------------------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # Mask rebuild of the sliding-window workload: 18 lists, a 3-of-4 vote over per-record top-15 % sets.  The
        # smallest call: launch and latency count.
        dict(name="mask-vote-window4", kind="mask", rule="vote", lists=18, I=4096, W=4, density=0.15),
        # Mask refresh of the large expert: exact top-20 % of one dense record per layer.
        dict(name="mask-topk-large", kind="mask", rule="topk", lists=18, I=16384, W=1, density=0.20),
        # One masked layer with a Bernoulli mask, for a model runtime that keeps the layer loop to itself.
        dict(name="layer-bernoulli30", kind="layer", H=1024, I=4096, T=51, density=0.30),
        # One denoising step of the base expert with a top-25 % mask: the ordinary call of a control loop.
        dict(name="step-top25", kind="step", H=1024, I=4096, L=18, T=51, B=1, density=0.25, runs=False, host=False),
        # The same expert on a 32-token chunk with run-structured masks of 15 %.
        dict(name="step-runs-T32", kind="step", H=1024, I=4096, L=18, T=32, B=1, density=0.15, runs=True, host=False),
        # The ordinary step for a caller whose activations are in (pinned) host memory: copies and wait included.
        dict(name="step-top25-host", kind="step", H=1024, I=4096, L=18, T=51, B=1, density=0.25, runs=False, host=True),
        # One step of the large expert with a top-20 % mask.
        dict(name="large-step-top20", kind="step", H=2048, I=16384, L=18, T=51, B=1, density=0.20, runs=False, host=False),
        # The large expert's dense step, which emits the activation records of the next masks.  The largest call.
        dict(name="large-dense-records", kind="dense", H=2048, I=16384, L=18, T=51),
        # Eight independent episodes served in one call, each with its own masks.
        dict(name="batch8-top25", kind="step", H=1024, I=4096, L=18, T=51, B=8, density=0.25, runs=False, host=False),
        # A step group of the anchor schedule: a dense anchor step, then four anchor-relative updates of the top half.
        dict(name="anchor-group-top50", kind="anchor", H=1024, I=4096, L=18, T=51, density=0.50, group=5),
        # Context Cache on one VLM layer: drift scores, the top quarter of the visual rows, their FFN and the scatter.
        dict(name="context-rho25", kind="context", H=2048, I=16384, P=768, S=48, density=0.25),
        # An expert of a width between the two configured ones.
        dict(name="width1536-top25", kind="step", H=1536, I=6144, L=12, T=51, B=1, density=0.25, runs=False, host=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["mask", "mask", "layer", "step", "step", "host", "large", "dense", "batch", "anchor", "context", "width"])
    density = round(math.exp(rng.uniform(math.log(0.06), math.log(0.6))), 3)
    T = rng.randint(4, 64)
    L = rng.randint(4, 18)
    if kind == "mask":
        rule = rng.choice(["vote", "topk", "group", "threshold", "bool"])
        W = 1 if rule in ("topk", "threshold", "bool") else rng.randint(2, 8)
        return dict(kind="mask", rule=rule, lists=_log_int(rng, 1, 64), I=_log_int(rng, 700, 16384), W=W, density=density)
    if kind == "layer":
        H = rng.choice([1024, 2048])
        return dict(kind="layer", H=H, I=rng.randint(2 * H, 4 * H), T=T, density=density)
    if kind in ("step", "host"):
        return dict(kind="step", H=1024, I=rng.randint(3000, 4096), L=L, T=T, B=1, density=density,
                    runs=rng.random() < 0.3, host=kind == "host")
    if kind == "large":
        return dict(kind="step", H=2048, I=rng.randint(8000, 16384), L=L, T=T, B=1, density=density,
                    runs=rng.random() < 0.3, host=False)
    if kind == "dense":
        H = rng.choice([1024, 2048])
        return dict(kind="dense", H=H, I=rng.randint(3 * H, 8 * H) if H == 2048 else rng.randint(3000, 4096), L=L, T=T)
    if kind == "batch":
        return dict(kind="step", H=1024, I=rng.randint(3000, 4096), L=L, T=T, B=rng.randint(2, 12), density=density,
                    runs=False, host=False)
    if kind == "anchor":
        return dict(kind="anchor", H=1024, I=rng.randint(3000, 4096), L=L, T=T, density=density, group=rng.randint(2, 5))
    if kind == "context":
        H = rng.choice([1024, 2048])
        return dict(kind="context", H=H, I=128 * rng.randint(4 * H // 128, 8 * H // 128), P=rng.randint(128, 900),
                    S=rng.randint(4, 64), density=density)
    # an expert of another width (any multiple of 64), or a chunk of more than 64 tokens; as much work as the listed one
    H = 64 * rng.randint(6, 30)
    T = rng.randint(65, 100) if H == 1024 or rng.random() < 0.25 else T
    I = rng.randint(3 * H, 4 * H)
    most = 12 * 1536 * 1536 * 51
    L = max(1, min(12, int(most / (H * I * density * T))))
    return dict(kind="step", H=H, I=I, L=L, T=T, B=1, density=density, runs=False, host=False)


# ------------------------------------------------------------------------------------------------ inputs
def _keep(case):
    """K = ceil(density * I), the number of neurons (rows) a ranking rule keeps."""
    n = case["P"] if case["kind"] == "context" else case["I"]
    return int(min(n, max(1, math.ceil(case.get("density", 1.0) * n - 1e-9))))


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _weights(g, H, I, sigma):
    """(W_gate [I,H], W_up [I,H], W_down [H,I]) bf16."""
    return tuple((_normal(g, *shape) * sigma).bfloat16() for shape in ((I, H), (I, H), (H, I)))


def _sigma(H):
    return 0.64 / math.sqrt(H)                       # 0.02 at H = 1024, 0.014 at H = 2048


def _run_scale(g, lists, I):
    """[lists, I]: 4 inside runs of 8 to 64 neighbouring neurons, 1 between them."""
    mark = torch.nn.functional.interpolate(_normal(g, lists, 1, max(2, I // 36)), size=I, mode="nearest")[:, 0]
    return torch.where(mark > 1.0, 4.0, 1.0)


def _lists(ctx, g, case, n_lists):
    """Index lists as a reference execution leaves them: exact top-k of one record per list."""
    I, k = case["I"], _keep(case)
    rec = _normal(g, n_lists, I).abs()
    if case.get("runs"):
        rec = rec * _run_scale(g, n_lists, I)
    stride = (I + 3) // 4 * 4
    idx = torch.zeros(n_lists, stride, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(n_lists, dtype=torch.int32, device="cuda")
    ctx.rm_mask_compact([rec], rm.RM_SRC_SCORE_F32, rm.RM_REDUCE_TOPK, idx, cnt, stride, n_lists=n_lists, k=k)
    return idx, cnt, stride


def _expert(case, g, B=1):
    """A context and its packed layers."""
    H, I, L = case["H"], case["I"], case.get("L", 1)
    ctx = rm.Context(L, H, I, case["T"], B)
    layers = []
    for _ in range(L):
        layers.append(ctx.rm_pack_weights(*_weights(g, H, I, _sigma(H))))
    return ctx, layers


def _activations(g, *shape):
    """A residual stream as the model hands it over: fp32 holding bf16 values."""
    return _normal(g, *shape).bfloat16().float()


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return {"case": case, **_PREPARE[case["kind"]](case, g)}


def _prepare_mask(case, g):
    lists, I, W = case["lists"], case["I"], case["W"]
    ctx = rm.Context(1, 64, I, 1)
    base = _normal(g, lists, I).abs() * _run_scale(g, lists, I)
    # the W records of a window are similar executions of one another
    recs = [(base * (1.0 + 0.1 * _normal(g, lists, I))).abs().contiguous() for _ in range(W)]
    threshold = 0.0
    if case["rule"] == "bool":
        recs = [(torch.rand(lists, I, generator=g, device="cuda") < case["density"]).to(torch.uint8) for _ in range(W)]
    elif case["rule"] == "threshold":
        threshold = float(recs[0].flatten().sort(descending=True).values[int(case["density"] * lists * I)])
    stride = (I + 3) // 4 * 4
    return dict(ctx=ctx, recs=recs, threshold=threshold, stride=stride,
                idx=torch.zeros(lists, stride, dtype=torch.int32, device="cuda"),
                cnt=torch.zeros(lists, dtype=torch.int32, device="cuda"))


def _prepare_layer(case, g):
    H, I, T = case["H"], case["I"], case["T"]
    ctx, layers = _expert(case, g)
    mask = (torch.rand(1, I, generator=g, device="cuda") < case["density"]).to(torch.uint8)
    stride = (I + 3) // 4 * 4
    idx = torch.zeros(stride, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    ctx.rm_mask_compact([mask], rm.RM_SRC_BOOL_U8, rm.RM_REDUCE_NONE, idx, cnt, stride, n_lists=1)
    ctx.rm_set_option("count_hint", _keep(case))
    return dict(ctx=ctx, layer=layers[0], idx=idx, cnt=cnt, x=_normal(g, T, H).bfloat16(), r=_activations(g, T, H),
                y=torch.zeros(T, H, device="cuda"))


def _prepare_step(case, g):
    H, L, T, B = case["H"], case["L"], case["T"], case["B"]
    ctx, layers = _expert(case, g, B)
    idx, cnt, stride = _lists(ctx, g, case, B * L)
    r, out = _activations(g, B, T, H), torch.zeros(B, T, H, device="cuda")
    if case["host"]:
        r, out = r.cpu().pin_memory(), out.cpu().pin_memory()
    return dict(ctx=ctx, layers=layers, idx=idx, cnt=cnt, stride=stride, r=r, out=out)


def _prepare_dense(case, g):
    H, I, L, T = case["H"], case["I"], case["L"], case["T"]
    ctx, layers = _expert(case, g)
    return dict(ctx=ctx, layers=layers, r=_activations(g, 1, T, H), out=torch.zeros(1, T, H, device="cuda"),
                rec=torch.zeros(1, L, I, device="cuda"))


def _prepare_anchor(case, g):
    H, I, L, T, n = case["H"], case["I"], case["L"], case["T"], case["group"]
    ctx, layers = _expert(case, g)
    idx, cnt, stride = _lists(ctx, g, case, L)
    hs = (T + 3) // 4 * 4
    x0, d = _normal(g, 1, T, H), _normal(g, 1, T, H)
    theta = math.acos(0.9) / 9.0                     # neighbouring denoising steps differ little
    return dict(ctx=ctx, layers=layers, idx=idx, cnt=cnt, stride=stride, h_stride=hs,
                r=[(math.cos(theta * s) * x0 + math.sin(theta * s) * d).bfloat16().float() for s in range(n)],
                gate=[1.0 + 0.25 * _normal(g, L, 1, H) for _ in range(n)],
                out=[torch.zeros(1, T, H, device="cuda") for _ in range(n)],
                ya=torch.zeros(L, 1, T, H, device="cuda"), ha=torch.zeros(L, 1, I, hs, device="cuda"))


def _prepare_context(case, g):
    H, I, P, S = case["H"], case["I"], case["P"], case["S"]
    ctx = rm.Context(1, H, I, 64)
    w = _weights(g, H, I, _sigma(H))
    ref = _normal(g, P + S, H)
    x = ref.clone()
    # most patches barely change between executions, a few change a lot
    x[:P] += 0.05 * torch.exp(1.2 * _normal(g, P, 1)) * _normal(g, P, H)
    k = _keep(case)
    return dict(ctx=ctx, w=w, x=x.bfloat16(), ref=ref[:P].bfloat16().contiguous(), y_ref=0.5 * _normal(g, P, H), k=k,
                R=min(1024, k + S), score=torch.zeros(P, device="cuda"),
                rows=torch.zeros((P + 3) // 4 * 4, dtype=torch.int32, device="cuda"),
                cnt=torch.zeros(1, dtype=torch.int32, device="cuda"), y=torch.zeros(P + S, H, device="cuda"))


_PREPARE = dict(mask=_prepare_mask, layer=_prepare_layer, step=_prepare_step, dense=_prepare_dense, anchor=_prepare_anchor,
                context=_prepare_context)


# ------------------------------------------------------------------------------------------------ one pass
def run(state):
    return _RUN[state["case"]["kind"]](state["case"], state)


def _run_mask(case, s):
    kind, reduce = {"vote": (rm.RM_SRC_SCORE_F32, rm.RM_REDUCE_TOPK), "topk": (rm.RM_SRC_SCORE_F32, rm.RM_REDUCE_TOPK),
                    "group": (rm.RM_SRC_SCORE_F32, rm.RM_REDUCE_GROUP),
                    "threshold": (rm.RM_SRC_SCORE_F32, rm.RM_REDUCE_THRESHOLD),
                    "bool": (rm.RM_SRC_BOOL_U8, rm.RM_REDUCE_NONE)}[case["rule"]]
    s["ctx"].rm_mask_compact(s["recs"], kind, reduce, s["idx"], s["cnt"], s["stride"], n_lists=case["lists"],
                             threshold=s["threshold"], k=_keep(case), min_votes=max(1, case["W"] * 3 // 4))
    return s["idx"], s["cnt"]


def _run_layer(case, s):
    return s["ctx"].rm_sparse_mlp(s["layer"], s["x"], s["r"], s["idx"], s["cnt"], s["y"])


def _run_step(case, s):
    call = s["ctx"].rm_action_expert_step_host if case["host"] else s["ctx"].rm_action_expert_step
    return call(s["layers"], s["r"], s["idx"], s["cnt"], s["stride"], s["out"], B=case["B"])


def _run_dense(case, s):
    s["ctx"].rm_action_expert_step(s["layers"], s["r"], None, None, case["I"], s["out"], records_out=s["rec"])
    return s["out"], s["rec"]


def _run_anchor(case, s):
    for i in range(case["group"]):
        first = i == 0
        s["ctx"].rm_action_expert_step_ex(s["layers"], s["r"][i], None if first else s["idx"], None if first else s["cnt"],
                                          s["stride"], s["out"][i], rm.RM_ANCHOR_WRITE if first else rm.RM_ANCHOR_UPDATE,
                                          s["ya"], s["ha"], s["h_stride"], out_gate=s["gate"][i])
    return s["out"], s["ya"], s["ha"]


def _run_context(case, s):
    ctx, P, S = s["ctx"], case["P"], case["S"]
    ctx.rm_context_drift(s["x"], s["ref"], P, s["score"])
    ctx.rm_mask_compact([s["score"]], rm.RM_SRC_SCORE_F32, rm.RM_REDUCE_TOPK, s["rows"], s["cnt"], s["rows"].numel(),
                        n_lists=1, k=s["k"], I=P)
    ctx.rm_context_ffn(*s["w"], s["x"], s["rows"], s["cnt"], P, S, s["R"], s["y_ref"], s["y"])
    return s["y"], s["score"], s["rows"], s["cnt"]


_RUN = dict(mask=_run_mask, layer=_run_layer, step=_run_step, dense=_run_dense, anchor=_run_anchor, context=_run_context)


# ------------------------------------------------------------------------------------------------ accounting
def work(case):
    kind = case["kind"]
    if kind == "mask":
        n = case["lists"] * case["I"]
        item = 1 if case["rule"] == "bool" else 4
        return {"bytes": n * case["W"] * item + 4 * case["lists"] * _keep(case), "flops": 0}
    H, I, K = case["H"], case["I"], _keep(case)
    if kind == "context":
        R, P, S = K + case["S"], case["P"], case["S"]
        return {"bytes": 6 * H * I + 2 * (2 * P + S) * H + 4 * (2 * P - K + S) * H, "flops": 6 * R * H * I}
    T, L, B = case["T"], case.get("L", 1), case.get("B", 1)
    if kind == "layer":
        return {"bytes": 6 * H * K + 4 * K + 2 * T * H + 8 * T * H, "flops": 6 * T * H * K}
    if kind == "dense":
        return {"bytes": L * (6 * H * I + 4 * I) + 8 * T * H, "flops": 6 * L * T * H * I}
    if kind == "anchor":
        n = case["group"] - 1
        anchor = 6 * H * I + 4 * I * T + 4 * T * H + 4 * H
        update = 6 * H * K + 4 * K + 4 * K * T + 4 * T * H + 4 * H
        return {"bytes": L * (anchor + n * update) + 8 * (n + 1) * T * H, "flops": 6 * L * T * H * (I + n * K)}
    union = I * (1.0 - (1.0 - K / I) ** B)           # neurons that at least one episode selects: read once
    return {"bytes": int(L * (6 * H * union + 4 * B * K)) + 8 * B * T * H, "flops": 6 * L * B * T * H * K}


def tolerance(case):
    kind = case["kind"]
    if kind == "mask":
        return "exact"
    if kind == "layer":
        return {"rel": 1e-4}                         # bf16 inputs taken as they are, fp32 sums, hidden values to 17 bits
    if kind == "context":
        return {"rel": 3e-3}                         # hidden activations rounded to bf16 between the two products
    # every layer rounds its normalised input to bf16: a last-bit difference of a sum moves single roundings, and the
    # following layers carry them on
    return {"rel": 5e-3}
