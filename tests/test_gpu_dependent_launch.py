"""Kernels of consecutive calls overlap at their edges (programmatic dependent launch).  A chain of mask rebuilds and masked passes,
each reading what the call in front wrote (list, count, activations) into buffers that are reused, has to give what the same
chain gives with the device idle between the calls."""
import pytest

from harness import REL_L2_TOL

pytestmark = pytest.mark.gpu

ROUNDS = 12


@pytest.mark.parametrize("H,I,L,T,B,in_place", [
    (1024, 2048, 3, 51, 1, False),        # whole-step kernel
    (1024, 2048, 3, 20, 1, True),         # layer kernels, the last buffer copied back
    (1024, 2048, 3, 20, 4, False),        # layer kernels, two cleared buffers
    (1024, 2048, 1, 32, 1, False),        # one layer
    (1024, 4096, 2, 51, 8, False),        # streaming kernel
    (2048, 4096, 2, 40, 1, True),
    (768, 2048, 2, 51, 1, False),         # slice kernel
])
def test_chain_without_host_waits(lib, H, I, L, T, B, in_place):
    import torch
    g = torch.Generator(device="cuda").manual_seed(H + I + L + T + B)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    ctx = lib.Context(L, H, I, T, B)
    layers = [ctx.rm_pack_weights(*[(0.64 / H ** 0.5 * rnd(*s)).bfloat16() for s in ((I, H), (I, H), (H, I))]) for _ in range(L)]
    recs = [rnd(B * L, I).abs() for _ in range(3)]
    ks = (I // 16, I // 3, I // 8)
    r0 = [rnd(B, T, H).bfloat16().float() for _ in range(3)]
    x = [rnd(T, H).bfloat16() for _ in range(3)]

    def chain(wait):
        idx = torch.zeros(B * L, I, dtype=torch.int32, device="cuda")
        cnt = torch.zeros(B * L, dtype=torch.int32, device="cuda")
        r, out, y = torch.empty_like(r0[0]), torch.empty_like(r0[0]), torch.empty(T, H, device="cuda")
        keep = []
        sync = torch.cuda.synchronize if wait else (lambda: None)
        torch.cuda.synchronize()
        for i in range(ROUNDS):
            ctx.rm_mask_compact([recs[i % 3]], lib.RM_SRC_SCORE_F32, lib.RM_REDUCE_TOPK, idx, cnt, I, n_lists=B * L, k=ks[i % 3])
            sync()
            # written by another library's kernel.  Every round has its own input: fed back through 12 rounds of L layers, last-bit
            # differences grow at every rounding to bf16 (0.8 % after 21 layers) and nothing could be told from them
            r.copy_(r0[i % 3])
            sync()
            ctx.rm_action_expert_step(layers, r, idx, cnt, I, r if in_place else out, B=B)
            sync()
            keep.append((r if in_place else out).clone())
            ctx.rm_mask_compact([recs[(i + 1) % 3]], lib.RM_SRC_SCORE_F32, lib.RM_REDUCE_TOPK, idx, cnt, I, n_lists=B * L, k=ks[(i + 1) % 3])
            sync()
            ctx.rm_sparse_mlp(layers[0], x[i % 3], y if i % 2 else r0[0][0], idx, cnt, y)
            sync()
            keep.append(y.clone())
            if i % 2 == 0:
                y.mul_(0.5)
        torch.cuda.synchronize()
        assert ctx.rm_device_status() == 0
        return keep

    want, got = chain(True), chain(False)
    for i, (a, b) in enumerate(zip(got, want)):
        assert torch.isfinite(a).all()
        # the order of the adds differs between runs; every layer (3 of a step, 2 of y in place) then rounds its input to bf16, which
        # the step bound covers for 18
        assert float((a - b).norm() / b.norm()) <= REL_L2_TOL, f"output {i}"
    ctx.close()


def both_ways(body):
    """What body(sync) returns with the device idle between the calls and without any wait: every output within the step bound."""
    import torch
    outs = []
    for sync in (torch.cuda.synchronize, lambda: None):
        torch.cuda.synchronize()
        outs.append(body(sync))
        torch.cuda.synchronize()
    for i, (want, got) in enumerate(zip(*outs)):
        assert torch.isfinite(got).all() and float((got - want).norm() / want.norm()) <= REL_L2_TOL, f"output {i}"


def weights(g, H, I, n):
    import torch
    return [[(0.64 / H ** 0.5 * torch.randn(*s, generator=g, device="cuda")).bfloat16() for s in ((I, H), (I, H), (H, I))] for _ in range(n)]


@pytest.mark.parametrize("H,I,T,L,variant", [(1024, 4096, 51, 1, 0), (2048, 4096, 20, 2, 0), (1024, 4096, 51, 1, 5), (1024, 4096, 51, 1, 4), (1024, 1000, 51, 1, 1)])
@pytest.mark.parametrize("front", ["pack", "copy", "drift"])
def test_dense_steps_behind_the_kernel_that_writes_their_weights(lib, H, I, T, L, variant, front):
    """Layer 0 is written by the kernel in front of the step, or by the one in front of that (a drift kernel, which lets the step in
    before it has waited itself)."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(H + T)
    ctx = lib.Context(L, H, I, T)
    ctx.rm_set_option("variant", variant)
    sets = weights(g, H, I, 3 + L - 1)
    ready = [ctx.rm_pack_weights(*w) for w in sets]
    layer0 = torch.empty_like(ready[0])
    layers = [layer0] + ready[3:]
    r = torch.randn(1, T, H, generator=g, device="cuda").bfloat16().float()
    out, rec, score = torch.empty_like(r), torch.zeros(1, L, I, device="cuda"), torch.zeros(8, device="cuda")
    small = torch.randn(8, H, generator=g, device="cuda").bfloat16()

    def body(sync):
        keep = []
        for i in range(ROUNDS):
            if front == "pack":
                ctx.rm_pack_weights(*sets[i % 3], packed_out=layer0)
            else:
                layer0.copy_(ready[i % 3])
            sync()
            if front == "drift":
                ctx.rm_context_drift(small, small, 8, score)
                sync()
            ctx.rm_action_expert_step(layers, r, None, None, I, out, records_out=rec)
            sync()
            keep += [out.clone(), rec.clone()]
        return keep

    both_ways(body)
    assert ctx.rm_get_info("last_variant") == (variant or 7) and ctx.rm_device_status() == 0
    ctx.close()


@pytest.mark.parametrize("H,I,T,host", [(1024, 4096, 51, False), (2048, 4096, 20, False), (1024, 2048, 51, True)])
def test_chain_of_the_anchor_schedule_and_of_host_steps(lib, H, I, T, host):
    """A group: anchor step, a mask of its records, updates with it.  With activations on the device, or host to host."""
    import torch
    L, hs = 3, (T + 3) // 4 * 4
    g = torch.Generator(device="cuda").manual_seed(H + I)
    ctx = lib.Context(L, H, I, T)
    layers = [ctx.rm_pack_weights(*w) for w in weights(g, H, I, L)]
    rs = [torch.randn(1, T, H, generator=g, device="cuda").bfloat16().float() for _ in range(3)]
    gate = 1.0 + 0.25 * torch.randn(L, 1, H, generator=g, device="cuda")
    pinned = [r.cpu().pin_memory() for r in rs]
    host_out = torch.empty(1, T, H).pin_memory()

    def body(sync):
        ya, ha, rec = torch.zeros(L, 1, T, H, device="cuda"), torch.zeros(L, 1, I, hs, device="cuda"), torch.zeros(1, L, I, device="cuda")
        idx, cnt = torch.zeros(L, I, dtype=torch.int32, device="cuda"), torch.zeros(L, dtype=torch.int32, device="cuda")
        out, keep = torch.empty_like(rs[0]), []
        for i in range(ROUNDS):
            ctx.rm_action_expert_step_ex(layers, rs[i % 3], None, None, I, out, lib.RM_ANCHOR_WRITE, ya, ha, hs, out_gate=gate, records_out=rec)
            sync()
            keep += [out.clone(), ya.clone()]
            # (the mask comes from other records than the step's: their last bits could move a tie)
            ctx.rm_mask_compact([ha[:, 0, :, :T].abs().sum(-1).bfloat16().float()], lib.RM_SRC_SCORE_F32, lib.RM_REDUCE_THRESHOLD, idx, cnt, I,
                                n_lists=L, threshold=-1.0)
            sync()
            if host:
                keep.append(ctx.rm_action_expert_step_host(layers, pinned[(i + 1) % 3], idx, cnt, I, host_out).clone())
            else:
                ctx.rm_action_expert_step_ex(layers, rs[(i + 1) % 3], idx, cnt, I, out, lib.RM_ANCHOR_UPDATE, ya, ha, hs, out_gate=gate)
                sync()
                keep.append(out.clone())
        return keep

    both_ways(body)
    assert ctx.rm_device_status() == 0
    ctx.close()


@pytest.mark.parametrize("H,I,P,S,R", [(1024, 2048, 300, 16, 96), (2048, 4096, 700, 40, 400)])
@pytest.mark.parametrize("with_drift", [True, False])
def test_context_cache_behind_the_kernels_that_write_its_weights(lib, H, I, P, S, R, with_drift):
    import torch
    g = torch.Generator(device="cuda").manual_seed(H + P)
    ctx = lib.Context(1, H, I, 64)
    sets = weights(g, H, I, 3)
    w = [torch.empty_like(t) for t in sets[0]]
    xs = [torch.randn(P + S, H, generator=g, device="cuda").bfloat16() for _ in range(3)]
    ref, y_ref = torch.randn(P, H, generator=g, device="cuda").bfloat16(), torch.randn(P, H, generator=g, device="cuda")
    fixed = torch.arange(0, 2 * (R - S), 2, dtype=torch.int32, device="cuda")[:R - S].clamp(max=P - 1)
    fixed = torch.unique(fixed).int()
    n_fixed = torch.tensor([fixed.numel()], dtype=torch.int32, device="cuda")

    def body(sync):
        x, score = torch.empty_like(xs[0]), torch.zeros(P, device="cuda")
        rows, cnt = torch.zeros((P + 3) // 4 * 4, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        y, keep = torch.empty(P + S, H, device="cuda"), []
        for i in range(ROUNDS):
            x.copy_(xs[i % 3])
            for t, new in zip(w, sets[(i + 1) % 3]):
                t.copy_(new)
            sync()
            if with_drift:
                ctx.rm_context_drift(x, ref, P, score)
                sync()
                ctx.rm_mask_compact([score], lib.RM_SRC_SCORE_F32, lib.RM_REDUCE_TOPK, rows, cnt, rows.numel(), n_lists=1, k=R - S, I=P)
                sync()
            ctx.rm_context_ffn(*w, x, rows if with_drift else fixed, cnt if with_drift else n_fixed, P, S, R, y_ref, y)
            sync()
            keep.append(y.clone())
        return keep

    both_ways(body)
    assert ctx.rm_device_status() == 0
    ctx.close()


def captured_edges(calls):
    """(programmatic, other) dependency edges of the calls, captured into a graph that is not run."""
    import ctypes

    import torch
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        calls()
    get = ctypes.CDLL("libcuda.so.1").cuGraphGetEdges_v2
    h, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert get(h, None, None, None, ctypes.byref(n)) == 0
    ends, data = [(ctypes.c_void_p * n.value)() for _ in range(2)], (ctypes.c_ubyte * 8 * n.value)()
    assert get(h, ends[0], ends[1], data, ctypes.byref(n)) == 0
    programmatic = sum(d[2] == 1 for d in data)                      # CUgraphEdgeData: from_port, to_port, type, 5 reserved bytes
    return programmatic, n.value - programmatic


@pytest.mark.parametrize("H,T,B,variant", [(1024, 51, 1, 5), (1024, 51, 1, 7), (1024, 51, 1, 6), (768, 51, 1, 6), (1024, 20, 1, 1), (1024, 51, 4, 4), (2048, 51, 2, 4)])
def test_option_pdl_governs_every_launch(lib, H, T, B, variant):
    import torch
    L, I, P, S = 2, 2048, 96, 8
    g = torch.Generator(device="cuda").manual_seed(H + T + B)
    ctx = lib.Context(L, H, I, T, B)
    ctx.rm_set_option("variant", variant)
    w = weights(g, H, I, 1)[0]
    layers = [ctx.rm_pack_weights(*w) for _ in range(L)]
    r = torch.randn(B, T, H, generator=g, device="cuda").bfloat16().float()
    out, y = torch.empty_like(r), torch.empty(T, H, device="cuda")
    rec = torch.rand(B * L, I, generator=g, device="cuda")
    idx, cnt = torch.zeros(B * L, I, dtype=torch.int32, device="cuda"), torch.zeros(B * L, dtype=torch.int32, device="cuda")
    x, x_ref = torch.randn(P + S, H, generator=g, device="cuda").bfloat16(), torch.randn(P, H, generator=g, device="cuda").bfloat16()
    score, rows, n = torch.zeros(P, device="cuda"), torch.zeros(P, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    y_ref, y_ctx = torch.zeros(P, H, device="cuda"), torch.zeros(P + S, H, device="cuda")

    def calls():
        for _ in range(2):
            ctx.rm_mask_compact([rec], lib.RM_SRC_SCORE_F32, lib.RM_REDUCE_TOPK, idx, cnt, I, n_lists=B * L, k=I // 4)
            dense = variant == 7
            ctx.rm_action_expert_step(layers, r, None if dense else idx, None if dense else cnt, I, out, B=B)
            assert ctx.rm_get_info("last_variant") == variant
            ctx.rm_sparse_mlp(layers[0], x[:min(T, P)], None, idx, cnt, y)
            ctx.rm_context_drift(x, x_ref, P, score)
            ctx.rm_mask_compact([score], lib.RM_SRC_SCORE_F32, lib.RM_REDUCE_TOPK, rows, n, P, n_lists=1, k=P // 4, I=P)
            ctx.rm_context_ffn(*w, x, rows, n, P, S, 64, y_ref, y_ctx)

    calls()                                                          # (workspaces, kernel attributes)
    torch.cuda.synchronize()
    on = captured_edges(calls)
    ctx.rm_set_option("pdl", 0)
    off = captured_edges(calls)
    assert on[0] >= 10 and off[0] == 0 and off[1] > 0, (on, off)
    ctx.close()
