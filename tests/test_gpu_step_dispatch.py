"""Which kernels a single-episode step takes follows its width, chunk length and list length; at the borders both sides agree."""
import pytest

from harness import REL_L2_TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,T,eq4,layers_up_to,stream_from", [
    (1024, 32, False, 29, None), (1024, 48, False, 16, None), (1024, 51, False, 15, None), (1024, 64, False, 8, None),
    (1024, 32, True, 32, None), (1024, 33, True, 20, None), (1024, 64, True, 13, None),
    (2048, 55, False, 15, 101), (2048, 56, False, 13, 101), (2048, 32, False, 15, 77), (2048, 64, True, 15, None),
])
def test_borders(lib, H, T, eq4, layers_up_to, stream_from):
    import torch
    L, I = 2, 2304 if stream_from is None else 6656
    g = torch.Generator(device="cuda").manual_seed(H + T)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    ctx = lib.Context(L, H, I, T)
    layers = [ctx.rm_pack_weights(*[(0.64 / H ** 0.5 * rnd(*s)).bfloat16() for s in ((I, H), (I, H), (H, I))]) for _ in range(L)]
    r, gate = rnd(1, T, H).bfloat16().float(), 1.0 + 0.25 * rnd(L, 1, H)
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    borders = [(layers_up_to, False), (layers_up_to + 1, True)]
    if stream_from:
        borders += [(stream_from - 1, True), (stream_from, sm < stream_from)]
    for tiles, whole_step in borders:
        K = 64 * tiles
        rec = torch.rand(L, I, generator=g, device="cuda")
        idx, cnt = torch.zeros(L, I, dtype=torch.int32, device="cuda"), torch.zeros(L, dtype=torch.int32, device="cuda")
        ctx.rm_mask_compact([rec], lib.RM_SRC_SCORE_F32, lib.RM_REDUCE_TOPK, idx, cnt, I, n_lists=L, k=K)
        outs = []
        for variant in (0, 1 if whole_step else 5):
            ctx.rm_set_option("variant", variant)
            for out in (torch.empty_like(r), r.clone()):           # into another buffer, in place
                src = r if out.data_ptr() != r.data_ptr() and not outs else out.copy_(r)
                if eq4:
                    ctx.rm_action_expert_step_ex(layers, src, idx, cnt, I, out, lib.RM_ANCHOR_NONE, None, None, 0, out_gate=gate)
                else:
                    ctx.rm_action_expert_step(layers, src, idx, cnt, I, out)
                if variant == 0:
                    assert (ctx.rm_get_info("last_variant") == 5) == whole_step, (tiles, ctx.rm_get_info("last_variant"))
                outs.append(out)
        for out in outs[1:]:
            # (the kernels add in different orders, then round every layer's input to bf16)
            assert torch.isfinite(out).all() and float((out - outs[0]).norm() / outs[0].norm()) <= REL_L2_TOL, tiles
    assert ctx.rm_device_status() == 0
    ctx.close()


@pytest.mark.parametrize("H", [1024, 2048])
def test_borders_of_dense_steps(lib, H):
    """One tile of 256 neurons per cluster of the whole-step kernel: up to there that kernel, from the next neuron the sweep kernel."""
    import torch
    L, T = 2, 51
    g = torch.Generator(device="cuda").manual_seed(H)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    clusters = lib.Context(L, H, 64, T).rm_get_info("persist_clusters")
    for I in (256 * clusters, 256 * clusters + 1):
        ctx = lib.Context(L, H, I, T)
        layers = [ctx.rm_pack_weights(*[(0.64 / H ** 0.5 * rnd(*s)).bfloat16() for s in ((I, H), (I, H), (H, I))]) for _ in range(L)]
        r, outs, recs = rnd(1, T, H).bfloat16().float(), [], []
        for variant in (0, 7 if I == 256 * clusters else 5):
            ctx.rm_set_option("variant", variant)
            out, rec = torch.empty_like(r), torch.zeros(1, L, I, device="cuda")
            ctx.rm_action_expert_step(layers, r, None, None, I, out, records_out=rec)
            if variant == 0:
                assert ctx.rm_get_info("last_variant") == (5 if I == 256 * clusters else 7)
            outs.append(out)
            recs.append(rec)
        for a, b in (outs, recs):
            assert torch.isfinite(b).all() and float((a - b).norm() / b.norm()) <= REL_L2_TOL, I
        assert ctx.rm_device_status() == 0
        ctx.close()


@pytest.mark.parametrize("H,T,mode,stream_from", [
    (1024, 20, "none", 33), (1024, 51, "none", 33), (1024, 60, "none", 17), (2048, 20, "none", 31), (2048, 60, "none", 31),
    (1024, 32, "write", 41), (1024, 33, "write", 57), (1024, 53, "write", 33), (2048, 52, "write", 31), (2048, 53, "write", 53),
    (1024, 20, "update", 33), (1024, 60, "update", 33), (2048, 32, "update", 64), (2048, 33, "update", 31),
])
def test_borders_of_batches(lib, H, T, mode, stream_from):
    """B episodes whose lists make one tile less than the streaming kernel takes, and as many: both kernels agree."""
    import torch
    L, I = 2, 4096
    g = torch.Generator(device="cuda").manual_seed(H + T)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    for tiles in (stream_from - 1, stream_from):
        B = next(b for b in range(2, 65) if tiles % b == 0)
        K = tiles // B * 64
        ctx = lib.Context(L, H, I, T, B)
        layers = [ctx.rm_pack_weights(*[(0.64 / H ** 0.5 * rnd(*s)).bfloat16() for s in ((I, H), (I, H), (H, I))]) for _ in range(L)]
        r, gate = rnd(B, T, H).bfloat16().float(), 1.0 + 0.25 * rnd(L, B, H)
        idx, cnt = torch.zeros(B * L, I, dtype=torch.int32, device="cuda"), torch.zeros(B * L, dtype=torch.int32, device="cuda")
        ctx.rm_mask_compact([rnd(B * L, I).abs()], lib.RM_SRC_SCORE_F32, lib.RM_REDUCE_TOPK, idx, cnt, I, n_lists=B * L, k=K)
        hs = (T + 3) // 4 * 4
        ya0, ha0 = rnd(L, B, T, H), rnd(L, B, I, hs)
        outs = []
        for variant in (0, 1 if tiles == stream_from else 4):
            ctx.rm_set_option("variant", variant)
            out, ya, ha = torch.empty_like(r), ya0.clone(), ha0.clone()
            if mode == "none":
                ctx.rm_action_expert_step(layers, r, idx, cnt, I, out, B=B)
            else:
                ctx.rm_action_expert_step_ex(layers, r, idx, cnt, I, out, lib.RM_ANCHOR_WRITE if mode == "write" else lib.RM_ANCHOR_UPDATE, ya, ha, hs,
                                             out_gate=gate, B=B)
            if variant == 0:
                assert (ctx.rm_get_info("last_variant") == 4) == (tiles == stream_from), (tiles, ctx.rm_get_info("last_variant"))
            outs.append((out, ya))
        for a, b in zip(*outs):
            assert torch.isfinite(a).all() and float((a - b).norm() / b.norm()) <= REL_L2_TOL, tiles
        assert ctx.rm_device_status() == 0
        ctx.close()
