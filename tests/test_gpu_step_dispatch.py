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
