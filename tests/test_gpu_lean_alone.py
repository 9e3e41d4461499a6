"""The lean layer kernel: lists of one tile, up to a cluster's one tile and more, and chunks of more than 52 tokens, where it is built for
one CTA per SM."""
import pytest

from test_gpu_edges import step_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,I,T,L,B,density,hint", [
    (1024, 256, 1, 3, 1, 0.05, 64), (1024, 512, 32, 3, 1, 0.8, 448), (1024, 512, 33, 3, 1, 0.875, 512), (1024, 512, 51, 4, 1, 1.0, 512),
    (1024, 300, 52, 2, 2, 0.3, 128), (1024, 512, 53, 3, 1, 1.0, 512), (1024, 960, 60, 3, 1, 1.0, 960), (1024, 1100, 64, 2, 1, 0.9, None),
    (1024, 256, 61, 2, 3, 0.5, 192), (2048, 700, 20, 2, 1, 0.9, 704), (2048, 420, 52, 2, 2, 0.8, 384), (2048, 960, 64, 2, 1, 1.0, 960)])
def test_lists_of_one_tile_to_a_cluster_match_the_oracle(lib, H, I, T, L, B, density, hint):
    """The hint is a bound of the lists here, so that every cluster has one tile: the build whose staged sums lie in the weight stage up to
    52 tokens and at 2048 columns, the one for one CTA per SM above."""
    step_case(lib, H=H, I=I, T=T, L=L, B=B, density=density, variant=1, hint=hint, config=98)


@pytest.mark.parametrize("H,I,T,B,density,hint", [
    (1024, 1600, 20, 1, 0.9, 600), (1024, 1600, 32, 2, 0.7, 512), (1024, 2200, 51, 1, 0.95, 1000), (1024, 1200, 52, 2, 0.9, 512),
    (1024, 900, 33, 3, 0.8, 320), (2048, 1500, 32, 1, 0.9, 64), (2048, 1500, 51, 2, 0.7, 400), (2048, 1900, 64, 1, 0.9, 960),
    (2048, 700, 52, 3, 0.9, 128)])
def test_lists_longer_than_the_hint_refill_the_stage_behind_the_sums(lib, H, I, T, B, density, hint):
    """The hint says one tile to a cluster, the lists make it two to many, with changes of the episode inside a run."""
    step_case(lib, H=H, I=I, T=T, L=2, B=B, density=density, variant=1, hint=hint, config=99)


@pytest.mark.parametrize("H,T,k,hint", [(1024, 20, 600, 600), (1024, 51, 600, 600), (1024, 51, 1500, 600), (1024, 60, 600, 600), (2048, 20, 700, 700),
                                        (2048, 51, 900, 900), (2048, 51, 1500, 640)])
def test_anchor_steps_of_one_tile_to_a_cluster(lib, H, T, k, hint):
    """An anchor step over the lists and an update with gate, against the CUDA-core kernels."""
    import torch
    from harness import REL_L2_TOL
    I, L, hs = 2048, 2, (T + 3) // 4 * 4
    g = torch.Generator(device="cuda").manual_seed(H + T + k)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    ctx = lib.Context(L, H, I, T)
    layers = [ctx.rm_pack_weights(*[(0.64 / H ** 0.5 * rnd(*s)).bfloat16() for s in ((I, H), (I, H), (H, I))]) for _ in range(L)]
    idx, cnt = torch.zeros(L, I, dtype=torch.int32, device="cuda"), torch.zeros(L, dtype=torch.int32, device="cuda")
    ctx.rm_mask_compact([rnd(L, I).abs()], lib.RM_SRC_SCORE_F32, lib.RM_REDUCE_TOPK, idx, cnt, I, n_lists=L, k=k)
    ctx.rm_set_option("count_hint", hint)
    r, gate = [rnd(1, T, H).bfloat16().float() for _ in range(2)], 1.0 + 0.25 * rnd(L, 1, H)
    got = {}
    for path in (1, 0):
        ctx.rm_set_option("path", path)
        ctx.rm_set_option("variant", 1 - path)
        ya, ha, outs = torch.zeros(L, 1, T, H, device="cuda"), torch.zeros(L, 1, I, hs, device="cuda"), []
        for mode, x in zip((lib.RM_ANCHOR_WRITE, lib.RM_ANCHOR_UPDATE), r):
            outs.append(ctx.rm_action_expert_step_ex(layers, x, idx, cnt, I, torch.empty_like(x), mode, ya, ha, hs, out_gate=gate))
            assert ctx.rm_get_info("last_variant") == 1 - path
        got[path] = (*outs, ya, ha)
    for a, b in zip(got[0], got[1]):
        # (the order of the sums differs, and every layer's input is rounded to bf16)
        assert torch.isfinite(a).all() and float((a - b).norm() / b.norm()) <= REL_L2_TOL
    assert ctx.rm_device_status() == 0
    ctx.close()


@pytest.mark.parametrize("T,k", [(20, 448), (51, 448), (51, 449), (53, 960), (64, 961)])
def test_repeated_layers_and_steps_agree_across_kernels(lib, T, k):
    """A stack of three layers 30 times, and one layer alone, against the two-tile kernel on the same lists."""
    import torch
    from harness import REL_L2_TOL
    H, I, L = 1024, 1024, 3
    g = torch.Generator(device="cuda").manual_seed(T + k)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    ctx = lib.Context(L, H, I, T)
    layers = [ctx.rm_pack_weights(*[(0.02 * rnd(*s)).bfloat16() for s in ((I, H), (I, H), (H, I))]) for _ in range(L)]
    idx, cnt = torch.zeros(L, I, dtype=torch.int32, device="cuda"), torch.zeros(L, dtype=torch.int32, device="cuda")
    ctx.rm_mask_compact([rnd(L, I).abs()], lib.RM_SRC_SCORE_F32, lib.RM_REDUCE_TOPK, idx, cnt, I, n_lists=L, k=k)
    r, out, x = rnd(1, T, H).bfloat16().float(), torch.empty(1, T, H, device="cuda"), rnd(T, H).bfloat16()
    got = {}
    for variant in (2, 1):
        ctx.rm_set_option("variant", variant)
        for i in range(30 if variant == 1 else 1):
            ctx.rm_action_expert_step(layers, r, idx, cnt, I, out)
            y = ctx.rm_sparse_mlp(layers[0], x, r[0], idx[0], cnt[:1], torch.empty(T, H, device="cuda"))
            got.setdefault(variant, (out.clone(), y))
            for a, b in zip((out, y), got[2]):
                # (the order of the sums differs, and every layer's input is rounded to bf16)
                assert torch.isfinite(a).all() and float((a - b).norm() / b.norm()) <= REL_L2_TOL, (variant, i)
    assert ctx.rm_device_status() == 0
    ctx.close()
