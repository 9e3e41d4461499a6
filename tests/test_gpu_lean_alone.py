"""The lean layer kernel: lists of one tile, up to a cluster's one tile and more, and chunks of more than 52 tokens, where it is built for
one CTA per SM."""
import pytest

from test_gpu_edges import step_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("I,T,L,B,density", [
    (256, 1, 3, 1, 0.05), (512, 32, 3, 1, 0.8), (512, 33, 3, 1, 0.875), (512, 51, 4, 1, 1.0), (300, 52, 2, 2, 0.3),
    (512, 53, 3, 1, 1.0), (960, 60, 3, 1, 1.0), (1100, 64, 2, 1, 0.9), (256, 61, 2, 3, 0.5)])
def test_lean_kernel_alone_on_its_sm_matches_the_oracle(lib, I, T, L, B, density):
    step_case(lib, H=1024, I=I, T=T, L=L, B=B, density=density, variant=1, max_clusters=0, config=98)


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
