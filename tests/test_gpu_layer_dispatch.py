"""Which kernel the one-layer entry takes follows width, chunk length and list length; at the borders both sides agree."""
import numpy as np
import pytest

import oracle
from paper_2609_19104_b200 import workloads as wl
from harness import Model, assert_close, dev, dev_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,T,borders", [
    (1024, 60, [(15, 1), (16, 2), (30, 2), (31, 4)]), (2048, 16, [(15, 1), (16, 2), (59, 2), (60, 4)]),
    (2048, 32, [(45, 2), (46, 5), (59, 5), (60, 4)]), (2048, 33, [(30, 2), (31, 5), (59, 5), (60, 4)]),
    (2048, 52, [(15, 1), (16, 2), (30, 2)]), (2048, 53, [(15, 1), (16, 1), (30, 1), (31, 5)]), (2048, 61, [(30, 1), (31, 5)])])
def test_borders_of_one_layer(lib, H, T, borders):
    import torch
    I = 3968
    g = torch.Generator(device="cuda").manual_seed(H + T)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    ctx = lib.Context(1, H, I, T)
    layer = ctx.rm_pack_weights(*[(0.64 / H ** 0.5 * rnd(*s)).bfloat16() for s in ((I, H), (I, H), (H, I))])
    x, r = rnd(T, H).bfloat16(), rnd(T, H)
    for tiles, kernel in borders:
        idx, cnt = torch.zeros(I, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        ctx.rm_mask_compact([rnd(1, I).abs()], lib.RM_SRC_SCORE_F32, lib.RM_REDUCE_TOPK, idx, cnt, I, n_lists=1, k=64 * tiles - 5)
        outs = []
        other = 1 if kernel != 1 else 2 if H == 1024 or T <= 52 else 5          # (another kernel than the chosen one)
        for variant in (0, other, 0):
            ctx.rm_set_option("variant", variant)
            y = r.clone() if len(outs) == 2 else torch.empty_like(r)           # (the last one in place)
            outs.append(ctx.rm_sparse_mlp(layer, x, y if len(outs) == 2 else r, idx, cnt, y))
            last = ctx.rm_get_info("last_variant")
            assert last == kernel if variant == 0 else last != kernel, (tiles, variant, last)
        for out in outs:
            # (one layer on the same bf16 input: only the order of fp32 sums of hidden values to 17 bits differs)
            assert torch.isfinite(out).all() and float((out - outs[1]).norm() / (outs[1] - r).norm()) <= 1e-4, tiles
    assert ctx.rm_device_status() == 0
    ctx.close()


@pytest.mark.parametrize("H,T,tiles,unset", [(2048, 20, 40, 2), (2048, 40, 40, 5), (1024, 60, 20, 2), (1024, 40, 20, 1)])
def test_streaming_threshold_of_one_layer_is_the_option_when_it_is_set(lib, H, T, tiles, unset):
    """From 1 (everything) to the largest int (nothing), on one layer and on a step of one."""
    import torch
    I = 2624
    g = torch.Generator(device="cuda").manual_seed(H + T)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    ctx = lib.Context(1, H, I, T)
    layer = ctx.rm_pack_weights(*[(0.64 / H ** 0.5 * rnd(*s)).bfloat16() for s in ((I, H), (I, H), (H, I))])
    x, r = rnd(T, H).bfloat16(), rnd(T, H)
    idx, cnt = torch.zeros(1, I, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    ctx.rm_mask_compact([rnd(1, I).abs()], lib.RM_SRC_SCORE_F32, lib.RM_REDUCE_TOPK, idx, cnt, I, n_lists=1, k=64 * tiles - 5)
    want = None
    for value in (None, 1, tiles, 2 * tiles + 1, 2 ** 31 - 1):
        if value is not None:
            ctx.rm_set_option("stream_min_tiles", value)
        y = ctx.rm_sparse_mlp(layer, x, r, idx, cnt, torch.empty_like(r))
        kernel = ctx.rm_get_info("last_variant")
        assert kernel == unset if value is None else (kernel == 4) == (value <= tiles), (value, kernel)
        want = y if want is None else want
        # (fp32 sums in another order, hidden values to 17 bits)
        assert torch.isfinite(y).all() and float((y - want).norm() / (want - r).norm()) <= 1e-4, value
    ctx.rm_set_option("persist_max_batch", 0)
    ctx.rm_action_expert_step([layer], r.view(1, T, H), idx, cnt, I, torch.empty_like(r))
    assert ctx.rm_get_info("last_variant") != 4
    assert ctx.rm_device_status() == 0
    ctx.close()


@pytest.mark.parametrize("T,tiles,kernel", [(48, 33, 5), (48, 57, 5), (20, 57, 5), (64, 33, 5), (20, 36, 2), (52, 16, 2), (60, 30, 1)])
def test_one_wide_layer_against_the_oracle(lib, T, tiles, kernel):
    """2048 columns: dense with records, a list without a residual, a compact layer, and a list far longer than the hint."""
    import torch
    H, I = 2048, 64 * tiles - 5
    w = wl.Workload(97, "wide-layer", 1, H, I, T, 1.0 / np.sqrt(H), 1, 0.5)
    model = Model(lib, w)
    ctx, x, r = model.ctx, wl.step_input(w, 0), wl.residual_input(w)
    W = model.Wg[0], model.Wu[0], model.Wd[0]

    def call(idx, cnt, residual, **kw):
        y = torch.full((T, H), 7.0, device="cuda")
        return ctx.rm_sparse_mlp(kw.pop("layer", model.packed[0]), dev_bf16(x), None if residual is None else dev(residual), idx, cnt, y, **kw).cpu().numpy()

    rec, scale = torch.zeros(I, device="cuda"), (1.0 + np.arange(I) % 3).astype(np.float32)
    got = call(None, None, r, record_out=rec, record_scale=dev(scale))
    assert ctx.rm_get_info("last_variant") == kernel
    want, want_rec = oracle.dense_mlp(x, *W, r, scale=scale, return_record=True)
    assert_close(got, want, "dense")
    assert np.all(np.abs(rec.cpu().numpy() - want_rec) <= 2e-2 + 1e-2 * np.abs(want_rec))

    lists = [np.flatnonzero(wl.uniform(wl.tensor_key(13, 97, 0, 2, i), I) < d).astype(np.int32) for i, d in enumerate((0.95, 0.4))]
    for sel, hint in ((lists[0], I), (lists[1], I), (np.arange(I, dtype=np.int32), I // 4)):     # (the hint decides on the kernel)
        ctx.rm_set_option("count_hint", hint)
        idx, cnt = np.zeros((I + 3) // 4 * 4, np.int32), dev(np.array([sel.size], np.int32))
        idx[:sel.size] = sel
        got = call(dev(idx), cnt, None)
        assert hint < I or ctx.rm_get_info("last_variant") == kernel
        assert_close(got, oracle.masked_mlp(x, *W, None, sel), f"{sel.size} neurons, hint {hint}")
    ctx.rm_set_option("count_hint", I)
    sel = lists[0]
    idx[:sel.size], cnt = sel, dev(np.array([sel.size], np.int32))
    compact = torch.full((ctx.packed_layer_bytes() // 2,), 0x7FC0, dtype=torch.int16, device="cuda").view(torch.uint8)      # (NaN behind the rows)
    ctx.rm_gather_weights(model.packed[0], dev(idx), cnt, I, compact_out=compact)
    got = call(None, cnt, r, layer=compact)
    assert ctx.rm_get_info("last_variant") == kernel
    assert_close(got, oracle.masked_mlp(x, *W, r, sel), "compact layer")
    assert ctx.rm_device_status() == 0
    model.close()
