"""The slice kernel (variant 6) against the oracle at the sizes where its tiles and splits end: widths that are no multiple
of 128, a single token, chunks of more than 64 tokens, lists shorter than the number of clusters, batches, in-place steps."""
import numpy as np
import pytest

import oracle
from harness import REL_L2_TOL, assert_close, dev, lists_to_padded
from test_gpu_anchor import make_case, run_write
from test_gpu_edges import step_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,I,T,L,B,density,clusters", [
    (64, 96, 9, 3, 1, 0.4, 0), (192, 333, 64, 2, 3, 0.5, 2), (320, 200, 1, 3, 1, 0.3, 0), (1024, 1000, 17, 2, 1, 0.37, 0),
    (1024, 600, 51, 4, 1, 0.01, 0), (1024, 700, 51, 3, 8, 0.2, 0), (1088, 300, 8, 2, 2, 0.5, 3), (1536, 520, 51, 3, 1, 0.6, 0),
    (2048, 712, 33, 2, 2, 0.5, 0), (512, 400, 65, 2, 2, 0.4, 0), (1024, 256, 100, 3, 1, 0.3, 0), (768, 300, 130, 2, 1, 0.9, 0)])
def test_slice_kernel_matches_the_oracle(lib, H, I, T, L, B, density, clusters):
    step_case(lib, H=H, I=I, T=T, L=L, B=B, density=density, variant=6, max_clusters=clusters, config=97)


@pytest.mark.parametrize("H,T,L,B", [(1024, 51, 3, 2), (384, 70, 2, 1)])
def test_slice_kernel_anchor_update_in_place(lib, H, T, L, B):
    """Eq. 4 through the slice kernel: write, update (one list empty, one full), and the update with input and output in
    one buffer, for stacks of one layer as well."""
    import torch
    for depth in (L, 1):
        w, model, r_a, r_t, gate, lists = make_case(lib, H, 300, T, depth, B)
        ctx = model.ctx
        ctx.rm_set_option("variant", 6)
        hs = (T + 3) // 4 * 4 + 4
        if T <= 64:
            out_a, y_an, h_an, _ = run_write(model, w, r_a, gate, B, hs)
        else:                                              # (records of long chunks go through the CUDA-core kernels)
            y_an = torch.full((depth, B, T, H), 7.0, dtype=torch.float32, device="cuda")
            h_an = torch.zeros(depth, B, w.I, hs, dtype=torch.float32, device="cuda")
            out_a = torch.empty(B, T, H, dtype=torch.float32, device="cuda")
            ctx.rm_action_expert_step_ex(model.packed, dev(r_a), None, None, 0, out_a, lib.RM_ANCHOR_WRITE, y_an, h_an, hs,
                                         out_gate=dev(gate), B=B, T=T)
        assert ctx.rm_get_info("last_variant") == 6
        idx, cnt = lists_to_padded([s for per_b in lists for s in per_b], w.I)
        buf = dev(r_t.copy())
        ctx.rm_action_expert_step_ex(model.packed, buf, dev(idx), dev(cnt), w.I, buf, lib.RM_ANCHOR_UPDATE, y_an, h_an, hs,
                                     out_gate=dev(gate), B=B, T=T)
        for b in range(B):
            want_a, want_y, want_h, _ = oracle.anchor_step_write(model.Wg, model.Wu, model.Wd, r_a[b], gate[:, b])
            assert_close(out_a.cpu().numpy()[b], want_a, f"anchor step, episode {b}")
            i_b, c_b = lists_to_padded(lists[b], w.I)
            want = oracle.anchor_step_update(model.Wg, model.Wu, model.Wd, r_t[b], i_b, c_b, want_y, want_h, gate[:, b])
            assert_close(buf.cpu().numpy()[b], want, f"update in place, episode {b}")
        assert ctx.rm_device_status() == 0
        model.close()


def test_slice_kernel_in_a_replayed_graph(lib):
    """The control block of a launch is set up and taken back by the launch itself: a captured step can be replayed."""
    import torch
    w, model, r_a, r_t, gate, lists = make_case(lib, 256, 200, 12, 3, 1)
    ctx = model.ctx
    ctx.rm_set_option("variant", 6)
    idx, cnt = lists_to_padded([s for per_b in lists for s in per_b], w.I)
    r, di, dc, out = dev(r_t), dev(idx), dev(cnt), torch.zeros(1, w.T, w.H, device="cuda")
    ctx.workspace(1, w.T)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ctx.rm_action_expert_step(model.packed, r, di, dc, w.I, out)
    want = oracle.step(model.Wg, model.Wu, model.Wd, r_t[0], idx, cnt)
    for _ in range(3):
        out.zero_()
        g.replay()
        assert_close(out.cpu().numpy()[0], want, "replay")
    assert ctx.rm_device_status() == 0
    del g
    model.close()


@pytest.mark.parametrize("H,I,T,L,B,density", [
    (384, 1300, 51, 1, 1, 0.25), (512, 2048, 51, 1, 1, 0.06), (1536, 6144, 51, 1, 1, 0.25), (1792, 3000, 33, 1, 1, 1.0), (2048, 4096, 90, 1, 1, 0.3),
    (1024, 3500, 70, 1, 1, 0.6), (1536, 6144, 51, 6, 1, 0.25), (1088, 900, 20, 3, 9, 0.5)])
def test_other_widths_lose_nothing_against_the_cuda_core_kernels(lib, H, I, T, L, B, density):
    """The CUDA-core kernels, which take the same shapes, sum in fp32 in one order: the same bits every time, and an error against
    64 bits that the slice kernel must not exceed.  (25 % for where the roundings that both share are the larger part.  Behind one
    layer single roundings of x to bf16 differ and hide the sums.)  Nine episodes: two launches."""
    import math

    import torch
    g = torch.Generator(device="cuda").manual_seed(H + I + T)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    ctx = lib.Context(L, H, I, T, B)
    W = [[(0.64 / H ** 0.5 * rnd(*s)).bfloat16() for s in ((I, H), (I, H), (H, I))] for _ in range(L)]
    layers = [ctx.rm_pack_weights(*w) for w in W]
    k, stride = max(1, int(density * I)), (I + 3) // 4 * 4
    idx = torch.zeros(B, L, stride, dtype=torch.int32, device="cuda")
    for b in range(B):
        for l in range(L):
            idx[b, l, :k] = torch.randperm(I, generator=g, device="cuda")[:k].sort().values.int()
    cnt = torch.full((B, L), k, dtype=torch.int32, device="cuda")
    r = rnd(B, T, H).bfloat16().float()

    def run(path):
        ctx.rm_set_option("path", path)
        out = torch.full_like(r, 7.0)
        ctx.rm_action_expert_step(layers, r, idx, cnt, stride, out, B=B)
        assert ctx.rm_get_info("last_variant") == (0 if path else 6)
        return out

    first, portable = run(0), run(1)
    for _ in range(3):
        assert torch.equal(first, run(0))
    in_place = r.clone()
    ctx.rm_action_expert_step(layers, in_place, idx, cnt, stride, in_place, B=B)
    assert torch.equal(first, in_place)
    assert ctx.rm_device_status() == 0
    if L == 1:
        gate, up, down = (w.double() for w in W[0])
        i = idx[0, 0, :k].long()
        x = (r[0].double() / torch.sqrt((r[0].double() ** 2).mean(-1, keepdim=True) + 1e-6)).float().bfloat16().double()
        z = x @ gate[i].T
        y = (0.5 * z * (1 + torch.tanh(math.sqrt(2 / math.pi) * (z + 0.044715 * z ** 3))) * (x @ up[i].T)) @ down[:, i].T
        err = [float((o[0].double() - r[0].double() - y).norm() / y.norm()) for o in (first, portable)]
        assert err[0] <= 1.25 * err[1], err
    else:
        assert float((first - portable).norm() / portable.norm()) <= REL_L2_TOL
    ctx.close()
