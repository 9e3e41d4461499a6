"""The slice kernel (variant 6) against the oracle at the sizes where its tiles and splits end: widths that are no multiple
of 128, a single token, chunks of more than 64 tokens, lists shorter than the number of clusters, batches, in-place steps."""
import numpy as np
import pytest

import oracle
from harness import assert_close, dev, lists_to_padded
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
