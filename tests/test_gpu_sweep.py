"""The sweep kernel (variant 7) against the oracle where its units, stages and splits end: neuron counts below, at and beside
multiples of 16 and 64, fewer units than CTAs, one token, the largest units per CTA, a small grid, the anchor step of Eq. 4."""
import numpy as np
import pytest

import oracle
from harness import Model, assert_close, dev
from paper_2609_19104_b200 import workloads as wl
from test_gpu_anchor import make_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,I,T,L,clusters", [(1024, 5, 9, 2, 0), (1024, 64, 64, 3, 0), (1024, 1000, 1, 2, 0), (2048, 129, 33, 2, 0),
                                              (2048, 712, 51, 3, 2), (1024, 1024, 51, 2, 1), (1024, 700, 17, 2, 1), (2048, 2400, 51, 1, 0)])
def test_dense_steps_match_the_oracle(lib, H, I, T, L, clusters):
    import torch
    w = wl.Workload(98, "sweep", L, H, I, T, 1.0 / np.sqrt(H), 1, 1.0)
    model = Model(lib, w)
    ctx = model.ctx
    ctx.rm_set_option("variant", 7)
    ctx.rm_set_option("max_clusters", clusters)
    r0 = wl.bf16_bits_to_f32(wl.step_input(w, 0))
    scale = (1.0 + wl.uniform(wl.tensor_key(3, 98, 0, 2), L * I)).astype(np.float32).reshape(L, I)
    want, want_rec = oracle.step(model.Wg, model.Wu, model.Wd, r0, return_records=True)
    rec = torch.zeros(1, L, I, dtype=torch.float32, device="cuda")
    r, out = dev(r0[None]), torch.full((1, T, H), 3.0, dtype=torch.float32, device="cuda")
    for _ in range(2):                                     # the second call finds the first one's control block
        ctx.rm_action_expert_step(model.packed, r, None, None, 0, out, records_out=rec, record_scale=dev(scale), B=1, T=T)
        assert ctx.rm_get_info("last_variant") == 7
        assert_close(out.cpu().numpy()[0], want, "dense step")
        got = rec.cpu().numpy()[0]
        assert np.all(np.abs(got - want_rec * scale) <= 4e-2 + 1e-2 * np.abs(want_rec * scale))
    ctx.rm_action_expert_step(model.packed, r, None, None, 0, r, B=1, T=T)      # in place
    assert_close(r.cpu().numpy()[0], want, "dense step in place")
    assert ctx.rm_device_status() == 0
    model.close()


@pytest.mark.parametrize("H,I,T,L", [(1024, 300, 51, 3), (2048, 200, 30, 2)])
def test_anchor_step_matches_the_oracle(lib, H, I, T, L):
    import torch
    w, model, r_a, _, gate, _ = make_case(lib, H, I, T, L, 1)
    ctx = model.ctx
    ctx.rm_set_option("variant", 7)
    hs = (T + 3) // 4 * 4 + 4
    y_an = torch.full((L, 1, T, H), 7.0, dtype=torch.float32, device="cuda")
    h_an = torch.zeros(L, 1, w.I, hs, dtype=torch.float32, device="cuda")
    out = torch.empty(1, T, H, dtype=torch.float32, device="cuda")
    ctx.rm_action_expert_step_ex(model.packed, dev(r_a), None, None, 0, out, lib.RM_ANCHOR_WRITE, y_an, h_an, hs, out_gate=dev(gate))
    assert ctx.rm_get_info("last_variant") == 7
    want, want_y, want_h, _ = oracle.anchor_step_write(model.Wg, model.Wu, model.Wd, r_a[0], gate[:, 0])
    assert_close(out.cpu().numpy()[0], want, "anchor step")
    for l in range(L):
        assert_close(y_an.cpu().numpy()[l, 0], want_y[l], "retained y_a")
        assert np.all(np.abs(h_an.cpu().numpy()[l, 0, :, :T].T - want_h[l]) <= 2e-2 + 1e-2 * np.abs(want_h[l]))
    assert ctx.rm_device_status() == 0
    model.close()


@pytest.mark.parametrize("H,I,T,L", [(1024, 4096, 51, 18), (2048, 4000, 64, 12), (1024, 18944, 64, 4)])
def test_records_of_every_layer_are_that_layers(lib, H, I, T, L):
    """All CTAs at work, the last of them (of 148: 144 to 147) with neurons but neither a split of the down sweep nor a row of x: nothing
    but the layers in turn keeps one layer's record sums from the next's."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(H + I)
    ctx = lib.Context(L, H, I, T)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    # Every layer has gate and up weights of its own, but adds next to nothing (columns of 1e-4), so that x differs between the two
    # kernels in single roundings to bf16 only.  One moves a hidden value by at most 2^-8 |x| |w| |u| = 2^-8 * 4 * 4.5 * 0.64 / sqrt(H) * 3
    # = 4e-3 at H = 1024; the fp32 sums add sqrt(H T) 2^-24 of a record.  Another layer's sum over the second token half is off by
    # about its size, 5 to 10.
    scale = lambda i: 1e-4 if i == 2 else 0.64 / H ** 0.5
    layers = [ctx.rm_pack_weights(*[(scale(i) * rnd(*s)).bfloat16() for i, s in enumerate(((I, H), (I, H), (H, I)))]) for _ in range(L)]
    r = rnd(1, T, H).bfloat16().float()
    out, rec, want = torch.empty_like(r), torch.zeros(1, L, I, device="cuda"), torch.zeros(1, L, I, device="cuda")
    ctx.rm_set_option("path", 1)
    ctx.rm_action_expert_step(layers, r, None, None, I, out, records_out=want)
    ctx.rm_set_option("path", 0)
    ctx.rm_set_option("variant", 7)
    for _ in range(5):
        rec.fill_(-1.0)
        ctx.rm_action_expert_step(layers, r, None, None, I, out, records_out=rec)
        assert ctx.rm_get_info("last_variant") == 7
        assert torch.all((rec - want).abs() <= 1e-3 * want + 5e-3)
    assert ctx.rm_device_status() == 0
    ctx.close()
