"""One context's workspace serves calls of every (B, T) and every kernel family, whose buffers lie over one another in it: no call may
count on what an earlier one left there.  The results are compared with the CUDA-core kernels', which keep nothing."""
import pytest

from harness import REL_L2_TOL

pytestmark = pytest.mark.gpu


class Steps:
    def __init__(self, lib, H, I, L, T_max, B_max):
        import torch
        self.lib, self.H, self.I, self.L = lib, H, I, L
        self.g = torch.Generator(device="cuda").manual_seed(H + I + L)
        self.ctx = lib.Context(L, H, I, T_max, B_max)
        self.layers = [self.ctx.rm_pack_weights(*[(0.64 / H ** 0.5 * self.rnd(*s)).bfloat16() for s in ((I, H), (I, H), (H, I))])
                       for _ in range(L)]

    def rnd(self, *s):
        import torch
        return torch.randn(*s, generator=self.g, device="cuda")

    def case(self, B, T, K):
        """Inputs of a step and what it has to give; K = 0: dense."""
        import torch
        r = self.rnd(B, T, self.H).bfloat16().float()
        idx = cnt = None
        if K:
            idx = torch.zeros(B * self.L, self.I, dtype=torch.int32, device="cuda")
            cnt = torch.zeros(B * self.L, dtype=torch.int32, device="cuda")
            self.ctx.rm_mask_compact([self.rnd(B * self.L, self.I).abs()], self.lib.RM_SRC_SCORE_F32, self.lib.RM_REDUCE_TOPK, idx, cnt,
                                     self.I, n_lists=B * self.L, k=K)
        c = dict(r=r, idx=idx, cnt=cnt, B=B, T=T, K=K, out=torch.empty_like(r))
        self.ctx.rm_set_option("path", 1)
        self.run(c)
        self.ctx.rm_set_option("path", 0)
        c["want"] = c["out"].clone()
        return c

    def run(self, c):
        self.ctx.rm_set_option("count_hint", c["K"])
        self.ctx.rm_action_expert_step(self.layers, c["r"], c["idx"], c["cnt"], self.I, c["out"], B=c["B"])

    def check(self, c, what):
        import torch
        assert torch.isfinite(c["out"]).all(), what
        assert float((c["out"] - c["want"]).norm() / c["want"].norm()) <= REL_L2_TOL, what
        assert self.ctx.rm_device_status() == 0, what


@pytest.mark.parametrize("calls", [
    [(1, 51, 1400, 5), (8, 51, 700, 4), (1, 51, 1400, 5)],          # the batch's residual buffers lie over the whole-step kernel's counters
    [(1, 20, 2048, 5), (1, 64, 500, 1), (1, 20, 2048, 5)],
    [(1, 51, 1400, 5), (1, 100, 500, 6), (1, 51, 1400, 5), (2, 70, 900, 6), (1, 51, 1400, 5)],
    [(1, 51, 0, 7), (8, 51, 700, 4), (1, 51, 0, 7), (1, 51, 1400, 5), (1, 100, 300, 6), (1, 51, 0, 7)],
])
def test_calls_of_other_sizes_in_between(lib, calls):
    s = Steps(lib, 1024, 4096, 3, 100, 8)
    s.ctx.workspace(8, 100)                                          # (one buffer for all of them, not a larger one on the way)
    cases = [s.case(B, T, K) for B, T, K, _ in calls]
    for _ in range(3):
        for c, (_, _, _, variant) in zip(cases, calls):
            c["out"].fill_(7.0)
            s.run(c)
            assert s.ctx.rm_get_info("last_variant") == variant, c
            s.check(c, (c["B"], c["T"], c["K"]))
    s.ctx.close()


@pytest.mark.parametrize("fill", [0xff, 0x01, 0x3f, 0x7f])
@pytest.mark.parametrize("B,T,K,variant", [(1, 51, 1400, 5), (3, 40, 300, 5), (1, 64, 1400, 6), (2, 100, 300, 6), (1, 51, 0, 7), (1, 20, 300, 1), (4, 51, 1100, 4)])
def test_workspace_of_any_content(lib, B, T, K, variant, fill):
    s = Steps(lib, 1024, 4096, 2, 100, 8)
    c = s.case(B, T, K)
    s.ctx.rm_set_option("variant", variant)
    for _ in range(2):
        s.ctx.workspace(B, T).fill_(fill)
        c["out"].fill_(7.0)
        s.run(c)
        assert s.ctx.rm_get_info("last_variant") == variant
        s.check(c, fill)
    s.ctx.close()


@pytest.mark.parametrize("T,K,variant", [(51, 1400, 5), (51, 0, 7), (100, 300, 6), (20, 300, 1)])
def test_captured_step_with_other_calls_between_its_replays(lib, T, K, variant):
    import torch
    s = Steps(lib, 1024, 4096, 3, 100, 8)
    s.ctx.workspace(8, 100)
    c, other = s.case(1, T, K), s.case(8, 51, 700)
    s.run(c)                                                         # (kernel attributes are set outside the capture)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        s.run(c)
    assert s.ctx.rm_get_info("last_variant") == variant
    for i in range(4):
        c["out"].fill_(7.0)
        graph.replay()
        s.check(c, f"replay {i}")
        if i % 2:
            s.run(other)
            s.check(other, "batch")
            s.run(c)
            s.check(c, "the step outside the graph")
    del graph
    s.ctx.close()


@pytest.mark.parametrize("H,T,tiles,variant", [(1024, 51, 15, 1), (1024, 60, 20, 2), (1024, 20, 40, 4), (1024, 51, 20, 5), (2048, 20, 40, 2),
                                               (2048, 40, 33, 5), (2048, 20, 50, 5), (2048, 51, 62, 4)])
def test_one_layer_alone_leaves_the_workspace_as_it_is(lib, H, T, tiles, variant):
    """Two streams may have one-layer calls of these widths on the device with one workspace between them: no kernel keeps anything there."""
    import torch
    s = Steps(lib, H, 4096, 1, T, 1)
    idx, cnt = torch.zeros(1, 4096, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    s.ctx.rm_mask_compact([s.rnd(1, 4096).abs()], lib.RM_SRC_SCORE_F32, lib.RM_REDUCE_TOPK, idx, cnt, 4096, n_lists=1, k=64 * tiles)
    x, r, y = s.rnd(T, H).bfloat16(), s.rnd(T, H), torch.empty(T, H, device="cuda")
    if variant == 5 and H == 1024:
        s.ctx.rm_set_option("variant", 5)
    ws = torch.full((s.ctx.workspace_bytes(1, T),), 0xa5, dtype=torch.uint8, device="cuda")
    s.ctx.rm_sparse_mlp(s.layers[0], x, r, idx, cnt, y, ws=ws)
    assert s.ctx.rm_get_info("last_variant") == variant
    assert s.ctx.rm_device_status() == 0
    assert bool((ws == 0xa5).all())
    s.ctx.rm_set_option("path", 1)
    want = torch.empty_like(y)
    s.ctx.rm_sparse_mlp(s.layers[0], x, r, idx, cnt, want)
    # (fp32 sums in another order, hidden values to 17 bits)
    assert float((y - want).norm() / (want - r).norm()) <= 1e-4
    s.ctx.close()
