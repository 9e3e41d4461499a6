"""What the native side of the binding does with argument lists that do not fit: Python errors, before anything is called."""
import numpy as np
import pytest


class FakeTensor:
    def data_ptr(self):
        return 4096


T = FakeTensor()
#                 ctx, layers, L, r_in, idx, cnt, stride, r_out, rec, scale, B, T, ws, bytes
STEP = lambda **kw: [kw.get("ctx", 0), kw.get("layers", [T, T]), kw.get("L", 2), T, None, None, kw.get("stride", 64), T, None, None,
                     kw.get("B", 1), kw.get("T", 8), T, 1 << 20]
MASK = lambda **kw: [0, kw.get("records", [T]), 1, 2, kw.get("threshold", 0.0), kw.get("k", 3), 1, None, kw.get("per_list", False),
                     kw.get("n_lists", 1), kw.get("I", 64), T, T, 64]


@pytest.fixture()
def native(lib):
    lib.load_library()
    return lib._native


@pytest.mark.parametrize("layers", [[], [T]])
def test_fewer_layers_than_the_model_has(lib, native, layers):
    extra = {"step": [], "step_ex": [0, T, T, 8, None], "step_host": []}
    for name, more in extra.items():
        args = STEP(layers=layers)
        if name == "step_host":
            del args[8:10]                                             # (no records)
        args[-2:-2] = more
        with pytest.raises(ValueError, match=f"{len(layers)} packed layers for a model of 2"):
            getattr(native, name)(*args)
    holder = lib.Context.__new__(lib.Context)
    holder.L = 2
    with pytest.raises(ValueError):
        holder._layer_ptrs(layers)


def test_too_few_and_too_many_arguments(native):
    for make, f in ((STEP, native.step), (MASK, native.mask_compact)):
        with pytest.raises(TypeError):
            f(*make()[:-1])
        with pytest.raises(TypeError):
            f(*make(), 7)
    for name in ("sparse_mlp", "sparse_mlp_static", "step_ex", "step_host", "context_drift", "context_ffn"):
        with pytest.raises(TypeError):
            getattr(native, name)()


@pytest.mark.parametrize("bad", [1 << 31, -(1 << 31) - 1, 1 << 40, 1 << 80])
def test_integers_beyond_32_bits(native, bad):
    for kw in ({"B": bad}, {"T": bad}):
        with pytest.raises(OverflowError):
            native.step(*STEP(**kw))
    for kw in ({"k": bad}, {"n_lists": bad}, {"I": bad}):
        with pytest.raises(OverflowError):
            native.mask_compact(*MASK(**kw))


def test_things_that_are_no_numbers(native):
    with pytest.raises(TypeError):
        native.mask_compact(*MASK(k=None))
    with pytest.raises(TypeError):
        native.mask_compact(*MASK(threshold=[1.0]))
    with pytest.raises(AttributeError):
        native.mask_compact(*MASK(records=[3]))
    with pytest.raises(TypeError):
        native.step(*STEP(layers=5))


@pytest.mark.gpu
def test_forms_that_are_accepted(lib):
    """More layers than the model has, any iterable, anything int(), float() or bool() takes."""
    import torch
    L, H, I, n = 2, 1024, 256, 8
    g = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    ctx = lib.Context(L, H, I, n)
    layers = [ctx.rm_pack_weights(*[(0.02 * rnd(*s)).bfloat16() for s in ((I, H), (I, H), (H, I))]) for _ in range(L + 1)]
    idx, cnt = torch.zeros(L, I, dtype=torch.int32, device="cuda"), torch.zeros(L, dtype=torch.int32, device="cuda")
    rec, r = rnd(L, I).abs(), rnd(1, n, H)
    outs = []
    for k, stride, per_list, threshold, more in ((64, I, False, 0.0, layers[:L]), (np.int64(64), torch.tensor(I), None, "0.5", layers),
                                                 (64.9, np.int32(I), [], torch.tensor(0.5), tuple(layers)), (torch.tensor(64), I, 0, 1, iter(layers))):
        ctx.rm_mask_compact(iter([rec]), lib.RM_SRC_SCORE_F32, lib.RM_REDUCE_TOPK, idx, cnt, stride, n_lists=L, k=k, threshold=threshold,
                            scale_per_list=per_list)
        out = torch.empty_like(r)
        ctx.rm_action_expert_step(more, r, idx, cnt, stride, out)
        outs.append((idx.clone(), cnt.clone(), out))
    for o in outs[1:]:
        assert torch.equal(o[0], outs[0][0]) and torch.equal(o[1], outs[0][1])
        assert float((o[2] - outs[0][2]).norm() / outs[0][2].norm()) <= 1e-3
    assert ctx.rm_device_status() == 0
    ctx.close()
