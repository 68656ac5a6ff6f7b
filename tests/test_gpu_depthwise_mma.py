"""The depthwise layers on tcgen05 against the oracle: rows of 32, 64 and 128 bytes, images around the tile, both
strides, concat window, per-layer and per-channel shifts, and tensors too little aligned for it (the other kernels)."""
import numpy as np
import pytest
import torch

from tests.helpers import gpu_conv, oracle_conv, rand_layer

pytestmark = pytest.mark.gpu

CASES = [  # N, H, W, C, stride
    (2, 9, 11, 32, 1), (1, 8, 14, 64, 1), (3, 7, 7, 128, 1), (2, 9, 15, 128, 1), (1, 1, 1, 64, 1), (2, 17, 130, 192, 1),
    (2, 14, 14, 64, 2), (1, 13, 9, 128, 2), (2, 9, 17, 48, 1), (1, 20, 15, 208, 1), (2, 7, 31, 112, 2), (1, 5, 5, 16, 1), (5, 3, 2, 96, 2), (1, 30, 61, 32, 2), (40, 14, 14, 256, 1), (40, 14, 14, 256, 2)]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("uniform", [0, 1])
def test_depthwise_on_tensor_cores_matches_the_oracle(case, uniform):
    from paper_1805_07941_b200 import binding
    N, H, W, C, st = case
    rng = np.random.default_rng(sum(case))
    x, w, bias, shift, _, _ = rand_layer(rng, N, H, W, C, C, 3, 3, groups=C, stride=(st, st), pad=(1, 1), per_channel_shift=not uniform)
    shift = (shift - 1).clip(4, 31)
    for relu in (0, 1):
        kw = dict(R=3, S=3, stride=(st, st), pad=(1, 1), groups=C, relu=relu)
        win = dict(kw, out_c_offset=16, out_c_pitch=C + 32)
        want, want_win = oracle_conv(x, w, bias, shift, **kw), oracle_conv(x, w, bias, shift, **win)
        for hints in (dict(), dict(bn_max=64), dict(patch_halo=0), dict(patch_halo=0, halo=0), dict(tma_store=1)):
            with binding.plan_hints(depthwise_form=3, **hints):
                got, desc = gpu_conv(x, w, bias, shift, **kw)
                assert "depthwise3x3/mma/" in desc and (got == want).all(), (hints, desc)
                got, desc = gpu_conv(x, w, bias, shift, **win)
                assert "depthwise3x3/mma/" in desc and (got == want_win).all(), (hints, desc)


# N, H, W, C, stride -> the form that the plan takes by itself: tcgen05 where narrow or short images leave the warps' groups partly
# empty or an SM gets a CTA more than its share, the warp level where tcgen05's tiles are the ones that waste
DISPATCH = [(212, 41, 9, 512, 2, "mma/"), (96, 28, 28, 256, 1, "mma/"), (200, 10, 10, 512, 1, "mma/"), (128, 36, 36, 128, 1, "mma/"),
            (128, 28, 28, 512, 1, "mma/"), (64, 56, 56, 112, 1, "mma/"), (64, 28, 28, 576, 1, "mma+tma"), (128, 14, 14, 512, 1, "mma+tma"),
            (32, 56, 56, 128, 1, "mma+tma"), (256, 14, 14, 512, 2, "mma+tma"), (64, 112, 112, 32, 1, "mma+tma"), (1, 28, 28, 256, 1, "mma+tma")]


@pytest.mark.parametrize("case", DISPATCH)
def test_the_form_is_chosen_by_what_it_costs(case):
    from paper_1805_07941_b200 import binding
    N, H, W, C, st, form = case
    conv = binding.QConv(np.ones((C, 3, 3, 1), np.int8), None, np.full(C, 6, np.int32), N=N, H=H, W=W, C=C, K=C, R=3, S=3, stride_h=st,
                         stride_w=st, pad_h=1, pad_w=1, groups=C)
    assert conv.describe().startswith("depthwise3x3/" + form), conv.describe()
    conv.destroy()


@pytest.mark.parametrize("case", [(200, 10, 10, 512, 1), (212, 41, 9, 512, 2), (64, 56, 56, 112, 1)])
def test_layers_that_take_tcgen05_by_themselves_match_the_oracle(case):
    """Whole and partial batches, and an output that is 8-byte aligned only: that run takes the warp level, or dp4a where 32 does not
    divide the channels."""
    from paper_1805_07941_b200 import binding
    N, H, W, C, st = case
    rng = np.random.default_rng(sum(case))
    x, w, bias, shift, _, _ = rand_layer(rng, N, H, W, C, C, 3, 3, groups=C, stride=(st, st), pad=(1, 1))
    shift = (shift - 1).clip(4, 31)
    conv = binding.QConv(w, bias, shift, N=N, H=H, W=W, C=C, K=C, R=3, S=3, stride_h=st, stride_w=st, pad_h=1, pad_w=1, groups=C)
    assert "depthwise3x3/mma/" in conv.describe()
    xd, want = torch.from_numpy(x).cuda(), oracle_conv(x, w, bias, shift, R=3, S=3, stride=(st, st), pad=(1, 1), groups=C)
    flat = torch.empty(want.size + 16, dtype=torch.int8, device="cuda")
    for n, off in ((N, 0), (N // 3, 0), (N, 8), (N // 2, 8), (N, 0)):
        flat.fill_(77)
        y = flat[off:off + want.size].view(want.shape)
        conv.run(xd, y, n_run=n)
        assert conv.status() == 0
        got = y.cpu().numpy()
        assert (got[:n] == want[:n]).all() and (got[n:] == 77).all() and (flat[:off] == 77).all() and (flat[off + want.size:] == 77).all()
    conv.destroy()


def test_less_aligned_tensors_take_the_other_kernels():
    from paper_1805_07941_b200 import binding
    N, H, W, C = 2, 9, 11, 64
    rng = np.random.default_rng(0)
    x, w, bias, shift, _, _ = rand_layer(rng, N, H, W, C, C, 3, 3, groups=C, pad=(1, 1))
    conv = binding.QConv(w, bias, shift, N=N, H=H, W=W, C=C, K=C, R=3, S=3, pad_h=1, pad_w=1, groups=C)
    want = oracle_conv(x, w, bias, shift, R=3, S=3, pad=(1, 1), groups=C)
    for off in (0, 4):
        xb, yb = (torch.zeros(x.size + 16, dtype=torch.int8, device="cuda") for _ in range(2))
        xd, yd = (b[off:off + x.size].view(N, H, W, C) for b in (xb, yb))
        xd.copy_(torch.from_numpy(x))
        conv.run(xd, yd)
        assert conv.status() == 0 and (yd.cpu().numpy() == want).all(), off


@pytest.mark.parametrize("case", [(2, 9, 11, 64, 1), (1, 13, 9, 128, 2), (3, 30, 31, 192, 1), (2, 21, 20, 256, 2)])
def test_plan_hints_never_change_a_depthwise_layer(case):
    """Every hint of the plan on a layer that the tensor cores take by themselves, and beside the depthwise forms; a hint that
    takes the fast epilogues away leaves the layer to the CUDA-core kernels."""
    from paper_1805_07941_b200 import binding
    N, H, W, C, st = case
    rng = np.random.default_rng(sum(case))
    x, w, bias, shift, _, _ = rand_layer(rng, N, H, W, C, C, 3, 3, groups=C, stride=(st, st), pad=(1, 1))
    shift = (shift - 1).clip(4, 31)
    kw = dict(R=3, S=3, stride=(st, st), pad=(1, 1), groups=C)
    want = oracle_conv(x, w, bias, shift, **kw)
    for form in (-1, 0, 1, 2, 3, 4):
        for hints in (dict(), dict(fast_epilogue=0), dict(float_rounding=0), dict(uniform_shift=0), dict(halo=0), dict(halo=1),
                      dict(resident_weights=0), dict(resident_weights=1), dict(tma_store=0), dict(tma_store=1), dict(group_taps=0),
                      dict(group_taps=1), dict(patch_halo=0), dict(patch_halo=1), dict(bn_max=32), dict(bn_max=256),
                      dict(ctas_per_sm=1), dict(ctas_per_sm=2), dict(pdl=0), dict(split_k=2), dict(pair_tiles=1), dict(fold=0)):
            with binding.plan_hints(depthwise_form=form, **hints):
                got, desc = gpu_conv(x, w, bias, shift, **kw)
            epilogue = "fast_epilogue" not in hints and "float_rounding" not in hints
            assert ("depthwise3x3/mma+tma" in desc) == (epilogue and form in (-1, 4)), (form, hints, desc)
            assert ("depthwise3x3/mma/" in desc) == (epilogue and form == 3), (form, hints, desc)
            assert form != 2 or "tap-packed+tma" in desc, (hints, desc)
            assert (got == want).all(), (form, hints, desc)
