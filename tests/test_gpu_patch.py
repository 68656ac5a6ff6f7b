"""The patch form of 3 x 3 layers (one activation box for all nine taps) against the oracle: images around the tile's
14 x 8 outputs, channel counts that fill a chunk or not, one and several channel tiles, staged and direct stores,
residual, concat window, pool, per-layer and per-channel shifts, both roundings' epilogues, several tiles per CTA."""
import numpy as np
import pytest

from oracle import ref
from tests.helpers import gpu_conv, oracle_conv, rand_layer

pytestmark = pytest.mark.gpu

CASES = [  # N, H, W, C, K
    (2, 8, 14, 64, 64), (1, 7, 13, 64, 128), (3, 9, 15, 128, 128), (2, 16, 28, 48, 64), (1, 17, 29, 96, 208), (2, 5, 3, 128, 256),
    (1, 1, 1, 64, 16), (2, 20, 43, 112, 80), (40, 28, 28, 64, 64), (30, 30, 30, 128, 128),
    # rows of 32 bytes: 16 and 32 channels, one and several channel tiles, images smaller than a tile, several tiles per CTA
    (1, 8, 14, 16, 16), (2, 7, 13, 32, 48), (3, 16, 28, 16, 208), (2, 6, 10, 32, 256), (5, 9, 15, 32, 112), (1, 1, 1, 32, 16), (2, 18, 30, 16, 128),
    (40, 28, 28, 32, 64), (24, 30, 30, 16, 32)]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("uniform", [0, 1])
def test_patch_form_matches_the_oracle(case, uniform):
    from paper_1805_07941_b200 import binding
    N, H, W, C, K = case
    for small in (0, 1):
        for with_res in (0, 1):
            rng = np.random.default_rng(sum(case) + uniform)
            x, w, bias, shift, res, t = rand_layer(rng, N, H, W, C, K, 3, 3, with_res=bool(with_res), pad=(1, 1), per_channel_shift=not uniform)
            if small:                                        # the float-rounding epilogue
                w, shift = (w // 16).astype(np.int8), np.maximum(shift - 4, 0).astype(np.int32)
                t = np.minimum(t, 5).astype(np.int32) if with_res else None
            if with_res and uniform:
                t = np.full(K, int(t[0]), np.int32)
            kw = dict(R=3, S=3, pad=(1, 1), relu=small)
            with binding.plan_hints(patch_halo=1):
                got, desc = gpu_conv(x, w, bias, shift, res, t, **kw)
                assert "patch=1" in desc and (got == oracle_conv(x, w, bias, shift, res, t, **kw)).all(), (desc, small, with_res)
                if with_res:
                    continue
                win = dict(kw, out_c_offset=16, out_c_pitch=K + 48)
                got, desc = gpu_conv(x, w, bias, shift, **win)
                assert "patch=1" in desc and (got == oracle_conv(x, w, bias, shift, **win)).all(), desc
                with binding.plan_hints(patch_halo=1, tma_store=0, ctas_per_sm=1):
                    got, desc = gpu_conv(x, w, bias, shift, **kw)
                want = oracle_conv(x, w, bias, shift, **kw)
                assert "patch=1" in desc and (got == want).all(), desc
                if H % 2 == 0 and W % 2 == 0:
                    with binding.plan_hints(patch_halo=1):
                        got, desc = gpu_conv(x, w, bias, shift, pool=2, **kw)
                    assert "patch=1" in desc and (got == ref.maxpool_i8(want, 2, 2, 2, 0)).all(), desc


# N, H, W, C, K -> whether the plan takes the patch form by itself (below a wave of tiles only at up to 32 channels), and its width:
# 64 channels only where 128-wide tiles are fewer than the SMs
PLANS = [(1, 32, 32, 16, 16, 1, 16), (1, 56, 56, 32, 32, 1, 32), (16, 7, 7, 32, 256, 1, 64), (32, 14, 14, 32, 128, 1, 64), (20, 28, 28, 32, 128, 1, 128),
         (1, 32, 32, 48, 64, 0, 64), (20, 28, 28, 64, 128, 1, 128), (10, 28, 28, 128, 256, 1, 128), (10, 28, 28, 96, 192, 1, 96)]


@pytest.mark.parametrize("N,H,W,C,K,patch,BN", PLANS)
def test_the_tiles_of_the_patch_form(N, H, W, C, K, patch, BN):
    rng = np.random.default_rng(N + C)
    x, w, bias, shift, _, _ = rand_layer(rng, N, H, W, C, K, 3, 3, pad=(1, 1))
    got, desc = gpu_conv(x, w, bias, shift, R=3, S=3, pad=(1, 1))
    assert ("patch=1" in desc) == bool(patch) and " BN=%d " % BN in desc, desc
    assert (got == oracle_conv(x, w, bias, shift, R=3, S=3, pad=(1, 1))).all(), desc


@pytest.mark.parametrize("N,H,W,C,K", [(64, 9, 5, 32, 256), (110, 5, 5, 32, 128), (33, 9, 9, 16, 64)])
def test_one_tile_to_a_cta_is_stored_without_staging(N, H, W, C, K):
    """Tiles leave straight from the registers while every CTA has one, whatever the plan holds for larger batches."""
    from paper_1805_07941_b200 import binding
    import torch
    rng = np.random.default_rng(N + K)
    x, w, bias, shift, _, _ = rand_layer(rng, N, H, W, C, K, 3, 3, pad=(1, 1))
    want = oracle_conv(x, w, bias, shift, R=3, S=3, pad=(1, 1))
    for hints, stores in ((dict(), "tma_store=0"), (dict(tma_store=1), "tma_store=2")):
        with binding.plan_hints(patch_halo=1, **hints):
            conv = binding.QConv(w, bias, shift, N=N, H=H, W=W, C=C, K=K, R=3, S=3, pad_h=1, pad_w=1)
        xd = torch.from_numpy(x).cuda()
        for n in (N, 3, N):
            y = torch.full((N, H, W, K), 77, dtype=torch.int8, device="cuda")
            conv.run(xd, y, n_run=n)
            assert conv.status() == 0 and "patch=1" in conv.describe() and stores in conv.describe(), conv.describe()
            got = y.cpu().numpy()
            assert (got[:n] == want[:n]).all() and (got[n:] == 77).all()
        conv.destroy()
