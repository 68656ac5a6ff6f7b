"""Staged output tiles of every width (the lean epilogue) against the oracle: channel tiles of 16 to 128 columns in every form
of the tensor-core kernel, tiles staged beside the ring, in it (one tile to a CTA) and stored directly, with the switch by the
batch of a run, residuals in registers and staged, windows of a wider tensor, per-layer and per-channel constants, and the
integer epilogue."""
import numpy as np
import pytest

from tests.helpers import oracle_conv, rand_layer

pytestmark = pytest.mark.gpu

# N, n_runs, H, W, C, K, R, stride: the second batch gives every CTA one tile where the first does not
CASES = [(9, (9, 1), 40, 40, 96, k, 1, 1) for k in (16, 32, 48, 80, 96, 112, 144, 224)] + [
    (3, (3, 1), 14, 14, 1024, 96, 1, 1), (2, (2, 1), 7, 7, 512, 2048, 1, 1), (40, (40, 2), 28, 28, 64, 80, 3, 1), (33, (33, 1), 28, 28, 128, 48, 3, 1),
    (3, (3, 2), 14, 14, 160, 112, 3, 1), (2, (2, 1), 7, 7, 256, 64, 3, 1), (4, (4, 1), 9, 5, 48, 176, 5, 1), (30, (30, 3), 31, 17, 64, 208, 1, 2),
    (2, (2, 1), 13, 11, 80, 240, 3, 2), (3, (3, 1), 12, 20, 16, 16, 3, 1)]


@pytest.mark.parametrize("case", CASES)
def test_staged_tiles_of_any_width_match_the_oracle(case):
    import torch
    from paper_1805_07941_b200 import binding
    N, n_runs, H, W, C, K, R, stride = case
    for with_res, uniform, small, window in ((0, 0, 1, 0), (0, 1, 1, 1), (1, 0, 1, 0), (1, 1, 0, 0), (0, 1, 0, 0), (1, 0, 0, 0), (1, 0, 0, 1)):
        rng = np.random.default_rng(N + H + K + with_res + 2 * uniform)
        x, w, bias, shift, res, t = rand_layer(rng, N, H, W, C, K, R, R, with_res=bool(with_res), stride=(stride, stride), pad=(R // 2, R // 2),
                                               per_channel_shift=not uniform)
        if with_res and uniform:
            t = np.full(K, int(t[0]), np.int32)
        if small:                                            # small weights: the float-rounding epilogue
            w = (w // 64).astype(np.int8)
            shift = np.maximum(shift - 6, 1).astype(np.int32)
            t = np.minimum(t, 5).astype(np.int32) if with_res else None
        kw = dict(R=R, S=R, stride=(stride, stride), pad=(R // 2, R // 2), relu=uniform)
        off, pitch = (16, K + 48) if window else (0, K)
        want = oracle_conv(x, w, bias, shift, res, t, **kw)
        xd, rd = torch.from_numpy(x).cuda(), None if res is None else torch.from_numpy(res).cuda()
        for hints in (dict(), dict(tma_store=0), dict(tma_store=1), dict(tma_residual=0), dict(halo=0, patch_halo=0), dict(halo=1)):
            with binding.plan_hints(split_k=0, **hints):
                conv = binding.QConv(w, bias, shift, t, None, N=N, H=H, W=W, C=C, K=K, R=R, S=R, stride_h=stride, stride_w=stride, pad_h=R // 2,
                                     pad_w=R // 2, relu=uniform, has_residual=with_res, out_c_offset=off, out_c_pitch=pitch)
            for n in n_runs + n_runs[:1]:
                y = torch.full((N, conv.P, conv.Q, pitch), 77, dtype=torch.int8, device="cuda")
                conv.run(xd, y, rd, n_run=n)
                assert conv.status() == 0, conv.describe()
                got = y.cpu().numpy()
                assert (got[:n, :, :, off:off + K] == want[:n]).all(), (conv.describe(), hints, n)
                assert (got[n:] == 77).all() and (got[..., :off] == 77).all() and (got[..., off + K:] == 77).all(), (conv.describe(), hints, n)
            conv.destroy()


# N, H, W, C, K, residual, {images in a run: whether its tiles are staged in the ring}: no room for staged tiles in the plan, one tile to
# a CTA, and more than a third of the SMs in tiles
RING = [(32, 28, 28, 512, 128, 0, {32: 1, 8: 0, 9: 1}), (32, 7, 7, 512, 2048, 1, {32: 1, 5: 0, 9: 1}), (32, 14, 14, 1024, 256, 0, {32: 1, 6: 0, 12: 1}),
        (70, 28, 28, 512, 128, 0, {70: 0, 32: 1, 3: 0}), (25, 13, 11, 736, 1024, 0, {25: 1, 2: 0})]


@pytest.mark.parametrize("case", RING)
@pytest.mark.parametrize("uniform", [0, 1])
def test_tiles_staged_in_the_ring_match_the_oracle(case, uniform):
    """... with the switch between ring and direct stores by the batch, both conversions, a window of a wider tensor, and a wait that
    expires: nothing is staged over operands still on their way, the status says so, and the next run is right."""
    import torch
    from paper_1805_07941_b200 import binding
    N, H, W, C, K, with_res, runs = case
    for small, window in ((0, 0), (1, 0), (1, 1)):
        rng = np.random.default_rng(N + K + uniform)
        x, w, bias, shift, res, t = rand_layer(rng, N, H, W, C, K, 1, 1, with_res=bool(with_res), per_channel_shift=not uniform)
        if small:                                            # the float-rounding epilogue
            w, shift = (w // 64).astype(np.int8), np.maximum(shift - 6, 1).astype(np.int32)
            t = np.minimum(t, 5).astype(np.int32) if with_res else None
        if with_res and uniform:
            t = np.full(K, int(t[0]), np.int32)
        off, pitch = (16, K + 48) if window else (0, K)
        want = oracle_conv(x, w, bias, shift, res, t, R=1, S=1, relu=uniform)
        conv = binding.QConv(w, bias, shift, t, None, N=N, H=H, W=W, C=C, K=K, R=1, S=1, relu=uniform, has_residual=with_res, out_c_offset=off,
                             out_c_pitch=pitch)
        xd, rd = torch.from_numpy(x).cuda(), None if res is None else torch.from_numpy(res).cuda()
        y = torch.empty((N, H, W, pitch), dtype=torch.int8, device="cuda")
        for n in list(runs) + list(runs)[:1]:
            y.fill_(77)
            conv.run(xd, y, rd, n_run=n)
            assert conv.status() == 0 and ("ring=1" in conv.describe()) == bool(runs[n]), (conv.describe(), n)
            got = y.cpu().numpy()
            assert (got[:n, :, :, off:off + K] == want[:n]).all(), (conv.describe(), n)
            assert (got[n:] == 77).all() and (got[..., :off] == 77).all() and (got[..., off + K:] == 77).all(), (conv.describe(), n)
        for n in [n for n in runs if runs[n]]:
            conv.set_wait_limit(0)
            conv.run(xd, y, rd, n_run=n)
            assert conv.status() == binding.ERR_TIMEOUT and "ring=1" in conv.describe()
            conv.set_wait_limit(1 << 22)
            conv.run(xd, y, rd, n_run=n)
            assert conv.status() == 0 and (y.cpu().numpy()[:n, :, :, off:off + K] == want[:n]).all()
        conv.destroy()


def test_an_expired_wait_with_direct_stores():
    """A wait that gives up reports its status, and the next run of the same handle is right."""
    import torch
    from paper_1805_07941_b200 import binding
    rng = np.random.default_rng(5)
    x, w, bias, shift, _, _ = rand_layer(rng, 2, 7, 7, 1024, 96, 1, 1)
    with binding.plan_hints(split_k=0):
        conv = binding.QConv(w, bias, shift, N=2, H=7, W=7, C=1024, K=96, R=1, S=1)
    xd, y = torch.from_numpy(x).cuda(), torch.empty((2, 7, 7, 96), dtype=torch.int8, device="cuda")
    conv.set_wait_limit(0)
    conv.run(xd, y)
    assert conv.status() == binding.ERR_TIMEOUT
    conv.set_wait_limit(1 << 22)
    conv.run(xd, y)
    assert conv.status() == 0 and (y.cpu().numpy() == oracle_conv(x, w, bias, shift, R=1, S=1)).all()
