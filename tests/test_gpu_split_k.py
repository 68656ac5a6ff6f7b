"""The split contraction (a cluster of CTAs per tile) against the oracle, forced through the plan hint and as the launch
chooses it: flat, strided, box and halo forms, ragged pixel counts, uneven stage counts, channel tiles with dead groups,
with and without a residual, per-layer and per-channel shifts, both roundings' epilogues, partial batches."""
import numpy as np
import pytest

from tests.helpers import oracle_conv, rand_layer

pytestmark = pytest.mark.gpu

CASES = [  # N, n_run, H, W, C, K, R, stride
    (1, 1, 7, 7, 512, 512, 3, 1), (1, 1, 7, 7, 2048, 512, 1, 1), (2, 1, 14, 14, 256, 256, 3, 1), (1, 1, 14, 14, 1024, 256, 1, 1),
    (1, 1, 9, 5, 640, 80, 1, 1), (1, 1, 14, 14, 512, 1024, 1, 2), (3, 2, 5, 5, 256, 48, 5, 1), (1, 1, 3, 3, 896, 208, 3, 2),
    (64, 33, 1, 1, 2048, 1008, 1, 1), (1, 1, 28, 28, 128, 128, 3, 1), (1, 1, 40, 30, 1152, 128, 1, 1)]
# CTAs that share a tile, forced to 2 and 4 and as the launch chooses: 1 where the column groups (3 of them) or the stages (3)
# do not divide, or where the clusters would fill the chip.
SPLITS = dict(zip(CASES, [(2, 4, 4), (2, 4, 4), (2, 4, 4), (2, 4, 4), (1, 1, 1), (2, 4, 1), (1, 1, 1), (2, 4, 4), (2, 4, 4), (2, 1, 1), (2, 4, 2)]))


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("split", [2, 4, -1, 0])
def test_split_contraction_matches_the_oracle(case, split):
    import torch
    from paper_1805_07941_b200 import binding
    N, n_run, H, W, C, K, R, stride = case
    pad = (R // 2, R // 2)
    for with_res in (0, 1):
        for uniform in (0, 1):
            for small in (0, 1):                             # small weights: the float-rounding epilogue
                rng = np.random.default_rng(sum(case) + 2 * with_res + uniform)
                x, w, bias, shift, res, t = rand_layer(rng, N, H, W, C, K, R, R, with_res=bool(with_res), stride=(stride, stride), pad=pad,
                                                       per_channel_shift=not uniform)
                if with_res and uniform:
                    t = np.full(K, int(t[0]), np.int32)
                if small:
                    w = (w // 64).astype(np.int8)
                    shift = np.maximum(shift - 6, 0).astype(np.int32)
                    t = np.minimum(t, 5).astype(np.int32) if with_res else None
                kw = dict(R=R, S=R, stride=(stride, stride), pad=pad, relu=with_res)
                want = oracle_conv(x[:n_run], w, bias, shift, None if res is None else res[:n_run], t, **kw)
                with binding.plan_hints(split_k=split):
                    conv = binding.QConv(w, bias, shift, t, None, N=N, H=H, W=W, C=C, K=K, R=R, S=R, stride_h=stride, stride_w=stride,
                                         pad_h=pad[0], pad_w=pad[1], relu=with_res, has_residual=with_res)
                y = torch.full((N, conv.P, conv.Q, K), 77, dtype=torch.int8, device="cuda")
                rd = torch.from_numpy(res).cuda() if with_res else None
                for _ in range(2):
                    conv.run(torch.from_numpy(x).cuda(), y, rd, n_run=n_run)
                assert conv.status() == 0, conv.describe()
                ran = dict(zip((2, 4, -1, 0), SPLITS[case] + (1,)))[split]
                assert ("split=%d" % ran in conv.describe()) if ran > 1 else ("split=" not in conv.describe()), conv.describe()
                got = y.cpu().numpy()
                assert (got[:n_run] == want).all() and (got[n_run:] == 77).all(), (conv.describe(), with_res, uniform, small)
                conv.destroy()


def test_expired_waits_leave_the_cluster_together():
    """Every wait gives up at once: all CTAs of a cluster still meet at its barrier, the status is reported, and the next run
    is right."""
    import torch
    from oracle import ref
    from paper_1805_07941_b200 import binding
    rng = np.random.default_rng(5)
    x, w, bias, shift, _, _ = rand_layer(rng, 1, 7, 7, 512, 128, 3, 3, pad=(1, 1))
    with binding.plan_hints(split_k=4):
        conv = binding.QConv(w, bias, shift, N=1, H=7, W=7, C=512, K=128, R=3, S=3, pad_h=1, pad_w=1)
    xd = torch.from_numpy(x).cuda()
    y = torch.empty((1, 7, 7, 128), dtype=torch.int8, device="cuda")
    conv.set_wait_limit(0)
    conv.run(xd, y)
    assert conv.status() == binding.ERR_TIMEOUT and "split=4" in conv.describe()
    conv.set_wait_limit(1 << 22)
    conv.run(xd, y)
    assert conv.status() == 0
    assert (y.cpu().numpy() == ref.qconv(x, w, bias, shift, R=3, S=3, pad=(1, 1))).all()
