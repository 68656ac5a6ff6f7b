"""Device memory that destroyed handles gave back is kept for later ones, but never in the way of a handle that needs it."""
import numpy as np
import pytest

from oracle import ref
from paper_1805_07941_b200 import binding

pytestmark = pytest.mark.gpu


def test_kept_blocks_make_room_on_a_full_device():
    import torch
    rng = np.random.default_rng(0)
    w = rng.integers(-128, 128, (16, 7, 7, 3), dtype=np.int8)
    shift = np.full(16, 12, np.int32)

    def stem(n):                                             # scratch: the images in space-to-depth form
        return binding.QConv(w, None, shift, N=n, H=224, W=224, C=3, K=16, R=7, S=7, stride_h=2, stride_w=2, pad_h=3, pad_w=3)

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    live = stem(1)                                           # (the last handle to go takes what is kept with it)
    torch.cuda.empty_cache()
    before = free()
    small = stem(1000)
    kept = before - free()
    assert 100 << 20 < kept <= 256 << 20
    small.destroy()
    assert before - free() == kept                           # still held
    needed = 5 * kept                                        # (no kept block is large enough for it)
    leave = needed - kept // 2
    filler = torch.empty(free() - leave, dtype=torch.uint8, device="cuda")
    try:
        assert free() < needed
        large = stem(5000)
        x = rng.integers(-128, 128, (1, 224, 224, 3), dtype=np.int8)
        xd, yd = torch.from_numpy(x).cuda(), torch.empty((1, 112, 112, 16), dtype=torch.int8, device="cuda")
        large.run(xd, yd)
        assert large.status() == 0
        got = yd.cpu().numpy()
        large.destroy()
    finally:
        del filler
        torch.cuda.empty_cache()
    assert (got == ref.qconv(x, w, None, shift, R=7, S=7, stride=(2, 2), pad=(3, 3))).all()
    live.destroy()
