"""Host weight conversion (vector form, several layers at once) against the oracle: counts around the vector width,
values at the ends of the range, non-finite weights, exponents outside the vector form's range."""
import os
import subprocess
import sys

import numpy as np
import pytest

from oracle import ref
from paper_1805_07941_b200 import binding


def _weights(rng, shape, scale):
    with np.errstate(over="ignore"):
        w = (rng.standard_normal(shape) * scale).astype(np.float32)
    flat = w.reshape(-1)
    for i, v in enumerate((np.nan, np.inf, -np.inf, 0.0, -0.0)):
        if i + 3 < flat.size:
            flat[i * (flat.size // 5)] = v
    return w


@pytest.mark.parametrize("n", [2, 5, 8])
@pytest.mark.parametrize("scale", [1.0, 1e-3, 3e-38, 1e-44, 1e38])
def test_list_equals_the_oracle_layer_by_layer(n, scale):
    rng = np.random.default_rng(n)
    layers, want = [], []
    for K, R, S, Cg in [(1, 1, 1, 1), (3, 1, 1, 15), (2, 1, 1, 16), (5, 3, 3, 17), (64, 3, 3, 33), (7, 1, 5, 31), (300, 3, 3, 100)]:
        for per_channel in (0, 1):
            w = _weights(rng, (K, R, S, Cg), scale)
            layers.append((w, K, R, S, Cg, per_channel))
            want.append(ref.quantize_weights(w, K=K, R=R, S=S, Cg=Cg, per_channel=per_channel, n=n))
    for (wq, e_w), (wq_ref, e_ref), layer in zip(binding.qquantize_weights_list(layers, n), want, layers):
        assert (e_w == e_ref).all() and (wq == wq_ref.reshape(wq.shape)).all(), layer[1:]


def test_ties_go_to_even():
    w = np.array([127, 0.5, 1.5, 2.5, -0.5, -1.5, -2.5, 126.5, -126.5, 3.5, 63.5, 64.5, 1e-45, -1e-45, 0.49999997, 0.50000006, 7.5],
                 np.float32).reshape(1, 1, 1, 17)
    [(wq, e_w)] = binding.qquantize_weights_list([(w, 1, 1, 1, 17, 1)])
    assert e_w[0] == 0 and (wq.reshape(-1) == np.rint(w.reshape(-1)).astype(np.int8)).all()


@pytest.mark.parametrize("n", [2, 8])
@pytest.mark.parametrize("per_channel", [0, 1])
def test_channels_last_equals_the_oracle(n, per_channel):
    w = _weights(np.random.default_rng(n), (3, 2, 17, 40), 0.3)
    wq, e_w = binding.qquantize_weights(w, 40, 3, 2, 17, layout=1, per_channel=per_channel, n=n)
    wq_ref, e_ref = ref.quantize_weights(w, K=40, R=3, S=2, Cg=17, layout=1, per_channel=per_channel, n=n)
    assert (e_w == e_ref).all() and (wq == wq_ref.reshape(wq.shape)).all()


def test_a_list_that_host_memory_cannot_hold_is_an_error():
    """The bookkeeping of 2^31 - 1 layers under a limit on the address space: an error code, not an exception through the C entry."""
    script = """
import resource
from paper_1805_07941_b200 import binding
jobs, lib = (binding.qweights_job * 1)(), binding.lib()
used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (used + (1 << 30), resource.RLIM_INFINITY))
assert lib.qquantize_weights_list(jobs, 2**31 - 1) == binding.ERR_BAD_ARG, "code"
assert b"2147483647 layers" in lib.qconv_last_error_string()
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    done = subprocess.run([sys.executable, "-c", script], cwd=root, capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, (done.returncode, done.stderr[-2000:])
