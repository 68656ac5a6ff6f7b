"""The host path of a network pass: an input read where it lies (captured graph pointed at it, or the native step
list) against the oracle, for inputs at every alignment and layout `QNetwork.run` takes."""
import numpy as np
import pytest

from oracle import network_ref
from paper_1805_07941_b200 import binding, workloads as wl

pytestmark = pytest.mark.gpu

NETS = {"s2d": lambda: wl.resnet50(batch=4, res=64, width=16, blocks=(1, 1, 1, 1)),        # stem converts the input
        "rows": lambda: wl.vgg16(batch=4, res=32, widths=(16, 32), reps=(2, 1)),            # padded-row stem converts
        "quantize": lambda: wl.inception(batch=4, res=14, cin=32, blocks=(("3a", 16, 24, 32, 8, 16, 16),))}


@pytest.mark.parametrize("name", sorted(NETS))
def test_input_is_read_where_it_lies(name):
    import torch
    from paper_1805_07941_b200.network import QNetwork
    net = NETS[name]()
    w = {nd["name"]: wl.gen_weights(nd, 0) for nd in net["nodes"] if nd["op"] == "conv"}
    xs = [wl.gen_input(net, seed=s) for s in range(3)]
    params, e_buf, _, _ = network_ref.calibrate(net, xs[0], w)
    want = [network_ref.run(net, x, params, e_buf)[next(reversed(net["nodes"]))["dst"]] for x in xs]
    qn = QNetwork(net, w).load_params(params, e_buf)

    def at_offset(x, floats):                              # the same batch at an address 4 * floats past a 16-byte boundary
        flat = torch.zeros(x.size + 4, dtype=torch.float32, device="cuda")
        t = flat[floats:floats + x.size].view(x.shape)
        t.copy_(torch.from_numpy(x))
        return t

    for form in (None, "chain", "split2"):
        if form:
            qn.capture(form)
            assert qn.graph.inputs.found
        for i in (1, 2, 1):
            layouts = [at_offset(xs[i], 0), at_offset(xs[i], 1), torch.from_numpy(xs[i]).cuda().double(),
                       torch.from_numpy(np.ascontiguousarray(xs[i].transpose(0, 2, 1, 3))).cuda().transpose(1, 2),
                       torch.from_numpy(xs[i])]
            for x in layouts:
                qn.bufs[qn.last].zero_()
                assert (qn.run(x).cpu().numpy() == want[i]).all(), (form, i, x.stride(), x.dtype)
            for n in (1, 3):
                assert (qn.run(layouts[0][:n]).cpu().numpy() == want[i][:n]).all()
        if form:                                           # a plain replay reads x_static again
            qn.x_static.copy_(torch.from_numpy(xs[0]))
            qn.graph.replay()
            assert (qn.bufs[qn.last].cpu().numpy() == want[0]).all()
    qn.check_status()
    qn.destroy()


def test_a_capture_is_a_cuda_graph():
    """What `capture` returns does all that torch's graph does; recorded work and a new executable read x_static."""
    import torch
    from paper_1805_07941_b200.network import QNetwork
    net = NETS["rows"]()
    w = {nd["name"]: wl.gen_weights(nd, 0) for nd in net["nodes"] if nd["op"] == "conv"}
    xs = [wl.gen_input(net, seed=s) for s in range(2)]
    params, e_buf, _, _ = network_ref.calibrate(net, xs[0], w)
    want = [network_ref.run(net, x, params, e_buf)[next(reversed(net["nodes"]))["dst"]] for x in xs]
    qn = QNetwork(net, w).load_params(params, e_buf)
    g = qn.capture("chain")
    assert isinstance(g, torch.cuda.CUDAGraph) and g is qn.graph and len(g.pool()) == 2
    qn.x_static.copy_(torch.from_numpy(xs[0]))
    other = torch.from_numpy(xs[1]).cuda()
    for again in range(2):
        assert (qn.run(other).cpu().numpy() == want[1]).all()
        if again:
            g.instantiate()
        g.replay()
        assert (qn.bufs[qn.last].cpu().numpy() == want[0]).all(), again
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        assert (qn.run(other).cpu().numpy() == want[1]).all()
    g.reset()
    with pytest.raises(RuntimeError):
        g.replay()
    qn.destroy()


def test_step_list_reports_the_first_error():
    steps = binding.Steps([dict(op=binding.NET_MAXPOOL, n=1, H=4, W=4, C=16, R=2, stride=2, pad=0)])
    with pytest.raises(binding.QconvError) as e:
        steps.run(0)
    assert e.value.code == binding.ERR_BAD_ARG
    with pytest.raises(binding.QconvError) as e:
        binding.Steps([dict(op=binding.NET_QUANTIZE, count=16, n_bits=8)]).run(None)
    assert e.value.code == binding.ERR_BAD_ARG


@pytest.mark.parametrize("K,C", [(16, 32), (64, 128), (128, 512), (96, 512), (100, 512)])
def test_handles_of_the_same_weights_share_them_in_any_order_of_destruction(K, C):
    """Below and above the size from which weights have a block of their own; layouts that agree and that do not."""
    import torch
    from oracle import ref
    rng = np.random.default_rng(K)
    x = rng.integers(-128, 128, (2, 6, 5, C), dtype=np.int8)
    w = rng.integers(-8, 8, (K, 3, 3, C), dtype=np.int8)
    acc_exp, shift = np.full(K, -10, np.int32), np.full(K, 9, np.int32)
    geom = dict(N=2, H=6, W=5, C=C, K=K, R=3, S=3, pad_h=1, pad_w=1)
    want_f = ref.qconv(x, w, None, None, None, None, acc_exp, R=3, S=3, pad=(1, 1), out_mode=2)
    want = ref.qconv(x, w, None, shift, R=3, S=3, pad=(1, 1))
    xd = torch.from_numpy(x).cuda()
    for first_gone in (0, 1):
        fl = binding.QConv(w, None, None, None, acc_exp, out_mode=binding.OUT_FLOAT, **geom)
        q8 = binding.QConv(w, None, shift, weights_of=fl, **geom)
        other = binding.QConv(np.zeros_like(w), None, shift, **geom)
        (fl, q8)[first_gone].destroy()
        junk = [binding.QConv(rng.integers(-8, 8, w.shape, dtype=np.int8), None, shift, **geom) for _ in range(3)]   # reuses what was given back
        if first_gone == 0:
            y = torch.empty(want.shape, dtype=torch.int8, device="cuda")
            assert (q8.run(xd, y).cpu().numpy() == want).all(), q8.describe()
        else:
            y = torch.empty(want.shape, dtype=torch.float32, device="cuda")
            assert (fl.run(xd, y).cpu().numpy() == want_f).all(), fl.describe()
        for h in [fl, q8, other] + junk:
            h.destroy()
