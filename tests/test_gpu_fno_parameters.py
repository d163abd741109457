"""The network's outputs belong to the parameters in force: after new parameters, training steps
(direct, and captured and replayed), and a capture that was refused.  A fresh handle with the same
parameters computes the same values (the same kernels on the same operands: equal bits)."""
import ctypes as ct

import numpy as np
import pytest
import torch

from paper_1104_4263_gb300 import die

pytestmark = pytest.mark.gpu
SHAPE = (3, 2, 8, 5, 2, 16, 24, 32, 2)        # c_in, c_out, width, modes, layers, hidden, H, W, batch


def _net(params=None):
    net = die.FNO(*SHAPE)
    if params is not None:
        net.set_params(params)
    return net


def _params(seed):
    return (0.3 * np.random.default_rng(seed).standard_normal(_net().n_params)).astype(np.float32)


def _capture(stream, body):
    """Records body() on the stream through the driver; the graph, or None if it was refused."""
    cu = ct.CDLL("libcuda.so.1")
    st, graph = ct.c_void_p(stream.cuda_stream), ct.c_void_p()
    torch.cuda.synchronize()
    assert cu.cuStreamBeginCapture_v2(st, 1) == 0
    body()
    ok = cu.cuStreamEndCapture(st, ct.byref(graph)) == 0
    return (cu, graph) if ok and graph.value else None


@pytest.mark.parametrize("event", ["set_params", "train_step", "replayed", "refused_first", "refused_later",
                                   "refused_precondition"])
def test_forward_uses_current_parameters(event):
    c_in, c_out, _, _, _, _, H, Wd, B = SHAPE
    g = torch.Generator("cuda").manual_seed(5)
    x = torch.randn((B, c_in, H, Wd), device="cuda", generator=g)
    t = torch.randn((B, c_out, H, Wd), device="cuda", generator=g)
    y = torch.empty_like(t)
    stream = torch.cuda.Stream()
    net = _net(_params(1))
    if event == "refused_precondition":
        net = die.FNO(6, 4, 8, 5, 2, 16, H, Wd, 1)
        p = (0.3 * np.random.default_rng(7).standard_normal(net.n_params)).astype(np.float32)
        net.set_params(p)
        op = die.Operator(np.full((H, Wd), 2.0 + 0.1j), 0.05)
        v = op.plane_wave(0.3)
        z = torch.empty_like(v)

        def refused():
            with pytest.raises(die.DieError):
                net.precondition(op, v, z, stream=stream)
        assert _capture(stream, refused) is None
        other = die.FNO(6, 4, 8, 5, 2, 16, H, Wd, 1)
        other.set_params(p)
        assert torch.equal(net.precondition(op, v), other.precondition(op, v))
        return
    if event != "refused_first":
        net.forward(x)
    if event == "set_params":
        net.set_params(_params(2))
    elif event == "train_step":
        net.train_step(x, t, 1e-2)
    elif event == "replayed":
        def step():
            assert die._lib().fno_train_step(net.handle, B, die._ptr(x), die._ptr(t), 1e-2, None,
                                             ct.c_void_p(stream.cuda_stream)) == 0
        cu, graph = _capture(stream, step)
        ex = ct.c_void_p()
        assert cu.cuGraphInstantiateWithFlags(ct.byref(ex), graph, ct.c_ulonglong(0)) == 0
        net.forward(x)
        before = net.get_params()
        for _ in range(2):
            assert cu.cuGraphLaunch(ex, ct.c_void_p(stream.cuda_stream)) == 0
        stream.synchronize()
        cu.cuGraphExecDestroy(ex)
        cu.cuGraphDestroy(graph)
        assert not np.array_equal(before, net.get_params())
    else:
        if event == "refused_later":
            net.set_params(_params(3))

        def refused():      # a forward pass ends with a synchronisation, which a capture refuses
            with pytest.raises(die.DieError):
                net.forward(x, y, stream=stream)
        assert _capture(stream, refused) is None
    got = net.forward(x)
    assert torch.equal(got, _net(net.get_params()).forward(x))
