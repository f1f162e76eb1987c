"""A handful of frames: the run of hidden layers as one launch and the kernels around it, on unit counts that are no multiple of
a block's, rows longer than what a lane holds ahead, more layers than one launch takes; every layer's bits against the
popcount kernel fed with the layer before, several streams at once, and a captured graph replayed."""
import dataclasses

import pytest

from paper_1706_09453_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available()
    from paper_1706_09453_b200 import build, binding, model
    build.build()
    return torch, binding, model


@pytest.mark.parametrize("hidden,n_hidden,values", [(17, 3, 0), (700, 4, 1), (1000, 12, 0), (2048, 6, 0), (4200, 3, 1), (4800, 3, 0)])
@pytest.mark.parametrize("frames", [1, 2, 4, 5, 16])
def test_hidden_bits(env, hidden, n_hidden, values, frames):
    torch, B, model = env
    cfg = dataclasses.replace(wl.CONFIGS["tiny"], hidden=hidden, n_hidden=n_hidden, classes=70)
    dn = model.DeviceNet(wl.make_model(cfg), act_values=values, prepare_xnor=False)
    X = model.to_dev(wl.make_frames(cfg, frames))
    outs = dn.layer_out_buffers(frames)
    logp = dn.forward(X, layer_out=outs).clone()
    words = (hidden + 31) // 32
    prev = B.bnn_set_option(B.OPT_XNOR_PATH, B.XNOR_POPC)
    try:
        for l in range(1, n_hidden):
            want = torch.zeros_like(outs[l])
            if values:
                B.bnn_gemm01(outs[l - 1], dn.Wp[l], hidden, thr=dn.thr[l], flip=dn.flip[l], out_bits=want)
            else:
                B.bnn_xnor_gemm(outs[l - 1], dn.Wp[l], hidden, thr=dn.thr[l], flip=dn.flip[l], out_bits=want)
            assert torch.equal(outs[l][:, :words], want[:, :words]), "hidden layer %d" % (l + 1)
    finally:
        B.bnn_set_option(B.OPT_XNOR_PATH, prev)
    prev = B.bnn_set_option(B.OPT_XNOR_STACK, 0)
    try:
        assert torch.equal(dn.forward(X), logp)
    finally:
        B.bnn_set_option(B.OPT_XNOR_STACK, prev)
    assert B.bnn_device_status() == 0


def test_streams_and_graph(env):
    torch, B, model = env
    cfg = dataclasses.replace(wl.CONFIGS["tiny"], hidden=2048, n_hidden=6, classes=500)
    net = wl.make_model(cfg)
    nets = [model.DeviceNet(net) for _ in range(4)]
    X = model.to_dev(wl.make_frames(cfg, 4))
    want = nets[0].forward(X).clone()
    outs = [torch.empty_like(want) for _ in nets]
    for dn in nets:
        dn.workspace(4)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in nets]
    for _ in range(50):
        for dn, st, o in zip(nets, streams, outs):
            with torch.cuda.stream(st):
                dn.forward(X, o)
    torch.cuda.synchronize()
    assert all(torch.equal(o, want) for o in outs)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        nets[0].forward(X, outs[0])
    outs[0].zero_()
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(outs[0], want)
    assert B.bnn_device_status() == 0
