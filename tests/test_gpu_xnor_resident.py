"""The run of binary hidden layers with resident weights, over the tile widths it chooses from (by frames and layer
size), even and odd numbers of stages of 256 positions, rings of weight stages that wrap inside a layer, ragged last stages
and tiles: the bits of every layer against those of the kernel that streams the weights, one launch per layer."""
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


@pytest.mark.parametrize("hidden,frames,values", [
    (2048, 33, 0), (2048, 129, 1),       # 32 units a tile
    (2048, 731, 0), (700, 300, 1),       # 96
    (2048, 1100, 0), (3072, 2500, 0),    # 128
    (2048, 5000, 1), (1800, 4500, 0),    # 192
    (200, 4000, 0), (1300, 900, 1), (2300, 200, 0), (1290, 9000, 0),   # 1, 6, 9 and 6 stages, ragged
    (1100, 9000, 1), (1100, 150, 0), (520, 12000, 0),                  # 5 and 3 stages, several frame tiles a block
])
def test_resident_run_equals_streamed_layers(env, hidden, frames, values):
    torch, B, model = env
    cfg = dataclasses.replace(wl.CONFIGS["tiny"], hidden=hidden, n_hidden=6, classes=64)
    dn = model.DeviceNet(wl.make_model(cfg), act_values=values)
    X = model.to_dev(wl.make_frames(cfg, frames))

    def layers(kind):
        prev = B.bnn_set_option(B.OPT_XNOR_PREPARED, kind)
        try:
            outs = dn.layer_out_buffers(frames)
            dn.forward(X, layer_out=outs)
            torch.cuda.synchronize()
            return outs
        finally:
            B.bnn_set_option(B.OPT_XNOR_PREPARED, prev)

    want, words = layers(B.PREPARED_STREAM), (hidden + 31) // 32
    for _ in range(3):
        for l, (a, b) in enumerate(zip(layers(B.PREPARED_RESIDENT), want)):
            assert torch.equal(a[:, :words], b[:, :words]), "hidden layer %d" % (l + 1)
    assert B.bnn_device_status() == 0


@pytest.mark.parametrize("k,n", [(256, 33), (512, 700), (2048, 2048), (3072, 256)])
def test_resident_layer_decides_sums_of_zeros(env, k, n):
    """(0,1) frames without a one on -1 weights: every product is a zero, and the sum 0 meets thresholds around it."""
    torch, B, model = env
    m = 200
    hp = torch.zeros((m, B.packed_pitch(k)), dtype=torch.int32, device="cuda:0")
    wp = torch.zeros((n, B.packed_pitch(k)), dtype=torch.int32, device="cuda:0")
    img = torch.empty(B.bnn_xnor_prepared_bytes(n, k), dtype=torch.uint8, device="cuda:0")
    B.bnn_xnor_prepare(wp, k, img)
    thr = (torch.arange(n, device="cuda:0", dtype=torch.int32) % 3 - 1)
    flip = torch.zeros((n + 31) // 32, dtype=torch.int32, device="cuda:0")
    out = torch.full((m, B.packed_pitch(n)), -1, dtype=torch.int32, device="cuda:0")
    prev = B.bnn_set_option(B.OPT_XNOR_PREPARED, B.PREPARED_RESIDENT)
    try:
        B.bnn_gemm01(hp, None, k, N=n, prepared=img, thr=thr, flip=flip, out_bits=out)
    finally:
        B.bnn_set_option(B.OPT_XNOR_PREPARED, prev)
    bits = (out.unsqueeze(2) >> torch.arange(32, device="cuda:0", dtype=torch.int32)) & 1
    want = (thr <= 0).int().expand(m, n)
    assert torch.equal(bits.reshape(m, -1)[:, :n], want)


@pytest.mark.parametrize("frames", [17, 100, 731, 3000])
def test_several_streams_at_once(env, frames):
    """Runs that do not fit the SMs side by side (32- to 192-unit tiles take 64 to 148 SMs each), on four streams."""
    torch, B, model = env
    cfg = dataclasses.replace(wl.CONFIGS["tiny"], hidden=2048, n_hidden=6, classes=500)
    net = wl.make_model(cfg)
    nets = [model.DeviceNet(net) for _ in range(4)]
    X = model.to_dev(wl.make_frames(cfg, frames))
    want = nets[0].forward(X).clone()
    outs = [torch.empty_like(want) for _ in nets]
    for dn in nets:
        dn.workspace(frames)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in nets]
    for _ in range(30):
        for dn, st, o in zip(nets, streams, outs):
            with torch.cuda.stream(st):
                dn.forward(X, o)
    torch.cuda.synchronize()
    assert all(torch.equal(o, want) for o in outs)
    assert B.bnn_device_status() == 0
