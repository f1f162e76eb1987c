"""The run of binary hidden layers on CTA pairs (large batches, fan-ins above 2048): 9 to 12 stages of 256 positions, whole and ragged,
an empty partner of an odd last one, rings of weight stages that wrap inside a layer, unit tiles and frame tiles that are cut
off, (0,1) activations; the bits of every layer against those of the kernel that streams the weights."""
import dataclasses

import pytest

from paper_1706_09453_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden,frames,values", [(2305, 9000, 0), (2100, 20000, 1), (2560, 5000, 0), (2900, 16385, 0), (3072, 9001, 1), (2817, 7000, 0)])
def test_pair_run_equals_streamed_layers(hidden, frames, values):
    import torch
    from paper_1706_09453_b200 import build, binding as B, model
    build.build()
    cfg = dataclasses.replace(wl.CONFIGS["tiny"], hidden=hidden, n_hidden=5, classes=64)
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
        for l, (a, b) in enumerate(zip(layers(B.PREPARED_AUTO), want)):
            assert torch.equal(a[:, :words], b[:, :words]), "hidden layer %d" % (l + 1)
    assert B.bnn_device_status() == 0
