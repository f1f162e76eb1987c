"""The forms in which a top layer's weights can be prepared (pairs or single weights, three or four digits), inside a forward pass: the
log-softmax that follows the logits tile by tile counts the tiles of the form that was chosen, and its results are those of a
log-softmax behind the last logit; with double precision beside them."""
import dataclasses

import numpy as np
import pytest

from paper_1706_09453_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weights", ["normal", "uniform", "outlier"])
@pytest.mark.parametrize("hidden,frames,classes", [(1000, 3000, 1801), (2048, 3000, 1804), (2048, 5000, 3307), (700, 400, 2000)])
@pytest.mark.parametrize("values", [0, 1])
def test_log_softmax_follows_every_form(weights, hidden, frames, classes, values):
    import torch
    from paper_1706_09453_b200 import build, binding as B, model
    build.build()
    cfg = dataclasses.replace(wl.CONFIGS["tiny"], hidden=hidden, n_hidden=2, classes=classes)
    net = wl.make_model(cfg)
    rng = np.random.default_rng(hidden + classes)
    if weights == "uniform":          # fill their range evenly, just below a power of two
        net.Wout = rng.uniform(-0.99, 0.99, (classes, hidden)).astype(np.float32) / 32
    elif weights == "outlier":
        net.Wout = np.array(net.Wout)
        net.Wout[:, hidden // 3] *= 1000
    dn = model.DeviceNet(net, act_values=values)
    x = model.to_dev(wl.make_frames(cfg, frames))
    outs = dn.layer_out_buffers(frames)

    def run(follow):
        prev = B.bnn_set_option(B.OPT_SOFTMAX_FOLLOW, follow)
        try:
            return dn.forward(x, layer_out=outs).clone()
        finally:
            B.bnn_set_option(B.OPT_SOFTMAX_FOLLOW, prev)

    got, apart = run(1), run(0)
    bits = outs[-1].cpu().numpy().view(np.uint8)
    a = torch.from_numpy(np.unpackbits(bits, axis=1, bitorder="little")[:, :hidden]).cuda().double()
    z = (a if values else 2 * a - 1) @ torch.from_numpy(np.asarray(net.Wout)).cuda().double().T + torch.from_numpy(np.asarray(net.bout)).cuda().double()
    want = torch.log_softmax(z, 1)
    # a logit's own error (the header's bound, with three digits) and its roundings, twice: once in the normaliser
    bound = 2 * hidden * 1.01 * 2.0 ** -24 * float(np.abs(net.Wout).max()) + 2.0 ** -21 * (want.abs().amax() + z.abs().amax())
    assert float((got.double() - want).abs().max()) <= float(bound)
    assert float((got - apart).abs().max()) <= 2.0 ** -21 * float(want.abs().max())       # the two kernels add a row up in another order
    assert B.bnn_device_status() == 0
