"""First layer with Sign units: a frame's bits do not depend on how many frames are in the batch, whichever width of unit tiles
the batch size selects (one or several turns of the persistent grid; ragged units, fan-ins and frames; spliced input)."""
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


@pytest.mark.parametrize("hidden,in_dim", [(2048, 440), (1000, 31), (129, 1300), (3072, 97), (513, 64)])
@pytest.mark.parametrize("mode", [0, 1])
def test_bits_do_not_depend_on_the_batch(env, hidden, in_dim, mode):
    torch, B, model = env
    cfg = dataclasses.replace(wl.CONFIGS["tiny"], hidden=hidden, in_dim=in_dim, n_hidden=2, classes=64)
    dn = model.DeviceNet(wl.make_model(cfg), mode)
    X = model.to_dev(wl.make_frames(cfg, 9000))
    X[5] = 0.0       # sums that are exactly zero

    def bits(n, at):
        outs = dn.layer_out_buffers(n)
        dn.forward(X[at:at + n], layer_out=outs)
        return outs[0][:, :(hidden + 31) // 32]

    want = bits(9000, 0)
    for n, at in ((17, 0), (128, 100), (731, 0), (1153, 3), (2000, 5), (2400, 1), (4700, 0)):
        assert torch.equal(bits(n, at), want[at:at + n]), n
    assert B.bnn_device_status() == 0
