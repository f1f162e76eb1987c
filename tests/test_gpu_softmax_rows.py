"""Log-softmax of rows that start anywhere in a 16-byte chunk, over widths around what the kernels hold in registers, alone and
following the top layer's kernel, against double precision."""
import dataclasses

import numpy as np
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


def check(got, z, prior):
    """Two roundings of results of magnitude up to |z| + lse, and a sum of exponentials good to 2^-20."""
    zd = z.astype(np.float64)
    mx = zd.max(1, keepdims=True)
    lse = mx + np.log(np.exp(zd - mx).sum(1, keepdims=True))
    want = zd - lse - (0.0 if prior is None else prior.astype(np.float64))
    bound = 2.0 ** -20 + 2.0 ** -22 * (np.abs(zd) + np.abs(lse) + np.abs(want))
    assert (np.abs(got - want) <= bound).all(), (np.abs(got - want) / bound).max()


@pytest.mark.parametrize("c", [1, 2, 3, 5, 129, 2047, 2049, 3307, 4093, 4095, 4097])
@pytest.mark.parametrize("m,extra,shift", [(1, 0, 0), (7, 1, 3), (1300, 2, 1)])
def test_rows_anywhere(env, c, m, extra, shift):
    torch, B, model = env
    h, pitch = 32, c + extra
    rng = np.random.default_rng(c + m)
    w, b = rng.normal(0, 1, (c, h)).astype(np.float32), rng.normal(0, 1, c).astype(np.float32)
    hp = model.to_dev(wl.make_bit_planes(m, h, 0.5, c, B.packed_pitch(h)))
    digits = torch.empty(B.bnn_output_digits_bytes(c, h), dtype=torch.uint8, device="cuda:0")
    B.bnn_output_prepare_digits(model.to_dev(w), digits)
    flat = torch.full((2, m * pitch + 8), 9.0, dtype=torch.float32, device="cuda:0")
    for i in (0, 1):
        view = flat[i, shift:shift + m * pitch].view(m, pitch)[:, :c]
        B.bnn_output_layer_digits(hp, digits, model.to_dev(b), view, h, log_softmax=bool(i))
    z, got = (flat[i, shift:shift + m * pitch].view(m, pitch).cpu().numpy() for i in (0, 1))
    check(got[:, :c], z[:, :c], None)
    np.testing.assert_array_equal(got[:, c:], 9.0)
    assert bool((flat[1, :shift] == 9.0).all()) and bool((flat[1, shift + m * pitch:] == 9.0).all())


@pytest.mark.parametrize("frames,classes,prior", [(2100, 3401, True), (4700, 2045, False), (2561, 4095, True)])
def test_rows_following(env, frames, classes, prior):
    torch, B, model = env
    cfg = dataclasses.replace(wl.CONFIGS["tiny"], hidden=256, n_hidden=2, classes=classes)
    rng = np.random.default_rng(frames)
    pr = np.log(rng.dirichlet(np.ones(classes) * 5.0)).astype(np.float32) if prior else None
    dn = model.DeviceNet(wl.make_model(cfg), log_prior=pr)
    outs = dn.layer_out_buffers(frames)
    got = dn.forward(model.to_dev(wl.make_frames(cfg, frames)), layer_out=outs).clone()
    z = torch.empty((frames, classes), dtype=torch.float32, device="cuda:0")
    B.bnn_output_layer_digits(outs[1], dn.Wout_digits, dn.bout, z, cfg.hidden, log_softmax=False)
    check(got.cpu().numpy(), z.cpu().numpy(), pr)
    assert B.bnn_device_status() == 0
