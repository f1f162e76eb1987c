"""Signs times numbers as byte digits: the top layer's as signs times sums and differences of pairs (2:4 sparse products), and layers with
binary weights, whose numbers stand by themselves, at the sizes where the layout of the digits can go wrong: fan-ins that end inside a pair, a word, a group of 64 or a stage of 256 positions, in
tiles of every width; and pairs whose sums are the largest numbers of their rows."""
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


FAN_INS = [15, 16, 17, 32, 47, 48, 64, 65, 95, 96, 128, 160, 176, 192, 224, 255, 256, 288, 320, 352, 511]


def signs(torch, p, k):
    return 2 * torch.from_numpy(np.unpackbits(p.view(np.uint8), axis=1, bitorder="little")[:, :k]).cuda().double() - 1


# (frames, classes): one turn of narrow, middle and wide tiles, and several of wide ones with a ragged end
@pytest.mark.parametrize("m,c", [(9, 100), (700, 520), (2600, 1000), (5000, 1090)])
@pytest.mark.parametrize("outlier", [False, True])
def test_top_layer_fan_ins(env, m, c, outlier):
    torch, B, model = env
    for h in FAN_INS:
        rng = np.random.default_rng(h + m)
        hp = wl.make_bit_planes(m, h, 0.5, 3 + h, B.packed_pitch(h))
        w = rng.normal(0, 1, (c, h)).astype(np.float32)
        w[0, 0] = 5.0
        w[0, min(16, h - 1)] = 5.0                   # a pair whose sum is twice the largest weight, and one whose difference is
        w[1, 0], w[1, min(16, h - 1)] = -6.0, 6.0
        if outlier:
            w[2] *= np.float32(1e-6)
            w[2, h // 2] = 1.0                       # four digits where h > 16
        wd, a = model.to_dev(w), signs(torch, hp, h)
        digits = torch.full((B.bnn_output_digits_bytes(c, h),), 255, dtype=torch.uint8, device="cuda:0")
        B.bnn_output_prepare_digits(wd, digits)
        four = bool((h * np.abs(w).max(1) > 16 * np.abs(w).sum(1)).any())
        for zo in (0, 1):
            z = torch.full((m, c), 9.0, device="cuda:0")
            B.bnn_output_layer_digits(model.to_dev(hp), digits, None, z, h, log_softmax=False, values=zo)
            want = (a if not zo else (a + 1) / 2) @ wd.double().T
            # half a unit per pair, whose scale lets twice the largest weight fit into 0x7F7F7F (2e9, a power of two, with four
            # digits); two roundings of the result
            bound = (h + 16) / 2 * wd.abs().amax(1).double() * (2 / 2e9 if four else 1.0001 / 0x7F7F7F) + 2.0 ** -23 * want.abs()
            err = (z.double() - want).abs()
            assert bool((err <= bound).all()), (h, zo, float((err / bound).max()))
    assert B.bnn_device_status() == 0


@pytest.mark.parametrize("m,n", [(9, 100), (300, 520), (1500, 1000), (4000, 1100)])
def test_binary_weights_fan_ins(env, m, n):
    """A layer on fp32 rows, then the same inputs handed on as digits by a layer in front of it."""
    torch, B, model = env
    g = torch.Generator("cuda:0").manual_seed(m)
    for k in FAN_INS:
        x = torch.randn((m, k), generator=g, device="cuda:0")
        x[0] = 1.0                                   # every pair's sum is the largest
        x[1, ::2], x[1, 1::2] = 1e-30, -1e-30        # far below 1
        wp = wl.make_bit_planes(n, k, 0.5, 5 + k, B.packed_pitch(k))
        w = signs(torch, wp, k)
        ws = torch.full((B.bnn_signw_workspace_bytes(m, k),), 255, dtype=torch.uint8, device="cuda:0")
        y = torch.empty((m, n), device="cuda:0")
        B.bnn_signw_gemm(x, model.to_dev(wp), k, Y=y, workspace=ws)
        want = x.double() @ w.T
        bound = (k + 16) / 2 * 1.0001 * x.abs().amax(1).double()[:, None] / 0x7F7F7F + 2.0 ** -22 * want.abs()
        assert bool(((y.double() - want).abs() <= bound).all()), k
        # k units in front, so that the digits of k outputs are written by an epilogue
        sc = torch.full((n,), 0.5, device="cuda:0")
        front = wl.make_bit_planes(k, 64, 0.5, 6, B.packed_pitch(64))
        fsc = torch.full((k,), 0.05, device="cuda:0")
        img = torch.empty(B.bnn_output_prepared_bytes(3, n), dtype=torch.uint8, device="cuda:0")
        wout = torch.randn((3, n), generator=g, device="cuda:0")
        B.bnn_output_prepare(wout, img)
        desc = B.ModelDesc([dict(kind=B.LAYER_SIGNW, K=64, N=k, Wp=model.to_dev(front), scale=fsc, shift=None, act=B.ACT_HARDTANH),
                            dict(kind=B.LAYER_SIGNW, K=k, N=n, Wp=model.to_dev(wp), scale=sc, shift=None, act=B.ACT_HARDTANH),
                            dict(kind=B.LAYER_REAL_OUT, K=n, N=3, W=wout, W_prepared=img)])
        x0 = torch.randn((m, 64), generator=g, device="cuda:0")
        outs = [torch.empty((m, k), device="cuda:0"), torch.empty((m, n), device="cuda:0")]
        B.bnn_forward(desc, x0, torch.empty((m, 3), device="cuda:0"), torch.empty(desc.workspace_bytes(m), dtype=torch.uint8, device="cuda:0"), outs)
        dot = outs[0].double() @ w.T
        # outputs of a hardtanh are written in units of 2^-22 at most
        bound = 0.5 * ((k + 16) / 2 * 128 / 127 * 2.0 ** -22 / 1.0 + 2.0 ** -22 * dot.abs()) + 2.0 ** -23
        err = (outs[1].double() - (0.5 * dot).clamp(-1, 1)).abs()
        assert bool((err <= bound).all()), (k, float((err / bound).max()))
    assert B.bnn_device_status() == 0
