"""How far sums of byte digits are from double precision: on no kind of row farther (root mean square) than with every number rounded by itself
to the finest power of two at which the row's largest stays within 0x7F7F7F, and one rounding of the sum to fp32.  Rows that fill their
range evenly are the hard ones: a sum of two of their numbers needs a bit more than either."""
import numpy as np
import pytest

from paper_1706_09453_b200 import workloads as wl

pytestmark = pytest.mark.gpu

# The error is a mean over 1e5 to 1e6 sums of K independent roundings, of rows that share the numbers: it varies by about a percent.
MARGIN = 1.03


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available()
    from paper_1706_09453_b200 import build, binding, model
    build.build()
    return torch, binding, model


def rows(torch, kind, m, k):
    g = torch.Generator("cuda:0").manual_seed(m + k)
    u = torch.rand((m, k), generator=g, device="cuda:0")
    sign = torch.where(torch.rand((m, k), generator=g, device="cuda:0") < 0.5, -1.0, 1.0)
    return {"normal": lambda: torch.randn((m, k), generator=g, device="cuda:0"),
            "uniform 0.7": lambda: (2 * u - 1) * 0.7, "uniform 0.99": lambda: (2 * u - 1) * 0.99, "uniform 0.033": lambda: (2 * u - 1) * 0.033,
            "positive": lambda: u, "shell": lambda: (0.9 + 0.1 * u) * 0.99 * sign,
            # one row in four is hard
            "mixed": lambda: torch.where(torch.arange(m, device="cuda:0")[:, None] % 4 == 0, (2 * u - 1) * 0.99, torch.randn((m, k), generator=g, device="cuda:0"))}[kind]()


def powers_of_two(torch, x, top):
    unit = torch.exp2(-torch.floor(torch.log2(0x7F7F7F / top.double())))[:, None]
    return torch.round(x.double() / unit) * unit


def signs(torch, p, k):
    return 2 * torch.from_numpy(np.unpackbits(p.view(np.uint8), axis=1, bitorder="little")[:, :k]).cuda().double() - 1


def rms(x):
    return float(x.square().mean().sqrt())


KINDS = ["normal", "uniform 0.7", "uniform 0.99", "uniform 0.033", "positive", "shell", "mixed"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("h", [440, 2048])
@pytest.mark.parametrize("values", [0, 1])
def test_top_layer(env, kind, h, values):
    torch, B, model = env
    m, c = 500, 1000
    w = rows(torch, kind, c, h)
    hp = wl.make_bit_planes(m, h, 0.5, h, B.packed_pitch(h))
    digits = torch.empty(B.bnn_output_digits_bytes(c, h), dtype=torch.uint8, device="cuda:0")
    B.bnn_output_prepare_digits(w, digits)
    z = torch.empty((m, c), device="cuda:0")
    B.bnn_output_layer_digits(model.to_dev(hp), digits, None, z, h, log_softmax=False, values=values)
    a = signs(torch, hp, h)
    if values:
        a = (a + 1) / 2
    want = a @ w.double().T
    ref = (a @ powers_of_two(torch, w, w.abs().amax(1)).T).float().double()
    assert rms(z.double() - want) <= MARGIN * rms(ref - want)
    assert B.bnn_device_status() == 0


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("k", [440, 2048])
@pytest.mark.parametrize("magnitude", [1.0, 1e-34])
def test_binary_weights(env, kind, k, magnitude):
    torch, B, model = env
    m, n = 1000, 500
    x = rows(torch, kind, m, k) * magnitude
    wp = wl.make_bit_planes(n, k, 0.5, k, B.packed_pitch(k))
    ws = torch.empty(B.bnn_signw_workspace_bytes(m, k), dtype=torch.uint8, device="cuda:0")
    y = torch.empty((m, n), device="cuda:0")
    B.bnn_signw_gemm(x, model.to_dev(wp), k, Y=y, workspace=ws)
    w = signs(torch, wp, k)
    want = x.double() @ w.T
    ref = (powers_of_two(torch, x, x.abs().amax(1)) @ w.T).float().double()
    assert rms((y.double() - want) / magnitude) <= MARGIN * rms((ref - want) / magnitude)
    assert B.bnn_device_status() == 0


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("top", [0.5, 0.8, 0.99, 1.0])
@pytest.mark.parametrize("act", [2, 3])
def test_rows_handed_on(env, kind, top, act):
    """The outputs of a layer, of given magnitudes and a bound on them (of `top`) that is known here: its inputs count for nothing beside its shifts."""
    torch, B, model = env
    m, k, n = 200, 2048, 500
    target = rows(torch, kind, 1, k)[0].abs()
    target = (target / target.max() * top).clamp(max=0.9999 if act == 3 else 1.0, min=1e-3)
    if act == 2:
        target *= torch.where(torch.rand(k, generator=torch.Generator("cuda:0").manual_seed(1), device="cuda:0") < 0.5, -1.0, 1.0)
        shift = target
    else:
        shift = torch.log(target.double() / (1 - target.double())).float()
    front, wp = (wl.make_bit_planes(r, c, 0.5, c, B.packed_pitch(c)) for r, c in ((k, 64), (n, k)))
    scale = torch.full((n,), 1 / 4096, device="cuda:0")
    w3 = torch.randn((3, n), device="cuda:0")
    img = torch.empty(B.bnn_output_prepared_bytes(3, n), dtype=torch.uint8, device="cuda:0")
    B.bnn_output_prepare(w3, img)
    tiny = torch.full((k,), 1e-20, device="cuda:0")
    desc = B.ModelDesc([dict(kind=B.LAYER_SIGNW, K=64, N=k, Wp=model.to_dev(front), scale=tiny, shift=shift, act=act),
                        dict(kind=B.LAYER_SIGNW, K=k, N=n, Wp=model.to_dev(wp), scale=scale, shift=None, act=B.ACT_HARDTANH),
                        dict(kind=B.LAYER_REAL_OUT, K=n, N=3, W=w3, W_prepared=img)])
    x = torch.randn((m, 64), device="cuda:0")
    outs = [torch.empty((m, k), device="cuda:0"), torch.empty((m, n), device="cuda:0")]
    B.bnn_forward(desc, x, torch.empty((m, 3), device="cuda:0"), torch.empty(desc.workspace_bytes(m), dtype=torch.uint8, device="cuda:0"), outs)
    w = signs(torch, wp, k)
    want = outs[0].double() @ w.T / 4096
    most = float(shift.abs().max()) if act == 2 else float(torch.exp(shift.max()))          # Sigmoid(x) < exp(x)
    bound = torch.full((m,), min(1.0, most * 1.0001), dtype=torch.float64, device="cuda:0")
    ref = (powers_of_two(torch, outs[0], bound) @ w.T / 4096).float().double()
    assert float(want.abs().max()) < 1
    # (one row of numbers here, so the mean is over 500 sums of 2048 roundings: 5 % or so)
    assert rms(outs[1].double() - want) <= 1.1 * rms(ref - want)
    assert B.bnn_device_status() == 0


def test_magnitudes_that_add_up_to_infinity(env):
    """The scale of the outputs comes from a bound on the sums; a row of finite numbers whose magnitudes overflow has none below one."""
    torch, B, model = env
    m, k, n = 40, 440, 300
    front, wp = (wl.make_bit_planes(r, c, 0.5, c, B.packed_pitch(c)) for r, c in ((n, k), (n, n)))
    w3 = torch.randn((3, n), device="cuda:0")
    img = torch.empty(B.bnn_output_prepared_bytes(3, n), dtype=torch.uint8, device="cuda:0")
    B.bnn_output_prepare(w3, img)
    small, scale = torch.full((n,), 1.2e-38, device="cuda:0"), torch.full((n,), 1 / 1024, device="cuda:0")
    desc = B.ModelDesc([dict(kind=B.LAYER_SIGNW, K=k, N=n, Wp=model.to_dev(front), scale=small, shift=None, act=B.ACT_HARDTANH),
                        dict(kind=B.LAYER_SIGNW, K=n, N=n, Wp=model.to_dev(wp), scale=scale, shift=None, act=B.ACT_HARDTANH),
                        dict(kind=B.LAYER_REAL_OUT, K=n, N=3, W=w3, W_prepared=img)])
    x = (0.5 + torch.rand((m, k), generator=torch.Generator("cuda:0").manual_seed(3), device="cuda:0")) * 1e37
    outs = [torch.empty((m, n), device="cuda:0") for _ in range(2)]
    B.bnn_forward(desc, x, torch.empty((m, 3), device="cuda:0"), torch.empty(desc.workspace_bytes(m), dtype=torch.uint8, device="cuda:0"), outs)
    assert bool(x.abs().sum(1).isinf().all())
    want = (x.double() @ signs(torch, front, k).T * small.double()).clamp(-1, 1)
    assert float(want.abs().max()) > 0.5 and float((outs[0].double() - want).abs().max()) < 1e-5
    want = outs[0].double() @ signs(torch, wp, n).T / 1024
    # half a unit per value, 1.01 * 2^-23 of one at most
    assert float((outs[1].double() - want).abs().max()) < n / 1024 * 1.01 * 2.0 ** -23 + 2.0 ** -22
    assert B.bnn_device_status() == 0
