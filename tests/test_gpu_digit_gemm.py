"""Products of packed signs with real-valued rows as exact integer products of byte digits, at the sizes where the
kernels can go wrong: edges of the 256-row x 64- (or 32-) column tiles, fan-ins around 32 / 128 / 256 positions, one
row, several turns of the persistent grid, and rows that need a fourth digit."""
import numpy as np
import pytest

from oracle import bnn_oracle as o
from paper_1706_09453_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available()
    from paper_1706_09453_b200 import build, binding, model
    build.build()
    return torch, binding, model


@pytest.mark.parametrize("m,h,c", [(1, 1, 1), (1, 32, 33), (255, 127, 63), (256, 128, 64), (257, 129, 65), (128, 255, 31),
                                   (129, 257, 97), (40, 2048, 3307), (2100, 300, 700), (513, 31, 193)])
@pytest.mark.parametrize("outlier", [False, True])
@pytest.mark.parametrize("values", [0, 1])
def test_output_layer_digits(env, m, h, c, outlier, values):
    torch, B, model = env
    rng = np.random.default_rng(1000 * m + h + c)
    hp = wl.make_bit_planes(m, h, 0.5, 7 + m + h, B.packed_pitch(h))
    w = rng.normal(0, 1 / np.sqrt(h), (c, h)).astype(np.float32)
    if outlier:      # one weight dwarfs the rest of its row: three digits would lose them
        w[c // 2] *= np.float32(1e-5)
        w[c // 2, h // 3] = 1.0
    b = rng.normal(0, 0.1, c).astype(np.float32)
    digits = torch.full((B.bnn_output_digits_bytes(c, h),), 255, dtype=torch.uint8, device="cuda:0")
    B.bnn_output_prepare_digits(model.to_dev(w), digits)
    z = torch.full((m, c + 1), 9.0, dtype=torch.float32, device="cuda:0")
    B.bnn_output_layer_digits(model.to_dev(hp), digits, model.to_dev(b), z[:, :c], h, log_softmax=False, values=values)
    a = np.unpackbits(hp.view(np.uint8), axis=1, bitorder="little")[:, :h].astype(np.float64)
    want = (a if values else 2 * a - 1) @ w.astype(np.float64).T + b
    # every weight is off by at most half a unit of its row's fixed-point scale: 2^-22 of the largest weight when three
    # digits are taken (the library's criterion; the scale may lose a bit to the power of two), 2^-30 with four;
    # then two roundings of the result and one of the bias addition
    mx, sm = np.abs(w).max(1).astype(np.float64), np.abs(w).sum(1, dtype=np.float64)
    four = bool((h * mx > 16 * sm).any())
    assert four or not outlier or h < 64
    bound = h * mx * (2.0 ** -30 if four else 2.0 ** -22) / 2 + 3 * 2.0 ** -24 * (np.abs(want) + np.abs(b))
    got = z.cpu().numpy()
    assert (np.abs(got[:, :c] - want) <= bound).all(), (np.abs(got[:, :c] - want) / bound).max()
    np.testing.assert_array_equal(got[:, c], 9.0)
    assert B.bnn_device_status() == 0


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (8, 33, 31), (7, 255, 32), (63, 256, 127), (64, 257, 128), (65, 31, 129),
                                   (9, 300, 257), (33, 2048, 440), (300, 129, 1300), (1100, 520, 96)])
@pytest.mark.parametrize("act", [0, 2, 3])
def test_signw_gemm_digits(env, m, n, k, act):
    torch, B, model = env
    rng = np.random.default_rng(m + 10 * n + 100 * k)
    x = (rng.standard_normal((m, k)) * 10.0 ** rng.uniform(-3, 3, (m, 1))).astype(np.float32)
    x[m // 2, k // 2] = 1e-30                      # far below its row's scale
    wp = wl.make_bit_planes(n, k, 0.5, 3 + m + n, B.packed_pitch(k))
    sc = rng.uniform(-1.5, 1.5, n).astype(np.float32)
    sh = rng.normal(0, 0.1, n).astype(np.float32)
    ws = torch.full((B.bnn_signw_workspace_bytes(m, k),), 255, dtype=torch.uint8, device="cuda:0")
    y = torch.full((m, n + 1), 9.0, dtype=torch.float32, device="cuda:0")
    B.bnn_signw_gemm(model.to_dev(x), model.to_dev(wp), k, Y=y[:, :n], act=act, scale=model.to_dev(sc), shift=model.to_dev(sh),
                     workspace=ws)
    ref, _ = o.signw_gemm(x, wp, k)
    mx = np.abs(x).max(1).astype(np.float64)[:, None]
    pre = sc.astype(np.float64) * ref + sh
    # every value is off by at most half a unit of its row's fixed-point scale (2^-22 of the largest); the sum, the
    # scale and the affine round once each
    bound = np.abs(sc) * (k * mx * 2.0 ** -22 / 2 + 2.0 ** -23 * np.abs(ref)) + 2.0 ** -23 * (np.abs(pre) + np.abs(sh))
    got = y.cpu().numpy()
    np.testing.assert_array_equal(got[:, n], 9.0)
    if act == B.ACT_HARDTANH:
        pre = np.clip(pre, -1, 1)
    elif act == B.ACT_SIGMOID:
        with np.errstate(over="ignore"):
            pre, bound = 1 / (1 + np.exp(-pre)), bound / 4 + 2e-7
    assert (np.abs(got[:, :n] - pre) <= bound).all(), (np.abs(got[:, :n] - pre) / bound).max()
    assert B.bnn_device_status() == 0


def test_signw_gemm_digits_rows_with_infinities_and_nans(env):
    """Such a row gives NaN everywhere; its neighbours are untouched."""
    torch, B, model = env
    m, n, k = 20, 70, 50
    rng = np.random.default_rng(5)
    x = rng.standard_normal((m, k)).astype(np.float32)
    clean = x.copy()
    x[3, 7], x[11, 0] = np.inf, np.nan
    wp = wl.make_bit_planes(n, k, 0.5, 8, B.packed_pitch(k))
    out = []
    for a in (clean, x):
        ws = torch.empty(B.bnn_signw_workspace_bytes(m, k), dtype=torch.uint8, device="cuda:0")
        y = torch.empty((m, n), dtype=torch.float32, device="cuda:0")
        B.bnn_signw_gemm(model.to_dev(a), model.to_dev(wp), k, Y=y, workspace=ws)
        out.append(y.cpu().numpy())
    bad = np.zeros(m, bool)
    bad[[3, 11]] = True
    np.testing.assert_array_equal(out[0][~bad], out[1][~bad])
    assert np.isnan(out[1][bad]).all()


# Several turns of the persistent grid on wide tiles with an odd number of 256-position stages per tile, where the two issuing
# warps change places from tile to tile and the two slots of widened bits with them; the last stage short or whole.
@pytest.mark.parametrize("m,h,c", [(8192, 1100, 3400), (6000, 520, 2000), (8192, 2100, 1500), (4096, 768, 3307)])
@pytest.mark.parametrize("outlier", [False, True])
@pytest.mark.parametrize("values", [0, 1])
def test_output_layer_digits_many_tiles(env, m, h, c, outlier, values):
    torch, B, model = env
    rng = np.random.default_rng(m + h + c)
    hp = wl.make_bit_planes(m, h, 0.5, 7 + m + h, B.packed_pitch(h))
    w = rng.normal(0, 1 / np.sqrt(h), (c, h)).astype(np.float32)
    if outlier:
        w[c // 2] *= np.float32(1e-5)
        w[c // 2, h // 3] = 1.0
    digits = torch.empty(B.bnn_output_digits_bytes(c, h), dtype=torch.uint8, device="cuda:0")
    wd = model.to_dev(w)
    B.bnn_output_prepare_digits(wd, digits)
    a = torch.from_numpy(np.unpackbits(hp.view(np.uint8), axis=1, bitorder="little")[:, :h]).cuda().double()
    want = (a if values else 2 * a - 1) @ wd.double().T
    # as above: half a unit of the row's scale per weight, then two roundings of the result
    bound = h * wd.abs().amax(1).double() * (2.0 ** -30 if outlier else 2.0 ** -22) / 2 + 2.0 ** -23 * want.abs()
    z = torch.empty((m, c), dtype=torch.float32, device="cuda:0")
    hpd = model.to_dev(hp)
    for _ in range(4):
        z.fill_(9.0)
        B.bnn_output_layer_digits(hpd, digits, None, z, h, log_softmax=False, values=values)
        assert bool(((z.double() - want).abs() <= bound).all()), float(((z.double() - want).abs() / bound).max())
    assert B.bnn_device_status() == 0


@pytest.mark.parametrize("m,n,k", [(8192, 2048, 600), (6000, 2048, 1100), (5001, 2500, 2100)])
def test_signw_gemm_digits_many_tiles(env, m, n, k):
    torch, B, model = env
    x = torch.randn((m, k), generator=torch.Generator("cuda:0").manual_seed(m + n + k), device="cuda:0")
    wp = wl.make_bit_planes(n, k, 0.5, 3 + m + n, B.packed_pitch(k))
    w = 2 * torch.from_numpy(np.unpackbits(wp.view(np.uint8), axis=1, bitorder="little")[:, :k]).cuda().double() - 1
    want = x.double() @ w.T
    bound = k * x.abs().amax(1).double()[:, None] * 2.0 ** -22 / 2 + 2.0 ** -23 * want.abs()     # as above
    ws = torch.empty(B.bnn_signw_workspace_bytes(m, k), dtype=torch.uint8, device="cuda:0")
    y = torch.empty((m, n), dtype=torch.float32, device="cuda:0")
    wd = model.to_dev(wp)
    for _ in range(4):
        y.fill_(9.0)
        B.bnn_signw_gemm(x, wd, k, Y=y, workspace=ws)
        assert bool(((y.double() - want).abs() <= bound).all()), float(((y.double() - want).abs() / bound).max())
    assert B.bnn_device_status() == 0


def test_chained_digit_layers_many_tiles(env):
    """Layers of 1100 units with binary weights only, each against double precision on the activations it was given."""
    torch, B, model = env
    cfg = wl.Config("chained", 3, 6000, 600, 1100, 4, 300, wl.ACT_HARDTANH, True)
    net = wl.make_model(cfg)
    dn = model.DeviceNet(net)
    x = model.to_dev(wl.make_frames(cfg, cfg.frames))
    outs = dn.layer_out_buffers(cfg.frames)
    for _ in range(4):
        dn.forward(x, layer_out=outs)
        below = x
        for l in range(cfg.n_hidden):
            w = torch.from_numpy(np.where(np.asarray(net.W[l]) < 0, -1.0, 1.0)).cuda()
            sc, sh = (torch.from_numpy(np.array(v, dtype=np.float64)).cuda() for v in (net.scale[l], net.shift[l]))
            dot = below.double() @ w.T
            # half a unit of the scale per value: 2^-22 of the frame's largest in the first layer, of 1 behind a hardtanh
            unit = below.abs().amax(1).double()[:, None] if l == 0 else 1.0
            bound = sc.abs() * (w.shape[1] * unit * 2.0 ** -22 / 2 + 2.0 ** -23 * dot.abs()) + 2.0 ** -23 * (sc * dot + sh).abs()
            err = (outs[l].double() - (sc * dot + sh).clamp(-1, 1)).abs()
            assert bool((err <= bound).all()), (l, float((err / bound).max()))
            below = outs[l]
    assert B.bnn_device_status() == 0
