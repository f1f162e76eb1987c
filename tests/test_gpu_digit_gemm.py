"""Products of packed signs with real-valued rows as exact integer products of byte digits, at the sizes where the
kernels can go wrong: edges of the 256-row tiles, of 128, 64 or 32 columns on pairs and 64 or 32 on single numbers, fan-ins around 32 / 128 / 256 positions, one
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
    # every weight is off by at most half a unit of its row's fixed-point scale, the finest power of two at which the largest
    # weight stays within 0x7F7F7F when three digits are taken (the library's criterion), within 2e9 with four; then two roundings of the result and one of the bias addition
    mx, sm = np.abs(w).max(1).astype(np.float64), np.abs(w).sum(1, dtype=np.float64)
    four = bool((h * mx > 16 * sm).any())
    assert four or not outlier or h < 64
    bound = h * mx / (2e9 if four else 0x7F7F7F) + 3 * 2.0 ** -24 * (np.abs(want) + np.abs(b))
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
    # every value is off by at most half a unit of its row's fixed-point scale (see above); the sum, the
    # scale and the affine round once each
    bound = np.abs(sc) * (k * mx / 0x7F7F7F + 2.0 ** -23 * np.abs(ref)) + 2.0 ** -23 * (np.abs(pre) + np.abs(sh))
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
    bound = h * wd.abs().amax(1).double() / (2e9 if outlier else 0x7F7F7F) + 2.0 ** -23 * want.abs()
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
    bound = k * x.abs().amax(1).double()[:, None] / 0x7F7F7F + 2.0 ** -23 * want.abs()     # as above
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
            # half a unit of the scale per value: of the frame's largest in the first layer, of 1 at most behind a hardtanh
            unit = below.abs().amax(1).double()[:, None] if l == 0 else 1.0
            bound = sc.abs() * (w.shape[1] * unit / 0x7F7F7F + 2.0 ** -23 * dot.abs()) + 2.0 ** -23 * (sc * dot + sh).abs()
            err = (outs[l].double() - (sc * dot + sh).clamp(-1, 1)).abs()
            assert bool((err <= bound).all()), (l, float((err / bound).max()))
            below = outs[l]
    assert B.bnn_device_status() == 0


def _chain(torch, B, model, widths, alphas, shift, act, classes=70, seed=0):
    """A network of layers with binary weights only: widths[0] inputs, one Sigmoid or hardtanh layer per further width."""
    g = torch.Generator("cuda:0").manual_seed(seed)
    layers, plain = [], []
    for l, (k, n) in enumerate(zip(widths, widths[1:])):
        w = torch.randn((n, k), generator=g, device="cuda:0")
        wp = model.packed_empty(n, k)
        B.bnn_pack_weights(w, wp)
        sc = torch.full((n,), alphas[l], device="cuda:0") * (0.5 + torch.rand((n,), generator=g, device="cuda:0"))
        sh = torch.full((n,), shift, device="cuda:0") * (0.5 + torch.rand((n,), generator=g, device="cuda:0"))
        layers.append(dict(kind=B.LAYER_SIGNW, K=k, N=n, Wp=wp, scale=sc, shift=sh, act=act))
        plain.append((torch.where(w < 0, -1.0, 1.0).double(), sc, sh))
    w = torch.randn((classes, widths[-1]), generator=g, device="cuda:0")
    img = torch.empty(B.bnn_output_prepared_bytes(classes, widths[-1]), dtype=torch.uint8, device="cuda:0")
    B.bnn_output_prepare(w, img)
    layers.append(dict(kind=B.LAYER_REAL_OUT, K=widths[-1], N=classes, W=w, W_prepared=img))
    return B.ModelDesc(layers), plain


@pytest.mark.parametrize("widths", [[440, 1024, 1024, 1024, 1024, 1024], [200, 700, 96, 1100, 64, 300]])
@pytest.mark.parametrize("act,alpha,shift", [(2, 0.001, 0.0), (2, 1e-5, 1e-4), (2, 0.05, 0.1), (3, 0.05, -7.0), (3, 0.5, -30.0)])
@pytest.mark.parametrize("frames", [3, 700])
def test_chained_layers_of_small_activations(env, widths, act, alpha, shift, frames):
    """Every layer against double precision on the activations it was given, however small these are; twice, with what the first
    pass left in the workspace."""
    torch, B, model = env
    desc, plain = _chain(torch, B, model, widths, [alpha] * (len(widths) - 1), shift, act)
    x = torch.randn((frames, widths[0]), generator=torch.Generator("cuda:0").manual_seed(1), device="cuda:0")
    x[1] *= 1e-3                                                    # one frame far below the others
    ws = torch.full((desc.workspace_bytes(frames),), 255, dtype=torch.uint8, device="cuda:0")
    for _ in range(2):
        outs = [torch.empty((frames, n), device="cuda:0") for n in widths[1:]]
        logp = torch.empty((frames, 70), device="cuda:0")
        B.bnn_forward(desc, x, logp, ws, outs)
        # a value is off by at most half a unit of its frame's scale, and the scale is the finest power of two at which the
        # bound below stays within 0x7F7F7F
        below, top = x.double(), x.abs().amax(1).double()
        for l, ((w, sc, sh), y) in enumerate(zip(plain, outs)):
            k = w.shape[1]
            off = k * top[:, None] / 0x7F7F7F
            dot = below @ w.T
            pre = sc.double() * dot + sh.double()
            want = pre.clamp(-1, 1) if act == B.ACT_HARDTANH else torch.sigmoid(pre)
            tol = sc.abs() * (off + 2.0 ** -22 * dot.abs()) + 2.0 ** -23 * (pre.abs() + sh.abs())
            if act == B.ACT_SIGMOID:     # its slope is at most its value, and within tol the value changes by a factor e^tol;
                # expf(-pre) is infinite where the value is below the normal numbers
                tol = want * torch.expm1(tol) + 2.0 ** -21 * want + 2.0 ** -126
            err = (y.double() - want).abs()
            assert bool((err <= tol).all()), float((err / tol).max())
            # the bound from which the next scale is chosen: sum |x| itself in the first layer, sqrt(k) |x|_2 in the others; it
            # is counted in high digits, 65536 units each, rounded at both ends
            d = below.abs().sum(1) if l == 0 else k ** 0.5 * below.norm(dim=1)
            d = sc.abs().max().double() * (d * 1.002 + 2 * 65536 * k * 2 * top / 0x7F7F7F)
            top = torch.exp(d + sh.max() + 1e-6 * (d + sh.abs().max())) if act == B.ACT_SIGMOID else d + sh.abs().max()
            top = (top * 1.0001).clamp(max=1.0)
            below = y.double()
    assert B.bnn_device_status() == 0


@pytest.mark.parametrize("widths", [[50, 70, 300], [440, 1024, 700, 1024, 96]])
@pytest.mark.parametrize("act", [2, 3])
@pytest.mark.parametrize("full", [True, False])
def test_chained_layers_carry_nans(env, widths, act, full):
    """Frames with an infinity or a NaN come out as NaN behind Sigmoid units (a hardtanh unit turns them into -1), whether
    the layers hand one another digits or fp32 rows, and a unit whose shift is a NaN spoils every frame from there on; the
    other frames are what they are without."""
    torch, B, model = env
    frames, bad = 200, [3, 64, 199]
    desc, plain = _chain(torch, B, model, widths, [0.1] * (len(widths) - 1), 0.1, act)
    x = torch.randn((frames, widths[0]), generator=torch.Generator("cuda:0").manual_seed(2), device="cuda:0")
    good = torch.ones(frames, dtype=torch.bool, device="cuda:0")
    good[bad] = False
    n = desc.workspace_bytes(frames) if full else desc.min_workspace_bytes(frames)

    def run():
        outs = [torch.empty((frames, w), device="cuda:0") for w in widths[1:]]
        logp = torch.empty((frames, 70), device="cuda:0")
        B.bnn_forward(desc, x, logp, torch.full((n,), 255, dtype=torch.uint8, device="cuda:0"), outs)
        return outs + [logp]

    clean = run()
    x[3, 7], x[64, 0], x[199, 49] = float("inf"), float("nan"), float("-inf")
    for a, b in zip(clean, run()):
        assert torch.equal(a[good], b[good])
        if act == B.ACT_SIGMOID:
            assert bool(b[~good].isnan().all())
        else:
            assert not bool(b.isnan().any())
    x[~good] = 0.0
    plain[0][2][69] = float("nan")          # the last unit's shift in the first layer
    spoilt = run()
    if act == B.ACT_SIGMOID:
        assert bool(spoilt[0][:, 69].isnan().all()) and not bool(spoilt[0][:, :69].isnan().any())
        for b in spoilt[1:]:
            assert bool(b.isnan().all())
    else:
        assert bool((spoilt[0][:, 69] == -1).all()) and not bool(spoilt[-1].isnan().any())


def test_unmarked_packed_weights_of_the_top_layer_are_ignored(env):
    """Whatever Wp of a top layer holds, the logits come from W and W_prepared unless ldwp marks a digit image."""
    torch, B, model = env
    cfg = wl.Config("wp", 4, 300, 100, 160, 2, 90)
    dn = model.DeviceNet(wl.make_model(cfg))
    x = model.to_dev(wl.make_frames(cfg))
    img = torch.empty(B.bnn_output_prepared_bytes(90, 160), dtype=torch.uint8, device="cuda:0")
    B.bnn_output_prepare(dn.Wout, img)
    junk = torch.full((1 << 16,), 0x5A5A5A5A, dtype=torch.int32, device="cuda:0")
    out = []
    for wp in (None, junk.view(-1, 8)):
        top = dict(dn.desc.layers[-1], W_prepared=img, W_digits=None, Wp=wp)
        desc = B.ModelDesc(dn.desc.layers[:-1] + [top])
        for frames in (8, 300):
            logp = torch.empty((frames, 90), device="cuda:0")
            ws = torch.empty(desc.workspace_bytes(frames), dtype=torch.uint8, device="cuda:0")
            out.append(B.bnn_forward(desc, x[:frames], logp, ws))
    assert torch.equal(out[0], out[2]) and torch.equal(out[1], out[3])
