"""Real-valued weights on real-valued activations over the tile shapes that the number of frames selects (64, 128 or 256
frames a tile, one, two or four CTAs to a tile), at their edges, against double precision; and Sigmoid units, whose
values must not depend on the tile at all."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available()
    from paper_1706_09453_b200 import build, binding, model
    build.build()
    return torch, binding, model


@pytest.mark.parametrize("c,h", [(3307, 520), (128, 127), (129, 2048), (999, 300)])
@pytest.mark.parametrize("m", [1, 63, 65, 129, 200, 257, 400, 1100, 2500])
def test_output_layer_tiles(env, c, h, m):
    torch, B, model = env
    rng = np.random.default_rng(m + c)
    w, b = rng.normal(0, 1, (c, h)).astype(np.float32), rng.normal(0, 1, c).astype(np.float32)
    a = rng.uniform(-1, 1, (m, h)).astype(np.float32)
    wd = model.to_dev(w)
    img = torch.empty(B.bnn_output_prepared_bytes(c, h), dtype=torch.uint8, device="cuda:0")
    B.bnn_output_prepare(wd, img)
    ws = torch.empty(B.bnn_output_workspace_bytes(m, h), dtype=torch.uint8, device="cuda:0")
    z = torch.full((m, c + 3), 9.0, dtype=torch.float32, device="cuda:0")
    B.bnn_output_layer(wd, model.to_dev(b), z[:, :c], h, Hf=model.to_dev(a), log_softmax=False, prepared=img, workspace=ws)
    got = z.cpu().numpy()
    want = a.astype(np.float64) @ w.astype(np.float64).T + b
    mag = np.abs(a).astype(np.float64) @ np.abs(w).astype(np.float64).T
    # two-term splits of both operands and the term left out, a rounding of the fp32 sum per position of K, the result's
    bound = (3 * 2.0 ** -22 + h * 2.0 ** -24) * mag + 2.0 ** -22 * (np.abs(want) + np.abs(b))
    assert (np.abs(got[:, :c] - want) <= bound).all(), (np.abs(got[:, :c] - want) / bound).max()
    np.testing.assert_array_equal(got[:, c:], 9.0)
    assert B.bnn_device_status() == 0


def test_sigmoid_units_do_not_depend_on_the_batch(env):
    torch, B, model = env
    rng = np.random.default_rng(0)
    k, n, m = 440, 700, 6000
    w, b = model.to_dev(rng.normal(0, 0.1, (n, k)).astype(np.float32)), model.to_dev(rng.normal(0, 0.1, n).astype(np.float32))
    x = model.to_dev(rng.normal(0, 1, (m, k)).astype(np.float32))
    img = torch.empty(B.bnn_output_prepared_bytes(n, k), dtype=torch.uint8, device="cuda:0")
    B.bnn_output_prepare(w, img)
    ws = torch.empty(B.bnn_output_workspace_bytes(m, k), dtype=torch.uint8, device="cuda:0")

    def run(at, rows):
        y = torch.empty((rows, n), dtype=torch.float32, device="cuda:0")
        B.bnn_real_layer(x[at:at + rows], w, b, y, prepared=img, workspace=ws)
        return y

    want = run(0, m)
    for at, rows in ((0, 1), (7, 64), (100, 130), (3, 400), (500, 1500), (1, 3100)):
        assert torch.equal(run(at, rows), want[at:at + rows]), rows
    assert B.bnn_device_status() == 0
