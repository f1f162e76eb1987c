"""The int32 product of packed planes, over pitches, offsets and widths that decide how a row is written: tile stores, a last
block of a width that is no multiple of 4, rows that start anywhere in a 32-byte sector; odd numbers of stages."""
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


@pytest.mark.parametrize("m,n,k", [(33, 31, 64), (128, 192, 256), (129, 193, 257), (300, 227, 513), (257, 384, 768),
                                   (1000, 387, 1500), (4000, 1100, 300)])
@pytest.mark.parametrize("extra,shift", [(0, 0), (5, 0), (4, 0), (9, 3)])
def test_int32_rows(env, m, n, k, extra, shift):
    torch, B, model = env
    ap = wl.make_bit_planes(m, k, 0.5, [1, m, n, k], B.packed_pitch(k))
    wp = wl.make_bit_planes(n, k, 0.5, [2, m, n, k], B.packed_pitch(k))
    pitch = n + extra + (-n % 4 if extra == 4 else 0)
    c = torch.full((m * pitch + 16,), -77, dtype=torch.int32, device="cuda:0")
    view = c[shift:shift + m * pitch].view(m, pitch)
    prev = B.bnn_set_option(B.OPT_XNOR_PATH, B.XNOR_TENSOR)
    try:
        B.bnn_xnor_gemm(model.to_dev(ap), model.to_dev(wp), k, C_out=view[:, :n])
    finally:
        B.bnn_set_option(B.OPT_XNOR_PATH, prev)
    got = c.cpu().numpy()
    rows = got[shift:shift + m * pitch].reshape(m, pitch)
    np.testing.assert_array_equal(rows[:, :n], o.xnor_gemm(ap, wp, k))
    np.testing.assert_array_equal(rows[:, n:], -77)
    np.testing.assert_array_equal(got[:shift], -77)
    np.testing.assert_array_equal(got[shift + m * pitch:], -77)
    assert B.bnn_device_status() == 0
