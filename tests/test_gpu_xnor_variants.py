"""The stand-alone binary product at sizes for which each of its variants is taken (CTA pairs with parts of 128 or of 64 units, single CTAs): cut-off
unit and frame tiles, a part that no unit is left for, fan-ins that end inside a word, a stage or behind an odd one, rows that start
anywhere in a sector, activations in (0,1), integers together with Sign bits; all bits against the kernel on the integer pipes."""
import os
import re

import pytest

from paper_1706_09453_b200 import build, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available()
    from paper_1706_09453_b200 import binding, model
    build.build()
    return torch, binding, model


def variants():
    """The table that the library chooses by: frames, units, CTAs per tile, clocks per stage, per epilogue and per launch."""
    text = open(os.path.join(os.path.dirname(build.__file__), "csrc", "xnor_gemm_tc.cu")).read()
    rows = re.search(r"variants\[\] = \{(.*)\};", text).group(1)
    numbers = [int(x) for x in re.findall(r"-?\d+", rows)]
    return dict(zip(("wide", "narrow", "single"), (numbers[i:i + 8] for i in range(0, 24, 8))))


def chosen(m, n, k, results):
    def up(a, b):
        return -(-a // b)

    cost = {name: up(up(m, frames) * up(n, units), 148 // per) * (up(k, 256) * stage + epilogue[results]) + fixed
            for name, (frames, units, per, stage, *epilogue, fixed) in variants().items()}
    return min(cost, key=cost.get)


# (frames, units, fan-in): unit tiles that end 98, 235 or 255 short or whole, odd and even numbers of stages
SHAPES = {"wide": [(5000, 3170, 1100), (4999, 3307, 1300), (8200, 4095, 2000), (16384, 2048, 2048), (5100, 3073, 513)],
          "narrow": [(1873, 930, 691), (257, 130, 127), (1000, 387, 1300), (33, 31, 64), (600, 1027, 2060)],
          "single": [(6270, 520, 2048), (6200, 513, 4100), (6272, 575, 1111)]}


@pytest.mark.parametrize("variant,shape", [(v, s) for v in SHAPES for s in SHAPES[v]])
@pytest.mark.parametrize("values", [0, 1])
@pytest.mark.parametrize("extra,shift", [(0, 0), (5, 0), (4, 0), (9, 3)])
def test_integers(env, variant, shape, values, extra, shift):
    torch, B, model = env
    m, n, k = shape
    a, w = (model.to_dev(wl.make_bit_planes(r, k, 0.5, [i, m, n, k], B.packed_pitch(k))) for i, r in ((1, m), (2, n)))
    pitch = n + extra + (-n % 4 if extra == 4 else 0)
    whole = n % 4 == 0 and pitch % 4 == 0 and shift % 4 == 0
    assert torch.cuda.get_device_properties(0).multi_processor_count != 148 or chosen(m, n, k, 1 if whole else 2) == variant

    def run(path):
        c = torch.full((m * pitch + 16,), -77, dtype=torch.int32, device="cuda:0")
        view = c[shift:shift + m * pitch].view(m, pitch)[:, :n]
        prev = B.bnn_set_option(B.OPT_XNOR_PATH, path)
        try:
            (B.bnn_gemm01(a, w, k, C_out=view) if values else B.bnn_xnor_gemm(a, w, k, C_out=view))
        finally:
            B.bnn_set_option(B.OPT_XNOR_PATH, prev)
        return c

    assert torch.equal(run(B.XNOR_TENSOR), run(B.XNOR_POPC))
    assert B.bnn_device_status() == 0


@pytest.mark.parametrize("variant,shape", [(v, s) for v in SHAPES for s in SHAPES[v]])
@pytest.mark.parametrize("values", [0, 1])
@pytest.mark.parametrize("integers", [False, True])
def test_sign_bits(env, variant, shape, values, integers):
    torch, B, model = env
    m, n, k = shape
    a, w = (model.to_dev(wl.make_bit_planes(r, k, 0.5, [i, m, n, k], B.packed_pitch(k))) for i, r in ((1, m), (2, n)))
    g = torch.Generator("cuda:0").manual_seed(m + n + k)
    thr = torch.randint(-40, 40, (n,), generator=g, device="cuda:0", dtype=torch.int32)
    flip = torch.randint(-2**31, 2**31 - 1, ((n + 31) // 32,), generator=g, device="cuda:0", dtype=torch.int32)
    if not integers:
        assert torch.cuda.get_device_properties(0).multi_processor_count != 148 or chosen(m, n, k, 0) == variant

    def run(path):
        bits = torch.full((m, B.packed_pitch(n)), 0x55, dtype=torch.int32, device="cuda:0")
        c = torch.zeros((m, n), dtype=torch.int32, device="cuda:0") if integers else None
        prev = B.bnn_set_option(B.OPT_XNOR_PATH, path)
        try:
            if values:
                B.bnn_gemm01(a, w, k, C_out=c, thr=thr, flip=flip, out_bits=bits)
            else:
                B.bnn_xnor_gemm(a, w, k, C_out=c, thr=thr, flip=flip, out_bits=bits)
        finally:
            B.bnn_set_option(B.OPT_XNOR_PATH, prev)
        return bits, c

    (x, cx), (y, cy) = run(B.XNOR_TENSOR), run(B.XNOR_POPC)
    assert torch.equal(x, y) and (cx is None or torch.equal(cx, cy))
    assert B.bnn_device_status() == 0
