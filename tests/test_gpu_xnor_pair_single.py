"""A prepared binary layer by itself on CTA pairs (fan-in above 2048), with more or fewer units than inputs: unit tiles and frame tiles cut off,
odd numbers of stages, a part that no unit is left for, (0,1) activations; its bits against the kernel on the integer pipes."""
import pytest

from paper_1706_09453_b200 import workloads as wl

pytestmark = pytest.mark.gpu


# (frames, units, fan-in), for which the estimate of the pairs is the smaller one by a quarter and more
@pytest.mark.parametrize("m,n,k", [(16550, 711, 2968), (27300, 1390, 2290), (9000, 3572, 2170), (16400, 5084, 2305), (20001, 1153, 3072), (12001, 1300, 2817)])
@pytest.mark.parametrize("values", [0, 1])
def test_single_layer(m, n, k, values):
    import torch
    from paper_1706_09453_b200 import build, binding as B, model
    build.build()
    a, w = (model.to_dev(wl.make_bit_planes(r, k, 0.5, [i, m, n, k], B.packed_pitch(k))) for i, r in ((1, m), (2, n)))
    g = torch.Generator("cuda:0").manual_seed(m + n + k)
    thr = torch.randint(-40, 40, (n,), generator=g, device="cuda:0", dtype=torch.int32)
    flip = torch.randint(-2**31, 2**31 - 1, ((n + 31) // 32,), generator=g, device="cuda:0", dtype=torch.int32)
    image = torch.empty(B.bnn_xnor_prepared_bytes(n, k), dtype=torch.uint8, device="cuda:0")
    B.bnn_xnor_prepare(w, k, image)
    got, want = (torch.full((m, B.packed_pitch(n)), 0x55, dtype=torch.int32, device="cuda:0") for _ in range(2))
    if values:
        B.bnn_gemm01(a, None, k, N=n, prepared=image, thr=thr, flip=flip, out_bits=got)
    else:
        B.bnn_xnor_gemm_prepared(a, image, n, k, thr=thr, flip=flip, out_bits=got)
    prev = B.bnn_set_option(B.OPT_XNOR_PATH, B.XNOR_POPC)
    try:
        (B.bnn_gemm01 if values else B.bnn_xnor_gemm)(a, w, k, thr=thr, flip=flip, out_bits=want)
    finally:
        B.bnn_set_option(B.OPT_XNOR_PATH, prev)
    assert torch.equal(got, want)
    assert B.bnn_device_status() == 0
