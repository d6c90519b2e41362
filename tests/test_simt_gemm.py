"""The SIMT matrix product on its own, against a float64 product (a library
routine, not the CUDA path).  Every output is one chain of K fused
multiply-adds, so |C - ref| <= K u (|A| |B|) entrywise with u the unit
roundoff (first order; the factor 1.01 covers the rest for K u < 1e-3)."""
import ctypes

import pytest
import torch

from paper_2504_06087_gb300 import fire

pytestmark = pytest.mark.gpu


# M, N, K, batch, transB, B offset (elements), accumulate
SHAPES = [
    (1, 1, 1, 1, 0, 0, 0), (3, 5, 2, 1, 1, 1, 0), (64, 64, 16, 1, 0, 0, 0), (65, 63, 17, 1, 0, 1, 0),
    (16, 64, 64, 1, 0, 0, 0), (64, 464, 144, 1, 1, 0, 0), (33, 31, 400, 1, 1, 0, 1), (130, 256, 256, 1, 0, 1, 1),
    (20000, 16, 64, 1, 1, 1, 0), (20000, 16, 64, 16, 0, 1, 0), (9000, 58, 128, 8, 0, 0, 0), (9000, 10, 64, 4, 0, 1, 0),
    (20011, 180, 256, 2, 0, 0, 0), (20011, 256, 58, 1, 1, 0, 1), (40000, 17, 33, 1, 0, 0, 0), (257, 7, 96, 3, 1, 0, 0),
]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("M,N,K,batch,tb,off,acc", SHAPES)
def test_simt_gemm_matches_float64_product(dtype, M, N, K, batch, tb, off, acc):
    g = torch.Generator(device="cpu").manual_seed(M + 7 * N + K)
    A = torch.randn(M, K, generator=g, dtype=torch.float64).to(dtype).cuda()
    flat = torch.randn(off + batch * N * K, generator=g, dtype=torch.float64).to(dtype).cuda()
    B = flat[off:].view(batch, N, K) if tb else flat[off:].view(batch, K, N)
    C = torch.randn(M, batch * N + 3, generator=g, dtype=torch.float64).to(dtype).cuda()
    C0 = C.clone()
    vp = ctypes.c_void_p
    rc = fire.lib().fire_selftest_simt_gemm(
        0 if dtype == torch.float64 else 1, M, N, K, batch, tb, acc, vp(A.data_ptr()), K, vp(B.data_ptr()),
        K if tb else N, N * K, vp(C.data_ptr()), C.stride(0), N, vp(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    torch.cuda.synchronize()
    Bd = B.double().transpose(1, 2) if tb else B.double()
    ref = torch.cat([A.double() @ b for b in Bd], 1)
    mag = torch.cat([A.double().abs() @ b.abs() for b in Bd], 1)
    u = 2.0 ** -53 if dtype == torch.float64 else 2.0 ** -24
    if acc:
        ref = ref + C0[:, :batch * N].double()
        mag = mag + C0[:, :batch * N].double().abs()
    # the float64 reference has a rounding of its own of the same form
    bound = 1.01 * (K + acc) * (u + 2.0 ** -53) * mag
    assert ((C[:, :batch * N].double() - ref).abs() <= bound).all()
    assert torch.equal(C[:, batch * N:], C0[:, batch * N:])   # nothing beyond the columns
