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


# M, N, K, residual, one, offset of R and C (elements: unaligned rows take scalar loads and stores)
LAYERS = [
    (1, 1, 1, 0, 0, 0), (33, 30, 17, 1, 0, 0), (64, 64, 64, 1, 1, 0), (65, 62, 64, 1, 1, 1), (300, 128, 128, 0, 0, 0),
    (257, 128, 96, 1, 0, 0), (20011, 256, 64, 1, 1, 0), (20011, 180, 33, 1, 0, 1), (40000, 17, 33, 1, 1, 0),
]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("M,N,K,res,one,off", LAYERS)
def test_simt_layer_matches_float64_layer(dtype, M, N, K, res, one, off):
    """The product's bound carried through SiLU (its slope is below 1.1), plus
    the rounding of bias, logistic (exp, sum, quotient), product and sum."""
    g = torch.Generator(device="cpu").manual_seed(3 * M + N + K)
    rnd = lambda *q: torch.randn(*q, generator=g, dtype=torch.float64).to(dtype).cuda()
    A, B, b = rnd(M, K), rnd(K, N), rnd(N)
    R, C = (rnd(off + M * (N + 4))[off:].view(M, N + 4) for _ in range(2))
    C0 = C.clone()
    vp = ctypes.c_void_p
    rc = fire.lib().fire_selftest_simt_layer(
        0 if dtype == torch.float64 else 1, M, N, K, one, vp(A.data_ptr()), K, vp(B.data_ptr()), vp(b.data_ptr()),
        vp(R.data_ptr()) if res else None, R.stride(0), vp(C.data_ptr()), C.stride(0),
        vp(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    torch.cuda.synchronize()
    x = A.double() @ B.double() + b.double()
    f = x * torch.sigmoid(x)
    ref = f + R[:, :N].double() if res else f
    u = (2.0 ** -53 if dtype == torch.float64 else 2.0 ** -24) + 2.0 ** -53
    mag = A.double().abs() @ B.double().abs() + b.double().abs()
    bound = 1.1 * 1.01 * (K + 2) * u * mag + 10 * u * f.abs() + 2 * u * ref.abs() + 1e-30
    assert ((C[:, :N].double() - ref).abs() <= bound).all()
    assert torch.equal(C[:, N:], C0[:, N:])
