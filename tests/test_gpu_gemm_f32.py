"""fp32 products on the tensor cores (three bf16 parts per value): every operand
layout, edges of tiles, K splits and non-finite values, against float64 and
against the CUDA-core kernel.

Tolerance: the six partial products kept leave 2^-24 of each product, a slice's
16-step accumulations and the fp32 sums over slices a few 2^-24 of the result's
scale; a chain of K fused multiply-adds in fp32 has a relative 2-norm error of
about sqrt(K) / 4 x 2^-24 here.  The test holds the tensor-core product to the
larger of that chain's measured error and 2^-22."""

import pytest
import torch

from tests.test_gpu_kernels import LAYOUTS, _operand

pytestmark = pytest.mark.gpu

# tile edges (128 rows, 64 / 128 columns, 64-deep slices), one row, and enough
# tiles for several per CTA (within and past the eight slices that share an accumulator)
SHAPES = [(128, 64, 64), (256, 384, 128), (1, 64, 512), (136, 192, 72), (1000, 512, 520),
          (8, 128, 1536), (6144, 768, 256), (6144, 768, 584)]


@pytest.fixture(scope="module")
def C(cuda_ok):
    from paper_2608_13578_gb300 import bcmt
    return bcmt


def _both(C, M, N, K, la, lb, splits=1, poison=None, scale=1.0):
    gen = torch.Generator().manual_seed(M * 7 + N * 3 + K)
    A, sam, sak, Al = _operand(M, K, la == "k", torch.float32, gen)
    B, sbk, sbn, Bl = _operand(K, N, lb == "n", torch.float32, gen)
    B *= scale
    Bl = Bl * scale
    if poison is not None:
        r, k, v = poison
        Al[r, k] = v
        A.as_strided((M, K), (sam, sak))[r, k] = v
    A, B = A.cuda(), B.cuda()
    out = []
    for impl in (6, 0):
        part = torch.full((splits, M, N), float("nan"), device="cuda")
        n = C.bcmt_test_gemm(impl, 0, 0, M, N, K, A, sam, sak, B, sbk, sbn, part, N, splits)
        C.bcmt_device_status()
        torch.cuda.synchronize()
        out.append(part[:n].cpu())
    return out[0], out[1], Al.double() @ Bl.double()


@pytest.mark.parametrize("la,lb", LAYOUTS)
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_gemm_f32(C, M, N, K, la, lb):
    if la == "m" and M % 8:
        pytest.skip("rows of an M-major operand come in groups of eight")
    tc, simt, ref = _both(C, M, N, K, la, lb, scale=K ** -0.5)
    rel = [((x[0].double() - ref).norm() / ref.norm()).item() for x in (tc, simt)]
    assert rel[0] <= max(rel[1], 2 ** -22), rel
    # the worst element, in units of the chain's bound K x 2^-24 x sum |a b|
    assert (tc[0].double() - ref).abs().max().item() <= K * 2 ** -24 * 8


@pytest.mark.parametrize("la,lb", [("m", "n"), ("k", "n")])
def test_gemm_f32_split_k(C, la, lb):
    tc, simt, ref = _both(C, 512, 256, 4040, la, lb, splits=6)
    assert 1 < len(tc) == len(simt)
    rel = [((x.double().sum(0) - ref).norm() / ref.norm()).item() for x in (tc, simt)]
    assert rel[0] <= max(rel[1], 2 ** -22), rel


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan"), 3.4e38, 1e-39])
def test_gemm_f32_extreme_values(C, value):
    tc, simt, ref = _both(C, 200, 128, 192, "k", "n", poison=(77, 100, value))
    a, b = tc[0], simt[0]
    assert torch.equal(torch.isnan(a), torch.isnan(b))
    assert torch.equal(a[torch.isinf(b)], b[torch.isinf(b)])
    fin = torch.isfinite(b)
    assert torch.equal(fin, torch.isfinite(a))
    assert ((a - b).abs()[fin] <= 1e-5 * b.abs()[fin].clamp(min=100.0)).all()
