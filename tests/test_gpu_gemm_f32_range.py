"""fp32 products on the tensor cores over the range of their operands and over K, in the
relative 2-norm against float64 and the CUDA-core kernel.

Tolerances.  N(0,1) operands at any scale from 2^-100 up are exact as three bf16 parts:
no further off than the CUDA-core chain.  Below 2^-110 an operand value is off by up to
2^-134: 2^-16 of values around 2^-118."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C(cuda_ok):
    from paper_2608_13578_gb300 import bcmt
    return bcmt


def _errors(C, K, scale_a, scale_b):
    M, N = 256, 192
    gen = torch.Generator(device="cuda").manual_seed(K)
    A = torch.randn(M, K, generator=gen, device="cuda") * scale_a
    B = torch.randn(K, N, generator=gen, device="cuda") * scale_b
    ref, out = A.double() @ B.double(), []
    for impl in (6, 0):
        c = torch.empty(M, N, device="cuda")
        C.bcmt_test_gemm(impl, 0, 0, M, N, K, A, K, 1, B, N, 1, c, N, 1)
        out.append(((c.double() - ref).norm() / ref.norm()).item())
    C.bcmt_device_status()
    return out


@pytest.mark.parametrize("K", [64, 192, 512, 1536, 2048, 4096, 16384])
def test_error_over_k(C, K):
    tc, simt = _errors(C, K, 1.0, K ** -0.5)
    assert tc <= simt, (tc, simt)


@pytest.mark.parametrize("log2a,log2b", [(-100, 60), (60, -100), (-60, -40), (60, 60)])
def test_error_over_scales(C, log2a, log2b):
    tc, simt = _errors(C, 512, 2.0 ** log2a, 2.0 ** log2b)
    assert tc <= simt, (tc, simt)


@pytest.mark.parametrize("log2a,log2b", [(-118, 60), (60, -118)])
def test_values_below_the_exact_range(C, log2a, log2b):
    tc, _ = _errors(C, 512, 2.0 ** log2a, 2.0 ** log2b)
    assert tc <= 2 ** -16, tc
