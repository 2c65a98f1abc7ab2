"""Non-finite values: what a product or an attention row costs when its inputs hold
some, and that no bounded wait runs out over it.

Limits.  A NaN makes the affected outputs be formed again from the operands: a walk
over K per row and column of a 32 x 32 run, at most a few times the product itself (its
three-part split reads each operand once per output tile).  40 times the finite call
leaves room for the timer; a chain of K terms per output took 10^3 times and more."""

import pytest
import torch

pytestmark = pytest.mark.gpu

NAN, INF = float("nan"), float("inf")


@pytest.fixture(scope="module")
def C(cuda_ok):
    from paper_2608_13578_gb300 import bcmt
    return bcmt


def _ms(f):
    """The shortest of three calls after one untimed."""
    f()
    best = 1e9
    for _ in range(3):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def _product(C, A, B, lay):
    """A[M, K] B[K, N] of fp32 operands stored K-major or M-major, N-major."""
    (M, K), N = A.shape, B.shape[1]
    a, sa = (A, (K, 1)) if lay == "k" else (A.t().contiguous(), (1, M))
    out = torch.empty(M, N, device="cuda")

    def run():
        C.bcmt_test_gemm(6, 0, 0, M, N, K, a, *sa, B, N, 1, out, N, 1)
    return run, out


@pytest.mark.parametrize("where", ["last k", "everywhere", "one row"])
@pytest.mark.parametrize("lay,M,N,K", [("m", 512, 256, 32768), ("k", 4096, 512, 512)])
def test_product_with_nan_costs_a_few_products(C, lay, M, N, K, where):
    gen = torch.Generator(device="cuda").manual_seed(K)
    A, B = (torch.randn(*s, generator=gen, device="cuda") for s in ((M, K), (K, N)))
    run, _ = _product(C, A, B, lay)
    finite = _ms(run)
    bad = torch.zeros(M, N, dtype=torch.bool, device="cuda")
    if where == "last k":
        A[:, K - 1] = NAN
        bad[:] = True
    elif where == "everywhere":
        A[:] = NAN
        bad[:] = True
    else:
        A[M // 2, K // 2] = NAN
        bad[M // 2] = True
    run, out = _product(C, A, B, lay)
    nan = _ms(run)
    C.bcmt_device_status()
    assert torch.equal(torch.isnan(out), bad)
    assert nan <= 40 * finite, (nan, finite)


def test_product_with_infinities(C):
    """The classes and signs of a chain in K order: an infinity beside finite terms, two
    that agree, two that do not, one against a zero; several at a time in row and column."""
    M, N, K = 192, 128, 256
    gen = torch.Generator(device="cuda").manual_seed(3)
    A = torch.randn(M, K, generator=gen, device="cuda")
    B = torch.randn(K, N, generator=gen, device="cuda")
    A[3, 0], A[64, 77], A[64, 200], A[130, 255] = INF, INF, -INF, -INF
    A[150, 10:20] = INF
    B[77, 5], B[200, 6], B[0, 7] = 0.0, INF, 0.0
    B[:, 100] = 1.0
    B[40, 127] = -INF
    outs = []
    for impl in (6, 0):
        c = torch.empty(M, N, device="cuda")
        C.bcmt_test_gemm(impl, 0, 0, M, N, K, A, K, 1, B, N, 1, c, N, 1)
        outs.append(c)
    C.bcmt_device_status()
    tc, simt = outs
    assert torch.equal(torch.isnan(tc), torch.isnan(simt)) and torch.isnan(tc).any()
    assert torch.equal(torch.isinf(tc), torch.isinf(simt))
    inf = torch.isinf(simt)
    assert inf.any() and torch.equal(tc[inf], simt[inf])


def test_long_chains_outlast_a_wait(C):
    """Two infinities that agree, 2^19 terms apart, against positive columns: every output
    is a chain of 2^19 terms, 64 one after the other in a lane, which takes 1.6 s, longer
    than a wait's bound of 2^31 cycles.  One CTA has a second tile, whose loads wait meanwhile:
    they go on, the result is complete and no wait has run out.  (Strides of 0: every row
    of A, and every row of B, is the same one.)"""
    K, M, N = 1 << 19, 128, 128 * 153
    a = torch.full((K,), 2.0 ** -19, device="cuda")
    b = torch.ones(N, device="cuda")
    a[0] = a[K - 1] = INF
    out = torch.zeros(M, N, device="cuda")
    C.bcmt_test_gemm(6, 0, 0, M, N, K, a, 0, 1, b, 0, 1, out, N, 1)
    C.bcmt_device_status()
    assert (out == INF).all()
