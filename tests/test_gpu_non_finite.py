"""Non-finite values: what a product or an attention row costs when its inputs hold
some, and that no bounded wait runs out over it.

Limits.  A NaN makes the affected outputs be formed again from the operands: a walk
over K per row and column of a 32 x 32 run, at most a few times the product itself (its
three-part split reads each operand once per output tile).  40 times the finite call
leaves room for the timer; a chain of K terms per output took 10^3 times and more.  An
attention row of NaN is known from its first keys: 8 times the finite call.  One token
that is not finite makes up to 128 rows, 16 a warp, walk 1024 keys, 32 at a time, with
up to four dot products of 128 each: 16 x 32 x (4 x 128 x 8 + 1500) cycles, 1.5 ms, in
each of two kernels, against 0.1 ms for the fastest finite backward; 60 times is the
limit, twice that (a thread per row and group of columns took 150 to 20000 times)."""

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


@pytest.mark.parametrize("what,limit", [("all", 8), ("key", 60), ("value", 60)])
@pytest.mark.parametrize("dtype,impl", [("fp32", 0), ("bf16", 0), ("bf16", 3)])
def test_non_finite_attention_costs_a_few_calls(C, dtype, impl, what, limit):
    B, T, H, dh, L = 2, 2048, 4, 128, 1024
    D, dt = H * dh, torch.float32 if dtype == "fp32" else torch.bfloat16
    p = C.make_params(B, T, D, H, L, dtype)
    gen = torch.Generator(device="cuda").manual_seed(5)
    ins = [torch.randn(B, T, D, generator=gen, device="cuda").to(dt) for _ in range(4)]
    o, lse = torch.empty_like(ins[0]), torch.empty(B, H, T, device="cuda")
    drow, g = torch.empty_like(lse), [torch.empty_like(ins[0]) for _ in range(3)]

    def both(q, k, v, dO):
        return (_ms(lambda: C.bcmt_test_attn(0, 0, p, q, k, v, D, o, lse)),
                _ms(lambda: C.bcmt_test_attn(impl, 1, p, q, k, v, D, o, lse, dO, drow, *g, D)))

    finite = both(*ins)
    if what == "all":
        ins = [torch.full_like(x, NAN) for x in ins]
    else:  # a token near the end of the first block
        ins[1 if what == "key" else 2][0, L - 2] = NAN if what == "key" else INF
    bad = both(*ins)
    C.bcmt_device_status()
    if what == "all":
        assert all(torch.isnan(x).all() for x in (o, lse, *g))
    else:  # the forward's rows that see it and no others
        rows = torch.zeros(B, T, dtype=torch.bool, device="cuda")
        rows[0, L - 2:L] = True
        assert torch.equal(torch.isfinite(o).all(-1), ~rows)
        assert torch.equal(torch.isfinite(g[0]).all(-1), ~rows)
    assert bad[0] <= limit * finite[0] and bad[1] <= limit * finite[1], (bad, finite)


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
