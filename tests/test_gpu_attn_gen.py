"""Attention of general shapes (any head width that is a multiple of 8, any block
size, any row stride): the CUDA-core kernels in fp32 and bf16 and the tcgen05
backward against the float64 oracle, and with non-finite tokens.

Tolerances.  fp32: the library's 1e-4.  bf16 forward: its own rounding, 2^-9 of
the value, bounded at 2^-8 of the largest.  bf16 gradients also carry
Drow = dO . O with O rounded to bf16: the library's 2e-2 against the oracle; the
tcgen05 backward, whose P and dS enter the products as two bf16 parts (2^-17),
within one rounding step, 2^-7 of the largest value, of the CUDA-core one."""

import numpy as np
import pytest
import torch

from tests.test_gpu_kernels import _attn_ref

pytestmark = pytest.mark.gpu

CASES = [
    # B, T, H, dh, L
    (2, 200, 2, 96, 48),      # two blocks a tile, ragged end
    (1, 256, 2, 128, 128),    # a block is a tile
    (2, 130, 8, 24, 100),     # one block and 28 idle rows a tile
    (1, 33, 8, 8, 1),         # every token its own block
    (1, 70, 2, 64, 7),
    (1, 129, 8, 40, 129),     # a block of one tile and one row
    (2, 300, 2, 128, 200),    # two tiles a block, ragged last block
    (1, 700, 4, 80, 256),     # walks whole tiles
    (1, 530, 4, 16, 500),
    (1, 1100, 8, 120, 1024),  # the largest block
    (1, 1, 8, 72, 64),        # a single token
    (3, 1000, 8, 96, 48),     # several CTAs per SM
]


@pytest.fixture(scope="module")
def C(cuda_ok):
    from paper_2608_13578_gb300 import bcmt
    return bcmt


def _run(C, impl, p, B, T, D, H, q, k, v, dO, ld=None):
    ld, dt = ld or D, q.dtype
    o = torch.full((B, T, D), float("nan"), dtype=dt, device="cuda")
    lse = torch.full((B, H, T), float("nan"), device="cuda")
    C.bcmt_test_attn(0, 0, p, q, k, v, ld, o, lse)
    drow = torch.empty(B, H, T, device="cuda")
    g = [torch.full((B, T, ld), float("nan"), dtype=dt, device="cuda") for _ in range(3)]
    C.bcmt_test_attn(impl, 1, p, q, k, v, ld, o, lse, dO, drow, *g, ld)
    C.bcmt_device_status()
    torch.cuda.synchronize()
    return o, lse, [x[..., :D] for x in g]


def _inputs(B, T, H, dh, dtype="bf16"):
    gen = torch.Generator().manual_seed(1000 * B + T + dh)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    return [torch.randn(B, T, H * dh, generator=gen).to(dt) for _ in range(4)]


def _err(got, ref):
    got = got.double().cpu().numpy()
    assert np.isfinite(got).all()
    return np.abs(got - ref).max(), np.abs(ref).max()


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,T,H,dh,L", CASES)
def test_general_attention(C, B, T, H, dh, L, dtype):
    q, k, v, dO = _inputs(B, T, H, dh, dtype)
    D = H * dh
    p = C.make_params(B, T, D, H, L, dtype)
    dev = [t.cuda() for t in (q, k, v, dO)]
    ref_o, ref_lse, *ref_g = _attn_ref(*(t.double().numpy() for t in (q, k, v)), L, H,
                                       dO.double().numpy())
    top = np.abs(ref_g[2]).max()  # a lone key's dQ and dK are 0 but for Drow's rounding
    runs = [_run(C, impl, p, B, T, D, H, *dev) for impl in ((0, 3) if dtype == "bf16" else (0,))]
    for o, lse, g in runs:
        e, m = _err(o, ref_o)
        assert e <= (2 ** -8 * m if dtype == "bf16" else 1e-4), ("o", e, m)
        assert _err(lse, ref_lse)[0] <= 1e-5 * (1 + np.abs(ref_lse).max())
        for n, x, r in zip(("dq", "dk", "dv"), g, ref_g):
            e, m = _err(x, r)
            assert e <= (2e-2 * max(m, top) if dtype == "bf16" else 1e-4), (n, e, m)
    if dtype == "bf16":
        top = max(x.float().abs().max() for x in runs[0][2])
        for x, y in zip(runs[0][2], runs[1][2]):
            assert (x.float() - y.float()).abs().max() <= 2 ** -7 * top


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("pad", [1, 2])
def test_rows_of_any_stride(C, dtype, pad):
    """Row strides that are no multiple of four elements: bit for bit the dense result."""
    B, T, H, dh, L = 2, 200, 2, 96, 48
    D = H * dh
    p = C.make_params(B, T, D, H, L, dtype)
    q, k, v, dO = (t.cuda() for t in _inputs(B, T, H, dh, dtype))
    dense = _run(C, 0, p, B, T, D, H, q, k, v, dO)
    wide = [torch.cat([t, torch.full((B, T, pad), 7.0, dtype=t.dtype, device="cuda")], 2)
            for t in (q, k, v)]
    strided = _run(C, 0, p, B, T, D, H, *wide, dO, ld=D + pad)
    for a, b in zip((dense[0], dense[1], *dense[2]), (strided[0], strided[1], *strided[2])):
        assert torch.equal(a, b)


NON_FINITE = [("v", float("inf")), ("dO", float("nan")), ("k", float("nan")), ("q", float("inf"))]


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("B,T,H,dh,L", [(1, 200, 2, 96, 48), (1, 300, 2, 128, 200)])
@pytest.mark.parametrize("which,value", NON_FINITE)
def test_non_finite_tokens_reach_the_rows_that_see_them(C, dtype, B, T, H, dh, L, which, value):
    """Token 60 of head 0 is not finite: the rows of its block that see it (or, for
    keys and values, that it sees) may be non-finite, every other row is the same
    as without it."""
    names = ("q", "k", "v", "dO")
    ins = dict(zip(names, (t.cuda() for t in _inputs(B, T, H, dh, dtype))))
    D = H * dh
    p = C.make_params(B, T, D, H, L, dtype)
    o0, lse0, g0 = _run(C, 0, p, B, T, D, H, *ins.values())
    ins[which][0, 60, 5] = value
    o, lse, g = _run(C, 0, p, B, T, D, H, *ins.values())
    t0, t1 = 60 // L * L, min((60 // L + 1) * L, T)
    # rows that may change: the forward's and dQ's from the token on, dK's and
    # dV's up to the last query that sees it
    for x, y in ((o, o0), (lse.transpose(1, 2), lse0.transpose(1, 2)), (g[0], g0[0]), (g[1], g0[1]),
                 (g[2], g0[2])):
        keep = torch.ones(T, dtype=torch.bool, device="cuda")
        keep[t0:t1] = False
        if x is o or x is g[0]:
            keep[t0:60] = True
        assert torch.equal(x[0][keep], y[0][keep])
        if x.shape[-1] == D:  # the other heads
            assert torch.equal(x[..., dh:], y[..., dh:])
    if which != "dO":  # the token's own row sees it
        assert not torch.isfinite(o[0, 60, :dh]).all()
    assert not torch.isfinite(g[2][0, t0:t1, :dh] if which == "dO" else g[0][0, 60, :dh]).all()


@pytest.mark.parametrize("B,T,H,dh,L", [(1, 200, 2, 96, 48), (1, 300, 2, 128, 200)])
@pytest.mark.parametrize("which,value", NON_FINITE)
def test_non_finite_tokens_tcgen05(C, B, T, H, dh, L, which, value):
    """The tcgen05 backward's non-finite values lie where the CUDA-core one's do."""
    ins = dict(zip(("q", "k", "v", "dO"), (t.cuda() for t in _inputs(B, T, H, dh))))
    ins[which][0, 60, 5] = value
    D = H * dh
    p = C.make_params(B, T, D, H, L, "bf16")
    g, g0 = (_run(C, impl, p, B, T, D, H, *ins.values())[2] for impl in (3, 0))
    for a, b in zip(g, g0):
        assert torch.equal(torch.isfinite(a), torch.isfinite(b))
