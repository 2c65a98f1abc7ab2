"""The allocation-free attention backward where a block has several tiles (L > 64: the
dK/dV kernel needs dO . O of queries that another kernel handles): equal to the regular
backward bit for bit, at the row limit, and with calls on two streams at once."""

import numpy as np
import pytest
import torch

from tests.test_gpu_kernels import _attn_ref
from tests.test_zz_no_alloc import ROWS_MAX, _inputs, _regular_and_noalloc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C(cuda_ok):
    from paper_2608_13578_gb300 import bcmt
    return bcmt


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("B,T,H,dh,L", [(2, 250, 2, 64, 100), (1, 300, 2, 128, 128), (2, 700, 4, 16, 512)])
def test_long_blocks(C, dtype, B, T, H, dh, L):
    D = H * dh
    tdt = torch.float32 if dtype == "fp32" else torch.bfloat16
    p = C.make_params(B, T, D, H, L, dtype)
    for seed in (31, 32):
        ins = _inputs(B, T, D, tdt, seed)
        ref, got = _regular_and_noalloc(C, p, B, T, D, H, tdt, *(t.cuda() for t in ins))
        q, k, v, dO = (t.double().numpy() for t in ins)
        _, _, *oracle = _attn_ref(q, k, v, L, H, dO)
        top = np.abs(oracle[2]).max()
        for name, a, r, o in zip(("dq", "dk", "dv"), got, ref, oracle):
            assert torch.equal(a, r), (seed, name)
            err = np.abs(a.double().cpu().numpy() - o).max()
            assert err <= (1e-4 if dtype == "fp32" else 2e-2 * max(np.abs(o).max(), top)), (seed, name)


def test_long_blocks_at_the_row_limit(C):
    B, T, H, dh, L = 1, ROWS_MAX // 16, 16, 8, 128
    D = H * dh
    p = C.make_params(B, T, D, H, L, "fp32")
    q, k, v, dO = (t.cuda() for t in _inputs(B, T, D, torch.float32, 41))
    ref, got = _regular_and_noalloc(C, p, B, T, D, H, torch.float32, q, k, v, dO)
    for a, r in zip(got, ref):
        assert torch.isfinite(a).all() and torch.equal(a, r)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_calls_on_two_streams(C, dtype):
    B, T, H, dh, L = 2, 2048, 4, 64, 256
    D = H * dh
    tdt = torch.float32 if dtype == "fp32" else torch.bfloat16
    p = C.make_params(B, T, D, H, L, dtype)
    sets = []
    for seed in (51, 52):
        q, k, v, dO = (t.cuda() for t in _inputs(B, T, D, tdt, seed))
        o, lse = torch.empty_like(q), torch.empty(B, H, T, device="cuda")
        C.bcmt_test_attn(0, 0, p, q, k, v, D, o, lse)
        sets.append((q, k, v, o, lse, dO, [torch.empty_like(q) for _ in range(3)], torch.cuda.Stream()))

    def call(i):
        q, k, v, o, lse, dO, out, s = sets[i]
        C.bcmt_attention_backward_noalloc(p, q, k, v, D, o, lse, dO, *out, D, s)

    torch.cuda.synchronize()
    want = []
    for i in range(2):
        call(i)
        torch.cuda.synchronize()
        want.append([t.clone() for t in sets[i][6]])
        for t in sets[i][6]:
            t.fill_(float("nan"))
    torch.cuda.synchronize()
    for _ in range(8):
        call(0)
        call(1)
    torch.cuda.synchronize()
    for i in range(2):
        for a, r in zip(sets[i][6], want[i]):
            assert torch.equal(a, r)
