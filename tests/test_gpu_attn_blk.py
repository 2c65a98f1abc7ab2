"""The one-pass attention backward of blocks of several 128-token tiles, against the
float64 oracle and the CUDA-core kernels.

Tolerances: the library's 2e-2 against the oracle; against the CUDA-core backward,
which holds P and dS in fp32 where the tensor cores take them as bf16 (2^-9 of each
term, and the sums' own bf16 rounding), 2^-6 of the largest value."""

import numpy as np
import pytest
import torch

from tests.test_gpu_attn_gen import _inputs, _run
from tests.test_gpu_kernels import _attn_ref

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C(cuda_ok):
    from paper_2608_13578_gb300 import bcmt
    return bcmt


@pytest.mark.parametrize("B,T,H,dh,L,pad", [
    (2, 512, 2, 64, 256, 0),
    (1, 700, 2, 64, 256, 64),     # ragged last block: a tile and 60 rows; strided rows
    (1, 129, 2, 32, 256, 0),      # the second tile holds one row
    (1, 1, 4, 16, 256, 0),        # one token
    (2, 1100, 2, 32, 384, 0),     # odd tile count, ragged
    (1, 900, 2, 32, 768, 0),      # the most tiles at this width
    (1, 2048, 4, 16, 1024, 0),
    (2, 1000, 4, 16, 896, 64),
    (8, 1024, 16, 16, 512, 0),    # more blocks than SMs
    (40, 300, 4, 16, 256, 0),     # and every second one a single tile
    (24, 1000, 8, 32, 384, 0),    # three, three, two tiles
    (30, 700, 6, 64, 256, 0),
])
def test_one_pass_backward(C, B, T, H, dh, L, pad):
    q, k, v, dO = _inputs(B, T, H, dh)
    D = H * dh
    p = C.make_params(B, T, D, H, L, "bf16")
    ld = D + pad
    wide = [torch.nn.functional.pad(t, (0, pad)).cuda() for t in (q, k, v)]
    _, _, got = _run(C, 4, p, B, T, D, H, *wide, dO.cuda(), ld)
    _, _, simt = _run(C, 0, p, B, T, D, H, *wide, dO.cuda(), ld)
    ref = _attn_ref(*(t.double().numpy() for t in (q, k, v)), L, H, dO.double().numpy())[2:]
    top = np.abs(ref[2]).max()
    for n, x, y, r in zip(("dq", "dk", "dv"), got, simt, ref):
        x = x.double().cpu().numpy()
        assert np.isfinite(x).all(), n
        assert np.abs(x - r).max() <= 2e-2 * max(np.abs(r).max(), top), n
        assert np.abs(x - y.double().cpu().numpy()).max() <= 2 ** -6 * top, n


@pytest.mark.parametrize("B,T,H,dh,L", [(1, 700, 2, 64, 256), (2, 600, 4, 16, 512), (1, 400, 2, 32, 384)])
@pytest.mark.parametrize("which,value", [("v", float("inf")), ("dO", float("nan")), ("k", float("nan")),
                                         ("q", float("inf"))])
def test_non_finite_tokens(C, B, T, H, dh, L, which, value):
    """A non-finite token reaches the rows that see it (where the CUDA-core kernels have
    it), nothing that it does not reach in the two-kernel form (hidden rows of its tile),
    and no other head, block or sequence: those are the same bit for bit."""
    ins = dict(zip(("q", "k", "v", "dO"), (t.cuda() for t in _inputs(B, T, H, dh))))
    D = H * dh
    p = C.make_params(B, T, D, H, L, "bf16")
    clean = _run(C, 4, p, B, T, D, H, *ins.values())[2]
    ins[which][0, 130, 5] = value
    blk, two, simt = (_run(C, impl, p, B, T, D, H, *ins.values())[2] for impl in (4, 2, 0))
    for x, y, s, z in zip(blk, two, simt, clean):
        assert not (torch.isfinite(x) & ~torch.isfinite(s)).any()
        assert not (~torch.isfinite(x) & torch.isfinite(y)).any()
        assert torch.equal(x[..., dh:], z[..., dh:]) and torch.equal(x[1:], z[1:])
        assert torch.equal(x[:, L:], z[:, L:])
    assert any(not torch.isfinite(x).all() for x in blk)
