"""The CUDA-core attention's one-dimensional grid: blocks longer than the sequence get
tiles for the sequence alone, many short sequences, and a grid beyond what a launch
takes, which is an error and not a smaller grid."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C(cuda_ok):
    from paper_2608_13578_gb300 import bcmt
    return bcmt


def _run(C, B, T, H, dh, L, ins):
    D, (q, k, v, dO) = H * dh, ins
    p = C.make_params(B, T, D, H, L, "fp32")
    o, lse = torch.empty_like(q), torch.empty(B, H, T, device="cuda")
    C.bcmt_test_attn(0, 0, p, q, k, v, D, o, lse)
    g, drow = [torch.empty_like(q) for _ in range(3)], torch.empty_like(lse)
    C.bcmt_test_attn(0, 1, p, q, k, v, D, o, lse, dO, drow, *g, D)
    torch.cuda.synchronize()
    return [o, lse, *g]


@pytest.mark.parametrize("B,T,H,dh", [(3, 70, 4, 32), (2, 130, 1, 128), (70000, 1, 8, 8), (2, 64, 8, 24)])
def test_blocks_longer_than_the_sequence(C, B, T, H, dh):
    """A block of T tokens and one of 1000 are the same for a sequence of T, where both
    run the kernels of long blocks (T > 64) bit for bit."""
    gen = torch.Generator(device="cuda").manual_seed(T)
    ins = [torch.randn(B, T, H * dh, generator=gen, device="cuda") for _ in range(4)]
    for a, b in zip(_run(C, B, T, H, dh, T, ins), _run(C, B, T, H, dh, 1000, ins)):
        assert torch.equal(a, b) if T > 64 else (a - b).abs().max() <= 1e-5 * (1 + b.abs().max())


def test_a_grid_too_large_is_refused(C):
    """2^18 tiles of 2^14 heads: refused on the host (the pointers are never used)."""
    a, D = 1 << 20, 8 << 14
    p = C.make_params(1 << 18, 1, D, 1 << 14, 64, "fp32")
    with pytest.raises(C.BCMTError):
        C.bcmt_test_attn(0, 0, p, a, a, a, D, a, a)
