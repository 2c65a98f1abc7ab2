"""The tcgen05 backward of general shapes holds P and dS to fp32's precision: of its bf16
gradients no more than twice as many differ from the rounded float64 result as of the
CUDA-core kernels', which hold both in fp32.  (What is left differs by the sums' order.
Values of 16 bits instead of 24, 2^-17 of each term, move about 2^-17 / 2^-9 = 0.4 % of
all roundings, four times the CUDA cores' own 0.1 %.)"""

import math

import pytest
import torch

pytestmark = pytest.mark.gpu


def _gradients(q, k, v, dO, o, L, H):
    """dQ, dK, dV in float64 from the given (rounded) O."""
    B, T, D = q.shape
    nb, dh = -(-T // L), D // H

    def blocks(z):
        z = torch.nn.functional.pad(z.double(), (0, 0, 0, nb * L - T))
        return z.view(B, nb, L, H, dh).transpose(2, 3)

    q, k, v, dO, o = map(blocks, (q, k, v, dO, o))
    hidden = torch.ones(L, L, dtype=torch.bool, device="cuda").triu(1)
    p = torch.softmax((q @ k.transpose(-1, -2) / math.sqrt(dh)).masked_fill(hidden, -math.inf), -1)
    ds = p * (dO @ v.transpose(-1, -2) - (dO * o).sum(-1, keepdim=True)) / math.sqrt(dh)
    out = (ds @ k, ds.transpose(-1, -2) @ q, p.transpose(-1, -2) @ dO)
    return [z.transpose(2, 3).reshape(B, nb * L, D)[:, :T] for z in out]


# one and two 64-column chunks, blocks of a part of a tile, a tile, several tiles
@pytest.mark.parametrize("B,T,H,dh,L", [(4, 1000, 8, 40, 48), (4, 1000, 8, 96, 48), (4, 1024, 8, 128, 128),
                                        (4, 1000, 8, 56, 200), (4, 1000, 8, 80, 256)])
def test_parts(cuda_ok, B, T, H, dh, L):
    from paper_2608_13578_gb300 import bcmt as C
    D = H * dh
    p = C.make_params(B, T, D, H, L, "bf16")
    gen = torch.Generator(device="cuda").manual_seed(dh + L)
    q, k, v, dO = (torch.randn(B, T, D, generator=gen, device="cuda").bfloat16() for _ in range(4))
    o, lse = torch.empty_like(q), torch.empty(B, H, T, device="cuda")
    C.bcmt_test_attn(0, 0, p, q, k, v, D, o, lse)
    want = [z.float().bfloat16() for z in _gradients(q, k, v, dO, o, L, H)]
    drow, off = torch.empty_like(lse), []
    for impl in (0, 3):
        g = [torch.empty_like(q) for _ in range(3)]
        C.bcmt_test_attn(impl, 1, p, q, k, v, D, o, lse, dO, drow, *g, D)
        C.bcmt_device_status()
        off.append(sum((x != w).double().mean().item() for x, w in zip(g, want)) / 3)
    assert off[1] <= 2 * off[0], off
