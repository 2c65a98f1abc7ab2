"""The one-launch bf16 decoding step over the shapes its layout depends on: more
heads than CTAs of a cluster, few heads in parts, column counts that do not divide
among the CTAs, more than eight sequences per cluster, blocks too long to stage,
HOnly; each token's row against the float64 oracle's forward (bf16: 2e-2)."""

import pytest
import torch

from paper_2608_13578_gb300.inputs import Workload, make_inputs
from tests.helpers import assert_close, oracle_run

pytestmark = pytest.mark.gpu

CASES = [
    # B, T, D, H, L, honly
    (1, 40, 64, 1, 16, False),        # one head in parts; CTAs without columns
    (1, 70, 64, 8, 32, False),        # heads of 8
    (2, 40, 640, 40, 16, False),      # 40 heads of 16: several per CTA
    (3, 40, 384, 4, 16, False),       # heads of 96
    (5, 66, 192, 3, 33, False),       # 24 column groups over 16 CTAs
    (17, 36, 128, 2, 12, False),      # uneven clusters
    (40, 20, 256, 4, 8, False),       # ten sequences per cluster
    (70, 6, 128, 1, 4, False),        # more clusters than four
    (2, 90, 1024, 8, 1024, False),    # a long block's cache stays in global memory
    (1, 600, 128, 2, 512, False),
    (9, 20, 512, 8, 8, True),
    (2, 20, 128, 2, 1, False),        # every token its own block
]


@pytest.mark.parametrize("B,T,D,H,L,honly", CASES)
def test_decode_shapes(cuda_ok, B, T, D, H, L, honly):
    from paper_2608_13578_gb300 import layer
    w = Workload("decode", B, T, D, H, L, "bf16", False, (0.5, 0.99), 31, True, honly)
    t = make_inputs(w)
    dev = {k: v.cuda() for k, v in t.items()}
    dec = layer.Decoder(dev, B, H, L, honly=honly)
    y = torch.stack([dec.step(dev["x"][:, i]) for i in range(T)], dim=1)
    torch.cuda.synchronize()
    fw, _ = oracle_run(w, t, backward=False)
    assert_close("Y", y, fw["Y"], "bf16")
