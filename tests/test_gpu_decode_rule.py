"""Which form a bf16 decoding step takes, on both sides of each line of the rule: sizes
whose staged step is the faster one take it (seen by the step temporaries that it alone
leaves in the state), the others the one launch; each gives bit for bit what that form
gives, and both are right wherever the rule lies."""

import pytest
import torch

from paper_2608_13578_gb300.inputs import Workload, make_inputs
from tests.helpers import assert_close, oracle_run

pytestmark = pytest.mark.gpu

CASES = [
    # B, D, H, L, staged
    (1, 1280, 20, 8, True), (1, 1024, 16, 8, False), (2, 1280, 20, 8, False),
    (1, 1280, 20, 256, False),
    (49, 320, 5, 4, True), (48, 320, 5, 4, False), (49, 384, 6, 4, False), (49, 128, 2, 256, False),
    (70, 128, 1, 4, True), (1000, 64, 8, 4, True), (1000, 576, 9, 4, True), (1000, 640, 10, 4, False),
]


@pytest.fixture()
def C(cuda_ok):
    from paper_2608_13578_gb300 import bcmt
    yield bcmt
    bcmt.bcmt_test_set_decode_one_launch(1)


@pytest.mark.parametrize("B,D,H,L,staged", CASES)
def test_form(C, B, D, H, L, staged):
    from paper_2608_13578_gb300 import layer
    T = 9 if L < 9 else 3
    w = Workload("decode", B, T, D, H, L, "bf16", False, (0.5, 0.99), 51)
    t = make_inputs(w)
    dev = {k: v.cuda() for k, v in t.items()}
    cache = -(-B * L * D * 2 // 256) * 256  # the keys, then the values; then the token's rows in fp32
    y, is_staged = {}, {}
    for mode in (0, 1, 2):
        C.bcmt_test_set_decode_one_launch(mode)
        dec = layer.Decoder(dev, B, H, L)
        y[mode] = torch.stack([dec.step(dev["x"][:, i]) for i in range(T)], dim=1)
        is_staged[mode] = bool(dec.state[2 * cache:2 * cache + B * D * 4].any())
    assert is_staged == {0: True, 1: staged, 2: False}
    assert torch.equal(y[1], y[0] if staged else y[2])
    rows = slice(0, min(B, 8)) if B <= 100 else slice(B - 8, B)
    fw, _ = oracle_run(w, t, backward=False, batch=rows)
    for mode in (0, 2):
        assert_close("Y", y[mode][rows], fw["Y"], "bf16")
