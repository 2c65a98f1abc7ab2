"""bf16 decoding as a launch per stage (the sizes that the one-launch step does not hold)
and non-finite tokens in either form."""

import pytest
import torch

from paper_2608_13578_gb300.inputs import Workload, make_inputs
from tests.helpers import assert_close, oracle_run

pytestmark = pytest.mark.gpu


@pytest.fixture()
def C(cuda_ok):
    from paper_2608_13578_gb300 import bcmt
    yield bcmt
    bcmt.bcmt_test_set_decode_one_launch(True)


def _decode(C, dev, B, T, H, L, honly, one_launch, x=None):
    from paper_2608_13578_gb300 import layer
    C.bcmt_test_set_decode_one_launch(one_launch)
    x = dev["x"] if x is None else x
    dec = layer.Decoder(dev, B, H, L, honly=honly)
    y = torch.stack([dec.step(x[:, i]) for i in range(T)], dim=1)
    torch.cuda.synchronize()
    return y


def _case(B, T, D, H, L, honly):
    w = Workload("decode", B, T, D, H, L, "bf16", False, (0.5, 0.99), 41, True, honly)
    t = make_inputs(w)
    return w, t, {k: v.cuda() for k, v in t.items()}


@pytest.mark.parametrize("honly", [False, True])
def test_size_beyond_the_one_launch_step(C, honly):
    """Sixteen sequences of 2048 columns per cluster: 131 KB of rows and 64 KB of partial
    sums leave no room for the rest.  The switch changes nothing there."""
    B, T, D, H, L = 64, 10, 2048, 32, 4
    w, t, dev = _case(B, T, D, H, L, honly)
    y = _decode(C, dev, B, T, H, L, honly, True)
    assert torch.equal(y, _decode(C, dev, B, T, H, L, honly, False))
    fw, _ = oracle_run(w, t, backward=False)
    assert_close("Y", y, fw["Y"], "bf16")


@pytest.mark.parametrize("B,T,D,H,L,honly", [
    (1, 40, 128, 2, 16, False),
    (3, 70, 256, 4, 64, False),
    (17, 36, 128, 1, 12, False),
    (2, 20, 128, 2, 1, False),
    (5, 24, 192, 3, 8, True),
])
def test_staged_steps(C, B, T, D, H, L, honly):
    w, t, dev = _case(B, T, D, H, L, honly)
    fw, _ = oracle_run(w, t, backward=False)
    assert_close("Y", _decode(C, dev, B, T, H, L, honly, False), fw["Y"], "bf16")


@pytest.mark.parametrize("one_launch", [True, False])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("B,T,D,H,L", [(5, 30, 128, 2, 8), (20, 20, 256, 4, 16), (2, 24, 64, 1, 8)])
def test_non_finite_tokens_stay_in_their_sequence(C, B, T, D, H, L, value, one_launch):
    """One value of one token of sequence 1: that sequence is non-finite from there on
    (its memory carries it), the others and its earlier tokens are the same bit for bit."""
    _, _, dev = _case(B, T, D, H, L, False)
    y0 = _decode(C, dev, B, T, H, L, False, one_launch)
    x = dev["x"].clone()
    x[1, 5, 3] = value
    y = _decode(C, dev, B, T, H, L, False, one_launch, x)
    keep = torch.ones(B, T, dtype=torch.bool, device="cuda")
    keep[1, 5:] = False
    assert torch.equal(y[keep], y0[keep])
    assert not torch.isfinite(y[1, 5]).any() and not torch.isfinite(y[1, T - 1]).all()
