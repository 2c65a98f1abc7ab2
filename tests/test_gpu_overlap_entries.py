"""Queued passes against passes alone (bit for bit, as in test_gpu_overlap.py) for the
other entries and kernels -- Q/K/V inputs, HOnly, the one-pass attention backward, a
learned decay, decoding -- and with every launch on the caller's stream."""

import pytest
import torch

from paper_2608_13578_gb300.inputs import Workload, make_inputs

pytestmark = pytest.mark.gpu

CASES = [
    # B, T, D, H, L, dtype, from x, honly
    (2, 256, 128, 2, 64, "bf16", False, False),
    (3, 200, 192, 3, 48, "fp32", False, False),
    (2, 256, 128, 2, 64, "bf16", True, True),
    (2, 512, 128, 2, 256, "bf16", True, False),   # one-pass backward, heads of 64
    (1, 700, 128, 8, 512, "bf16", True, False),   # and of 16
    (2, 256, 512, 8, 64, "bf16", True, False),    # grouped weight gradients
    (2, 100, 1088, 17, 32, "bf16", True, False),  # D beyond the register-held pooling backward
    (2, 256, 128, 4, 32, "fp32", True, False),
]


@pytest.fixture(params=[True, False], ids=["side streams", "one stream"])
def C(request, cuda_ok):
    from paper_2608_13578_gb300 import bcmt
    bcmt.bcmt_test_set_side_streams(request.param)
    yield bcmt
    bcmt.bcmt_test_set_side_streams(True)


def _setup(B, T, D, H, L, dtype, from_x, honly, seeds):
    from paper_2608_13578_gb300 import layer
    w = Workload("overlap", B, T, D, H, L, dtype, decay=(0.5, 0.99), input_is_x=from_x, honly=honly)
    ins = [{k: v.cuda() for k, v in make_inputs(w, seed=s).items()} for s in seeds]
    return layer, layer.params_for(B, T, D, H, L, dtype, from_x, honly), ins


@pytest.mark.parametrize("case", CASES)
def test_queued_passes(C, case):
    layer, p, ins = _setup(*case, seeds=(1, 2))
    ws = layer._buffer(C.bcmt_workspace_size(p), "cuda")
    scratch = layer._buffer(C.bcmt_scratch_size(p), "cuda")

    def step(t):
        y, _ = layer.forward(p, t, workspace=ws)
        return {"y": y, **layer.backward(p, t, ws, t["dy"], scratch=scratch)}

    torch.cuda.synchronize()
    alone = step(ins[0])
    torch.cuda.synchronize()
    for _ in range(4):
        step(ins[1])
        queued = step(ins[0])
    torch.cuda.synchronize()
    for n in alone:
        assert torch.equal(alone[n], queued[n]), n


@pytest.mark.parametrize("case", [c for c in CASES if c[6]])
def test_stacked_layers(C, case):
    """dX of one layer is dY of the layer below with nothing in between."""
    layer, p, (t,) = _setup(*case, seeds=(3,))
    y1, ws1 = layer.forward(p, t)
    t2 = dict(t, x=y1)
    _, ws2 = layer.forward(p, t2)
    torch.cuda.synchronize()
    g2 = layer.backward(p, t2, ws2, t["dy"])
    torch.cuda.synchronize()
    want = layer.backward(p, t, ws1, g2["dx"])
    torch.cuda.synchronize()
    dx = torch.full_like(g2["dx"], float("nan"))
    for _ in range(4):
        dx.fill_(float("nan"))
        layer.backward(p, t2, ws2, t["dy"], out=dict(g2, dx=dx))
        got = layer.backward(p, t, ws1, dx)
    torch.cuda.synchronize()
    for n in want:
        assert torch.equal(want[n], got[n]), n


@pytest.mark.parametrize("B,T,D,H,L,dtype", [(1, 40, 128, 2, 16, "bf16"), (5, 40, 256, 2, 8, "bf16"),
                                             (2, 24, 128, 4, 8, "fp32")])
def test_queued_tokens(cuda_ok, B, T, D, H, L, dtype):
    """Tokens decoded one behind the other, each layer's output the next one's input."""
    layer, _, (t,) = _setup(B, T, D, H, L, dtype, True, False, seeds=(4,))
    x = t["x"].transpose(0, 1).contiguous()

    def run(wait):
        decs = [layer.Decoder(t, B, H, L) for _ in range(2)]
        ys = []
        for x_t in x:
            for dec in decs:
                x_t = dec.step(x_t)
                if wait:
                    torch.cuda.synchronize()
            ys.append(x_t)
        torch.cuda.synchronize()
        return torch.stack(ys)

    want = run(True)
    for _ in range(3):
        assert torch.equal(run(False), want)
