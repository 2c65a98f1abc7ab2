"""Passes queued one behind the other on one stream, on the same workspace and
scratch with other inputs in between, give bit for bit what a pass alone gives:
every kernel reads what earlier kernels wrote only after its wait for them,
however early it is launched.  Small shapes, whose kernels are resident together."""

import pytest
import torch

from paper_2608_13578_gb300.inputs import Workload, make_inputs

pytestmark = pytest.mark.gpu

SHAPES = [
    # B, T, D, H, L, dtype
    (10, 64, 384, 12, 16, "fp32"),
    (7, 1024, 64, 4, 64, "fp32"),
    (1, 256, 128, 4, 32, "fp32"),
    (2, 256, 128, 2, 64, "bf16"),
    (2, 200, 256, 4, 32, "bf16"),
    (2, 300, 384, 4, 48, "bf16"),
    (1, 600, 256, 4, 512, "bf16"),
]


@pytest.mark.parametrize("decay_grad", [False, True])
@pytest.mark.parametrize("B,T,D,H,L,dtype", SHAPES)
def test_queued_passes_match_a_pass_alone(cuda_ok, B, T, D, H, L, dtype, decay_grad):
    from paper_2608_13578_gb300 import layer
    w = Workload("overlap", B, T, D, H, L, dtype, decay=(0.5, 0.99))
    ins = [{k: v.cuda() for k, v in make_inputs(w, seed=s).items()} for s in (1, 2)]
    p = layer.params_for(B, T, D, H, L, dtype)
    ws = layer._buffer(layer.C.bcmt_workspace_size(p), "cuda")
    scratch = layer._buffer(layer.C.bcmt_scratch_size(p), "cuda")

    def step(t, dy):
        y, _ = layer.forward(p, t, workspace=ws)
        return {"y": y, **layer.backward(p, t, ws, dy, scratch=scratch, decay_grad=decay_grad)}

    torch.cuda.synchronize()
    alone = step(ins[0], ins[0]["dy"])
    torch.cuda.synchronize()
    for _ in range(4):
        step(ins[1], ins[1]["dy"])
        queued = step(ins[0], ins[0]["dy"])
    torch.cuda.synchronize()
    for n in alone:
        assert torch.equal(alone[n], queued[n]), n


@pytest.mark.parametrize("B,T,D,H,L,dtype", SHAPES)
def test_stacked_layers(cuda_ok, B, T, D, H, L, dtype):
    """dX of one layer is dY of the layer below with nothing in between."""
    from paper_2608_13578_gb300 import layer
    w = Workload("stacked", B, T, D, H, L, dtype, decay=(0.5, 0.99))
    t = {k: v.cuda() for k, v in make_inputs(w, seed=3).items()}
    p = layer.params_for(B, T, D, H, L, dtype)
    y1, ws1 = layer.forward(p, t)
    t2 = dict(t, x=y1)
    _, ws2 = layer.forward(p, t2)
    torch.cuda.synchronize()
    g2 = layer.backward(p, t2, ws2, t["dy"])
    torch.cuda.synchronize()
    want = layer.backward(p, t, ws1, g2["dx"])
    torch.cuda.synchronize()
    dx = torch.full_like(g2["dx"], float("nan"))
    out = dict(g2, dx=dx)
    for _ in range(4):
        dx.fill_(float("nan"))
        layer.backward(p, t2, ws2, t["dy"], out=out)
        got = layer.backward(p, t, ws1, dx)
    torch.cuda.synchronize()
    for n in want:
        assert torch.equal(want[n], got[n]), n
