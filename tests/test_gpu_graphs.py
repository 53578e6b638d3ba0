"""The layer's calls under stream capture: a graph computes anew each time it runs, whatever ran between."""
import pytest
import torch

from paper_2605_23764_b200 import MoeLayer
from tests.gpu_util import small_problem

pytestmark = pytest.mark.gpu
T, d, E, k, S, F = 640, 136, 12, 3, 1, 72


def _problem():
    x, W1, W2, logits, dout = small_problem(T, d, E, k, S, F, 8)
    douts = [dout, (dout.float() * -0.5).to(torch.bfloat16), dout.flip(0).contiguous()]
    return x, W1, W2, logits, douts


def _capture(fn):
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        res = fn()
    return g, res


@pytest.mark.parametrize("serial", [False, True])
@pytest.mark.parametrize("forward", ["eager", "graph", "same graph"])
def test_captured_backward_runs_again(forward, serial):
    x, W1, W2, logits, douts = _problem()
    ref = MoeLayer(T, d, E, k, S, F, save_for_bwd=True, serial=serial)
    layer = MoeLayer(T, d, E, k, S, F, save_for_bwd=True, serial=serial)
    ids, w = ref.route(logits)
    ids[5, 1] = E + 7   # a dropped slot: its weight's gradient is zero
    ref.ffn_fwd(x, ids, w, W1, W2)
    want = [[t.clone() for t in ref.ffn_bwd(g, x, ids, w, W1, W2)] for g in douts]
    dout = douts[0].clone()
    # (the first launches of a kernel set its attributes: once outside the capture)
    layer.ffn_fwd(x, ids, w, W1, W2)
    layer.ffn_bwd(dout, x, ids, w, W1, W2)
    if forward == "same graph":
        def both():
            layer.ffn_fwd(x, ids, w, W1, W2)
            return layer.ffn_bwd(dout, x, ids, w, W1, W2)
        graph, res = _capture(both)
    else:
        if forward == "graph":
            fwd, _ = _capture(lambda: layer.ffn_fwd(x, ids, w, W1, W2))
            fwd.replay()
        else:
            layer.ffn_fwd(x, ids, w, W1, W2)
        graph, res = _capture(lambda: layer.ffn_bwd(dout, x, ids, w, W1, W2))
    for g, expect in zip(douts, want):   # several gradients behind one forward
        dout.copy_(g)
        for t in res:
            t.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        for got, exp, name in zip(res, expect, ("dx", "dW_gate_up", "dW_down", "d_topk_w")):
            assert torch.equal(got, exp), name
    # and an eager backward behind a replayed forward
    if forward == "graph":
        fwd.replay()
        for got, exp in zip(layer.ffn_bwd(dout.copy_(douts[1]), x, ids, w, W1, W2), want[1]):
            assert torch.equal(got, exp)
    layer.close()
    ref.close()
