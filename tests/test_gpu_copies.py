"""Gradient rows summed over copies: the update cell's gradient against the oracle where a few rows get most of the additions
(32 copies) and where rows and additions are about as many (8), for both models and the smallest and a wide row."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("model", ["tgn", "jodie"])
@pytest.mark.parametrize("nodes,batch,d,k", [(3, 64, 4, 10), (40, 200, 100, 10), (1500, 200, 100, 5), (12, 100, 160, 20)])
def test_cell_gradient_is_the_sum_over_the_copies(model, nodes, batch, d, k):
    from paper_2608_16305_b200 import binding as B, trainer as T, workload as wl
    cfg = wl.WorkloadConfig("copies", nodes, 0, 6 * batch, 0, "f32", d, k, 2, batch, 0.0, False, 1.1, 1.1, 5)
    dw = T.DeviceWorkload(wl.make_stream(cfg))
    tr = T.Trainer(dw, wl.make_weights(d, 0, 5, bias_scale=0.1, model=model), model=model, lr=0.0)
    lay, P = B.param_layout(tr.tcfg), tr.params.numel()
    names = ("rnn_w_i", "rnn_w_h") if model == "jodie" else ("gru_w_i", "gru_w_h")
    sizes = [(3 * d if model == "jodie" else 3 * d) * d * (1 if model == "jodie" else 3), d * d * (1 if model == "jodie" else 3)]
    snap, grads = [], []
    for b in range(5):      # the same steps from the same state twice: whatever the additions' order, the sums agree
        tr.step(b)
    state = [x.clone() for x in (tr.memory, tr.last_update)]
    for _ in range(3):
        tr.memory.copy_(state[0]); tr.last_update.copy_(state[1])
        tr.step(5)
        g = torch.zeros(P, device="cuda")
        tr.lib.debug_get_grads(g)
        grads.append(g.double())
    torch.cuda.synchronize()
    assert tr.lib.status() == 0
    for n, s in zip(names, sizes):
        a = [g[lay[n]:lay[n] + s] for g in grads]
        assert a[0].abs().max() > 0
        for x in a[1:]:
            # fp32 sums of up to batch * k terms in another order: 1e-6 of their magnitude, which cancellation may raise tenfold;
            # a copy left out or counted twice moves them by its share, at least 1 / 32 of the terms
            assert (x - a[0]).norm() <= 1e-4 * a[0].norm()
