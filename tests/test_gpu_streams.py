"""How a step's inputs and scalars travel: pinned and pageable hosts."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def make(model="tgn", embed_aux=False):
    from paper_2608_16305_b200 import binding as B, trainer as T, workload as wl
    cfg = wl.scaled(wl.CONFIGS["reddit"], num_events=3000)
    dw = T.DeviceWorkload(wl.make_stream(cfg), embed_aux=embed_aux)
    return T.Trainer(dw, wl.make_weights(cfg.d, cfg.d_e, 3, bias_scale=0.1, model=model), math_mode=B.TGNN_MATH_TF32,
                     model=model)


def state(tr):
    return [x.clone() for x in (tr.memory, tr.last_update, tr.adam_m, tr.loss, tr.gradnorm, tr.dw.mb_keep)]


def close(a, b):
    for x, y in zip(a, b):
        x, y = x.double(), y.double()
        assert (x - y).norm() <= 1e-4 * y.norm() + 1e-12    # gradients: fp32 atomics in another order, with a ReLU kink now and then


@pytest.mark.parametrize("model", ["tgn", "jodie"])
@pytest.mark.parametrize("embed_aux", [False, True])
def test_host_scalars_pinned_pageable_and_absent(model, embed_aux):
    trs = [make(model, embed_aux) for _ in range(3)]
    pin = [torch.full((4,), -7.0).pin_memory(), torch.full((4,), -7.0).pin_memory()]
    page = [torch.full((4,), -7.0), torch.full((4,), -7.0)]
    for i in range(4):      # one element per step, so that a step that wrote through a stale address would show
        trs[0].step_host(i, trs[0].host_batch(i), pin[0][i:i + 1], pin[1][i:i + 1])
        trs[1].step_host(i, trs[1].host_batch(i), page[0][i:i + 1], page[1][i:i + 1])
        trs[2].step_host(i, trs[2].host_batch(i), None, pin[1].new_empty(1) if i == 3 else None)
    torch.cuda.synchronize()
    for p, q in zip(pin, page):
        assert (p > 0).all() and np.allclose(p.numpy(), q.numpy(), rtol=1e-4)
    close([trs[2].memory, trs[2].adam_m], [trs[0].memory, trs[0].adam_m])
    trs[0].lib.set_state(trs[0].memory, trs[0].last_update, trs[0].params, trs[0].adam_m, trs[0].adam_v, trs[0].step_count)
    last = pin[0].clone()
    trs[0].step(4)                          # a step from device arrays leaves the host's scalars alone
    torch.cuda.synchronize()
    assert torch.equal(pin[0], last)
