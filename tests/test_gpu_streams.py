"""Where a step may run and how its inputs and scalars travel: any stream, a caller's recording, pinned and pageable hosts."""
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


@pytest.mark.parametrize("on_default", [True, False])
def test_a_replayed_step_on_any_stream_equals_plain_launches(on_default):
    a, b = make(), make()
    a.lib.set_graph_replay(False)
    s = torch.cuda.Stream()
    for i in range(5):
        a.step(i)
        if on_default:
            b.step(i)
        else:
            s.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(s):
                b.step(i)
            torch.cuda.current_stream().wait_stream(s)
    torch.cuda.synchronize()
    close(state(b), state(a))
    assert a.lib.status() == 0 and b.lib.status() == 0
    assert a.lib.kernel_launches() == b.lib.kernel_launches()


def test_a_step_inside_a_callers_recording_joins_it():
    a, b = make(), make()
    s = torch.cuda.Stream()
    for tr in (a, b):                       # replay has started in both before one of them is recorded by its caller
        for i in range(3):
            tr.step(i)
    torch.cuda.synchronize()
    upd, tgt = b.dw.mb_slice(2), b.dw.targets(3)
    dw = b.dw
    g = torch.cuda.CUDAGraph()
    before = b.memory.clone()
    with torch.cuda.graph(g, stream=s):
        b.lib.train_step(dw.mb_src[upd], dw.mb_dst[upd], dw.mb_t[upd], dw.mb_eid[upd], dw.mb_keep[upd], *tgt, None, b.loss,
                         b.gradnorm)
    torch.cuda.synchronize()
    assert torch.equal(b.memory, before)    # recorded, not run
    g.replay()
    a.step(3)
    torch.cuda.synchronize()
    close(state(b)[:5], state(a)[:5])


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


def test_a_prune_behind_a_host_step_on_its_stream_counts_alone():
    """The host step's own prune runs beside it and counts endpoints in the context's table; what the caller enqueues next on the same
    stream comes behind it."""
    a, b = make(), make()
    loss, norm = torch.zeros(1).pin_memory(), torch.zeros(1).pin_memory()
    for i in range(1, 5):
        a.step_host(i, a.host_batch(i), loss, norm)
        a.prune(i - 1)
        b.prune(i - 1)
    torch.cuda.synchronize()
    cut = a.dw.mb_slice(3).stop
    assert torch.equal(a.dw.mb_keep[:cut], b.dw.mb_keep[:cut]) and torch.equal(a.dw.heavy[:4], b.dw.heavy[:4])
    assert a.lib.status() == 0
