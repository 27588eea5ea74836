"""The link-prediction head's forms at the edges of their blocks, against the same formulas in fp64.

The time-projection model without a memory update: its embedding is one product, so the head's part of the gradient and
d loss / d h (through w_p and b_p) are all there is to a step."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("d", [4, 36, 100, 128, 256])
@pytest.mark.parametrize("n_q", [1, 3, 4, 5, 299, 600, 743, 889, 1185, 2367, 2368, 4900])
@pytest.mark.parametrize("masked", [False, True])
def test_head_forward_and_backward(d, n_q, masked):
    from paper_2608_16305_b200 import binding as B, workload as wl
    if n_q > 600 and masked and d != 100 or n_q > 4000 and d not in (36, 100):
        pytest.skip("the same code at every size")
    N = 500
    cfg = B.make_config(N, d, 0, 5, 2, max_events=4, max_roots=3 * n_q, model=B.TGNN_MODEL_JODIE)
    lib, lay = B.Tgnn(cfg), B.param_layout(cfg)
    weights = wl.make_weights(d, 0, 5, bias_scale=0.1, model="jodie")
    g = torch.Generator(device="cuda").manual_seed(n_q * 1000 + d)
    z = lambda *s, dt=torch.float32: torch.zeros(s, dtype=dt, device="cuda")
    memory = torch.randn((N, d), device="cuda", generator=g)
    last, step = z(N, dt=torch.float64), z(1, dt=torch.int64)
    params = torch.from_numpy(B.pack_params(cfg, weights)).cuda()
    m, v = z(lay["total"]), z(lay["total"])
    lib.set_graph(z(N + 1, dt=torch.int64), z(1, dt=torch.int32), z(1, dt=torch.int32), z(1, dt=torch.float64))
    lib.set_edge_features(None, 0)
    lib.set_state(memory, last, params, m, v, step)
    nodes = torch.randint(0, N, (3 * n_q,), device="cuda", generator=g, dtype=torch.int32)
    times = torch.rand(n_q, device="cuda", generator=g, dtype=torch.float64).repeat(3)
    h, loss, gn, grads = z(3 * n_q, d), z(1), z(1), z(lay["total"])
    mask = (torch.rand(n_q, device="cuda", generator=g) < 0.6).to(torch.uint8) if masked else None
    lib.embed(nodes, times, None, None, None, None, h)
    p64 = {n: torch.from_numpy(np.asarray(weights[n], dtype=np.float64)).cuda().requires_grad_() for n in ("w_1", "b_1", "w_2", "b_2")}
    h64 = h.double().requires_grad_()
    hs, hd, hn = h64[:n_q], h64[n_q:2 * n_q], h64[2 * n_q:]
    pre = lambda a, b: torch.cat((a, b), 1) @ p64["w_1"].reshape(d, 2 * d).T + p64["b_1"]
    pos, neg = pre(hs, hd), pre(hs, hn)
    score = lambda x: torch.relu(x) @ p64["w_2"].reshape(-1) + p64["b_2"]
    w = torch.ones(n_q, device="cuda", dtype=torch.float64) if mask is None else mask.double()
    w = w / w.sum().clamp(min=1)
    ref = (w * (torch.nn.functional.softplus(-score(pos)) + torch.nn.functional.softplus(score(neg)))).sum()
    ref.backward()
    # one sum of n_q d terms per entry in fp32, with atomics: a few 1e-7 of its terms' magnitude; a hidden unit whose
    # pre-activation is within 1e-6 of zero may take the other branch, which moves an entry by at most its own term
    near = sum(int((x.abs() < 2e-6).sum()) for x in (pos, neg))
    tol = 2e-5 if near == 0 else 2e-3
    lib.backward_step(n_q, mask, loss, gn)
    lib.debug_get_grads(grads)
    torch.cuda.synchronize()
    assert lib.status() == 0
    assert abs(loss.item() - ref.item()) <= 1e-5 * max(ref.item(), 1e-3)
    mem64 = memory.double()[nodes.long()]
    dt = times.float().double()[:, None]
    want = {n: p64[n].grad.reshape(-1) for n in p64}
    want["proj_w"], want["proj_b"] = (h64.grad * mem64 * dt).sum(0), (h64.grad * mem64).sum(0)
    for n, x in want.items():
        got = grads[lay[n]:lay[n] + x.numel()].double()
        if n == "b_2":      # one number, a difference of sums that nearly cancel: measured by its terms
            assert (got - x).abs().item() <= 1e-5
            continue
        assert (got - x).norm() <= tol * x.norm() + 1e-9, (n, ((got - x).norm() / x.norm()).item(), near)
