"""The step's first launch forgets which rows the step before has updated: the gradients of a step behind another with other nodes are those of the same step in
a context that has run nothing before it."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

D, DE, K, E, UPDATES = 32, 6, 5, 70000, 4000


# the nodes of the step before: some, more than the 4 x 1 024 that are asked for ahead; a table in shared memory and one that does not fit (51 200 nodes)
@pytest.mark.parametrize("math,model", [("FP32", "TGN"), ("F16X3", "TGN"), ("FP32", "JODIE")])
@pytest.mark.parametrize("N,before", [(3000, 300), (20000, UPDATES), (60000, UPDATES)])
def test_a_step_behind_another_is_the_step_alone(N, before, math, model):
    from paper_2608_16305_b200 import binding as B, workload as wl
    g = torch.Generator(device="cuda").manual_seed(N + before)
    ints = lambda n, hi: torch.randint(0, hi, (n,), device="cuda", generator=g, dtype=torch.int32)
    times = lambda n: torch.rand(n, device="cuda", generator=g, dtype=torch.float64).sort().values
    z = lambda *s, dt=torch.float32: torch.zeros(s, dtype=dt, device="cuda")
    per = 2 * E // N + 1
    graph = (torch.arange(N + 1, device="cuda") * per, ints(N * per, N), ints(N * per, E), times(N * per).reshape(per, N).T.reshape(-1).contiguous())
    feat, memory = torch.randn((E, DE), device="cuda", generator=g), torch.randn((N, D), device="cuda", generator=g)
    cfg = B.make_config(N, D, DE, K, 2, max_events=UPDATES, max_roots=900, math_mode=getattr(B, "TGNN_MATH_" + math), model=getattr(B, "TGNN_MODEL_" + model))
    params = torch.from_numpy(B.pack_params(cfg, wl.make_weights(D, DE, 7, bias_scale=0.1, model=model.lower()))).cuda()
    batch = lambda n_u: (ints(n_u, N), ints(n_u, N), times(n_u), torch.arange(n_u, device="cuda", dtype=torch.int32))
    first, second = batch(before), batch(50)
    if before == UPDATES:
        assert torch.cat(first[:2]).unique().numel() > 4 * 1024
    q = (ints(300, N), ints(300, N), ints(300, N), 1.0 + times(300))
    grads = []
    for steps in ((first, second), (second,)):
        lib = B.Tgnn(cfg)
        state = [x.clone() for x in (memory, z(N, dt=torch.float64), params, torch.zeros_like(params), torch.zeros_like(params), z(1, dt=torch.int64))]
        start = [x.clone() for x in state]
        loss, norm, grad = z(1), z(1), torch.zeros_like(params)
        lib.set_graph(*graph)
        lib.set_edge_features(feat, E)
        lib.set_state(*state)
        for u in steps:
            for x, y in zip(state, start):
                x.copy_(y)
            lib.train_step(*u, None, *q, None, loss, norm)
        lib.debug_get_grads(grad)
        torch.cuda.synchronize()
        assert lib.status() == 0
        grads.append(grad.double())
    # the same sums in another order: 2^-24 of the magnitudes of a few thousand terms of both signs
    assert (grads[0] - grads[1]).norm() <= 2e-5 * grads[1].norm()
