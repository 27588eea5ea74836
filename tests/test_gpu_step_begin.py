"""The step's first launch (staging, roots, latest-event reduction, weight images) at the edges of its blocks of 1 024 threads:
a step leaves the state and the embeddings that its parts leave when they are called one by one."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N, D, DE, K = 3000, 32, 6, 5


class Context:
    def __init__(self, math, n_u, n_q, seed=11):
        from paper_2608_16305_b200 import binding as B, workload as wl
        cfg = B.make_config(N, D, DE, K, 2, max_events=2100, max_roots=3 * 2100, math_mode=getattr(B, "TGNN_MATH_" + math))
        self.lib = B.Tgnn(cfg)
        g = torch.Generator(device="cuda").manual_seed(seed)
        E, z = 5000, lambda *s, dt=torch.float32: torch.zeros(s, dtype=dt, device="cuda")
        ints = lambda n, hi: torch.randint(0, hi, (n,), device="cuda", generator=g, dtype=torch.int32)
        times = lambda n: torch.rand(n, device="cuda", generator=g, dtype=torch.float64).sort().values
        per = 2 * E // N + 1                                                     # an adjacency of equal lists
        self.graph = (torch.arange(N + 1, device="cuda") * per, ints(N * per, N), ints(N * per, E), times(N * per).reshape(per, N).T.reshape(-1).contiguous())
        self.feat = torch.randn((E, DE), device="cuda", generator=g)
        self.memory = torch.randn((N, D), device="cuda", generator=g)
        self.last, self.step = z(N, dt=torch.float64), z(1, dt=torch.int64)
        self.params = torch.from_numpy(B.pack_params(cfg, wl.make_weights(D, DE, 7, bias_scale=0.1))).cuda()
        self.m, self.v, self.loss, self.gn = z(self.params.numel()), z(self.params.numel()), z(1), z(1)
        self.lib.set_graph(*self.graph)
        self.lib.set_edge_features(self.feat, E)
        self.lib.set_state(self.memory, self.last, self.params, self.m, self.v, self.step)
        self.u = (ints(n_u, N), ints(n_u, N), times(n_u), torch.arange(n_u, device="cuda", dtype=torch.int32))
        self.keep = (torch.rand(n_u, device="cuda", generator=g) < 0.8).to(torch.uint8)
        self.q = (ints(n_q, N), ints(n_q, N), ints(n_q, N), 1.0 + times(n_q))


@pytest.mark.parametrize("math", ["FP32", "F16X3"])
@pytest.mark.parametrize("n_u,n_q", [(1, 1), (0, 5), (1023, 1025), (1024, 1024), (1025, 1023), (2100, 7), (7, 2100)])
def test_a_step_is_its_parts(math, n_u, n_q):
    a, b = Context(math, n_u, n_q), Context(math, n_u, n_q)
    z = lambda *s, dt=torch.int32: torch.zeros(s, dtype=dt, device="cuda")
    if n_u:
        node, uniq, win, cnt = z(2 * n_u), z(2 * n_u), z(2 * n_u), z(1)
        b.lib.build_messages(*b.u, b.keep, None, node)
        b.lib.reduce_latest(node, b.u[2], b.u[3], uniq, win, cnt)
        b.lib.memory_update(None, uniq, win, cnt)
    nodes, times = torch.cat(b.q[:3]), b.q[3].repeat(3)
    nbr, eid, ts, c, h = z(3 * n_q, K), z(3 * n_q, K), z(3 * n_q, K, dt=torch.float64), z(3 * n_q), z(3 * n_q, D, dt=torch.float32)
    b.lib.sample_recent(nodes, times, nbr, eid, ts, c)
    b.lib.embed(nodes, times, nbr, eid, ts, c, h)
    start = [x.clone() for x in (a.memory, a.last, a.params, a.m, a.v, a.step)]
    for _ in range(3):                                  # plain launches, the recording, a replay
        for x, y in zip((a.memory, a.last, a.params, a.m, a.v, a.step), start):
            x.copy_(y)
        a.lib.train_step(*a.u, a.keep, *a.q, None, a.loss, a.gn)
        got = torch.zeros_like(h)
        a.lib.debug_get_embeddings(got)
        torch.cuda.synchronize()
        assert a.lib.status() == 0 and b.lib.status() == 0
        assert torch.equal(a.last, b.last)
        # the same products in both, in an order that does not depend on the launch
        assert torch.equal(a.memory, b.memory) and torch.equal(got, h)


@pytest.mark.parametrize("math", ["FP32", "F16X3"])
@pytest.mark.parametrize("model", ["TGN", "JODIE"])
def test_steps_without_an_update_are_replayed(model, math):
    """A recorded step joins the side streams that it has forked and no others: without update events some of them carry nothing."""
    from paper_2608_16305_b200 import binding as B, workload as wl
    c = Context(math, 0, 40)
    cfg = B.make_config(N, D, DE, K, 2, max_events=64, max_roots=192, math_mode=getattr(B, "TGNN_MATH_" + math), model=getattr(B, "TGNN_MODEL_" + model))
    losses = []
    for replay in (False, True):
        lib = B.Tgnn(cfg)
        lib.set_graph_replay(replay)
        lib.set_graph(*c.graph)
        lib.set_edge_features(c.feat, c.feat.shape[0])
        p = torch.from_numpy(B.pack_params(cfg, wl.make_weights(D, DE, 7, bias_scale=0.1, model=model.lower()))).cuda()
        m, v, step = torch.zeros_like(p), torch.zeros_like(p), torch.zeros(1, dtype=torch.int64, device="cuda")
        lib.set_state(c.memory, c.last, p, m, v, step)
        out = []
        for _ in range(4):
            lib.train_step(None, None, None, None, None, *c.q, None, c.loss, c.gn)
            out += [c.loss.clone(), c.gn.clone()]
        torch.cuda.synchronize()
        assert lib.status() == 0 and int(step) == 4
        losses.append(torch.cat(out).double())
    assert (losses[0] - losses[1]).norm() <= 1e-4 * losses[0].norm()      # (gradients are summed by atomics, in another order each time)
