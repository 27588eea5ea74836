"""Gradient rows summed over copies: steps against the oracle where a few rows get most of the additions (32 copies), where a row
gets several (8) and where rows and additions are about as many (2), for both models, with the smallest and a wide row.  A copy that
is left out or counted twice changes the update cell's gradients by its share, a thirty-second part at least, hundreds of times the
tolerance of 1e-4."""
import pytest
import torch

from paper_2608_16305_b200 import workload as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", ["tgn", "jodie"])
@pytest.mark.parametrize("nodes,batch,d,k", [(3, 64, 4, 10), (40, 200, 100, 10), (1500, 200, 100, 5), (12, 100, 160, 20)])
def test_cell_gradient_is_the_sum_over_the_copies(oracle, model, nodes, batch, d, k):
    from paper_2608_16305_b200 import binding as B
    from tests.test_gpu_parity import Rig
    B.load_library()
    c = wl.scaled(wl.CONFIGS["tiny"], num_nodes=nodes, num_events=6 * batch, d_e=0, d=d, k=k, batch=batch)
    rig = Rig(B, oracle, c, model=model)
    for b in range(6):
        pre = rig.snapshot() if b in (2, 5) else None
        rig.tr.step(b)
        if pre is not None:
            res, _ = rig.oracle_step(pre, b, rig.gpu_gates(b))
            rig.check_step(b, pre, res, what=f"[batch {b}]")


def contexts(model, capacities, N=5000, d=32, k=3):
    """A context for each capacity in events, all on one graph of N nodes, each with a state of its own."""
    from paper_2608_16305_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(11)
    E = 20000
    ends = torch.randint(0, N, (2, E), device="cuda", generator=g, dtype=torch.int32)
    ends[0, ::3] = 7                                     # a hub
    node = torch.stack((ends[0], ends[1]), 1).reshape(-1)
    order = torch.sort(node.long(), stable=True).indices
    indptr = torch.zeros(N + 1, dtype=torch.int64, device="cuda")
    indptr[1:] = torch.cumsum(torch.bincount(node.long(), minlength=N), 0)
    t = torch.arange(E, device="cuda", dtype=torch.float64) / 100
    eid = (order // 2).int()
    graph = indptr, torch.stack((ends[1], ends[0]), 1).reshape(-1)[order].contiguous(), eid, t[eid.long()].contiguous()
    memory = torch.rand((N, d), device="cuda", generator=g) - 0.5
    out = []
    for cap in capacities:
        cfg = B.make_config(N, d, 0, k, 2, max_events=cap, max_roots=3 * cap, lr=1e-3,
                            model=B.TGNN_MODEL_JODIE if model == "jodie" else B.TGNN_MODEL_TGN)
        lib, lay = B.Tgnn(cfg), B.param_layout(cfg)
        z = lambda *s, dt=torch.float32: torch.zeros(s, dtype=dt, device="cuda")
        state = dict(memory=memory.clone(), last_update=z(N, dt=torch.float64), m=z(lay["total"]), v=z(lay["total"]), step=z(1, dt=torch.int64),
                     params=torch.from_numpy(B.pack_params(cfg, wl.make_weights(d, 0, 3, bias_scale=0.1, model=model))).cuda())
        lib.set_graph(*graph)
        lib.set_edge_features(None, E)
        lib.set_state(*(state[n] for n in ("memory", "last_update", "params", "m", "v", "step")))
        out.append((lib, state, z(lay["total"]), z(1), z(1)))
    return out, ends, t, g


@pytest.mark.parametrize("model", ["tgn", "jodie"])
def test_steps_of_many_sizes_in_a_context_for_far_more_events(model):
    """The copies are as many rows as the step at hand can write: after steps of other sizes nothing of those is left in them.  A
    context for exactly the step's events takes the same steps from the same state."""
    sizes = [(600, 600), (3, 600), (600, 3), (1, 1), (0, 40), (250, 900), (3, 600), (900, 2), (600, 600), (3, 600), (1, 1), (600, 600)]
    pairs, ends, t, g = contexts(model, [16384] + sorted({max(s) for s in sizes}))
    tight = dict(zip(sorted({max(s) for s in sizes}), pairs[1:]))
    at = 1000
    for n_u, n_q in sizes:
        u, q = slice(at, at + n_u), slice(at + n_u, at + n_u + n_q)
        at += 700
        neg = torch.randint(0, 5000, (n_q,), device="cuda", generator=g, dtype=torch.int32)
        eid = torch.arange(at, at + n_u, device="cuda", dtype=torch.int32)
        upd = (ends[0, u].contiguous(), ends[1, u].contiguous(), t[u].contiguous(), eid, None) if n_u else (None,) * 5
        got = []
        for lib, state, grads, loss, norm in (pairs[0], tight[max(n_u, n_q)]):
            if lib is not pairs[0][0]:
                for n, x in pairs[0][1].items():
                    state[n].copy_(before[n])
            before = {n: x.clone() for n, x in state.items()}
            lib.train_step(*upd, ends[0, q].contiguous(), ends[1, q].contiguous(), neg, t[q].contiguous(), None, loss, norm)
            lib.debug_get_grads(grads)
            torch.cuda.synchronize()
            assert lib.status() == 0
            got.append((grads.clone(), loss.item(), state["memory"].clone()))
        # the same terms, added in the order in which the blocks come by: fp32 sums of some thousand terms
        assert (got[0][0] - got[1][0]).norm() <= 2e-5 * got[1][0].norm() and abs(got[0][1] - got[1][1]) <= 1e-5 * got[1][1]
        assert torch.equal(got[0][2], got[1][2])


def test_workspace_for_the_copies_is_bounded():
    """262 144 events on as many nodes twice over: a copy of the rows is 210 MB, all copies together 512 MB."""
    from paper_2608_16305_b200 import binding as B

    def used(num_nodes):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        lib = B.Tgnn(B.make_config(num_nodes, 100, 0, 10, 2, max_events=1 << 18, max_roots=3 << 12))
        taken = before - torch.cuda.mem_get_info()[0]
        lib.close()
        return taken
    used(8)
    rows = 1 << 19
    tables = 40 * rows                                   # per node, beside the copies
    assert used(rows) - used(8) <= (512 << 20) + tables + (8 << 20)
