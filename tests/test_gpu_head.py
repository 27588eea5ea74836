"""The link-prediction head's forms at the edges of their blocks, against the same formulas in fp64.

The time-projection model without a memory update: its embedding is one product, so the head's part of the gradient and
d loss / d h (through w_p and b_p) are all there is to a step."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# events on both sides of each form's lines and of its blocks' edges; larger batches at fewer widths, masked ones among them
SIZES = [(d, n, m) for d in (4, 36, 100, 128, 256) for n in (1, 3, 4, 5, 299, 600) for m in (False, True)]
SIZES += [(d, n, d == 100) for d in (4, 36, 100, 128, 256) for n in (743, 889, 1185, 2367, 2368)] + [(100, n, False) for n in (743, 889, 1185, 2367, 2368)]
SIZES += [(d, n, True) for d in (36, 128, 256) for n in (2367, 2368)] + [(d, 4900, m) for d in (36, 100) for m in (False, True)]


class Head:
    """A context whose last embedding has 3 n_q rows, and what the head is expected to leave for them."""

    def __init__(self, d, n_q, masked, math="FP32", edit=None):
        from paper_2608_16305_b200 import binding as B, workload as wl
        self.d, self.n_q, N = d, n_q, 500
        cfg = B.make_config(N, d, 0, 5, 2, max_events=4, max_roots=3 * n_q, model=B.TGNN_MODEL_JODIE, math_mode=getattr(B, "TGNN_MATH_" + math))
        self.lib, self.lay = B.Tgnn(cfg), B.param_layout(cfg)
        self.weights = wl.make_weights(d, 0, 5, bias_scale=0.1, model="jodie")
        if edit is not None:
            edit(self.weights)
        g = torch.Generator(device="cuda").manual_seed(n_q * 1000 + d)
        z = lambda *s, dt=torch.float32: torch.zeros(s, dtype=dt, device="cuda")
        self.memory, self.last, self.step = torch.randn((N, d), device="cuda", generator=g), z(N, dt=torch.float64), z(1, dt=torch.int64)
        self.params = torch.from_numpy(B.pack_params(cfg, self.weights)).cuda()
        self.m, self.v = z(self.lay["total"]), z(self.lay["total"])
        self.graph = z(N + 1, dt=torch.int64), z(1, dt=torch.int32), z(1, dt=torch.int32), z(1, dt=torch.float64)
        self.lib.set_graph(*self.graph)
        self.lib.set_edge_features(None, 0)
        self.lib.set_state(self.memory, self.last, self.params, self.m, self.v, self.step)
        self.nodes = torch.randint(0, N, (3 * n_q,), device="cuda", generator=g, dtype=torch.int32)
        self.times = torch.rand(n_q, device="cuda", generator=g, dtype=torch.float64).repeat(3)
        self.h, self.loss, self.gn, self.grads = z(3 * n_q, d), z(1), z(1), z(self.lay["total"])
        self.close = 2e-6 if math == "FP32" else 1e-5      # (products of 21-bit operands: 5e-7 of their terms)
        self.mask = (torch.rand(n_q, device="cuda", generator=g) < 0.6).to(torch.uint8) if masked else None
        self.lib.embed(self.nodes, self.times, None, None, None, None, self.h)

    def reference(self, h):
        """Loss, gradients and the number of pre-activations close to zero, in fp64, for these embedding rows."""
        d, n_q = self.d, self.n_q
        p64 = {n: torch.from_numpy(np.asarray(self.weights[n], dtype=np.float64)).cuda().requires_grad_() for n in ("w_1", "b_1", "w_2", "b_2")}
        h64 = h.double().requires_grad_()
        hs, hd, hn = h64[:n_q], h64[n_q:2 * n_q], h64[2 * n_q:]
        pre = lambda a, b: torch.cat((a, b), 1) @ p64["w_1"].reshape(d, 2 * d).T + p64["b_1"]
        pos, neg = pre(hs, hd), pre(hs, hn)
        score = lambda x: torch.relu(x) @ p64["w_2"].reshape(-1) + p64["b_2"]
        w = torch.ones(n_q, device="cuda", dtype=torch.float64) if self.mask is None else self.mask.double()
        w = w / w.sum().clamp(min=1)
        loss = (w * (torch.nn.functional.softplus(-score(pos)) + torch.nn.functional.softplus(score(neg)))).sum()
        loss.backward()
        want = {n: p64[n].grad.reshape(-1) for n in p64}
        mem64, dt = self.memory.double()[self.nodes.long()], self.times.float().double()[:, None]
        want["proj_w"], want["proj_b"] = (h64.grad * mem64 * dt).sum(0), (h64.grad * mem64).sum(0)
        return loss.item(), want, sum(int((x.abs() < self.close).sum()) for x in (pos, neg))

    def check(self, loss, want, near):
        # one sum of n_q d terms per entry in fp32, with atomics: a few 1e-7 of its terms' magnitude; a hidden unit whose
        # pre-activation is within 1e-6 of zero may take the other branch, which moves an entry by at most its own term
        tol = 2e-5 if near == 0 else 2e-3
        self.lib.debug_get_grads(self.grads)
        torch.cuda.synchronize()
        assert self.lib.status() == 0
        assert abs(self.loss.item() - loss) <= 1e-5 * max(loss, 1e-3)
        for n, x in want.items():
            got = self.grads[self.lay[n]:self.lay[n] + x.numel()].double()
            if n == "b_2":      # one number, a difference of sums that nearly cancel: measured by its terms
                assert (got - x).abs().item() <= 1e-5
                continue
            assert (got - x).norm() <= tol * x.norm() + 1e-9, (n, ((got - x).norm() / x.norm()).item(), near)


@pytest.mark.parametrize("d,n_q,masked", SIZES)
def test_head_forward_and_backward(d, n_q, masked):
    r = Head(d, n_q, masked)
    expected = r.reference(r.h)
    r.lib.backward_step(n_q, r.mask, r.loss, r.gn)
    r.check(*expected)


@pytest.mark.parametrize("math,d,n_q,one_launch", [
    ("FP32", 116, 2368, True), ("FP32", 160, 2400, True), ("FP32", 244, 2368, True), ("FP32", 256, 2368, False),
    ("F16X3", 116, 2368, True), ("F16X3", 128, 3552, True), ("F16X3", 128, 3553, False), ("TF32", 120, 3001, True), ("TF32", 116, 4100, False),
    ("F16X3", 132, 2367, True), ("F16X3", 132, 2368, False), ("TF32", 256, 2367, True), ("TF32", 256, 2369, False), ("F16X3", 100, 2368, True)])
def test_form_of_the_head_by_width_events_and_mode(math, d, n_q, one_launch):
    r = Head(d, n_q, masked=n_q % 2 == 1, math=math)
    expected = r.reference(r.h)
    r.lib.profile_begin()
    r.lib.backward_step(n_q, r.mask, r.loss, r.gn)
    names = r.lib.profile_report()
    assert ("head_fused" in names) == one_launch and ("head_gather" in names) != one_launch
    r.check(*expected)


@pytest.mark.parametrize("d,n_q", [(36, 7), (36, 2400), (136, 4000)])
def test_events_without_weight_leave_nothing_whatever_their_scores(d, n_q):
    """Two hidden units of masked events overflow and meet in the score with opposite signs: it is not a number.  (Small head, tiled
    head, separate products.)"""
    def edit(w):
        w["w_1"] = np.array(w["w_1"], dtype=np.float32).reshape(d, 2 * d)
        w["w_1"][:2] = 0.5
        w["w_2"] = np.array(w["w_2"], dtype=np.float32).reshape(-1)
        w["w_2"][:2] = 1.0, -1.0
    r = Head(d, n_q, masked=True, edit=edit)
    r.mask[0], r.mask[1] = 0, 1
    out = torch.nonzero(r.mask == 0).reshape(-1)
    finite = r.h.clone()
    for block in range(3):
        finite[block * n_q + out] = 0.0
        r.h[block * n_q + out] = 3e38
    loss, want, near = r.reference(finite)
    r.lib.backward_step(n_q, r.mask, r.loss, r.gn)
    r.check(loss, want, near)
