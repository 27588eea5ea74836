"""Attention on the query side (heads <= 8, feature columns <= 256) and the per-slot path of the other shapes, step against
the oracle at the edges of the kernels' column pieces, slot batches and head groups."""
import pytest
import torch

from paper_2608_16305_b200 import workload as wl

pytestmark = pytest.mark.gpu
TINY = wl.CONFIGS["tiny"]


@pytest.fixture(scope="module")
def B():
    from paper_2608_16305_b200 import binding
    binding.load_library()
    return binding


@pytest.mark.parametrize("d,d_e,k,heads,dtype,odd,batch", [
    (4, 0, 1, 1, "f32", False, 50),        # one lane's columns, one slot, no features
    (32, 2, 5, 2, "f32", True, 50),        # one pair of features, table off the pair alignment
    (100, 186, 10, 2, "bf16", False, 750), # a row pitch with two columns of padding; more roots than warps
    (128, 64, 16, 4, "f32", False, 50),    # full piece of columns; a second batch of slots
    (132, 90, 11, 3, "f32", True, 50),     # two pieces; one head at a time; one slot in the second batch
    (256, 256, 32, 8, "bf16", False, 60),  # the widest rows, the most slots
    (40, 172, 32, 10, "f32", False, 50),   # per-slot path: heads
    (32, 258, 10, 2, "bf16", False, 50),   # per-slot path: feature columns
    (100, 300, 10, 2, "f32", False, 50),   # the same at the width of its compile-time kernels, attention inputs of two 256-column halves
    (100, 258, 10, 2, "bf16", False, 750), # and in a batch large enough for CTA pairs; key/value weight gradient in one pass
    (160, 20, 7, 10, "f32", False, 400),   # encoding columns that no longer fit the gather's registers
])
def test_attention_edges(B, oracle, d, d_e, k, heads, dtype, odd, batch):
    from tests.test_gpu_parity import Rig
    c = wl.scaled(TINY, num_events=5 * batch, d=d, d_e=d_e, k=k, heads=heads, feat_dtype=dtype, batch=batch)
    per_slot = heads > 8 or d_e > 256        # only there does f16x3 differ from tf32: fp16 planes for the products over slots
    for math in ("fp32", "tf32", "f16x3") if per_slot else ("fp32", "tf32"):
        rig = Rig(B, oracle, c, math=math)
        if odd:
            tab = rig.dw.efeat
            flat = torch.zeros(tab.numel() + 1, dtype=tab.dtype, device="cuda")
            flat[1:] = tab.reshape(-1)
            rig.dw.efeat = flat[1:].view(tab.shape)
            rig.tr.lib.set_edge_features(rig.dw.efeat, c.num_events)
        for b in range(5):
            pre = rig.snapshot() if b in (0, 2, 4) else None
            rig.tr.step(b)
            if pre is not None:
                res, _ = rig.oracle_step(pre, b, rig.gpu_gates(b))
                rig.check_step(b, pre, res, what=f"[{math} batch {b}]")


def off_by_one_word(t):
    """A contiguous copy of t that starts 4 bytes past an alignment boundary."""
    n = 4 // t.element_size()
    flat = torch.zeros(t.numel() + n, dtype=t.dtype, device=t.device)
    out = flat[n:].view(t.shape)
    out.copy_(t)
    assert out.data_ptr() % 16 == 4 and out.is_contiguous()
    return out


@pytest.mark.parametrize("d,d_e,k,heads,dtype,math", [
    (32, 0, 10, 2, "f32", "fp32"), (32, 0, 10, 2, "f32", "tf32"),          # no features
    (100, 18, 7, 2, "f32", "fp32"), (100, 18, 7, 2, "f32", "tf32"),        # fp32 features
    (132, 34, 12, 4, "bf16", "fp32"), (132, 34, 12, 4, "bf16", "tf32"),    # bf16 features, two pieces of columns, a second batch of slots
    (36, 258, 10, 2, "f32", "f16x3"),                                      # per-slot path on fp16 planes: feature columns,
    (160, 6, 5, 10, "f32", "f16x3"),                                       # heads
])
def test_tables_off_the_vector_alignment(B, oracle, d, d_e, k, heads, dtype, math):
    """The state's and the features' tables may start at any float: nothing is said about their alignment but that of their
    type.  (The feature table in fp32 here; in bf16 it has to start at a pair.)"""
    from tests.test_gpu_parity import Rig
    c = wl.scaled(TINY, num_events=250, d=d, d_e=d_e, k=k, heads=heads, feat_dtype=dtype, batch=50)
    rig = Rig(B, oracle, c, math=math)
    tr = rig.tr
    if d_e and dtype == "f32":
        rig.dw.efeat = off_by_one_word(rig.dw.efeat)
        tr.lib.set_edge_features(rig.dw.efeat, c.num_events)
    tr.memory = off_by_one_word(tr.memory)
    tr.lib.set_state(tr.memory, tr.last_update, tr.params, tr.adam_m, tr.adam_v, tr.step_count)
    for b in range(5):
        pre = rig.snapshot()
        tr.step(b)
        res, _ = rig.oracle_step(pre, b, rig.gpu_gates(b))
        rig.check_step(b, pre, res, what=f"[{math} batch {b}]")


@pytest.mark.parametrize("math", ["fp32", "tf32"])
@pytest.mark.parametrize("which", ["memory", "params", "output"])
def test_time_projection_off_the_vector_alignment(B, oracle, math, which):
    from tests.test_gpu_parity import Rig, dev, relerr
    from oracle import jodie as oj
    c = wl.scaled(TINY, num_events=250, d=36, d_e=6, batch=50)
    rig = Rig(B, oracle, c, math=math, model="jodie")
    tr = rig.tr
    if which == "memory":
        tr.memory = off_by_one_word(tr.memory)
    if which == "params":
        tr.params = off_by_one_word(tr.params)
    tr.lib.set_state(tr.memory, tr.last_update, tr.params, tr.adam_m, tr.adam_v, tr.step_count)
    for b in range(5):
        pre = rig.snapshot()
        tr.step(b)
        res, _ = rig.oracle_step(pre, b, rig.gpu_gates(b))
        rig.check_step(b, pre, res, what=f"[{math} batch {b}]")
    n = rig.stream.src[:40]
    h = torch.zeros((40, c.d), device="cuda")
    h = off_by_one_word(h) if which == "output" else h
    t = rig.stream.t[-1] + 2.5
    tr.lib.embed(dev(n, torch.int32), torch.full((40,), t, dtype=torch.float64, device="cuda"), None, None, None, None, h)
    post = rig.snapshot()
    W = oj.unpack(c.d, c.d_e, post["params"])
    dt = (t - post["last_update"][n]).astype("float32").astype("float64")
    assert relerr(h.cpu().numpy(), oj.time_projection(post["memory"][n], dt, W["proj_w"], W["proj_b"])) <= 1e-6


@pytest.mark.parametrize("math", ["fp32", "tf32"])
@pytest.mark.parametrize("k,heads,d_e,dtype", [(5, 2, 0, "f32"), (10, 2, 18, "bf16"), (13, 4, 18, "f32"), (7, 1, 6, "f32")])
def test_rows_that_are_not_finite_stay_with_the_roots_that_name_them(B, math, k, heads, d_e, dtype):
    """Roots with fewer than k neighbors, none of which is node 0 or event 0, from a memory table and a feature table whose
    rows 0 are infinite and NaN: the empty slots weigh nothing, so embeddings, loss, gradient and update are those of tables
    with ordinary rows 0, up to the order of the atomic sums (1e-5 of the largest entry)."""
    import numpy as np
    from tests.test_gpu_parity import relerr
    N, d, n_q, E = 60, 32, 20, 400
    rng = np.random.default_rng(k)
    cfg = B.make_config(N, d, d_e, k, heads, feat_dtype=B.TGNN_BF16 if dtype == "bf16" else B.TGNN_F32, max_events=64,
                        max_roots=3 * n_q, math_mode=B.TGNN_MATH_TF32 if math == "tf32" else B.TGNN_MATH_FP32)
    W = wl.make_weights(d, d_e, 3, bias_scale=0.1)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    nodes = rng.integers(1, N, 3 * n_q).astype(np.int32)
    cnt = rng.integers(0, k, 3 * n_q).astype(np.int32)          # at most k - 1: every root has an empty slot
    held = np.arange(k)[None] < cnt[:, None]
    nbr = np.where(held, rng.integers(1, N, (3 * n_q, k)), -1).astype(np.int32)
    eid = np.where(held, rng.integers(1, E, (3 * n_q, k)), -1).astype(np.int32)
    ts = np.where(held, rng.random((3 * n_q, k)) * 50, 0.0)
    times = np.full(3 * n_q, 60.0)
    mem = rng.normal(size=(N, d)).astype(np.float32) * 0.3
    feat = torch.from_numpy(rng.normal(size=(E, d_e)).astype(np.float32)).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    got = {}
    for bad in (False, True):
        lib = B.Tgnn(cfg)
        m, f = torch.from_numpy(mem.copy()), feat.clone()
        if bad:
            m[0, ::2], m[0, 1::2] = float("inf"), float("nan")
            f[0] = float("nan")
        m, f = m.cuda(), f.cuda()
        par = dev(B.pack_params(cfg, W))
        am, av = torch.zeros_like(par), torch.zeros_like(par)
        st = torch.zeros(1, dtype=torch.int64, device="cuda")
        lib.set_edge_features(f if d_e else None, E)
        lib.set_state(m, torch.zeros(N, dtype=torch.float64, device="cuda"), par, am, av, st)
        h, loss, gn = torch.zeros((3 * n_q, d), device="cuda"), torch.zeros(1, device="cuda"), torch.zeros(1, device="cuda")
        args = [dev(x) for x in (nodes, times, nbr, eid, ts, cnt)]
        lib.embed(*args, h)
        lib.backward_step(n_q, None, loss, gn)
        g = torch.zeros_like(par)
        lib.debug_get_grads(g)
        torch.cuda.synchronize()
        assert lib.status() == 0
        got[bad] = [x.cpu().numpy() for x in (h, loss, gn, g)]
        assert all(np.isfinite(x).all() for x in got[bad]), bad
        lib.close()
    for x, y in zip(got[True], got[False]):
        assert relerr(x, y) <= 1e-5


@pytest.mark.parametrize("d,k,heads", [(32, 13, 2), (32, 20, 1), (132, 32, 4)])
@pytest.mark.parametrize("which", ["first", "last"])
def test_slots_whose_logit_is_minus_infinity(B, d, k, heads, which):
    """Logits beyond fp32's range on the negative side weigh nothing, also where they fill a whole batch of slots: the
    embedding is that of the root's other slots alone."""
    import numpy as np
    N, n = 8, 5
    cfg = B.make_config(N, d, 0, k, heads, max_events=8, max_roots=3 * n)
    W = {x: np.zeros_like(y) for x, y in wl.make_weights(d, 0, 3).items()}
    rng = np.random.default_rng(d + k)
    eye = np.eye(d, dtype=np.float32)
    W["w_q"] = np.concatenate([eye, 0 * eye], 1)
    W["w_k"] = np.concatenate([-1e3 * eye, 0 * eye], 1)
    W["w_v"] = np.concatenate([0 * eye, eye], 1)
    W["w_o"] = rng.random((d, 2 * d)).astype(np.float32)
    W["time_w"] = rng.random(d).astype(np.float32)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    mem = (1.0 + 1e-4 * rng.random((N, d))).astype(np.float32)
    mem[7] = 1e37
    bad = np.arange(k) < 10 if which == "first" else np.arange(k) >= 10
    keep = np.flatnonzero(~bad)
    nbr = np.broadcast_to(np.where(bad, 7, np.arange(k) % 7), (n, k)).astype(np.int32)
    ts = rng.random((n, k)) * 3
    less = np.full((n, k), -1, np.int32), np.zeros((n, k))
    less[0][:, :keep.size], less[1][:, :keep.size] = nbr[:, keep], ts[:, keep]
    lib = B.Tgnn(cfg)
    par = dev(B.pack_params(cfg, W))
    lib.set_state(dev(mem), torch.zeros(N, dtype=torch.float64, device="cuda"), par, torch.zeros_like(par), torch.zeros_like(par),
                  torch.zeros(1, dtype=torch.int64, device="cuda"))
    out = []
    for nb, t, c in ((nbr, ts, k), (*less, keep.size)):
        h = torch.zeros((n, d), device="cuda")
        lib.embed(dev(np.arange(n, dtype=np.int32)), dev(np.full(n, 4.0)), dev(nb), dev(nb), dev(t), dev(np.full(n, c, np.int32)), h)
        torch.cuda.synchronize()
        out.append(h.cpu().numpy())
    assert lib.status() == 0
    assert np.isfinite(out[0]).all() and np.abs(out[1]).max() > 0.1
    assert np.abs(out[0] - out[1]).max() <= 1e-5 * np.abs(out[1]).max()
    lib.close()


@pytest.mark.parametrize("d,k,heads", [(128, 1, 2), (132, 3, 1)])
def test_time_encoding_of_either_sign(B, d, k, heads):
    """Phi as the attention kernels form it (pairs of columns), for arguments from -1e5 to 1e5, through an attention layer
    that hands it on unchanged: one neighbor, W_v picks the encoding, W_o = +-identity.  Bound: the hardware cosine's
    2^-21.19 on [-pi, pi] and three roundings of a remainder below pi, half an ulp (2^-23) each."""
    import numpy as np
    N, n = 4, 3 * 400
    cfg = B.make_config(N, d, 0, k, heads, max_events=8, max_roots=n)
    rng = np.random.default_rng(d)
    W = {x: np.zeros_like(y) for x, y in wl.make_weights(d, 0, 3).items()}
    sign = np.where(np.arange(d) % 2, -1.0, 1.0)
    W["time_w"] = sign.astype(np.float32)
    W["time_b"] = (0.5 * rng.random(d) - 0.25).astype(np.float32)
    eye = np.eye(d, dtype=np.float32)
    W["w_v"] = np.concatenate([0 * eye, eye], 1)
    dt = np.concatenate([np.zeros(1), 10.0 ** rng.uniform(-2, 5, n - 1)]).astype(np.float32).astype(np.float64)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    z = torch.zeros(n, dtype=torch.int32, device="cuda")
    phi = 0.0
    for s in (1.0, -1.0):                                        # (the layer ends in a ReLU)
        W["w_o"] = np.concatenate([np.float32(s) * eye, 0 * eye], 1)
        lib = B.Tgnn(cfg)
        par = dev(B.pack_params(cfg, W))
        lib.set_state(torch.zeros((N, d), device="cuda"), torch.zeros(N, dtype=torch.float64, device="cuda"), par,
                      torch.zeros_like(par), torch.zeros_like(par), torch.zeros(1, dtype=torch.int64, device="cuda"))
        h = torch.zeros((n, d), device="cuda")
        lib.embed(z, dev(dt), z[:1].expand(n, k).contiguous(), z[:1].expand(n, k).contiguous(),
                  torch.zeros((n, k), dtype=torch.float64, device="cuda"), z + 1, h)
        torch.cuda.synchronize()
        assert lib.status() == 0
        phi = phi + s * h.cpu().numpy().astype(np.float64)
        lib.close()
    arg = (sign[None] * dt[:, None] + W["time_b"].astype(np.float64)[None]).astype(np.float32).astype(np.float64)
    assert arg.min() < -5e4 and arg.max() > 5e4
    assert np.abs(phi - np.cos(arg)).max() <= 2.0 ** -21.19 + 3 * 2.0 ** -23
