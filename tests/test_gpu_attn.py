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
])
def test_attention_edges(B, oracle, d, d_e, k, heads, dtype, odd, batch):
    from tests.test_gpu_parity import Rig
    c = wl.scaled(TINY, num_events=5 * batch, d=d, d_e=d_e, k=k, heads=heads, feat_dtype=dtype, batch=batch)
    for math in ("fp32", "tf32"):
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
