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
