"""Attention over 11 to 16 slots in one batch: a step against the oracle at the edges of that range and of the column pieces."""
import pytest

from paper_2608_16305_b200 import workload as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,d_e,k,heads,dtype,batch,math", [
    (4, 0, 11, 2, "f32", 50, "fp32"),         # one lane's columns, no features, the fewest slots
    (36, 66, 12, 4, "bf16", 50, "tf32"),      # a pair of features into the second piece
    (100, 172, 15, 2, "f32", 650, "tf32"),    # more roots than warps
    (128, 256, 16, 8, "bf16", 50, "fp32"),    # the widest rows, every slot of the batch
    (128, 2, 17, 2, "f32", 50, "fp32"),       # one slot too many: two batches of ten
])
def test_one_batch_of_sixteen_slots(oracle, d, d_e, k, heads, dtype, batch, math):
    from paper_2608_16305_b200 import binding as B
    from tests.test_gpu_parity import Rig
    B.load_library()
    c = wl.scaled(wl.CONFIGS["tiny"], num_events=5 * batch, d=d, d_e=d_e, k=k, heads=heads, feat_dtype=dtype, batch=batch)
    rig = Rig(B, oracle, c, math=math)
    for b in range(5):
        pre = rig.snapshot() if b in (0, 2, 4) else None
        rig.tr.step(b)
        if pre is not None:
            res, _ = rig.oracle_step(pre, b, rig.gpu_gates(b))
            rig.check_step(b, pre, res, what=f"[batch {b}]")
