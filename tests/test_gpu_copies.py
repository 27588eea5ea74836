"""Gradient rows summed over copies: steps against the oracle where a few rows get most of the additions (32 copies) and where
rows and additions are about as many (8), for both models, with the smallest and a wide row.  A copy that is left out or counted
twice changes the update cell's gradients by its share, a thirty-second part at least, hundreds of times the tolerance of 1e-4."""
import pytest

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
