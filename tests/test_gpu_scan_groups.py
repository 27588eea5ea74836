"""The backward scan of four workers at once at the edges of its groups, chunks and node tables, against the oracle (bit-exact)."""
import numpy as np
import pytest

from tests.test_gpu_scan import B, _check_against_oracle  # noqa: F401

pytestmark = pytest.mark.gpu


# more than 148 pairs of a worker and a window: groups of one to four workers; windows around 1 024 (the smallest for groups) and
# 4 096 events (one or several per thread), the last one short; node tables around 200 KB for a group (12 800 nodes)
@pytest.mark.parametrize("P,N,E,batch,K", [(P, 40, 1024 * (150 // P + 1) + 3, b, 1) for P in (3, 4, 5, 9, 38) for b in (1023, 1024)] +
                         [(40, 60, 16400, 4095, 1), (50, 60, 16390, 1024, 4), (53, 700, 13000, 1025, 4), (75, 12800, 3000, 1030, 1),
                          (75, 12801, 3000, 1030, 1)])
def test_groups_chunks_and_tables(B, P, N, E, batch, K):  # noqa: F811
    rng = np.random.default_rng(N + E + P)
    src = np.minimum(rng.zipf(1.3, size=E) - 1, N - 1).astype(np.int32)
    dst = np.minimum(rng.zipf(1.2, size=E) - 1, N - 1).astype(np.int32)
    _check_against_oracle(B, src, dst, rng.integers(0, P, size=N).astype(np.int32), P, batch, K)


@pytest.mark.parametrize("n", [1100, 5000])
def test_a_chain_through_a_whole_chunk(B, n):  # noqa: F811
    # a path walked backward one event per round: as many rounds as events, for every worker of a group that has the path remote
    owner = np.full(n + 2, 3, np.int32)
    owner[0] = 0
    src = np.concatenate([np.arange(n, 0, -1), [0]]).astype(np.int32)
    dst = np.concatenate([np.arange(n, 0, -1) - 1, [1]]).astype(np.int32)
    _check_against_oracle(B, src, dst, owner, 149, n + 1, 1)
