"""Stored fp32 products whose contraction is split over the blocks of a cluster, at the edges of their tiles of 64 x 64, against fp64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# clusters of 2, 3, 4 and 8 (48 contraction elements a block at least, and all of a cluster's blocks on the machine at once); one row beyond a tile, one
# row, whole tiles; 100 columns (28 of the second tile's are beyond the matrix), columns that end inside a run of four; more clusters than SMs.  gap: the
# output's rows are longer than its columns, and what lies between stays.
@pytest.mark.parametrize("K,split", [(96, 2), (101, 2), (144, 3), (150, 3), (192, 4), (223, 4), (384, 8), (845, 8)])
@pytest.mark.parametrize("M,N,gap", [(65, 100, 0), (1, 100, 5), (64, 64, 0), (129, 67, 1), (193, 3, 0), (63, 129, 4)])
def test_a_cluster_adds_up_its_parts(M, N, gap, K, split):
    from paper_2608_16305_b200 import binding as B
    assert -(-M // 64) * -(-N // 64) * split <= 3 * 148 and K >= 48 * split and (split == 8 or K < 48 * {2: 3, 3: 4, 4: 8}[split])
    lib = B.Tgnn(B.make_config(100, 32, 16, 10, 2, math_mode=B.TGNN_MATH_FP32))
    rng = np.random.default_rng(M * 100003 + N * 1009 + K)
    A, W, bias = (rng.normal(size=s).astype(np.float32) for s in ((M, K), (N, K), (N,)))
    a, w, b = (torch.from_numpy(x).cuda() for x in (A, W, bias))
    want = A.astype(np.float64) @ W.astype(np.float64).T + bias
    for relu in (False, True):
        C = torch.full((M, N + gap), 7.0, device="cuda")
        for _ in range(3):
            lib.debug_gemm(a, K, 1, w, 1, K, C, N + gap, M, N, K, bias=b, relu=relu)
        torch.cuda.synchronize()
        assert lib.status() == 0
        got = C.cpu().numpy()
        # K products in fp32, added in a chain per team of each block and then over teams and blocks: K 2^-24 of the sum of their magnitudes bounds it
        bound = (K + 2 * split + 1) * 2.0 ** -24 * (np.abs(A).astype(np.float64) @ np.abs(W).astype(np.float64).T + np.abs(bias))
        assert (np.abs(got[:, :N] - (np.maximum(want, 0) if relu else want)) <= bound).all()
        assert (got[:, N:] == 7.0).all()


def test_clusters_fill_the_machine():
    """As many blocks as run at once and rows that a device-side count ends inside a tile."""
    from paper_2608_16305_b200 import binding as B
    lib = B.Tgnn(B.make_config(100, 32, 16, 10, 2, math_mode=B.TGNN_MATH_FP32))
    M, N, K, used = 1800, 100, 845, 1729
    rng = np.random.default_rng(3)
    A, W = rng.normal(size=(M, K)).astype(np.float32), rng.normal(size=(N, K)).astype(np.float32)
    a, w, m = torch.from_numpy(A).cuda(), torch.from_numpy(W).cuda(), torch.tensor([used], dtype=torch.int32, device="cuda")
    for count, rows in ((None, M), (m, used)):
        C = torch.full((M, N), 7.0, device="cuda")
        lib.debug_gemm(a, K, 1, w, 1, K, C, N, M, N, K, dev_M=count)
        torch.cuda.synchronize()
        assert lib.status() == 0
        got = C.cpu().numpy()
        bound = (K + 17) * 2.0 ** -24 * (np.abs(A[:rows]).astype(np.float64) @ np.abs(W).astype(np.float64).T)
        assert (np.abs(got[:rows] - A[:rows].astype(np.float64) @ W.astype(np.float64).T) <= bound).all()
        assert (got[rows:] == 7.0).all()
