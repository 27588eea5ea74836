"""Error of the tensor-core weight gradients (a long contraction split into parts, the parts' sums added by atomics) against fp64."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# The tensor core truncates the accumulator at its last bit with every MMA, over 8 rows of the contraction: half an ulp, 2^-24 of the sum so far (3/4 of that for a
# mean mantissa), always towards zero.  A part of P rows whose sum grows as sqrt(i) (operands of both signs) ends with about 2/3 of the bias of P / 8 such
# steps, one whose sum grows as i with half of it.  Beside it: 2^-22 of the operands' dropped bits, 2^-25 sqrt(parts) of the parts' rounded additions.
# A part has 4 blocks of 32 rows until the tiles' parts fill half the machine.
@pytest.mark.parametrize("M,N,K", [(100, 200, 8000), (128, 256, 8000), (100, 200, 2474), (32, 64, 1200), (101, 200, 9411)])
@pytest.mark.parametrize("one_sign", [False, True])
def test_parts_are_short(M, N, K, one_sign):
    from paper_2608_16305_b200 import binding as B
    lib = B.Tgnn(B.make_config(100, 32, 16, 10, 2, math_mode=B.TGNN_MATH_F16X3))
    g = torch.Generator(device="cuda").manual_seed(K + M)
    a, b = (torch.randn((K, n), device="cuda", generator=g) for n in (M, N))
    if one_sign:
        a, b = a.abs(), b.abs()
    C = torch.zeros((M, N), device="cuda")
    lib.debug_gemm(a, 1, M, b, N, 1, C, N, M, N, K, accumulate=True, split_k=8, precise=True)
    torch.cuda.synchronize()
    assert lib.status() == 0
    want = a.double().T @ b.double()
    steps, parts = 128 / 8, -(-K // 128)
    bound = (0.5 if one_sign else 2 / 3) * steps * 0.75 * 2.0 ** -24 + 2.0 ** -22 + 2.0 ** -25 * parts ** 0.5
    # (twice the sum: the means above are of the ulp's place in a sum's binade, which all sums of a product of one sign share)
    assert (C.double() - want).norm() <= 2 * bound * want.norm()
