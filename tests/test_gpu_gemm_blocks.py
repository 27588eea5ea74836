"""Stored products with prepared weight images (half blocks of the contraction, split over clusters or not; short contractions) at the edges of
their tiles: a memory update and an embedding in the tensor-core mode against the same in the fp32 mode."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def parts(math, d, de, heads, k, n_u, n_q, N=4000, E=6000):
    from paper_2608_16305_b200 import binding as B, workload as wl
    cfg = B.make_config(N, d, de, k, heads, max_events=max(n_u, 1), max_roots=3 * n_q, math_mode=getattr(B, "TGNN_MATH_" + math))
    lib = B.Tgnn(cfg)
    g = torch.Generator(device="cuda").manual_seed(1000 * n_q + d)
    z = lambda *s, dt=torch.int32: torch.zeros(s, dtype=dt, device="cuda")
    ints = lambda n, hi: torch.randint(0, hi, (n,), device="cuda", generator=g, dtype=torch.int32)
    times = lambda n: torch.rand(n, device="cuda", generator=g, dtype=torch.float64)
    memory = torch.randn((N, d), device="cuda", generator=g).tanh_()
    feat = torch.randn((E, de), device="cuda", generator=g) if de else None
    params = torch.from_numpy(B.pack_params(cfg, wl.make_weights(d, de, 7, bias_scale=0.1))).cuda()
    last, step, m, v = z(N, dt=torch.float64), z(1, dt=torch.int64), torch.zeros_like(params), torch.zeros_like(params)
    graph = (z(N + 1, dt=torch.int64), z(1), z(1), z(1, dt=torch.float64))
    lib.set_graph(*graph)
    lib.set_edge_features(feat, E if de else 0)
    lib.set_state(memory, last, params, m, v, step)
    src, dst, t = ints(n_u, N), ints(n_u, N), times(n_u).sort().values
    eid = torch.arange(n_u, device="cuda", dtype=torch.int32)
    node, uniq, win, cnt = z(2 * n_u), z(2 * n_u), z(2 * n_u), z(1)
    lib.build_messages(src, dst, t, eid, None, None, node)
    lib.reduce_latest(node, t, eid, uniq, win, cnt)
    lib.memory_update(None, uniq, win, cnt)
    R = 3 * n_q
    h = z(R, d, dt=torch.float32)
    lib.embed(ints(R, N), 1.0 + times(R), ints(R * k, N).view(R, k), ints(R * k, E).view(R, k), times(R * k).view(R, k),
              torch.randint(0, k + 1, (R,), device="cuda", generator=g, dtype=torch.int32), h)
    torch.cuda.synchronize()
    assert lib.status() == 0
    return memory, h


# contraction lengths that end in a full half block, in its middle and behind it; rows that end on, before and behind a tile; few tiles (split over
# 2 to 8 CTAs), and more than run as clusters at once
@pytest.mark.parametrize("d,de,heads,k,n_u,n_q", [(100, 172, 2, 10, 600, 43), (100, 0, 2, 5, 1, 1), (32, 6, 2, 5, 128, 128), (36, 10, 2, 4, 65, 171),
                                                  (128, 90, 4, 15, 300, 300), (100, 186, 2, 3, 3000, 3300), (160, 16, 2, 4, 500, 129),
                                                  (44, 2, 1, 3, 63, 3201), (112, 48, 2, 2, 700, 600), (120, 30, 2, 2, 64, 640)])
def test_tensor_core_products_with_images(d, de, heads, k, n_u, n_q):
    (m1, h1), (m0, h0) = parts("F16X3", d, de, heads, k, n_u, n_q), parts("FP32", d, de, heads, k, n_u, n_q)
    for x, y in ((m1, m0), (h1, h0)):
        # operands of 21 bits in every product (2^-21 each, independent over the terms), through three products in a row and the softmax
        assert (x - y).double().norm() <= 2e-5 * y.double().norm()
        assert (x - y).abs().max() <= 2e-4 * y.double().pow(2).mean().sqrt().clamp(min=1e-6) + 1e-6 * y.abs().max()
