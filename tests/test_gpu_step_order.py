"""How a step's launches depend on one another and how they are split, read from a recording that its caller makes of it."""
import re

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def recorded(tmp_path, math, n_u, n_q, d=100, de=172, heads=2, k=10, N=3000, E=6000):
    """The nodes of a step of plain launches: name, grid, and the nodes that each comes directly behind."""
    from paper_2608_16305_b200 import binding as B, workload as wl
    lib = B.Tgnn(B.make_config(N, d, de, k, heads, max_events=max(n_u, 1), max_roots=3 * n_q, math_mode=getattr(B, "TGNN_MATH_" + math)))
    g = torch.Generator(device="cuda").manual_seed(n_q)
    z = lambda *s, dt=torch.float32: torch.zeros(s, dtype=dt, device="cuda")
    ints = lambda n, hi: torch.randint(0, hi, (n,), device="cuda", generator=g, dtype=torch.int32)
    times = lambda n: torch.rand(n, device="cuda", generator=g, dtype=torch.float64).sort().values
    per = 2 * E // N
    graph = (torch.arange(N + 1, device="cuda") * per, ints(N * per, N), ints(N * per, E), times(N * per).reshape(per, N).T.reshape(-1).contiguous())
    params = torch.from_numpy(B.pack_params(lib.cfg, wl.make_weights(d, de, 7, bias_scale=0.1))).cuda()
    state = (torch.randn((N, d), device="cuda", generator=g), z(N, dt=torch.float64), params, z(params.numel()), z(params.numel()), z(1, dt=torch.int64))
    feat = torch.randn((E, de), device="cuda", generator=g)
    lib.set_graph(*graph)
    lib.set_edge_features(feat, E)
    lib.set_state(*state)
    u = (ints(n_u, N), ints(n_u, N), times(n_u), torch.arange(n_u, device="cuda", dtype=torch.int32))
    q = (ints(n_q, N), ints(n_q, N), ints(n_q, N), 1.0 + times(n_q))
    loss, norm = z(1), z(1)
    lib.train_step(*u, None, *q, None, loss, norm)
    torch.cuda.synchronize()
    rec = torch.cuda.CUDAGraph(keep_graph=True)
    rec.enable_debug_mode()
    with torch.cuda.graph(rec, stream=torch.cuda.Stream()):
        lib.train_step(*u, None, *q, None, loss, norm)
    rec.debug_dump(str(tmp_path / "step.dot"))
    text = (tmp_path / "step.dot").read_text()
    assert lib.status() == 0
    nodes = {}
    for at, body in re.findall(r'"(\w+_node_\d+)"\[[^\]]*?label="\{(.*?)\}"\];', text, re.S):
        m = re.search(r"(\w+)\\<\\<\\<(\\?\{[^}]*\\?\}|\d+),", body)
        if m:
            grid = [int(x) for x in re.findall(r"\d+", m.group(2))]
            nodes[at] = dict(name=m.group(1), grid=tuple(grid + [1] * (3 - len(grid))), behind=set())
    for a, b in re.findall(r'"(\w+_node_\d+)" -> "(\w+_node_\d+)"', text):
        nodes[b]["behind"].add(a)
    return nodes


def the(nodes, name):
    at = [a for a, n in nodes.items() if name in n["name"]]
    assert len(at) == 1, (name, at)
    return at[0]


def directly_behind(nodes, at):
    return {a: n for a, n in nodes.items() if at in n["behind"]}


def test_the_gradient_of_the_queries_is_split_as_the_output_product_is(tmp_path):
    """Both are stored products of 15 tiles over 700 to 900 columns: eight CTAs of a cluster each.  Fewer for the one, to leave SMs to the gradient
    of the folded weights, would be longer chains of an accumulator that every MMA truncates."""
    nodes = recorded(tmp_path, "F16X3", 300, 600)
    products = lambda at: [n["grid"] for n in directly_behind(nodes, at).values() if "gemm_tf32_kernel" in n["name"] and n["grid"][1] == 15]
    out = products(the(nodes, "attn_fwd_kernel"))
    assert out == [(1, 15, 8)]
    assert products(the(nodes, "attn_bwd_kernel")) == out


def test_the_fp32_mode_keeps_the_products_behind_the_attention_in_a_row(tmp_path):
    """Beside each other the two fp32 products share SMs, and the one that the chain waits for ends later than both in a row."""
    nodes = recorded(tmp_path, "FP32", 100, 100)
    assert len([n for n in directly_behind(nodes, the(nodes, "attn_bwd_kernel")).values() if "gemm_fp32_kernel" in n["name"]]) == 1


@pytest.mark.parametrize("math", ["FP32", "F16X3"])
def test_what_runs_beside_the_memory_update_of_plain_launches_follows_the_begin(tmp_path, math):
    """Outside the library's own recordings nothing tells when a kernel has begun: what needs nothing of the memory update waits for none of its kernels."""
    nodes = recorded(tmp_path, math, 300, 100)
    begin = the(nodes, "step_begin_kernel")
    for name in ("gather_winner_kernel", "sample_recent_kernel", "fold_weights_kernel"):
        assert nodes[the(nodes, name)]["behind"] == {begin}, name
