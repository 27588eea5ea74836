"""Cases of the training path for timing: what a user's program calls, over the sizes that it calls it with.

A case names one call pattern (`kind`):

  step      Trainer.step: one training step from device-resident batches (prune mask, memory update, neighbor
            search, embedding, loss, backward, Adam)
  host      Trainer.step_host: the same from pinned host arrays, one call of the streaming entry point per batch
  forward   the scoring half of a step by its entry points (messages, latest-event reduction, memory update,
            neighbor search, embedding), as an evaluation pass runs it
  scan      offline preprocessing of one worker: backward dependency scan over all workers' windows, then its
            mixed batches
  refresh   boundary refresh of a worker: pack the owed state rows, unpack the received ones

The model is in the middle of training (non-zero memory and Adam moments) near the end of its stream, where the
neighbor lists are full; every pass takes the next batch of the stream, as a training loop does.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_16305_b200 import binding as B
from paper_2608_16305_b200 import trainer as T
from paper_2608_16305_b200 import workload as wl

MATH = {"fp32": B.TGNN_MATH_FP32, "tf32": B.TGNN_MATH_TF32, "f16x3": B.TGNN_MATH_F16X3}
SPAN = 12            # consecutive batches that a state steps through before it starts over


def _model(name, kind, like, **kw):
    """A case with the shape of one of the package's workload configurations, with some fields replaced."""
    c = wl.CONFIGS[like]
    case = dict(name=name, kind=kind, nodes=c.num_nodes, sources=c.num_src, events=c.num_events, d_e=c.d_e,
                feat=c.feat_dtype, d=c.d, k=c.k, heads=c.heads, batch=c.batch, replay=c.replay_frac, prune=c.prune,
                zipf_src=c.zipf_src, zipf_dst=c.zipf_dst, math="f16x3", model="tgn", embed_aux=False)
    case.update(kw)
    return case


def listed():
    return [
        # the smallest step, in the trainer's default arithmetic: launches and latency are what it costs
        _model("tiny_fp32", "step", "tiny", math="fp32"),
        # Wikipedia-shaped training, fp32 edge features, small batches: tensor-core mode and the default mode
        _model("wiki", "step", "wiki"),
        _model("wiki_fp32", "step", "wiki", math="fp32"),
        # Reddit-shaped training with replay events and pruning, TF32 operands
        _model("reddit_tf32", "step", "reddit", math="tf32"),
        # no edge features, a few hub nodes in every batch, large batches
        _model("lastfm", "step", "lastfm"),
        # the headline shape: bf16 edge features, large batches (a stream long enough to fill the neighbor lists)
        _model("large", "step", "large", events=6_000_000),
        # the headline shape fed from host memory, every event of the mixed batch embedded and scored
        _model("large_host_aux", "host", "large", events=6_000_000, embed_aux=True),
        # the time-projection model, fed from host memory
        _model("wiki_jodie_host", "host", "wiki", model="jodie"),
        # a generic wider model with more neighbors and heads, odd batch and feature sizes
        _model("wide_ragged", "step", "wiki", d=128, d_e=90, k=15, heads=4, batch=1237, replay=0.13, prune=True),
        # scoring of a Reddit-shaped batch in an evaluation pass
        _model("reddit_forward", "forward", "reddit"),
        # offline preprocessing for 8 workers, windows of 6 batches
        dict(name="preprocess", kind="scan", nodes=2_000, sources=0, events=1_300_000, batch=4_000, zipf_src=1.5,
             zipf_dst=1.5, workers=8, window=6),
        # boundary refresh of a large node table
        dict(name="refresh", kind="refresh", nodes=600_000, d=100, rows=400_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(("step", "host", "forward", "scan", "refresh"), (55, 15, 14, 8, 8))[0]
    if kind == "refresh":
        nodes = _log(rng, 9_000, 600_000)
        return dict(kind=kind, nodes=nodes, d=rng.choice((32, 64, 100, 128, 172)), rows=min(nodes, _log(rng, 1_000, 400_000)))
    if kind == "scan":
        events = _log(rng, 20_000, 1_300_000)
        zipf = round(rng.uniform(1.0, 1.5), 2)
        return dict(kind=kind, nodes=_log(rng, 1_000, 17_000), sources=0, events=events,
                    batch=min(_log(rng, 200, 4_000), events // 8), zipf_src=zipf, zipf_dst=zipf,
                    workers=rng.choice((2, 4, 8)), window=rng.choice((2, 4, 6)))
    mode = rng.choices(("f16x3", "fp32", "tf32"), (6, 3, 2))[0]
    d, heads = rng.choice(((32, 2), (64, 2), (100, 2), (100, 2), (100, 2), (128, 4), (160, 2)))
    d_e = rng.choice((0, 16, 172, 172, 186, 2 * rng.randint(1, 93)))
    nodes = _log(rng, 1_000, 17_000)
    replay = rng.choice((0.0, 0.13, 0.2, 0.3))
    case = dict(kind=kind, nodes=nodes, sources=rng.choice((0, nodes * 8 // 9)), events=0, d_e=d_e,
                feat=rng.choice(("f32", "f32", "bf16")) if d_e else "f32", d=d, k=rng.choice((5, 10, 10, 10, 15, 20)),
                heads=heads, batch=_log(rng, 100, 4_000), replay=replay, prune=replay > 0 and rng.random() < 0.7,
                zipf_src=round(rng.uniform(1.0, 1.5), 2), zipf_dst=round(rng.uniform(1.0, 1.5), 2), math=mode,
                model="jodie" if kind != "forward" and rng.random() < 0.15 else "tgn",
                embed_aux=kind == "host" and replay > 0 and rng.random() < 0.5)
    # no more work than the largest listed case; in the fp32 mode, which has no tensor cores, no more than its own
    most = next(c for c in listed() if c["name"] == ("wiki_fp32" if mode == "fp32" else "large_host_aux"))
    case["events"] = max(20_000, 24 * case["batch"])
    while case["batch"] > 100 and work(case)["flops"] > work(most)["flops"]:
        case["batch"] = int(case["batch"] * 0.83)
    case["events"] = _log(rng, max(20_000, 24 * case["batch"]), 1_300_000)
    return case


# ---- what a user's program has in hand ---------------------------------------------------------
def _config(case, seed):
    return wl.WorkloadConfig(case.get("name", "drawn"), case["nodes"], case["sources"], case["events"],
                             case.get("d_e", 0), case.get("feat", "f32"), case.get("d", 100), case.get("k", 10),
                             case.get("heads", 2), case["batch"], case.get("replay", 0.0), case.get("prune", False),
                             case["zipf_src"], case["zipf_dst"], seed)


def _zipf(n, s, size, gen):
    """Zipf-distributed node indices by inverse CDF, drawn on the device."""
    cdf = torch.from_numpy(np.cumsum(1.0 / np.arange(1, n + 1, dtype=np.float64) ** s)).cuda()
    u = torch.rand(size, dtype=torch.float64, device="cuda", generator=gen) * cdf[-1]
    return torch.searchsorted(cdf, u, right=True).clamp_(max=n - 1).int()


def _stream(cfg, gen):
    """An event stream with its time-sorted adjacency, drawn on the device (workload.make_stream's recipe)."""
    E, N, ns = cfg.num_events, cfg.num_nodes, cfg.num_src
    gaps = -torch.log1p(-torch.rand(E, dtype=torch.float64, device="cuda", generator=gen))
    # times in days, 5 000 events a day; integer sums are exact, hence the same on every call
    t = torch.cumsum((gaps * (1 << 20)).long(), 0).double() / (1 << 20) / 5000
    src = _zipf(ns or N, cfg.zipf_src, E, gen)
    if ns:
        dst = _zipf(N - ns, cfg.zipf_dst, E, gen) + ns
    else:
        dst = _zipf(N, cfg.zipf_dst, E, gen)
        dst = torch.where(dst == src, (dst + 1) % N, dst)      # no self-loops
    neg = torch.randint(ns, N, (E,), dtype=torch.int32, device="cuda", generator=gen)
    node = torch.stack((src, dst), 1).reshape(-1)               # both directions of every event, in time order
    order = torch.sort(node, stable=True).indices
    indptr = torch.zeros(N + 1, dtype=torch.int64, device="cuda")
    indptr[1:] = torch.cumsum(torch.bincount(node, minlength=N), 0)
    nbr = torch.stack((dst, src), 1).reshape(-1)[order]
    eid = (order // 2).int()
    h = lambda x: x.cpu().numpy()
    return wl.EventStream(cfg, h(src), h(dst), h(t), h(neg), h(indptr), h(nbr), h(eid), h(t[eid.long()]))


def _trainer(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    cfg = _config(case, seed)
    stream = _stream(cfg, gen)
    efeat = None
    if cfg.d_e:
        efeat = torch.empty((cfg.num_events, cfg.d_e), device="cuda",
                            dtype=torch.float32 if cfg.feat_dtype == "f32" else torch.bfloat16).normal_(generator=gen)
    last = cfg.num_batches - 1 if cfg.num_events % cfg.batch else cfg.num_batches      # full batches only
    dw = T.DeviceWorkload(stream, efeat=efeat, batches=range(last - SPAN - 1, last), embed_aux=case["embed_aux"])
    weights = wl.make_weights(cfg.d, cfg.d_e, seed, bias_scale=0.1, model=case["model"])
    tr = T.Trainer(dw, weights, math_mode=MATH[case["math"]], model=case["model"])
    # the state of a model in the middle of its training: memory and last-update times as the events so far leave
    # them, Adam moments of the size of this model's gradients
    tr.memory.normal_(0.0, 0.3, generator=gen).tanh_()
    lo = dw.batches.start * cfg.batch
    lu = np.zeros(cfg.num_nodes)
    for ends in (stream.src[:lo], stream.dst[:lo]):
        seen = np.zeros(cfg.num_nodes)
        seen[ends] = stream.t[:lo]
        np.maximum(lu, seen, out=lu)
    tr.last_update.copy_(torch.from_numpy(lu))
    tr.adam_m.normal_(0.0, 1e-5, generator=gen)
    tr.adam_v.uniform_(1e-7, 1e-6, generator=gen)
    tr.step_count.fill_(1000)
    return tr


def prepare(case, seed):
    if case["kind"] == "scan":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        s = _stream(_config(case, seed), gen)
        N, E, P, K, batch = case["nodes"], case["events"], case["workers"], case["window"], case["batch"]
        nb = (E + batch - 1) // batch
        dev = lambda a: torch.from_numpy(a).cuda()
        z = lambda *shape, dtype=torch.int32: torch.zeros(shape, dtype=dtype, device="cuda")
        return dict(kind="scan", batch=batch, K=K, P=P, src=dev(s.src), dst=dev(s.dst), t=dev(s.t), neg=dev(s.neg),
                    owner=torch.randint(0, P, (N,), dtype=torch.int32, device="cuda", generator=gen),
                    role=z(P, E, dtype=torch.uint8), n_sync=z(P, (nb + K - 1) // K),
                    sync=z(P, (nb + K - 1) // K, N, dtype=torch.uint8),
                    scratch=z(B.backward_scan_scratch(E, batch, K, N, P)), status=z(2), off=z(nb + 1), toff=z(nb + 1),
                    mb=(z(E), z(E), z(E, dtype=torch.float64), z(E), z(E, dtype=torch.uint8)),
                    tgt=(z(E), z(E), z(E, dtype=torch.float64), z(E), z(E)))
    if case["kind"] == "refresh":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        N, d, n = case["nodes"], case["d"], case["rows"]
        r = lambda *shape, dtype=torch.float32: torch.rand(shape, dtype=dtype, device="cuda", generator=gen)
        pick = lambda: torch.randperm(N, device="cuda", generator=gen)[:n].sort().values.int()
        times = r(n, dtype=torch.float64).view(n, 1).view(torch.float32)        # two floats hold a row's fp64 time
        return dict(kind="refresh", memory=r(N, d), last_update=r(N, dtype=torch.float64), send=pick(), recv=pick(),
                    packed=torch.zeros((n, d + 2), device="cuda"), received=torch.cat((r(n, d), times), 1).contiguous(),
                    status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    tr = _trainer(case, seed)
    dw = tr.dw
    s = dict(kind=case["kind"], tr=tr, at=0)
    if case["kind"] == "host":
        s["batches"] = {b: tr.host_batch(b) for b in dw.batches}
        s["loss"], s["gradnorm"] = torch.zeros(1).pin_memory(), torch.zeros(1).pin_memory()
    if case["kind"] == "forward":
        z = lambda *shape, dtype=torch.int32: torch.zeros(shape, dtype=dtype, device="cuda")
        n_u, R, k = case_mixed(case), 3 * case["batch"], case["k"]
        s.update(msg_node=z(2 * n_u), uniq=z(2 * n_u), winner=z(2 * n_u), n_uniq=z(1), nbr=z(R, k), eid=z(R, k),
                 ts=z(R, k, dtype=torch.float64), cnt=z(R), h=z(R, case["d"], dtype=torch.float32))
    return s


def case_mixed(case):
    """Events of a full mixed batch."""
    return case["batch"] + int(round(case["replay"] * case["batch"]))


# ---- one pass ----------------------------------------------------------------------------------
def _forward(s, b):
    tr = s["tr"]
    dw, lib = tr.dw, tr.lib
    u = dw.mb_slice(b - 1)
    lib.build_messages(dw.mb_src[u], dw.mb_dst[u], dw.mb_t[u], dw.mb_eid[u], dw.mb_keep[u], None, s["msg_node"])
    lib.reduce_latest(s["msg_node"], dw.mb_t[u], dw.mb_eid[u], s["uniq"], s["winner"], s["n_uniq"])
    lib.memory_update(None, s["uniq"], s["winner"], s["n_uniq"])
    src, dst, neg, t = dw.targets(b)
    s["nodes"], s["times"] = torch.cat((src, dst, neg)), t.repeat(3)
    lib.sample_recent(s["nodes"], s["times"], s["nbr"], s["eid"], s["ts"], s["cnt"])
    lib.embed(s["nodes"], s["times"], s["nbr"], s["eid"], s["ts"], s["cnt"], s["h"])
    return [s["h"], s["nbr"], s["eid"], s["ts"], s["cnt"], s["n_uniq"], s["uniq"], s["winner"], tr.memory, tr.last_update]


def run(s):
    if s["kind"] == "scan":
        B.backward_scan(s["src"], s["dst"], s["batch"], s["K"], s["owner"], s["P"], s["role"], s["n_sync"], s["sync"],
                        s["scratch"], s["status"][:1])
        B.build_mixed(s["src"], s["dst"], s["t"], s["neg"], s["batch"], s["role"][0], s["off"], s["toff"], s["mb"],
                      s["tgt"], s["status"][1:])
        return [s["role"], s["n_sync"], s["sync"], s["off"], s["toff"], *s["mb"], *s["tgt"], s["status"]]
    if s["kind"] == "refresh":
        B.pack_rows(s["memory"], s["last_update"], s["send"], s["packed"], s["status"])
        B.unpack_rows(s["memory"], s["last_update"], s["recv"], s["received"], s["status"])
        return [s["packed"].view(torch.int32), s["memory"], s["last_update"], s["status"]]
    tr = s["tr"]
    b = tr.dw.batches.start + 1 + s["at"]
    s["at"] = (s["at"] + 1) % SPAN
    if s["kind"] == "forward":
        return _forward(s, b)
    if s["kind"] == "host":
        tr.step_host(b, s["batches"][b], s["loss"], s["gradnorm"])
        scalars = [s["loss"], s["gradnorm"]]
    else:
        tr.step(b)
        scalars = [tr.loss, tr.gradnorm, tr.dw.mb_keep, tr.dw.heavy]
    return [*scalars, tr.memory, tr.last_update, tr.params, tr.adam_m, tr.adam_v, tr.step_count]


# ---- what a pass cannot do without -------------------------------------------------------------
def _distinct(n, s, draws):
    """Expected number of different values among `draws` Zipf(s) draws of n."""
    p = 1.0 / np.arange(1, n + 1, dtype=np.float64) ** s
    return float(np.sum(-np.expm1(draws * np.log1p(-np.minimum(p / p.sum(), 1 - 1e-12)))))


def work(case):
    """Bytes: each distinct row, record and parameter read once, each result written once.  Flops: the products of
    the method (forward; and for a training step the weight gradients and the input gradients it needs)."""
    if case["kind"] == "refresh":
        row = 4 * case["d"] + 8
        return {"bytes": case["rows"] * (4 * row + 8), "flops": 0}
    if case["kind"] == "scan":
        E, P, N = case["events"], case["workers"], case["nodes"]
        Q = -(-E // (case["batch"] * case["window"]))
        mine = E / P                                 # target events of one worker; its mixed batches hold at least these
        return {"bytes": 12 * E + P * E + P * Q * (N + 4) + E + 8 * E + mine * (21 + 24), "flops": 0}
    d, de, k, n_u, jodie = case["d"], case["d_e"], case["k"], case_mixed(case), case["model"] == "jodie"
    n_q = n_u if case["embed_aux"] else case["batch"]
    train = case["kind"] != "forward"
    R, NB, f = 3 * n_q, 3 * n_q * k, 4 if case["feat"] == "f32" else 2
    ns, N = case["sources"], case["nodes"]
    seen = lambda draws: (_distinct(ns, case["zipf_src"], draws) + _distinct(N - ns, case["zipf_dst"], draws) if ns
                          else _distinct(N, (case["zipf_src"] + case["zipf_dst"]) / 2, 2 * draws))
    U = seen(n_u)                                    # updated nodes
    roots = min(N, seen(n_q) + min(N - ns, n_q))     # embedded nodes, negatives among them
    recent = 0 if jodie else min(NB, roots * k + R)  # different neighbor records: k per node, then one more per event
    d_msg, d_kv, g = 3 * d + de, 2 * d + de, 1 if jodie else 3
    P = sum(int(np.prod(x)) for x in wl.param_shapes(d, de, case["model"]).values())
    by = n_u * 21 + n_q * 20 + U * (de * f + 2 * (4 * d + 8)) + recent * (16 + de * f) + min(N, roots + recent) * 4 * d
    by += 24 * P if train else 4 * P + R * 4 * d + NB * 16
    cell, attn = U * 2.0 * g * d * (d_msg + d), 0.0
    if not jodie:
        attn = 2.0 * NB * 2 * d * d_kv + 2 * (2.0 * R * d * 2 * d) + 4.0 * R * k * d
    flops = cell + attn
    if train:
        head = 2.0 * (2 * n_q) * d * 2 * d
        flops += cell + U * 2.0 * g * d * d + 3 * head   # update cell: weight gradients, gradient of the encoded time
        if not jodie:                                    # weight gradients, input gradients without the feature columns
            flops += 2.0 * NB * 2 * d * d_kv + 2.0 * NB * 2 * d * 2 * d + 4 * (2.0 * R * d * 2 * d) + 8.0 * R * k * d
    return {"bytes": by, "flops": flops}


def tolerance(case):
    """Index work and copied rows are the same to the bit.  Embeddings and memory come from fp32 sums of operands of 21
    bits and more (a few 1e-6 between the modes).  Gradients differ by about 1e-5 between correct summation orders, and
    by up to 5e-4 where a hidden unit whose pre-activation is zero to rounding takes the other branch of its ReLU: that
    unit's row of the gradient then moves by a few percent of its largest entry."""
    if case["kind"] in ("scan", "refresh"):
        return "exact"
    return {"rel": 2e-5, "max": 2e-4} if case["kind"] == "forward" else {"rel": 1e-3, "max": 5e-2}
