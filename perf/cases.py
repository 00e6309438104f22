"""What this framework is used for, as cases that can be timed and compared.

Each case is one call sequence of a user's program through the public entry
points: training steps over a resident or a host store, screening forwards,
requests to the inference server, the aggregation operator under autograd and
the collation of a batch.  Sizes follow the configurations of bench.py and the
tests: molecules of 3-51 atoms (log-normal, mean 18) for training, 5-30 for the
small parity model, 5-80 for screening; hidden 200 and 6 layers for the
benchmark model, hidden 256 with batches of 1,024 for the recomputation study.

A molecule is a random spanning tree plus extra bonds up to 1.1 n + 0.5, at
most four bonds per atom, every bond stored in both directions.
"""
import math
import os
import tempfile

import numpy as np
import torch

import paper_2207_11333_gb300 as gcnn
from paper_2207_11333_gb300 import autograd

TYPES = 7
TYPE_PROB = (.45, .33, .08, .08, .02, .02, .02)
STEPS = 4          # a training state's store holds the molecules of this many steps
LR = 1e-4          # a rate at which the synthetic model's training is stable
STD_EPS = 1e-5


def listed():
    return [
        # one optimisation step of the benchmark model, the work of a training run
        dict(name="train_bf16_b128", kind="train", precision="bf16", H=200, L=6, G=128, sizes="lognormal",
             F=0, node_head=False, recompute=False, host=False),
        # a short last batch of an epoch, or one process's share of a step spread over many
        dict(name="train_bf16_b13", kind="train", precision="bf16", H=200, L=6, G=13, sizes="lognormal",
             F=0, node_head=False, recompute=False, host=False),
        # the benchmark step with bond features and a node-level head (multitask training)
        dict(name="train_bf16_bonds_nodes_b128", kind="train", precision="bf16", H=200, L=6, G=128, sizes="lognormal",
             F=4, node_head=True, recompute=False, host=False),
        # large batches of a wider model, aggregates recomputed in the backward to save memory
        dict(name="train_bf16_b1024_recompute", kind="train", precision="bf16", H=256, L=6, G=1024, sizes="lognormal",
             F=0, node_head=False, recompute=True, host=False),
        # the full-precision training path, the one that precision studies compare with
        dict(name="train_fp32_b128", kind="train", precision="fp32", H=200, L=6, G=128, sizes="lognormal",
             F=0, node_head=False, recompute=False, host=False),
        # the small model of the parity workload, batches loaded from host memory at every step
        dict(name="train_fp32_small_host", kind="train", precision="fp32", H=32, L=2, G=64, sizes="small",
             F=0, node_head=False, recompute=False, host=True),
        # screening a large collection offline, in both precisions
        dict(name="screen_bf16_3600", kind="forward", precision="bf16", H=200, L=6, G=3600, sizes="lognormal"),
        dict(name="screen_fp32_1100", kind="forward", precision="fp32", H=200, L=6, G=1100, sizes="lognormal"),
        # an interactive request to the server: one molecule, where latency counts
        dict(name="serve_bf16_one", kind="serve", precision="bf16", H=200, L=6, requests=1, most=1),
        # a burst of requests of very different sizes, at the server's default precision
        dict(name="serve_fp32_burst", kind="serve", precision="fp32", H=200, L=6, requests=12, most=257),
        # the aggregation operator composed in PyTorch, forward and gradient, a batch far above the L2 cache
        dict(name="aggregate_300k_atoms", kind="aggregate", H=200, G=16500, sizes="lognormal"),
        # assembling one batch from host memory, the loading phase of every step
        dict(name="collate_host_b128", kind="collate", G=128, sizes="lognormal"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train", "train", "train", "forward", "forward", "serve", "aggregate", "collate"])
    if kind == "train":
        precision = rng.choice(["bf16", "bf16", "fp32"])
        H = rng.choice([32, 64, 104, 200, 256] if precision == "bf16" else [24, 32, 104, 200])
        G = _log_int(rng, 5, 900 if precision == "bf16" else 120)
        F = rng.choice([0, 0, 1, 4, 7])
        return dict(kind="train", precision=precision, H=H, L=rng.randint(1, 6), G=G,
                    sizes=rng.choice(["lognormal", "lognormal", "small"]), F=F, node_head=rng.random() < .25,
                    recompute=rng.random() < .25, host=rng.random() < .3)
    if kind == "forward":
        precision = rng.choice(["bf16", "fp32"])
        return dict(kind="forward", precision=precision, H=rng.choice([32, 104, 200]), L=rng.randint(1, 6),
                    G=_log_int(rng, 1, 3500 if precision == "bf16" else 1000), sizes="lognormal")
    if kind == "serve":
        return dict(kind="serve", precision=rng.choice(["bf16", "fp32"]), H=200, L=rng.randint(2, 6),
                    requests=rng.randint(1, 12), most=_log_int(rng, 1, 250))
    if kind == "aggregate":
        return dict(kind="aggregate", H=4 * _log_int(rng, 2, 50), G=_log_int(rng, 3, 16000), sizes="lognormal")
    return dict(kind="collate", G=_log_int(rng, 2, 2000), sizes=rng.choice(["lognormal", "screen"]))


# ---------------------------------------------------------------- molecules

def _counts(rng, G, sizes):
    """Atoms per molecule: the same sizes for every seed, in another order."""
    own = _rng(G)
    if sizes == "small":
        return rng.permutation(own.integers(5, 31, G))
    if sizes == "screen":
        return rng.permutation(own.integers(5, 81, G))
    n = np.exp(own.normal(2.80, .45, 4 * G + 64))  # about 18 atoms on average within [3, 51]
    n = np.rint(n[(n >= 2.5) & (n < 51.5)]).astype(np.int64)
    return rng.permutation(n[:G])


def molecules(rng, G, sizes, F=0, node_y=False):
    """G molecules as global arrays (node_ptr, edge_ptr, types, edges, y, and bond features and atom targets)."""
    n = _counts(rng, G, sizes)
    most = int(n.max())
    deg = np.zeros((G, most), np.int64)
    adj = np.zeros((G, most, most), bool)
    rows = np.arange(G)
    bonds = []  # (graph, u, v)

    def bond(at, u, v):
        adj[at, u, v] = adj[at, v, u] = True
        deg[at, u] += 1
        deg[at, v] += 1
        bonds.append(np.stack([at, u, v], 1))

    for v in range(1, most):  # spanning tree: each atom joins an earlier one with a free place
        at = rows[n > v]
        free = np.where(deg[at, :v] < 4, rng.random((len(at), v)), -1.)
        bond(at, free.argmax(1), np.full(len(at), v))
    wanted = np.floor(1.1 * n + .5).astype(np.int64) - (n - 1)
    for _ in range(1000):  # rings: random pairs that are free and not yet bonded
        at = rows[wanted > 0]
        if not len(at):
            break
        u, v = (np.minimum((rng.random(len(at)) * n[at]).astype(np.int64), n[at] - 1) for _ in range(2))
        ok = (u != v) & (deg[at, u] < 4) & (deg[at, v] < 4) & ~adj[at, u, v]
        bond(at[ok], u[ok], v[ok])
        wanted[at[ok]] -= 1
    b = np.concatenate(bonds)
    b = b[np.argsort(b[:, 0], kind="stable")]
    node_ptr = np.concatenate([[0], np.cumsum(n)]).astype(np.int64)
    edge_ptr = np.concatenate([[0], np.cumsum(2 * np.bincount(b[:, 0], minlength=G))]).astype(np.int64)
    edges = np.empty((2 * len(b), 2), np.uint8)
    edges[0::2] = b[:, 1:]
    edges[1::2] = b[:, :0:-1]
    N = int(node_ptr[-1])
    return dict(node_ptr=node_ptr, edge_ptr=edge_ptr, types=rng.choice(TYPES, N, p=TYPE_PROB).astype(np.uint8),
                edges=edges, y=rng.uniform(1, 10, G).astype(np.float32),
                eattr=np.repeat(rng.uniform(-1, 1, (len(b), F)), 2, 0).astype(np.float32) if F else None,
                ynode=rng.uniform(-1, 1, N).astype(np.float32) if node_y else None)


def open_store(m):
    """The molecules as a packed store file, opened (the file is not needed afterwards)."""
    G, N, E = len(m["y"]), len(m["types"]), len(m["edges"])
    arrays = [m["node_ptr"], m["edge_ptr"], m["types"], m["edges"], m["y"]]
    more = [m["eattr"], m["ynode"]]
    at, pos = [], 128
    for a in arrays + more:
        pos = (pos + 63) // 64 * 64
        at.append(pos if a is not None else 0)
        pos += 0 if a is None else a.nbytes
    size = (pos + 63) // 64 * 64
    data = np.zeros(size, np.uint8)
    version = 2 if any(a is not None for a in more) else 1
    data[:8] = np.frombuffer(b"GCNNPKD1", np.uint8)
    data[8:16] = np.array([version, TYPES], "<u4").view(np.uint8)
    data[16:88] = np.array([G, N, E] + at[:5] + [size], "<i8").view(np.uint8)
    if version == 2:
        F = 0 if m["eattr"] is None else m["eattr"].shape[1]
        data[88:112] = np.array([F, at[5], at[6]], "<i8").view(np.uint8)
    for o, a in zip(at, arrays + more):
        if a is not None:
            data[o:o + a.nbytes] = np.ascontiguousarray(a).reshape(-1).view(np.uint8)
    fd, path = tempfile.mkstemp(suffix=".gcnn")
    try:
        with os.fdopen(fd, "wb") as f:
            f.write(data.tobytes())
        return gcnn.Store(path)
    finally:
        os.unlink(path)


def layout(H, L, F=0, node_head=False):
    """Name -> (offset, shape, fan-in) of the flat parameter vector, and its length."""
    v, at = {}, 0

    def take(name, *shape, fan=None):
        nonlocal at
        v[name] = (at, shape, fan)
        at += math.prod(shape)

    take("emb", TYPES, H)
    for k in range(L):
        take("msg_w%d" % k, H, 2 * H, fan=2 * H + F)
        take("msg_b%d" % k, H, fan=2 * H + F)
        take("upd_w%d" % k, 16 * H, H, fan=16 * H)
        take("upd_b%d" % k, H, fan=16 * H)
    take("w1", H, H, fan=H)
    take("b1", H, fan=H)
    take("w2", H, fan=H)
    take("b2", 1, fan=H)
    if F:
        at = (at + 3) // 4 * 4
        for k in range(L):
            take("edge_w%d" % k, F, H, fan=2 * H + F)
    if node_head:
        at = (at + 3) // 4 * 4
        take("w1n", H, H, fan=H)
        take("b1n", H, fan=H)
        take("w2n", H, fan=H)
        take("b2n", 1, fan=H)
    return v, at


def parameters(rng, H, L, F=0, node_head=False):
    v, size = layout(H, L, F, node_head)
    p = np.zeros(size, np.float32)
    for at, shape, fan in v.values():
        n = math.prod(shape)
        p[at:at + n] = rng.normal(size=n) if fan is None else (2 * rng.random(n, np.float32) - 1) / math.sqrt(fan)
    return p


def _rng(seed):
    return np.random.default_rng(seed)


def _train_inputs(c, seed):
    rng = _rng(seed)
    m = molecules(rng, STEPS * c["G"], c["sizes"], c["F"], c["node_head"])
    return m, parameters(rng, c["H"], c["L"], c["F"], c["node_head"]), rng.permutation(STEPS * c["G"])


def _serve_inputs(c, seed):
    rng = _rng(seed)
    k = np.rint(np.geomspace(c["most"], 1, c["requests"])).astype(np.int64)  # the largest first
    return [molecules(rng, int(q), "screen") for q in k], parameters(rng, c["H"], c["L"])


def _batch_inputs(c, seed):
    rng = _rng(seed)
    return rng, molecules(rng, c["G"], c["sizes"])


def _delta(m):
    d = np.bincount((np.repeat(m["node_ptr"][:-1], np.diff(m["edge_ptr"])) + m["edges"][:, 1]).astype(np.int64),
                    minlength=len(m["types"]))
    return float(np.mean(np.log(d + 1.)))


# ---------------------------------------------------------------- the calls

def _precision(c):
    return gcnn.PREC_BF16 if c["precision"] == "bf16" else gcnn.PREC_FP32


def _held(view, ctx):
    """A view of a context's memory that keeps the context: results are read after the state is gone."""
    view.owner = ctx
    return view


def prepare(c, seed):
    if c["kind"] == "train":
        m, params, order = _train_inputs(c, seed)
        st = open_store(m)
        sizes = [st.batch_size(order[k * c["G"]:(k + 1) * c["G"]]) for k in range(STEPS)]
        ctx = gcnn.Context(gcnn.make_config(
            c["H"], c["L"], c["G"], max(s[0] for s in sizes), max(s[1] for s in sizes), delta=st.delta(),
            precision=_precision(c), recompute=int(c["recompute"]), edge_features=c["F"],
            node_head=int(c["node_head"])))
        ctx.set_params(params)
        if not c["host"]:
            st.to_device()
            ctx.set_order(st, order)
        loss = torch.zeros(5 if c["node_head"] else 3, dtype=torch.float64, device="cuda")
        return dict(case=c, st=st, ctx=ctx, order=order, loss=loss, at=0, grads=_held(ctx.grads_tensor(), ctx))
    if c["kind"] == "forward":
        rng, m = _batch_inputs(c, seed)
        st = open_store(m)
        st.to_device()
        ctx = gcnn.Context(gcnn.make_config(c["H"], c["L"], c["G"], st.n_nodes, st.n_edges, delta=st.delta(),
                                            precision=_precision(c)))
        ctx.set_params(parameters(rng, c["H"], c["L"]))
        ctx.set_order(st, np.arange(c["G"]))
        return dict(case=c, st=st, ctx=ctx, pred=torch.empty(c["G"], device="cuda"))
    if c["kind"] == "serve":
        reqs, params = _serve_inputs(c, seed)
        model = gcnn.Context(gcnn.make_config(c["H"], c["L"], 1, 256, 1024, delta=1.1, precision=_precision(c)))
        model.set_params(params)
        srv = gcnn.Server(model, n_slots=2, buckets=(1024, 4096, 16384), max_graphs=1024, precision=_precision(c),
                          queue_nodes=1 << 20)
        return dict(case=c, model=model, srv=srv, reqs=[
            (np.diff(m["node_ptr"]).astype(np.int32), np.diff(m["edge_ptr"]).astype(np.int32), m["types"], m["edges"])
            for m in reqs])
    rng, m = _batch_inputs(c, seed)
    st = open_store(m)
    ctx = gcnn.Context(gcnn.make_config(8, 1, c["G"], st.n_nodes, st.n_edges, delta=st.delta()))
    b = ctx.collate(st, np.arange(c["G"]))
    if c["kind"] == "collate":  # a batch's arrays stay where they are; each call fills them
        return dict(case=c, st=st, ctx=ctx, ids=rng.permutation(c["G"]), views={k: _held(b.tensor(k), ctx) for k in (
            "node_off", "edge_off", "graph_id", "row_ptr", "col", "rev", "deg", "types", "amp", "att", "y")})
    PQ, dagg = _aggregate_inputs(c, seed, st.n_nodes)
    return dict(case=c, st=st, ctx=ctx, PQ=PQ.requires_grad_(), dagg=dagg,
                csr=[b.tensor(k) for k in ("row_ptr", "col", "rev", "node_off")])


def _aggregate_inputs(c, seed, N):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn(N, w * c["H"], device="cuda", generator=gen) for w in (2, 5)]


def run(s):
    c = s["case"]
    if c["kind"] == "train":
        first, G = s["at"] * c["G"], c["G"]
        s["at"] = (s["at"] + 1) % STEPS
        if c["host"]:
            s["ctx"].train_step(s["ctx"].collate(s["st"], s["order"][first:first + G]), LR, s["loss"])
        else:
            s["ctx"].train_step_range(s["st"], first, G, LR, s["loss"])
        return {"grads": s["grads"], "loss": s["loss"]}
    if c["kind"] == "forward":
        b = s["ctx"].collate_range(s["st"], 0, c["G"])
        s["ctx"].forward(b, s["pred"], train=False)
        return s["pred"]
    if c["kind"] == "serve":
        tickets = [s["srv"].submit(*r) for r in s["reqs"]]
        return [s["srv"].wait(t)[0] for t in tickets]
    if c["kind"] == "collate":
        s["ctx"].collate(s["st"], s["ids"])
        return s["views"]
    row_ptr, col, rev, node_off = s["csr"]
    agg = autograd.aggregate(s["PQ"], row_ptr, col, rev, STD_EPS, node_off)
    return [agg.detach(), torch.autograd.grad(agg, s["PQ"], s["dagg"])[0]]


def _mean_atoms(sizes):
    return {"small": 17.5, "screen": 42.5, "lognormal": 18.}[sizes]


def work(c):
    """Weights and molecules read once, results (and a training step's state) written once; the dense layers' operations."""
    if c["kind"] == "serve":
        mols = float(np.rint(np.geomspace(c["most"], 1, c["requests"])).sum())
        N, P = 42.5 * mols, layout(c["H"], c["L"])[1]
        return {"bytes": (2 if c["precision"] == "bf16" else 4) * P + 5.4 * N + 4 * mols,
                "flops": 36. * c["H"] ** 2 * N * c["L"]}
    N = c["G"] * _mean_atoms(c["sizes"])
    E = 2.2 * N
    if c["kind"] == "collate":  # types and bonds in; offsets, graph ids, CSR, reverse slots, degrees and scalers out
        return {"bytes": N + 2 * E + 20. * c["G"] + N * (4 * 5 + 1) + 8 * E + 12. * c["G"], "flops": 0}
    if c["kind"] == "aggregate":  # P|Q and CSR in, aggregates out; then their gradient and P|Q in, P|Q's gradient out
        return {"bytes": 4. * c["H"] * N * (2 + 5 + 5 + 2 + 2) + 4 * (N + 2 * E), "flops": 30. * E * c["H"]}
    H, L = c["H"], c["L"]
    if c["kind"] == "forward":
        return {"bytes": (2 if c["precision"] == "bf16" else 4) * layout(H, L)[1] + N + 2 * E + 4. * c["G"],
                "flops": 36. * H * H * N * L}
    P = layout(H, L, c["F"], c["node_head"])[1]
    return {"bytes": 28. * P + N + 2 * E + 4. * E * c["F"],
            "flops": (108. * H * H * L + 4. * E / N * c["F"] * H * L + (6. * H * H if c["node_head"] else 0.)) * N}


# ---------------------------------------------------------------- in 64 bits

def _batch(m, ids=None):
    """The molecules ids as one graph: atom types, sources and destinations, molecule of each atom, on the GPU."""
    ids = np.arange(len(m["y"])) if ids is None else ids
    n, e = np.diff(m["node_ptr"])[ids], np.diff(m["edge_ptr"])[ids]

    def spread(ptr, cnt):
        return np.repeat(ptr[ids] - np.concatenate([[0], np.cumsum(cnt)[:-1]]), cnt) + np.arange(cnt.sum())

    atoms, bonds = spread(m["node_ptr"], n), spread(m["edge_ptr"], e)
    base = np.repeat(np.concatenate([[0], np.cumsum(n)[:-1]]), e)
    ed = m["edges"][bonds].astype(np.int64)
    g = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    return dict(types=g(m["types"][atoms].astype(np.int64)), src=g(ed[:, 0] + base), dst=g(ed[:, 1] + base),
                mol=g(np.repeat(np.arange(len(ids)), n)), n=g(n.astype(np.float64)), y=g(m["y"][ids].astype(np.float64)),
                eattr=None if m["eattr"] is None else g(m["eattr"][bonds].astype(np.float64)),
                ynode=None if m["ynode"] is None else g(m["ynode"][atoms].astype(np.float64)))


def _aggregates(m, dst, N, deg):
    idx = dst[:, None].expand_as(m)
    z = m.new_zeros(N, m.shape[1])
    mean = z.index_add(0, dst, m) / deg
    var = z.index_add(0, dst, (m - mean[dst]) ** 2) / deg
    return [mean * deg, mean, z.scatter_reduce(0, idx, m, "amin", include_self=False),
            z.scatter_reduce(0, idx, m, "amax", include_self=False), torch.sqrt(torch.relu(var) + STD_EPS)]


def _model(c, p, b, delta, node_head=False):
    """Predictions per molecule (and per atom) of the flat parameters p."""
    w = {k: p[at:at + math.prod(shape)].view(shape) for k, (at, shape, _) in
         layout(c["H"], c["L"], c.get("F", 0), node_head)[0].items()}
    N, H = len(b["types"]), c["H"]
    deg = torch.bincount(b["dst"], minlength=N).double()[:, None]
    s = torch.log(deg + 1) / delta
    x = w["emb"][b["types"]]
    for k in range(c["L"]):
        pq = x @ w["msg_w%d" % k]
        m = (pq[:, :H] + w["msg_b%d" % k])[b["dst"]] + pq[:, H:][b["src"]]
        if b["eattr"] is not None:
            m = m + b["eattr"] @ w["edge_w%d" % k]
        a = torch.cat(_aggregates(m, b["dst"], N, deg), 1)
        x = torch.relu(torch.cat([x, a, s * a, a / s], 1) @ w["upd_w%d" % k] + w["upd_b%d" % k])
    g = x.new_zeros(len(b["n"]), H).index_add(0, b["mol"], x) / b["n"][:, None]
    pred = torch.relu(g @ w["w1"] + w["b1"]) @ w["w2"] + w["b2"]
    return pred, torch.relu(x @ w["w1n"] + w["b1n"]) @ w["w2n"] + w["b2n"] if node_head else None


def exact(c, seed):
    if c["kind"] == "train":
        m, params, order = _train_inputs(c, seed)
        b = _batch(m, order[:c["G"]])
        p = torch.from_numpy(params).cuda().double().requires_grad_()
        pred, atom = _model(c, p, b, _delta(m), c["node_head"])
        off = pred - b["y"]
        loss, sums = (off ** 2).mean(), [(off ** 2).sum(), off.abs().sum(), off.new_tensor(len(off))]
        if c["node_head"]:
            off = atom - b["ynode"]
            loss, sums = loss + (off ** 2).mean(), sums + [(off ** 2).sum(), off.new_tensor(len(off))]
        return {"grads": torch.autograd.grad(loss, p)[0], "loss": torch.stack(sums).detach()}
    if c["kind"] == "forward":
        rng, m = _batch_inputs(c, seed)
        p = torch.from_numpy(parameters(rng, c["H"], c["L"])).cuda().double()
        with torch.no_grad():
            return _model(c, p, _batch(m), _delta(m))[0]
    if c["kind"] == "serve":
        reqs, params = _serve_inputs(c, seed)
        p = torch.from_numpy(params).cuda().double()
        with torch.no_grad():
            return [_model(c, p, _batch(m), 1.1)[0].cpu().numpy() for m in reqs]
    rng, m = _batch_inputs(c, seed)
    if c["kind"] == "collate":
        b = _batch(m, rng.permutation(c["G"]))
        s = torch.log(torch.bincount(b["dst"], minlength=len(b["types"])).double() + 1) / _delta(m)
        whole = ("node_off", "edge_off", "graph_id", "row_ptr", "col", "rev", "deg", "types")
        return {**{k: None for k in whole}, "amp": s, "att": 1 / s, "y": b["y"]}
    b = _batch(m)
    N, H = len(b["types"]), c["H"]
    PQ, dagg = (t.double() for t in _aggregate_inputs(c, seed, N))
    PQ.requires_grad_()
    deg = torch.bincount(b["dst"], minlength=N).double()[:, None]
    agg = torch.cat(_aggregates(PQ[:, :H][b["dst"]] + PQ[:, H:][b["src"]], b["dst"], N, deg), 1)
    return [agg.detach(), torch.autograd.grad(agg, PQ, dagg)[0]]
