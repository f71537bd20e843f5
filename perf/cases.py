"""Workloads of the band-GGNN library as its users run them, for timing and for checking results.

Every case is one call sequence through the public binding (`paper_1906_11786_gb300.lib`): node
states and gradients come in the caller's own node order, are packed into band order, go through
the propagation, the GGNN layer or the training step, and come back in the caller's order.  Sizes
are those of this repository's workloads (`synth.WORKLOADS`) and tests, with smaller and ragged
batches between them.  Graphs are the program-shaped ones of `synth`, whose short-range edges reach
three eighths of a block, so that after the reordering every edge lies inside the three block
diagonals and the 64-bit reference is a plain sum over all edges.

Case fields: op (see `run`), dtype, graphs drawn with node counts in [lo, hi] until `nodes` is
reached (one graph of exactly `nodes` nodes when lo = 0), S block size, H state size, F edge
families (P = 2 F types with `reverse`, else F), lam edges per node of a short-range family, T steps.
"""
import math

import numpy as np
import torch

from paper_1906_11786_gb300 import lib as L
from paper_1906_11786_gb300 import synth

KEYS = ("W", "b", "W_ih", "W_hh", "b_ih", "b_hh")
LR, B1, B2, EPS, STEP = 1e-3, 0.9, 0.999, 1e-8, 100


def _case(name, op, dtype, nodes, lo, hi, S, H, F, reverse, T=1, lam=3.0):
    c = dict(op=op, dtype=dtype, nodes=nodes, lo=lo, hi=hi, S=S, H=H, F=F, reverse=reverse, T=T,
             lam=lam)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small graph in fp32, one propagation: the interactive call, all latency
        _case("f32_512_fwd", "fwd", "f32", 512, 0, 0, 64, 64, 4, False, lam=1.0),
        _case("f32_512_bwd", "bwd", "f32", 512, 0, 0, 64, 64, 4, False, lam=1.0),
        # a ragged fp32 batch through a two-step model: full-precision inference, state size off
        # the powers of two
        _case("f32_batch_infer", "infer", "f32", 3001, 100, 900, 64, 96, 6, True, T=2, lam=2.0),
        # a handful of graphs through the whole model: serving latency
        _case("small_infer", "infer", "bf16", 800, 100, 300, 128, 64, 10, True, T=8),
        # a narrow-band batch whose padded size is not a whole number of 128-row tiles
        _case("ragged_S32_fwd", "fwd", "bf16", 30011, 200, 2000, 32, 64, 10, True),
        # the packed batch of 64 graphs (70k nodes): one propagation in each direction
        _case("packed64_fwd", "fwd", "bf16", 72000, 200, 2000, 128, 64, 10, True),
        _case("packed64_bwd", "bwd", "bf16", 72000, 200, 2000, 128, 64, 10, True),
        # ... and the whole eight-step model over it: batch inference
        _case("packed64_infer", "infer", "bf16", 72000, 200, 2000, 128, 64, 10, True, T=8),
        # one large graph with a wide band
        _case("single20k_bwd", "bwd", "bf16", 20000, 0, 0, 256, 128, 10, True),
        # the widest band of the block-size sweep, at its full node count
        _case("sweep131k_S512_fwd", "fwd", "bf16", 131072, 200, 2000, 512, 64, 10, True),
        # one GGNN layer's backward at the largest state size
        _case("layer_H256_bwd", "layer_bwd", "bf16", 40000, 200, 5000, 128, 256, 10, True),
        # the training step: forward, readout loss, backward, Adam
        _case("train100k_H128", "train", "bf16", 100000, 200, 5000, 128, 128, 10, True, T=8),
    ]


def draw(rng):
    """One more case of the same ranges; sizes spread over their logarithm, odd ones among them."""
    op = rng.choice(["fwd", "fwd", "bwd", "bwd", "infer", "layer_bwd", "train"])
    dtype = "f32" if rng.random() < 0.2 else "bf16"
    S = rng.choice([32, 64, 128, 128, 256, 512])
    H = rng.choice([32, 64, 64, 128, 256] if dtype == "bf16" else [32, 64, 96])
    top = 6000 if dtype == "f32" else {32: 130000, 64: 130000, 128: 90000, 256: 30000}[H]
    nodes = int(round(math.exp(rng.uniform(math.log(400), math.log(top)))))
    F = rng.choice([4, 10, 10])
    reverse = F == 10 or rng.random() < 0.5
    T = rng.choice([2, 4, 8]) if op in ("infer", "train") else 1
    lo, hi = (0, 0) if nodes <= 20000 and rng.random() < 0.25 else (min(200, nodes), min(2000, nodes))
    return _case(None, op, dtype, nodes, lo, hi, S, H, F, reverse, T, rng.choice([1.0, 2.0, 3.0]))


# ---------------------------------------------------------------------------------- inputs


def _sizes(c, seed):
    if c["lo"] == 0:
        return [c["nodes"]]
    rng = np.random.default_rng([seed, 1])
    out, left = [], c["nodes"]
    while left > 0:
        x = min(int(rng.integers(c["lo"], c["hi"] + 1)), left)
        out.append(x)
        left -= x
    return out


def _graphs(c, seed):
    reach = 3 * c["S"] // 8
    return [synth.gen_graph(n, c["F"], c["reverse"], reach, reach, c["lam"], 1000003 * seed + 17 * g)
            for g, n in enumerate(_sizes(c, seed))]


def _inputs(c, seed, graphs):
    """Everything random but the graphs, on the GPU, in the caller's node order."""
    n, H = sum(g.n_nodes for g in graphs), c["H"]
    P = graphs[0].n_types
    wdt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = {"E": torch.randn((n, H), generator=gen, device="cuda").to(wdt)}
    # gradients arriving at the states, and the readout's targets
    x["dY"] = torch.randn((n, H), generator=gen, device="cuda")
    x["target"] = torch.randn(len(graphs), generator=gen, device="cuda")
    deg = sum(g.n_edges for g in graphs) / n
    prm = synth.gen_params(P, H, seed, mean_in_degree=deg)
    w = {k: torch.from_numpy(np.asarray(prm[k], np.float32)).cuda() for k in KEYS + ("w_out",)}
    x["w32"] = w
    x["w"] = {k: (v.to(wdt) if k in ("W", "W_ih", "W_hh") else v) for k, v in w.items()}
    if c["op"] == "train":
        # optimizer state of a run under way
        m = sum(w[k].numel() for k in KEYS)
        x["m"] = 0.01 * torch.randn(m, generator=gen, device="cuda")
        x["v"] = 1e-4 * torch.rand(m, generator=gen, device="cuda") + 1e-5
    return x


def _bytes(n):
    return torch.empty(max(int(n), 16), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    c = case
    graphs = _graphs(c, seed)
    x = _inputs(c, seed, graphs)
    dt, H, T, op = c["dtype"], c["H"], c["T"], c["op"]
    P = graphs[0].n_types
    plan = L.band_plan(graphs, P, c["S"])
    plan.upload()
    N = plan.info()["n_pad"]
    n = x["E"].shape[0]
    s = dict(c=c, x=x, plan=plan)
    s["Eb"] = torch.empty((N, H), dtype=x["E"].dtype, device="cuda")
    f32 = dict(dtype=torch.float32, device="cuda")
    if op in ("fwd", "bwd"):
        which = L.BG_OP_PROPAGATE_FWD if op == "fwd" else L.BG_OP_PROPAGATE_BWD
        s["ws"] = _bytes(L.workspace_bytes(plan, dt, H, which))
    else:
        s["saved"] = _bytes(L.ggnn_saved_bytes(plan, dt, H, T))
        s["ws"] = _bytes(max(L.ggnn_workspace_bytes(plan, dt, H, T, o)
                             for o in (L.BG_OP_GGNN_FWD, L.BG_OP_GGNN_BWD)))
    if op == "fwd":
        s["Yb"], s["Y"] = torch.empty((N, H), **f32), torch.empty((n, H), **f32)
    if op in ("bwd", "layer_bwd"):
        s["dYb"], s["dEb"] = torch.empty((N, H), **f32), torch.empty((N, H), **f32)
        s["dE"] = torch.empty((n, H), **f32)
        L.pack_states(plan, dt, H, x["E"], s["Eb"])  # the forward's packed states
    if op in ("infer", "train"):
        s["ETb"], s["ET"] = torch.empty_like(s["Eb"]), torch.empty_like(x["E"])
    names = {"bwd": KEYS[:2], "layer_bwd": KEYS, "train": KEYS}.get(op, ())
    if op == "train":
        # one flat buffer each for master weights, working weights and gradients, as an optimizer
        # that updates everything in one call keeps them
        s["master"] = torch.cat([x["w32"][k].reshape(-1) for k in KEYS])
        s["work"] = s["master"].to(torch.bfloat16) if dt == "bf16" else s["master"].clone()
        s["grad"] = torch.zeros_like(s["master"])
        s["m"], s["v"] = x["m"], x["v"]
        s["prm"], s["g"], o = {}, {}, 0
        for k in KEYS:
            w = x["w"][k]
            flat = s["work"] if k in ("W", "W_ih", "W_hh") else s["master"]
            s["prm"][k] = flat[o:o + w.numel()].view(w.shape)
            s["g"]["d" + k] = s["grad"][o:o + w.numel()].view(w.shape)
            o += w.numel()
        s["loss"], s["dw_out"] = torch.empty(1, **f32), torch.empty(H, **f32)
        s["dEb"] = torch.empty((N, H), **f32)
        s["dEb0"] = torch.empty((N, H), **f32)
        s["rws"] = _bytes(L.workspace_bytes(plan, dt, H, L.BG_OP_READOUT))
    else:
        s["prm"] = x["w"]
        s["g"] = {"d" + k: torch.empty(x["w"][k].shape, **f32) for k in names}
    if op == "layer_bwd":
        L.ggnn_step(plan, dt, H, T, s["prm"], s["Eb"], None, s["saved"], s["ws"])
    return s


# ---------------------------------------------------------------------------------- one pass


def run(state):
    s, c, x, plan = state, state["c"], state["x"], state["plan"]
    dt, H, T, op = c["dtype"], c["H"], c["T"], c["op"]
    if op == "fwd":
        L.pack_states(plan, dt, H, x["E"], s["Eb"])
        L.band_propagate_fwd(plan, dt, H, s["Eb"], s["prm"]["W"], s["prm"]["b"], s["Yb"], s["ws"])
        L.unpack_states(plan, "f32", H, s["Yb"], s["Y"])
        return {"Y": s["Y"]}
    if op == "bwd":
        L.pack_states(plan, "f32", H, x["dY"], s["dYb"])
        L.band_propagate_bwd(plan, dt, H, s["Eb"], s["prm"]["W"], s["dYb"], s["dEb"],
                             s["g"]["dW"], s["g"]["db"], s["ws"])
        L.unpack_states(plan, "f32", H, s["dEb"], s["dE"])
        return dict(s["g"], dE=s["dE"])
    if op == "infer":
        L.pack_states(plan, dt, H, x["E"], s["Eb"])
        L.ggnn_step(plan, dt, H, T, s["prm"], s["Eb"], s["ETb"], s["saved"], s["ws"])
        L.unpack_states(plan, dt, H, s["ETb"], s["ET"])
        return {"ET": s["ET"]}
    if op == "layer_bwd":
        L.pack_states(plan, "f32", H, x["dY"], s["dYb"])
        L.ggnn_step_bwd(plan, dt, H, T, s["prm"], s["saved"], s["dYb"], s["dEb"], s["g"], s["ws"])
        L.unpack_states(plan, "f32", H, s["dEb"], s["dE"])
        return dict(s["g"], dE=s["dE"])
    # train
    L.pack_states(plan, dt, H, x["E"], s["Eb"])
    L.ggnn_step(plan, dt, H, T, s["prm"], s["Eb"], s["ETb"], s["saved"], s["ws"])
    L.readout_loss(plan, dt, H, s["ETb"], x["w"]["w_out"], x["target"], s["loss"], s["dEb"],
                   s["dw_out"], s["rws"])
    L.ggnn_step_bwd(plan, dt, H, T, s["prm"], s["saved"], s["dEb"], s["dEb0"], s["g"], s["ws"])
    L.adam_step(s["master"], s["work"], s["m"], s["v"], s["grad"], LR, B1, B2, EPS, STEP)
    return {"loss": s["loss"], "master": s["master"], "work": s["work"], "m": s["m"], "v": s["v"]}


# ---------------------------------------------------------------------------------- accounting


def work(case):
    """Bytes and operations one pass cannot do without: node arrays, weights and results once, two
    bytes per edge and propagation (its endpoint within the band), one multiply-add per edge and
    state column, the per-node products with the edge-type and GRU weights."""
    c = case
    n, H, T, F = c["nodes"], c["H"], c["T"], c["F"]
    P = 2 * F if c["reverse"] else F
    edges = n * (2 + c["lam"] * (F - 2)) * (2 if c["reverse"] else 1)
    e = 2 if c["dtype"] == "bf16" else 4
    wb, gb = P * H * H * e + P * H * 4, 6 * H * H * e + 24 * H
    prop = 2 * H * edges + 2 * n * P * H * H
    gru = 12 * n * H * H
    op = c["op"]
    if op == "fwd":
        return {"bytes": n * H * (e + 4) + 2 * edges + wb, "flops": prop}
    if op == "bwd":
        return {"bytes": n * H * (e + 8) + 2 * edges + wb + 4 * P * H * (H + 1),
                "flops": prop + 2 * n * P * H * H}
    if op == "infer":
        return {"bytes": 2 * n * H * e + T * 2 * edges + wb + gb, "flops": T * (prop + gru)}
    bwd = prop + 2 * n * P * H * H + 3 * gru
    if op == "layer_bwd":
        return {"bytes": n * H * (2 * e + 8) + 2 * edges + wb + gb + 4 * P * H * (H + 1) + 24 * H * H,
                "flops": bwd}
    params = P * H * (H + 1) + 6 * H * H + 6 * H
    return {"bytes": 2 * T * (n * H * 2 * e + 2 * edges) + wb + gb + params * (7 * 4 + e),
            "flops": T * (prop + gru + bwd)}


# ---------------------------------------------------------------------------------- 64 bits


def _edges64(graphs):
    """Per edge type (dst, src) over the concatenated graphs, on the GPU; repeats already removed."""
    off = np.cumsum([0] + [g.n_nodes for g in graphs[:-1]])
    src = np.concatenate([g.src.astype(np.int64) + o for g, o in zip(graphs, off)])
    dst = np.concatenate([g.dst.astype(np.int64) + o for g, o in zip(graphs, off)])
    et = np.concatenate([g.etype for g in graphs])
    out = []
    for p in range(graphs[0].n_types):
        k = et == p
        out.append((torch.from_numpy(dst[k]).cuda(), torch.from_numpy(src[k]).cuda()))
    return out


def _prop64(edges, E, W, b):
    Y = torch.zeros_like(E)
    for p, (dst, src) in enumerate(edges):
        M = E @ W[p] + b[p]
        Y = Y + torch.zeros_like(E).index_add_(0, dst, M[src])
    return Y


def _prop64_bwd(edges, E, W, dY):
    dE, dW, db = torch.zeros_like(E), torch.zeros_like(W), []
    for p, (dst, src) in enumerate(edges):
        dM = torch.zeros_like(E).index_add_(0, src, dY[dst])
        dE += dM @ W[p].T
        dW[p] = E.T @ dM
        db.append(dM.sum(0))
    return dE, dW, torch.stack(db)


def _gru64(w, Y, E):
    H = E.shape[1]
    gi, gh = Y @ w["W_ih"].T + w["b_ih"], E @ w["W_hh"].T + w["b_hh"]
    r = torch.sigmoid(gi[:, :H] + gh[:, :H])
    z = torch.sigmoid(gi[:, H:2 * H] + gh[:, H:2 * H])
    hn = gh[:, 2 * H:]
    n = torch.tanh(gi[:, 2 * H:] + r * hn)
    return (1 - z) * n + z * E, (r, z, n, hn)


def _layer64_bwd(edges, w, E, Y, dH, g):
    _, (r, z, n, hn) = _gru64(w, Y, E)
    dan = dH * (1 - z) * (1 - n * n)
    dar = dan * hn * r * (1 - r)
    daz = dH * (E - n) * z * (1 - z)
    dgi, dgh = torch.cat([dar, daz, dan], 1), torch.cat([dar, daz, dan * r], 1)
    g["dW_ih"] += dgi.T @ Y
    g["dW_hh"] += dgh.T @ E
    g["db_ih"] += dgi.sum(0)
    g["db_hh"] += dgh.sum(0)
    dE, dW, db = _prop64_bwd(edges, E, w["W"], dgi @ w["W_ih"])
    g["dW"] += dW
    g["db"] += db
    return dE + dgh @ w["W_hh"] + dH * z


def exact(case, seed):
    c = case
    graphs = _graphs(c, seed)
    x = _inputs(c, seed, graphs)
    edges = _edges64(graphs)
    E = x["E"].double()
    w = {k: v.double() for k, v in x["w"].items()}
    op, T = c["op"], c["T"]
    if op == "fwd":
        return {"Y": _prop64(edges, E, w["W"], w["b"])}
    if op == "bwd":
        dE, dW, db = _prop64_bwd(edges, E, w["W"], x["dY"].double())
        return {"dW": dW, "db": db, "dE": dE}
    Es, Ys = [E], []
    for _ in range(T):
        Ys.append(_prop64(edges, Es[-1], w["W"], w["b"]))
        Es.append(_gru64(w, Ys[-1], Es[-1])[0])
    if op == "infer":
        return {"ET": Es[T]}
    g = {"d" + k: torch.zeros_like(w[k]) for k in KEYS}
    if op == "layer_bwd":
        dE = _layer64_bwd(edges, w, E, Ys[0], x["dY"].double(), g)
        return dict(g, dE=dE)
    # mean-pool readout with a linear output and half the squared error
    cnt = torch.tensor([gr.n_nodes for gr in graphs], device="cuda")
    idx = torch.repeat_interleave(torch.arange(len(graphs), device="cuda"), cnt)
    pool = torch.zeros((len(graphs), c["H"]), dtype=torch.float64, device="cuda")
    pool.index_add_(0, idx, Es[T])
    pool /= cnt[:, None]
    resid = pool @ w["w_out"] - x["target"].double()
    d = (resid / cnt)[idx][:, None] * w["w_out"][None, :]
    for t in range(T - 1, -1, -1):
        d = _layer64_bwd(edges, w, Es[t], Ys[t], d, g)
    grad = torch.cat([g["d" + k].reshape(-1) for k in KEYS])
    m = B1 * x["m"].double() + (1 - B1) * grad
    v = B2 * x["v"].double() + (1 - B2) * grad * grad
    master = torch.cat([x["w32"][k].double().reshape(-1) for k in KEYS])
    master = master - LR * (m / (1 - B1 ** STEP)) / ((v / (1 - B2 ** STEP)).sqrt() + EPS)
    return {"loss": (0.5 * resid * resid).sum().reshape(1), "master": master, "work": master, "m": m,
            "v": v}
