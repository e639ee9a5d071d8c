"""The work a user of this framework has it do, as cases that can be timed and compared.

A case is one call of an agent's program through the package's public entry points: a rewrite step (pack the current
graph and its candidates, encode, policy and value heads, draw), the same from host arrays, a step with delta
encoding, or the gradient of a training step.  Graphs are synthetic computation graphs (transformer- and CNN-shaped,
power-law, random DAGs); a candidate is the current graph with one run of nodes rewritten.

`exact` restates the method in 64-bit torch (paper Eq. 3-8) from the same inputs; for a bf16 model the shape features
and the matrices of Eq. 6 and Eq. 7 are rounded to bf16 first, as the model stores them, and nothing else is.
"""
import math

import numpy as np
import torch

import paper_2304_14698_b200 as xrl

S = 8                      # shape features per node
WINDOW = 256               # a power-law graph's consumers sit among the next WINDOW nodes
GAMMA, LAMBDA = 0.99, 0.95
EPS, C1, C2 = 0.2, 0.5, 0.01


def _case(name, kind, family, dtype, H, K, L, T, Hm, Hm2, nodes, candidates, envs, slots, **more):
    c = dict(kind=kind, family=family, dtype=dtype, H=H, K=K, L=L, T=T, Hm=Hm, Hm2=Hm2, nodes=nodes,
             candidates=candidates, envs=envs, slots=slots, ragged=False, edge_attr=False, both_ways=False)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest step an agent makes: eight graphs of 64 operators, fp32; latency and launches count
        _case("tiny_step", "step", "random", "fp32", 64, 1, 2, 32, 64, 0, 64, 7, 1, 8),
        # one rewrite step on a transformer-shaped graph, an fp32 model
        _case("transformer_step", "step", "transformer", "fp32", 128, 4, 3, 32, 128, 0, 570, 63, 1, 64),
        # one rewrite step on a CNN-shaped graph, a bf16 model of hidden 128
        _case("cnn_step", "step", "cnn", "bf16", 128, 4, 3, 32, 128, 0, 1170, 255, 1, 256),
        # a step of the paper's size with its hyper-parameters (5 layers, MLP heads [256, 64], 26 candidates) as the
        # environment hands it over: host arrays, which the call rounds, copies and packs
        _case("paper_step_host", "host", "transformer", "bf16", 256, 8, 5, 40, 256, 64, 570, 26, 1, 32),
        # the same step with the graphs already on the GPU
        _case("paper_step", "step", "transformer", "bf16", 256, 8, 5, 40, 256, 64, 570, 26, 1, 32),
        # the largest single step: 1,024 power-law graphs of 4,000 operators
        _case("large_step", "step", "powerlaw", "bf16", 256, 8, 4, 64, 256, 0, 4000, 1023, 1, 1024),
        # a rollout batch: 64 environments with different numbers of candidates
        _case("rollout_batch", "step", "mixed", "bf16", 256, 8, 4, 64, 256, 0, 980, 60, 64, 128, ragged=True),
        # the same kind of batch with delta encoding: only what a rewrite can reach is computed again
        _case("rollout_delta", "delta", "mixed", "bf16", 256, 8, 4, 64, 256, 0, 980, 127, 16, 128),
        # other options: a width without a power of two, attributes on the edges, neighbourhoods read both ways
        _case("options_step", "step", "cnn", "bf16", 192, 6, 3, 40, 96, 0, 700, 95, 2, 128, ragged=True,
              edge_attr=True, both_ways=True),
        # the training step's gradient on a mini-batch of 16 of the paper's transitions
        _case("paper_train", "train", "transformer", "bf16", 256, 8, 5, 40, 256, 64, 570, 26, 16, 32, ragged=True),
        # the same for a small fp32 model
        _case("transformer_train", "train", "transformer", "fp32", 128, 4, 3, 32, 128, 0, 570, 15, 4, 16),
        # a large mini-batch
        _case("rollout_train", "train", "mixed", "bf16", 256, 8, 4, 64, 256, 0, 980, 63, 16, 64),
    ]


def draw(rng):
    """Any of these calls, on any model the library is built for, from a few hundred nodes to a million."""
    log = lambda lo, hi: math.exp(rng.uniform(math.log(lo), math.log(hi)))
    kind = rng.choice(["step", "step", "step", "host", "delta", "train", "train"])
    H = rng.choice([64, 96, 128, 128, 192, 256, 256, 256, 512])
    K = rng.choice([k for k in (1, 2, 3, 4, 6, 8, 16) if H % k == 0 and (H // k) % 8 == 0 and H // k >= 16])
    total = log(600, 1_000_000 if kind in ("step", "delta") else 250_000) * min(1.0, 256 / H)
    envs = rng.choice([1, 1, 1, 2, 16, 64] if kind != "train" else [4, 8, 16, 32])
    envs = max(envs if total > 400 * envs else 1, 4 if kind == "train" else 1)
    nodes = int(log(40, min(4000, max(60, total / (6 * envs)))))
    candidates = int(min(1023, max(2, total / (nodes * envs) - 1)))
    plain = kind == "delta" or rng.random() < 0.7
    return _case(None, kind, rng.choice(["random", "transformer", "cnn", "powerlaw", "mixed"]),
                 rng.choice(["fp32", "bf16", "bf16"]), H, K, rng.randint(1, 5), rng.choice([20, 32, 40, 64]),
                 rng.choice([48, 64, 128, 256]), rng.choice([0, 0, 64]), nodes, candidates, envs,
                 candidates + rng.choice([0, 1, 5, 32]), ragged=rng.random() < 0.5,
                 edge_attr=not plain and rng.random() < 0.7, both_ways=not plain and rng.random() < 0.7)


# ---- inputs ----------------------------------------------------------------------------------------------------
def _template(nrng, family, nodes, T):
    """(operators, producers, consumers) of one graph of about `nodes` nodes; every edge goes to a higher id."""
    if family == "transformer":                       # blocks: attention heads written out, then the feed-forward part
        heads = 6 if nodes >= 800 else 3
        ops, es = [7], []                             # node 0 of a block: the reshape of its input

        def node(op, *producers):
            ops.append(op)
            es.extend((p, len(ops) - 1) for p in producers)
            return len(ops) - 1
        ctx = []
        for _ in range(heads):
            q, k, v = (node(2, 0, node(1)) for _ in range(3))
            ctx.append(node(2, node(4, node(8, node(2, q, node(6, k)))), v))
        x = node(5, node(3, 0, node(2, node(7, node(13, *ctx)), node(1))))
        node(5, node(3, x, node(2, node(9, node(2, x, node(1))), node(1))))
        n, blocks = len(ops), max(1, round(nodes / len(ops)))
        es = np.asarray(es, np.int64)
        es = np.concatenate([es + n * b for b in range(blocks)] + [np.array([[n * b - 1, n * b]]) for b in range(1, blocks)])
        return np.tile(np.asarray(ops), blocks) % T, es[:, 0], es[:, 1]
    if family == "cnn":                               # residual blocks of one to four branches
        ops, es, x = [0], [], 0

        def node(op, *producers):
            ops.append(op)
            es.extend((p, len(ops) - 1) for p in producers)
            return len(ops) - 1
        while len(ops) < nodes - 20 or len(ops) < 12:
            outs = []
            depth = int(nrng.integers(1, 4))
            for _ in range(int(nrng.integers(1, 5))):
                y = x
                for _ in range(depth):
                    y = node(12, node(11, node(10, y, node(1))))
                outs.append(y)
            y = node(13, *outs) if len(outs) > 1 else outs[0]
            x = node(12, node(3, x, node(11, node(10, y, node(1)))))
        es = np.asarray(es, np.int64)
        return np.asarray(ops) % T, es[:, 0], es[:, 1]
    n = max(12, nodes)
    if family == "powerlaw":                          # out-degree k with P(k) ~ k^-2.2, at most 64
        k = np.arange(1, 65)
        p = k ** -2.2
        deg = nrng.choice(k, size=n, p=p / p.sum())
        src = np.repeat(np.arange(n), deg)
        dst = src + nrng.integers(1, min(WINDOW, n // 2) + 1, size=len(src))
    else:                                             # in-degree Binomial(4, 1/2) from the sixteen nodes before
        dst = np.repeat(np.arange(n), nrng.binomial(4, 0.5, size=n))
        src = dst - nrng.integers(1, 17, size=len(dst))
    ok = (src >= 0) & (dst < n)
    code = np.unique(src[ok] * n + dst[ok])
    return nrng.integers(0, T, size=n), code // n, code % n


def _shape(g, *size):
    """log2(dim) / 12 with dim log-uniform in [1, 4096]."""
    return torch.exp2(12 * torch.rand(*size, generator=g, device="cuda")).floor().clamp_(1, 4096).log2_() / 12


def _environment(g, nrng, family, nodes, T, C):
    """The current graph and C candidates, flat on the GPU: a candidate replaces a run of 2-6 nodes by 1-6 fresh ones."""
    op, src, dst = (torch.from_numpy(np.ascontiguousarray(a, np.int32)).cuda() for a in _template(nrng, family, nodes, T))
    n, m = len(op), len(src)
    shape = _shape(g, n, S)
    ints = lambda lo, hi, *size: torch.randint(lo, hi, size, generator=g, device="cuda", dtype=torch.int32)
    length, r = ints(2, 7, C, 1), ints(1, 7, C, 1)
    s = 1 + (torch.rand(C, 1, generator=g, device="cuda") * (n - 1 - length)).int()
    e, shift = s + length, r - length
    j = torch.arange(n + 4, device="cuda", dtype=torch.int32)[None, :]
    live, new = j < n + shift, (j >= s) & (j < s + r)
    old = torch.where(j < s, j, j - shift).clamp_(0, n - 1)
    ops = torch.where(new, ints(0, T, C, n + 4), op[old.long()])[live]
    twin = torch.where(new, -1, old)[live]
    shapes = torch.where(new[live][:, None], _shape(g, len(ops), S), shape[old[live].long()])
    # edges of the graph that stay, then up to three producers among the sixteen nodes before each fresh node
    keep = ((dst < s) | (dst >= e))
    es = torch.where((src >= s) & (src < e), s + (torch.rand(C, m, generator=g, device="cuda") * r).int(),
                     src + torch.where(src >= e, shift, 0))
    ed = dst + torch.where(dst >= e, shift, 0)
    k = torch.arange(6, device="cuda", dtype=torch.int32)[None, :, None]
    off = 1 + torch.rand(C, 6, 16, generator=g, device="cuda").argsort(-1)[..., :3].int()
    fs, fd = s[..., None] + k - off, (s[..., None] + k).expand(C, 6, 3)
    fresh = (k < r[..., None]) & (torch.arange(3, device="cuda") < ints(1, 4, C, 6, 1)) & (fs >= 0)
    mask = torch.cat([keep.expand(C, m), fresh.reshape(C, 18)], 1)
    es, ed = torch.cat([es, fs.reshape(C, 18)], 1)[mask], torch.cat([ed, fd.reshape(C, 18)], 1)[mask]
    first = torch.tensor([n], device="cuda"), torch.tensor([m], device="cuda")
    return dict(op=torch.cat([op, ops]), shape=torch.cat([shape, shapes]), src=torch.cat([src, es]),
                dst=torch.cat([dst, ed]), twin=torch.cat([torch.full((n,), -1, device="cuda", dtype=torch.int32), twin]),
                n=torch.cat([first[0], live.sum(1)]), m=torch.cat([first[1], mask.sum(1)]))


def _model(c):
    return dict(T=c["T"], S=S, H=c["H"], K=c["K"], L=c["L"], Hm=c["Hm"], Hm2=c["Hm2"], Dg=1, dtype=c["dtype"],
                A_max=c["slots"], edge_attr=c["edge_attr"], both_ways=c["both_ways"])


def _layout(c):
    H, last = c["H"], c["Hm2"] or c["Hm"]
    out = [("We", (2 * S + c["T"], H)), ("be", (H,))]
    for l in range(c["L"]):
        out += [("W%d" % l, (H, H)), ("as%d" % l, (H,)), ("ad%d" % l, (H,)), ("b%d" % l, (H,))]
    out += [("Wg", (H + 1, H)), ("bg", (H,))]
    for h, width in (("p", H), ("v", 2 * H)):
        out += [(h + "W1", (width, c["Hm"])), (h + "b1", (c["Hm"],))]
        if c["Hm2"]:
            out += [(h + "Wh", (c["Hm"], c["Hm2"])), (h + "bh", (c["Hm2"],))]
        out += [(h + "w2", (last,)), (h + "b2", (1,))]
    return out


def _weights(c, nrng, mean_nodes):
    """Xavier-uniform matrices and attention vectors, biases U(-0.1, 0.1); the readout rows are scaled by the graphs'
    size, as training would, so that sums over thousands of nodes leave the softmax a distribution."""
    parts = []
    for name, shape in _layout(c):
        fan = sum(shape) if len(shape) == 2 else c["H"] // c["K"] + 1 if name[0] == "a" else shape[0] + 1
        w = nrng.uniform(-1, 1, shape) * (math.sqrt(6 / fan) if len(shape) == 2 or name[0] == "a" or name[1:] == "w2" else 0.1)
        if name == "Wg":
            w[:c["H"]] /= mean_nodes
        parts.append(w.astype(np.float32).ravel())
    return np.concatenate(parts)


def _inputs(c, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    nrng = np.random.default_rng(seed)
    envs = []
    for e in range(c["envs"]):
        C = max(1, c["candidates"] - (e * 37 + 11) % (c["candidates"] // 2 + 1)) if c["ragged"] else c["candidates"]
        family = ("transformer", "cnn")[e % 2] if c["family"] == "mixed" else c["family"]
        envs.append(_environment(g, nrng, family, c["nodes"], c["T"], C))
    cat = lambda k: torch.cat([v[k] for v in envs])
    i32 = lambda a: np.ascontiguousarray(a, np.int32)
    b = dict(op=cat("op"), shape=cat("shape"), edge_src=cat("src").contiguous(), edge_dst=cat("dst").contiguous(),
             n_nodes=i32(cat("n").cpu().numpy()), n_edges=i32(cat("m").cpu().numpy()),
             env_off=i32(np.concatenate([[0], np.cumsum([len(v["n"]) for v in envs])])))
    start = np.concatenate([[0], np.cumsum([len(v["op"]) for v in envs])])
    if c["kind"] == "delta":
        b["base_id"] = torch.cat([torch.where(v["twin"] >= 0, v["twin"] + int(o), -1) for v, o in zip(envs, start)]).int()
    if c["edge_attr"]:                                # a tensor's dimensions divided by 4096, ranks below four padded
        dims = torch.exp2(12 * torch.rand(len(b["edge_src"]), 4, generator=g, device="cuda")).floor() / 4096
        rank = torch.randint(1, 5, (len(dims), 1), generator=g, device="cuda")
        dims *= torch.arange(4, device="cuda") >= 4 - rank
        b["edge_attr"] = torch.cat([dims, torch.zeros_like(dims)], 1)
    mask = np.zeros((c["envs"], c["slots"]), np.uint8)
    for e, v in enumerate(envs):                      # about one candidate in a hundred is invalid
        mask[e, :len(v["n"]) - 1] = nrng.random(len(v["n"]) - 1) >= 0.01
    x = dict(batch=b, mask=mask, weights=_weights(c, nrng, float(b["n_nodes"].mean())))
    if c["kind"] == "train":                          # envs = steps x trajectories of a rollout
        ne, steps = c["envs"], 4 if c["envs"] % 4 == 0 else 1
        f32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
        action = np.array([nrng.choice(np.append(np.flatnonzero(mask[e]), c["slots"])) for e in range(ne)], np.int32)
        x.update(action=torch.from_numpy(action).cuda(),
                 logp_old=f32(-np.log(1.0 + mask.sum(1)) + nrng.uniform(-0.3, 0.3, ne)),
                 reward=f32(0.3 * nrng.normal(size=(steps, ne // steps))),
                 values=f32(0.5 * nrng.normal(size=(steps + 1, ne // steps))),
                 done=torch.from_numpy((nrng.random((steps, ne // steps)) < 0.1).astype(np.uint8)).cuda())
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    b = x["batch"]
    agent = xrl.Agent(_model(case), len(b["n_nodes"]), case["envs"], len(b["op"]), max(1, len(b["edge_src"])))
    agent.set_weights(x["weights"])
    if case["kind"] == "host":
        for k in ("op", "shape", "edge_src", "edge_dst", "edge_attr"):
            if k in b:
                b[k] = b[k].cpu().numpy()
    elif case["dtype"] == "bf16":
        for k in ("shape", "edge_attr"):
            if k in b:
                b[k] = b[k].to(torch.bfloat16)
    x.update(case=case, agent=agent, mask=torch.from_numpy(x["mask"]).cuda(), step=0)
    if case["kind"] == "train":
        x.update(loss=torch.empty(4, device="cuda"), grad=torch.empty(len(x["weights"]), device="cuda"),
                 logp=torch.empty(case["envs"], device="cuda"))
    return x


def run(state):
    agent, b = state["agent"], state["batch"]
    if state["case"]["kind"] != "train":
        return agent.step(b, state["mask"], sample=True, seed=1234, step=7, base_id=b.get("base_id"))
    adv, ret = xrl.xrl_gae(state["reward"], state["values"], state["done"], GAMMA, LAMBDA)
    agent.pack(b)
    xrl.xrl_ppo_grad(agent.ctx, agent.batch, state["mask"], state["action"], state["logp_old"], adv.view(-1),
                     ret.view(-1), state["loss"], state["grad"], eps=EPS, c1=C1, c2=C2, logp_out=state["logp"])
    return dict(loss=state["loss"], grad=state["grad"], logp=state["logp"], adv=adv, ret=ret)


# ---- what a pass cannot do without -------------------------------------------------------------------------------
def work(case):
    c = case
    per_graph = {"transformer": 1.23, "cnn": 1.1, "powerlaw": 2.1, "random": 1.9, "mixed": 1.16}[c["family"]]
    graphs = c["envs"] * (1 + c["candidates"] * (0.75 if c["ragged"] else 1.0))
    N, H = graphs * c["nodes"], c["H"]
    E = N * per_graph
    size = 2 if c["dtype"] == "bf16" and c["kind"] != "host" else 4
    weights = sum(math.prod(shape) for _, shape in _layout(c))
    nbytes = N * (4 + S * size) + E * (8 + (S * size if c["edge_attr"] else 0)) + 4 * weights + 4 * graphs * H
    rows = N if c["kind"] != "delta" else c["envs"] * c["nodes"]         # (delta: the current graphs at least)
    edges = rows * per_graph * (2 if c["both_ways"] else 1)
    flops = rows * (2 * 2 * S * H + c["L"] * 2 * H * H) + c["L"] * (edges + rows) * 2 * H + graphs * 2 * H * (H + c["Hm"])
    if c["kind"] == "delta":
        nbytes += 4 * N
    if c["kind"] == "train":
        flops, nbytes = 3 * flops, nbytes + 4 * weights
    return {"bytes": int(nbytes), "flops": int(flops)}


def tolerance(case):
    """About four times the largest distance from `exact` that was measured over the ranges: fp32 sums of thousands of
    terms, 5e-6 (a value near zero); bf16, whose Z and layer outputs keep 8-bit mantissas, 3e-4 of the embeddings, up
    to 6e-3 of a value near zero and 2e-2 of a gradient (a hidden unit within rounding of zero moves its column).  An
    action may differ where the draw falls between two probabilities."""
    rel = {"fp32": 2e-5, "bf16": 1e-2} if case["kind"] != "train" else {"fp32": 2e-5, "bf16": 2e-2}
    return {"rel": rel[case["dtype"]], "differ": 0.01}


# ---- the same in 64 bits ---------------------------------------------------------------------------------------
def _features(c, w, op, x_edge, shape, es, ed):
    """Eq. 6 and the layers of Eq. 7 for the nodes of some whole graphs, float64."""
    n, K, H = len(op), c["K"], c["H"]
    agg = torch.zeros(n, S, dtype=torch.float64, device=op.device).index_add_(0, ed, x_edge)
    h = torch.relu(agg @ w["We"][:S] + w["We"][S + op] + shape @ w["We"][S + c["T"]:] + w["be"])
    me = torch.arange(n, device=op.device)
    j, i = (torch.cat([es, ed, me]), torch.cat([ed, es, me])) if c["both_ways"] else (torch.cat([es, me]), torch.cat([ed, me]))
    for l in range(c["L"]):
        z = (h @ w["W%d" % l]).view(n, K, H // K)
        s = (z * w["as%d" % l].view(K, -1)).sum(-1)[j] + (z * w["ad%d" % l].view(K, -1)).sum(-1)[i]
        s = torch.where(s > 0, s, 0.2 * s)
        top = torch.full((n, K), -math.inf, dtype=torch.float64, device=op.device)
        top = top.scatter_reduce(0, i[:, None].expand(-1, K), s.detach(), "amax")
        p = torch.exp(s - top[i])
        p = p / torch.zeros(n, K, dtype=torch.float64, device=op.device).index_add(0, i, p)[i]
        out = torch.zeros(n, K, H // K, dtype=torch.float64, device=op.device).index_add(0, i, p[..., None] * z[j])
        h = torch.relu(out.reshape(n, H) + w["b%d" % l])
    return h


def _mlp(c, w, head, x):
    x = torch.relu(x @ w[head + "W1"] + w[head + "b1"])
    if c["Hm2"]:
        x = torch.relu(x @ w[head + "Wh"] + w[head + "bh"])
    return x @ w[head + "w2"] + w[head + "b2"][0]


def exact(case, seed):
    c, x = case, _inputs(case, seed)
    b, f64 = x["batch"], torch.float64
    stored = (lambda a: a.to(torch.bfloat16).to(f64)) if c["dtype"] == "bf16" else (lambda a: a.to(f64))
    w, at = {}, 0
    blob = torch.from_numpy(x["weights"]).cuda()
    for name, shape in _layout(c):
        part = blob[at:at + math.prod(shape)].view(shape)
        at += math.prod(shape)
        w[name] = (stored(part) if name[0] == "W" and name != "Wg" else part.to(f64)).requires_grad_(c["kind"] == "train")
    nn, ne, env_off = b["n_nodes"].astype(np.int64), b["n_edges"].astype(np.int64), b["env_off"]
    no, eo = np.concatenate([[0], np.cumsum(nn)]), np.concatenate([[0], np.cumsum(ne)])
    shape = stored(b["shape"])
    edge_attr = stored(b["edge_attr"]) if c["edge_attr"] else None
    G = len(nn)
    cuts, room = [0], max(1, 30_000_000 // c["H"])    # groups of whole graphs that fit
    for g in range(G):
        if no[g + 1] - no[cuts[-1]] > room and g > cuts[-1]:
            cuts.append(g)
    cuts.append(G)

    def sums(g0, g1):
        """Sums of the last layer's features over graphs g0 .. g1 - 1."""
        r, q = slice(no[g0], no[g1]), slice(eo[g0], eo[g1])
        lift = torch.from_numpy(np.repeat(no[g0:g1] - no[g0], ne[g0:g1])).cuda()
        es, ed = b["edge_src"][q].long() + lift, b["edge_dst"][q].long() + lift
        x_edge = edge_attr[q] if c["edge_attr"] else shape[r][es]
        h = _features(c, w, b["op"][r].long(), x_edge, shape[r], es, ed)
        seg = torch.from_numpy(np.repeat(np.arange(g1 - g0), nn[g0:g1])).cuda()
        return torch.zeros(g1 - g0, c["H"], dtype=f64, device="cuda").index_add(0, seg, h)

    with torch.no_grad():
        total = torch.cat([sums(a, z) for a, z in zip(cuts, cuts[1:])])
    total.requires_grad_(c["kind"] == "train")
    emb = torch.relu(total @ w["Wg"][:c["H"]] + w["bg"])             # (the global attribute is zero)
    logit = _mlp(c, w, "p", emb)
    logs, values = [], []
    for e in range(c["envs"]):
        a, z = int(env_off[e]), int(env_off[e + 1])
        valid = torch.from_numpy(x["mask"][e, :z - a - 1]).cuda().bool()
        row = torch.full((c["slots"] + 1,), -math.inf, dtype=f64, device="cuda")
        row = torch.cat([torch.where(valid, logit[a + 1:z], -math.inf), row[z - a - 1:-1], logit[a:a + 1]])
        logs.append(torch.log_softmax(row, 0))
        mean = (emb[a + 1:z] * valid[:, None]).sum(0) / max(1, int(valid.sum()))
        values.append(_mlp(c, w, "v", torch.cat([emb[a], mean])))
    logs, values = torch.stack(logs), torch.stack(values)
    if c["kind"] != "train":
        return dict(emb=emb, probs=logs.exp(), value=values, action=None)
    # advantages and targets, backwards over the trajectory; then Eq. 3-5
    reward, v, done = (x[k].to(f64) for k in ("reward", "values", "done"))
    adv, run_ = torch.zeros_like(reward), torch.zeros_like(reward[0])
    for t in reversed(range(len(reward))):
        run_ = reward[t] + GAMMA * v[t + 1] * (1 - done[t]) - v[t] + GAMMA * LAMBDA * (1 - done[t]) * run_
        adv[t] = run_
    ret = adv + v[:-1]
    A = adv.view(-1)
    logp = logs.gather(1, x["action"].long()[:, None])[:, 0]
    ratio = torch.exp(logp - x["logp_old"].to(f64))
    clip = -torch.minimum(ratio * A, ratio.clamp(1 - EPS, 1 + EPS) * A).mean()
    vf = ((values - ret.view(-1)) ** 2).mean()
    ent = torch.where(logs > -math.inf, logs.exp() * torch.where(logs > -math.inf, logs, 0.0), 0.0).sum(1).mean()
    J = clip + C1 * vf + C2 * ent
    J.backward()
    for a, z in zip(cuts, cuts[1:]):
        sums(a, z).backward(total.grad[a:z])
    grad = torch.cat([w[name].grad.reshape(-1) if w[name].grad is not None else torch.zeros(math.prod(s), dtype=f64, device="cuda")
                      for name, s in _layout(c)])
    return dict(loss=torch.stack([J, clip, vf, ent]).detach(), grad=grad, logp=logp.detach(), adv=adv, ret=ret)
