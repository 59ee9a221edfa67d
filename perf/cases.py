"""The work that users of this library have it do, as cases to be timed.

Five forms of use, each through the public entry points of the Python binding:

``stream``   one forest fed minibatch by minibatch: a reset, then a Bulk-Update and a Bulk-Query
             (or a Bulk-Find, ``ask="find"``) each, and the component labels at the end.
``batch``    many small graphs with minibatches of their own, in one ``submit``.
``resume``   a forest loaded from a checkpoint's labels, one more minibatch, and the new labels.
``served``   a request loop over one mature graph: a burst of mixed requests, until all are done.

``options`` are launch options by name and value, as a program passes them to ``Forest``; an empty
text means the defaults, on the current stream, as a program that tunes nothing uses the library.
The other sets are what the autotuner stores for streams of that kind, and run on a stream of
their own, as programs that overlap kernels do.
"""
import numpy as np
import torch

from paper_1602_05232_gb300 import cc

# What the autotuner stores for streams of small uniform graphs, R-MAT graphs, meshes, a served
# R-MAT graph and many small graphs.
UNIFORM = "update_variant=1 edges_per_thread=2 block=256 hook=2 compress_every=0 query_halving=1 pdl=2"
RMAT = ("update_variant=5 edges_per_thread=2 block=128 hook=2 compress_every=0 query_halving=1 "
        "query_pairs_per_thread=2 pdl=2")
MESH = ("update_variant=5 edges_per_thread=2 block=128 hook=1 compress_every=6 big_filter=640 "
        "edge_order=7 pdl=2")
SERVED = ("update_variant=2 edges_per_thread=1 block=512 hook=1 compress_every=0 "
          "query_pairs_per_thread=2 pdl=2")
MANY = "seg_block=1024 seg_edges_per_thread=2"


def listed():
    return [
        # The smallest use: a graph of a few thousand vertices, minibatches of 4096. Launches count.
        dict(name="tiny", form="stream", kind="uniform", n=4096, m=16384, batch=4096, ask="query",
             asked=4096, uneven=False, shifted=False, options=""),
        # The plain method on a small graph: 2^20 uniform edges on 2^16 vertices, 16 minibatches.
        dict(name="uniform", form="stream", kind="uniform", n=1 << 16, m=1 << 20, batch=1 << 16,
             ask="query", asked=1 << 16, uneven=False, shifted=False, options=""),
        # The same by a program that uses the tuned options.
        dict(name="uniform_tuned", form="stream", kind="uniform", n=1 << 16, m=1 << 20,
             batch=1 << 16, ask="query", asked=1 << 16, uneven=False, shifted=False, options=UNIFORM),
        # Minibatches as they come: of any size, out of a buffer that is only 4-byte aligned.
        dict(name="ragged", form="stream", kind="uniform", n=1_000_003, m=3_000_001, batch=1 << 18,
             ask="query", asked=50_001, uneven=True, shifted=True, options=""),
        # A social or web graph with the defaults: R-MAT, each minibatch followed by as many queries.
        dict(name="rmat", form="stream", kind="rmat", n=1 << 22, m=1 << 25, batch=1 << 20,
             ask="query", asked=1 << 20, uneven=False, shifted=False, options=""),
        # The plain method at scale, tuned: R-MAT on 2^24 vertices, 2^27 edges in minibatches of 2^20.
        dict(name="rmat_tuned", form="stream", kind="rmat", n=1 << 24, m=1 << 27, batch=1 << 20,
             ask="query", asked=1 << 20, uneven=False, shifted=False, options=RMAT),
        # A mesh (long paths, half of the edges join two trees) with the defaults.
        dict(name="mesh", form="stream", kind="grid", n=3001 * 3001, m=2 * 3001 * 3000,
             batch=1 << 20, ask="query", asked=1 << 20, uneven=False, shifted=False, options=""),
        # The high-diameter stream: an 8192 x 8192 mesh, larger than L2, tuned. The largest case.
        dict(name="mesh_tuned", form="stream", kind="grid", n=8192 * 8192, m=2 * 8192 * 8191,
             batch=1 << 22, ask="query", asked=1 << 22, uneven=False, shifted=False, options=MESH),
        # A program that asks for component ids of some vertices after each minibatch.
        dict(name="find", form="stream", kind="rmat", n=1 << 20, m=1 << 22, batch=1 << 18,
             ask="find", asked=1 << 16, uneven=False, shifted=False, options=""),
        # 1024 independent graphs of 2^8 to 2^16 vertices, uneven minibatches, one submit.
        dict(name="many_graphs", form="batch", graphs=1024, low=8, high=16, degree=4, shape=1,
             options=MANY),
        # A restart: labels from a checkpoint, then the next minibatch.
        dict(name="resume", form="resume", kind="rmat", n=1 << 25, m=1 << 26, batch=1 << 21,
             asked=1 << 20, options=""),
        # A service: 256 requests at once, three updates to a query, sizes log-uniform.
        dict(name="served", form="served", kind="rmat", n=1 << 24, requests=256, largest=20,
             shape=1, options=SERVED),
    ]


def draw(rng):
    def size(low, high):  # spread over the logarithm, odd sizes among them
        return int(2.0 ** rng.uniform(low, high)) | rng.randint(0, 1)

    form = rng.choice(["stream"] * 8 + ["find", "batch", "resume", "served"])
    if form == "batch":
        low = rng.randint(6, 10)
        return dict(form=form, graphs=size(4, 10), low=low, high=low + rng.randint(2, 6),
                    degree=rng.randint(1, 6), shape=rng.randint(2, 1 << 20),
                    options=rng.choice(["", MANY]))
    if form == "served":
        return dict(form=form, kind="rmat", n=1 << rng.randint(16, 24), requests=size(5, 8.5),
                    largest=rng.randint(12, 20), shape=rng.randint(2, 1 << 20),
                    options=rng.choice(["", SERVED]))
    kind = rng.choice(["uniform", "rmat", "grid"])
    n = size(10, 20) if form == "find" else size(14, 25) if form == "resume" else size(10, 24)
    if kind == "rmat":
        n = 1 << (n.bit_length() - 1)
    if kind == "grid":
        rows = max(8, int(n ** 0.5))
        cols = n // rows
        n, m = rows * cols, rows * (cols - 1) + (rows - 1) * cols
    else:
        m = min(int(n * 2.0 ** rng.uniform(0, 3)), 1 << 26)
    batch = min(max(m // rng.randint(2, 96), min(m, 256)), 1 << 22)
    if form == "resume":
        return dict(form=form, kind=kind, n=n, m=m, batch=batch, asked=size(8, 20), options="")
    uneven = rng.random() < 0.5
    ask = "find" if form == "find" else "query"
    tuned = dict(uniform=UNIFORM, rmat=RMAT, grid=MESH)[kind]
    return dict(form="stream", kind=kind, n=n, m=m, batch=batch, ask=ask,
                asked=min(size(8, 17 if ask == "find" else 22), 4 * batch,
                          (1 << 26) // len(_cuts(m, batch, uneven))),
                uneven=uneven, shifted=rng.random() < 0.25,
                options="" if ask == "find" or rng.random() < 0.5 else tuned)


# ------------------------------------------------------------------------------------- inputs

def _made(seed, *more):
    """A generator for one purpose of one seed."""
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1_000_003 + sum((i + 1) * 7_919 * int(x) for i, x in enumerate(more)))
                  % (1 << 62))
    return g


def _buffer(k, shifted):
    """Room for k pairs; shifted: 4 bytes past a 16-byte boundary."""
    return torch.empty(2 * k + 4, dtype=torch.int32, device="cuda")[1 if shifted else 0:][:2 * k].view(k, 2)


def _uniform(n, k, g, shifted=False):
    return _buffer(k, shifted).copy_(torch.randint(0, n, (k, 2), dtype=torch.int32, device="cuda", generator=g))


def _rmat(n, k, g, shifted=False):
    """R-MAT edges (0.57, 0.19, 0.19, 0.05) on n = 2^scale vertices, ids permuted."""
    names = torch.randperm(n, device="cuda", generator=g).to(torch.int32)
    out = _buffer(k, shifted)
    for lo in range(0, k, 1 << 24):
        part = min(k - lo, 1 << 24)
        u = torch.zeros(part, dtype=torch.int32, device="cuda")
        v = torch.zeros_like(u)
        for _ in range(n.bit_length() - 1):
            r = torch.rand(part, device="cuda", generator=g)
            down = r >= 0.76
            u.mul_(2).add_(down)
            v.mul_(2).add_(((r >= 0.57) & ~down) | (r >= 0.95))
        out[lo:lo + part, 0] = names[u.long()]
        out[lo:lo + part, 1] = names[v.long()]
    return out


def _grid(n, m, g, shifted=False):
    """The first m edges, shuffled, of the 4-neighbour mesh with n vertices numbered row by row."""
    cols = max(8, int(n ** 0.5))
    while n % cols:
        cols -= 1
    ids = torch.arange(n, dtype=torch.int32, device="cuda").view(n // cols, cols)
    edges = torch.cat([torch.stack([ids[:, :-1].reshape(-1), ids[:, 1:].reshape(-1)], 1),
                       torch.stack([ids[:-1].reshape(-1), ids[1:].reshape(-1)], 1)])
    order = torch.randperm(edges.shape[0], device="cuda", generator=g)[:m]
    return _buffer(order.numel(), shifted).copy_(edges[order])


def _edges(case, m, seed, shifted=False):
    g = _made(seed, 1)
    return {"uniform": _uniform, "rmat": _rmat, "grid": _grid}[case["kind"]](case["n"], m, g, shifted)


def _cuts(total, batch, uneven):
    """Where the minibatches start and end: all of `batch`, or log-uniform from 1 to `batch`."""
    at, rng = [0], np.random.RandomState(total % 9973)
    while at[-1] < total:
        k = int(batch ** rng.uniform(0.4, 1)) if uneven else batch
        at.append(min(total, at[-1] + max(k, 1)))
    return at


def _forest(options, make, *args):
    kw = {k: int(v) for k, v in (w.split("=") for w in options.split())}
    return make(*args, stream=torch.cuda.Stream() if kw else None, **kw)


def _steps(case, seed):
    """The minibatches of a stream, and what is asked after each."""
    edges = _edges(case, case["m"], seed, case["shifted"])
    at = _cuts(edges.shape[0], case["batch"], case["uneven"])
    if len(at) > 200:  # a stream of very small minibatches: its first ones
        at = at[:200]
    g = _made(seed, 2)
    if case["ask"] == "find":
        asked = torch.randint(0, case["n"], (len(at) - 1, case["asked"]), dtype=torch.int32, device="cuda", generator=g)
    else:
        asked = _uniform(case["n"], (len(at) - 1) * case["asked"], g, case["shifted"]).view(len(at) - 1, -1, 2)
    return [(edges[a:b], asked[i]) for i, (a, b) in enumerate(zip(at, at[1:]))]


def _many(case, seed):
    """Sizes, edges, pairs and (graph, first, last) minibatches of many graphs."""
    rng = np.random.RandomState(case["shape"])
    n = np.floor(2.0 ** rng.uniform(case["low"], case["high"], case["graphs"])).astype(np.int64)
    m = case["degree"] * n
    first = np.concatenate([[0], np.cumsum(m)])
    own = torch.from_numpy(np.repeat(n, m)).cuda()[:, None]
    g = _made(seed, 3)
    both = [(torch.rand(own.shape[0], 2, dtype=torch.float64, device="cuda", generator=g) * own).to(torch.int32)
            for _ in range(2)]
    cuts = []
    for i in range(case["graphs"]):
        a = 0
        while a < m[i]:
            b = min(int(m[i]), a + int(2.0 ** rng.uniform(6, 14)))
            cuts.append((i, int(first[i]) + a, int(first[i]) + b))
            a = b
    return n, both[0], both[1], cuts


def _trace(case):
    """(kind, first, last) of a burst of requests; first and last count edges or pairs."""
    rng, at, out = np.random.RandomState(case["shape"]), [0, 0], []
    for i in range(case["requests"]):
        kind = cc.OP_QUERY if rng.random_sample() < 0.25 or i == 0 else cc.OP_UPDATE
        high = case["largest"] - (2 if kind == cc.OP_QUERY else 0)
        k = int(2.0 ** rng.uniform(8, high))
        out.append((kind, at[kind], at[kind] + k))
        at[kind] += k
    return out, at


class _Served:
    """A server over its forest, closed when the program drops it."""

    def __init__(self, forest):
        self.forest, self.server = forest, cc.Server(forest, ring_pairs=1 << 23)

    def __del__(self):
        self.server.close()
        self.forest.close()


def prepare(case, seed):
    form, s = case["form"], {"form": case["form"]}
    if form == "stream":
        s["steps"] = _steps(case, seed)
        s["forest"] = _forest(case["options"], cc.Forest, case["n"])
        count, find = len(s["steps"]), case["ask"] == "find"
        s["find"] = find
        s["out"] = torch.empty(count, case["asked"], dtype=torch.int32 if find else torch.uint8, device="cuda")
        s["outs"] = list(s["out"])
        s["labels"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
    elif form == "batch":
        n, edges, pairs, cuts = _many(case, seed)
        s["forest"] = _forest(case["options"], cc.Forest.segmented, n)
        s["out"] = torch.empty(edges.shape[0], dtype=torch.uint8, device="cuda")
        s["labels"] = torch.empty(int(n.sum()), dtype=torch.int32, device="cuda")
        ops = np.zeros(2 * len(cuts), dtype=cc.OP_DTYPE)
        for i, (graph, a, b) in enumerate(cuts):
            ops[2 * i] = (graph, cc.OP_UPDATE, edges.data_ptr() + 8 * a, b - a, 0)
            ops[2 * i + 1] = (graph, cc.OP_QUERY, pairs.data_ptr() + 8 * a, b - a, s["out"].data_ptr() + a)
        s.update(ops=ops, edges=edges, pairs=pairs)
    elif form == "resume":
        edges = _edges(case, case["m"], seed)
        s["old"], s["edges"] = edges[:-case["batch"]].contiguous(), edges[-case["batch"]:].clone()
        s["pairs"] = _uniform(case["n"], case["asked"], _made(seed, 2))
        s["forest"] = _forest(case["options"], cc.Forest, case["n"])
        s["out"] = torch.empty(case["asked"], dtype=torch.uint8, device="cuda")
        s["labels"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        if s["old"].numel():
            s["forest"].bulk_update(s["old"])
        s["saved"] = s["forest"].labels()
        del s["old"]
    else:
        trace, (edges, pairs) = _trace(case)
        s["edges"] = _edges(case, edges, seed).cpu().pin_memory()
        s["pairs"] = _uniform(case["n"], pairs, _made(seed, 2)).cpu().pin_memory()
        s["out"] = torch.empty(pairs, dtype=torch.uint8, pin_memory=True)
        forest = _forest(case["options"], cc.Forest, case["n"])
        forest.bulk_update(s["edges"].cuda())  # a graph that has been served for long
        forest.sync()
        base = [s["edges"].data_ptr(), s["pairs"].data_ptr()]
        s["kinds"] = np.array([k for k, _, _ in trace], dtype=np.int32)
        s["data"] = np.array([base[k] + 8 * a for k, a, _ in trace], dtype=np.uint64)
        s["sizes"] = np.array([b - a for _, a, b in trace], dtype=np.int64)
        s["to"] = np.array([s["out"].data_ptr() + a if k == cc.OP_QUERY else 0 for k, a, _ in trace], dtype=np.uint64)
        s["served"] = _Served(forest)
    torch.cuda.synchronize()
    return s


def run(s):
    if s["form"] == "served":
        server = s["served"].server
        server.enqueue_many(s["kinds"], s["data"], s["sizes"], s["to"])
        server.drain()
        return s["out"]
    f = s["forest"]
    if s["form"] == "stream":
        f.reset()
        ask = f.bulk_find if s["find"] else f.bulk_query
        for (edges, asked), out in zip(s["steps"], s["outs"]):
            f.bulk_update(edges)
            ask(asked, out)
    elif s["form"] == "batch":
        f.reset()
        f.submit(s["ops"])
    else:
        f.load_labels(s["saved"])
        f.bulk_update(s["edges"])
        f.bulk_query(s["pairs"], s["out"])
    return [s["out"], f.labels(s["labels"])]


def work(case):
    """Each edge, pair, vertex id or saved label read once; each answer and label written once."""
    if case["form"] == "stream":
        m = case["m"]
        steps = min(199, len(_cuts(m, case["batch"], case["uneven"])) - 1)
        m = _cuts(m, case["batch"], case["uneven"])[steps]
        b = 8 * m + (8 if case["ask"] == "find" else 9) * steps * case["asked"] + 4 * case["n"]
    elif case["form"] == "batch":
        rng = np.random.RandomState(case["shape"])
        n = np.floor(2.0 ** rng.uniform(case["low"], case["high"], case["graphs"])).sum()
        b = (8 + 9) * case["degree"] * n + 4 * n
    elif case["form"] == "resume":
        b = 8 * case["batch"] + 9 * case["asked"] + 8 * case["n"]
    else:
        edges, pairs = _trace(case)[1]
        b = 8 * edges + 9 * pairs
    return {"bytes": float(b), "flops": 0.0}


# -------------------------------------------------------------------- the same, in plain torch

def _fold(label, edges):
    """Minimum-id labels (int64) after `edges` joined the components of `label`."""
    a, b = label[edges[:, 0].long()], label[edges[:, 1].long()]
    up = torch.arange(label.numel(), device="cuda")
    while True:
        a, b = up[a], up[b]
        apart = a != b
        if not bool(apart.any()):
            break
        a, b = a[apart], b[apart]
        up.scatter_reduce_(0, torch.maximum(a, b), torch.minimum(a, b), "amin")
        while True:
            further = up[up]
            if torch.equal(further, up):
                break
            up = further
    return up[label]


def exact(case, seed):
    if case["form"] == "stream":
        label, out = torch.arange(case["n"], device="cuda"), []
        for edges, asked in _steps(case, seed):
            label = _fold(label, edges)
            if case["ask"] == "find":
                out.append(label[asked.long()].to(torch.int32))
            else:
                out.append((label[asked[:, 0].long()] == label[asked[:, 1].long()]).to(torch.uint8))
        return [torch.stack(out), label.to(torch.int32)]
    if case["form"] == "batch":
        n, edges, pairs, cuts = _many(case, seed)
        base, seen, level = np.concatenate([[0], np.cumsum(n)]), {}, []
        for graph, a, b in cuts:  # the j-th minibatches of all graphs together
            j = seen[graph] = seen.get(graph, -1) + 1
            level.extend([[]] if j == len(level) else [])
            level[j].append((int(base[graph]), a, b))
        label = torch.arange(int(n.sum()), device="cuda")
        out = torch.empty(edges.shape[0], dtype=torch.uint8, device="cuda")
        for parts in level:
            label = _fold(label, torch.cat([edges[a:b].long() + o for o, a, b in parts]))
            ask = torch.cat([pairs[a:b].long() + o for o, a, b in parts])
            got = (label[ask[:, 0]] == label[ask[:, 1]]).to(torch.uint8)
            for (_, a, b), x in zip(parts, torch.split(got, [b - a for _, a, b in parts])):
                out[a:b] = x
        return [out, label.to(torch.int32)]
    if case["form"] == "resume":
        label = _fold(torch.arange(case["n"], device="cuda"), _edges(case, case["m"], seed))
        pairs = _uniform(case["n"], case["asked"], _made(seed, 2))
    else:
        edges, pairs = _trace(case)[1]
        label = _fold(torch.arange(case["n"], device="cuda"), _edges(case, edges, seed))
        pairs = _uniform(case["n"], pairs, _made(seed, 2))
    got = (label[pairs[:, 0].long()] == label[pairs[:, 1].long()]).to(torch.uint8)
    return [got, label.to(torch.int32)] if case["form"] == "resume" else got
