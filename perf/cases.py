"""Timed cases of the compression library: the calls its users make, through the
package's public functions, over the range of sizes they are made on.

A case names a generated graph (R-MAT with the quadrant probabilities of the
benchmark, a Chung-Lu power-law graph, or a 3-D random geometric graph), a call
and its parameters.  Graphs are made on the GPU from the seed alone.
"""
import math

import torch

import paper_1912_08950_gb300 as sg

DEV = "cuda"
_CTX = None


def _ctx():
    """The one context of the program."""
    global _CTX
    if _CTX is None:
        _CTX = sg.Context(0)
    return _CTX


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the latency of one compression of a small graph, as a server gets them
        dict(name="union-1k", call="compress", graph="rmat", n=1000, ef=16, kernel="tr_random", p=0.5),
        # Triangle 0.5-1-Reduction at the benchmark's smaller size
        dict(name="union-4m", call="compress", graph="rmat", n=1 << 22, ef=16, kernel="tr_random", p=0.5),
        # the headline: the same on a graph of a billion edges
        dict(name="union-64m", call="compress", graph="rmat", n=1 << 26, ef=16, kernel="tr_random", p=0.5),
        # edge-once reduction (keeps the components) of a graph of modest size
        dict(name="edge-once-16k", call="compress", graph="rmat", n=1 << 14, ef=16, kernel="tr_eo", p=0.2),
        # edge-once reduction at the benchmark's smaller size
        dict(name="edge-once-4m", call="compress", graph="rmat", n=1 << 22, ef=16, kernel="tr_eo", p=0.5),
        # max-weight (MST-preserving) reduction of a weighted power-law graph
        dict(name="max-weight-2m", call="compress", graph="chung_lu", n=1 << 21, ef=16, kernel="tr_maxw", p=1.0,
             weighted=True),
        # uniform edge sampling of a large graph
        dict(name="uniform-16m", call="compress", graph="rmat", n=1 << 24, ef=16, kernel="uniform", p=0.5),
        # spectral sparsification with its 1/p weights, an odd vertex count
        dict(name="spectral-3m", call="compress", graph="rmat", n=3000017, ef=16, kernel="spectral_avgdeg", p=0.5,
             want_weights=True),
        # a batch of small graphs of uneven sizes, each with its own kernel, p and seed
        dict(name="batch-28", call="batch", count=28, lo=256, hi=65536),
        # judging one result: KL divergence of the PageRanks and the components of both graphs
        dict(name="divergence-1m", call="divergence", graph="rmat", n=1 << 20, ef=16, kernel="tr_eo", p=0.5),
        # the PageRank vector of the benchmark's smaller graph
        dict(name="pagerank-4m", call="pagerank", graph="rmat", n=1 << 22, ef=16),
        # triangles per vertex of a triangle-dense graph without hubs
        dict(name="triangles-rgg-1m", call="vertex_triangles", graph="rgg", n=1 << 20, ef=24),
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["compress"] * 6 + ["batch", "divergence", "pagerank", "vertex_triangles"])
    if call == "batch":
        return dict(call="batch", count=rng.randint(8, 28), lo=_between(rng, 100, 1000), hi=_between(rng, 20000, 65536))
    ef = rng.randint(8, 24)
    if call == "divergence":
        kernel = rng.choice(["uniform", "tr_random", "tr_eo"])
        return dict(call=call, graph=rng.choice(["rmat", "chung_lu"]), n=_between(rng, 1000, 1 << 21), ef=ef,
                    kernel=kernel, p=rng.choice([0.2, 0.5, 0.8]))
    if call in ("pagerank", "vertex_triangles"):
        return dict(call=call, graph=rng.choice(["rmat", "chung_lu", "rgg"]), n=_between(rng, 1000, 1 << 21), ef=ef)
    kernel = rng.choice(["uniform", "spectral_logn", "spectral_avgdeg", "tr_random", "tr_random", "tr_p2", "tr_mincount",
                         "tr_maxw", "tr_eo", "tr_eo", "tr_eo_maxw", "tr_eo_mincount"])
    triangles = kernel.startswith("tr_")
    case = dict(call=call, graph=rng.choice(["rmat", "rmat", "chung_lu", "rgg"]), kernel=kernel, ef=ef,
                n=_between(rng, 1000, (1 << 22) if triangles else (1 << 24)), p=round(rng.uniform(0.1, 1.0), 2))
    case["weighted"] = kernel.endswith("maxw") or rng.random() < 0.25
    if kernel.startswith("spectral"):
        case["want_weights"] = rng.random() < 0.5
    if case["graph"] == "rgg":
        case["n"] = min(case["n"], 1 << 22)
    return case


# --------------------------------------------------------------------- graphs
def _generator(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + stream) % (1 << 62))
    return g


def _csr(n, src, dst):
    """Symmetric CSR (int64 offsets, int32 columns) of the edges, without loops or duplicates."""
    ok = src != dst
    src, dst = src[ok], dst[ok]
    keys = torch.unique(torch.cat([src * n + dst, dst * n + src]))
    del src, dst, ok
    rows = torch.div(keys, n, rounding_mode="floor")
    col = (keys - rows * n).to(torch.int32)
    del keys
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return off, col


def _rmat(n, ef, seed, a=0.57, b=0.19, c=0.19):
    """R-MAT on the next power of two, ids permuted, restricted to the first n ids."""
    scale = max(1, (n - 1).bit_length())
    full = 1 << scale
    total = int(ef * n * (full / n) ** 2)
    gen = _generator(seed, 1)
    perm = torch.randperm(full, generator=gen, device=DEV)
    srcs, dsts = [], []
    for start in range(0, total, 1 << 27):
        k = min(total - start, 1 << 27)
        s = torch.zeros(k, dtype=torch.int64, device=DEV)
        d = torch.zeros(k, dtype=torch.int64, device=DEV)
        for _ in range(scale):
            u = torch.rand(k, generator=gen, device=DEV)
            low = u >= a + b
            right = torch.where(low, u >= a + b + c, u >= a)
            s = s * 2 + low
            d = d * 2 + right
        s, d = perm[s], perm[d]
        if full != n:
            ok = (s < n) & (d < n)
            s, d = s[ok], d[ok]
        srcs.append(s)
        dsts.append(d)
    src, dst = torch.cat(srcs)[:ef * n], torch.cat(dsts)[:ef * n]
    del srcs, dsts
    return _csr(n, src, dst)


def _chung_lu(n, ef, seed, gamma=2.1):
    """ef * n endpoint pairs drawn by weights (i + 10)^(-1 / (gamma - 1)), capped at the root of their sum."""
    gen = _generator(seed, 2)
    w = (torch.arange(n, dtype=torch.float64, device=DEV) + 10.0) ** (-1.0 / (gamma - 1.0))
    w *= 2.0 * ef * n / w.sum()
    w = torch.minimum(w, w.sum().sqrt())
    cum = torch.cumsum(w, 0)
    perm = torch.randperm(n, generator=gen, device=DEV)
    ends = []
    for _ in range(2):
        r = torch.rand(ef * n, generator=gen, device=DEV, dtype=torch.float64) * cum[-1]
        ends.append(perm[torch.searchsorted(cum, r, right=True).clamp_(max=n - 1)])
    return _csr(n, ends[0], ends[1])


def _rgg(n, ef, seed):
    """Points on the unit torus joined below the radius that gives mean degree 2 ef."""
    gen = _generator(seed, 3)
    radius = (2.0 * ef * 3.0 / (4.0 * math.pi * n)) ** (1.0 / 3.0)
    if radius >= 1.0 / 3.0:
        radius = 1.0 / 3.0 - 1e-6
    side = int(1.0 / radius)
    pts = torch.rand(n, 3, generator=gen, device=DEV, dtype=torch.float64)
    cell3 = (pts * side).long().clamp_(max=side - 1)
    cell = (cell3[:, 0] * side + cell3[:, 1]) * side + cell3[:, 2]
    order = torch.argsort(cell)
    starts = torch.searchsorted(cell[order], torch.arange(side**3 + 1, device=DEV))
    ids = torch.arange(n, device=DEV)
    srcs, dsts = [], []
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dz in (-1, 0, 1):
                shift = torch.tensor([dx, dy, dz], device=DEV)
                c3 = (cell3 + shift) % side
                c = (c3[:, 0] * side + c3[:, 1]) * side + c3[:, 2]
                lo, cnt = starts[c], starts[c + 1] - starts[c]
                p = torch.repeat_interleave(ids, cnt)
                q = order[torch.arange(p.numel(), device=DEV) + torch.repeat_interleave(lo - torch.cumsum(cnt, 0) + cnt, cnt)]
                diff = (pts[p] - pts[q]).abs()
                diff = torch.minimum(diff, 1.0 - diff)
                ok = ((diff * diff).sum(1) < radius * radius) & (p < q)
                srcs.append(p[ok])
                dsts.append(q[ok])
    return _csr(n, torch.cat(srcs), torch.cat(dsts))


def _weights(n, off, col, seed):
    """Edge weights k 2^-24 with k in {1 .. 2^24}, the same on both arcs of an edge."""
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), off[1:] - off[:-1])
    c = col.long()
    key = torch.minimum(rows, c) * n + torch.maximum(rows, c)
    h = (key ^ (key >> 29)) * 0x3F58476D1CE4E5B9 + int(seed) * 0x1E3779B97F4A7C15 % (1 << 62)
    h = (h ^ (h >> 27)) * 0x14D049BB133111EB
    return (((h >> 33) & 0xFFFFFF) + 1).to(torch.float32) * 2.0**-24


def _graph(case, seed):
    off, col = {"rmat": _rmat, "chung_lu": _chung_lu, "rgg": _rgg}[case["graph"]](case["n"], case["ef"], seed)
    w = _weights(case["n"], off, col, seed) if case.get("weighted") else None
    return off, col, w


def _resident(n, off, col, w=None):
    """The graph in the library's own device arrays; the tensors may go once the copies are done."""
    g = sg.Graph.from_tensors(_ctx(), n, off, col, w, copy=True)
    _ctx().synchronize()
    return g


def _most_arcs(case):
    return 2 * case["ef"] * case["n"] * 5 // 4


def _key(seed):
    return (int(seed) * 0x9E3779B97F4A7C15 + 12345) % (1 << 64)


def _batch_members(case):
    """Sizes, edge factors, kernels and p of a batch, in a fixed spread over its range."""
    k = case["count"]
    sizes = [int(case["lo"] * (case["hi"] / case["lo"]) ** (i / max(k - 1, 1))) for i in range(k)]
    efs = [8 + (7 * i) % 25 for i in range(k)]
    kernels = [("uniform", "spectral_avgdeg", "tr_random")[i % 3] for i in range(k)]
    ps = [(0.2, 0.5, 0.8)[(i // 3) % 3] for i in range(k)]
    return sizes, efs, kernels, ps


# -------------------------------------------------------------- the interface
def prepare(case, seed):
    call = case["call"]
    if call == "batch":
        sizes, efs, kernels, ps = _batch_members(case)
        graphs = []
        for i, n in enumerate(sizes):
            off, col = _rmat(n, efs[i], seed * 64 + i)
            graphs.append(_resident(n, off, col))
        batch = sg.Batch(_ctx(), graphs)
        return dict(call=call, batch=batch, kernels=kernels, ps=ps, seeds=[_key(seed * 64 + i) for i in range(len(sizes))],
                    own=[_own(n, 2 * ef * n, False) for n, ef in zip(sizes, efs)])
    state = dict(call=call, G=_resident(case["n"], *_graph(case, seed)), key=_key(seed), kernel=case.get("kernel"), p=case.get("p"),
                 want_weights=bool(case.get("want_weights")))
    if call == "compress":
        state["own"] = _own(case["n"], _most_arcs(case), case.get("weighted") or state["want_weights"])
    if call == "divergence":
        state["H"] = sg.compress(state["G"], state["kernel"], state["p"], state["key"])
    return state


def _own(n, arcs, weighted):
    """Tensors of the program's own for a result of n vertices and at most `arcs` arcs."""
    return (torch.zeros(n + 1, dtype=torch.int64, device=DEV), torch.full((arcs,), -1, dtype=torch.int32, device=DEV),
            torch.zeros(arcs, dtype=torch.float32, device=DEV) if weighted else None)


def _keep(h, own):
    """The result copied into them, in the order of the library's stream (the graph may go after it)."""
    with torch.cuda.stream(h.ctx.torch_stream):
        for mine, t in zip(own, h.tensors()):
            if mine is not None and t is not None:
                mine[:t.numel()].copy_(t, non_blocking=True)
    return [t for t in own if t is not None]


def run(state):
    call, G = state["call"], state.get("G")
    if call == "compress":
        return _keep(sg.compress(G, state["kernel"], state["p"], state["key"], state["want_weights"]), state["own"])
    if call == "batch":
        outs = state["batch"].compress(state["kernels"], state["ps"], state["seeds"])
        return [_keep(h, own) for h, own in zip(outs, state["own"])]
    if call == "divergence":
        return sg.divergence(G, state["H"])
    if call == "pagerank":
        x, residual = sg.pagerank(G)
        return {"x": x, "residual": residual}
    return sg.vertex_triangle_counts(G)


def work(case):
    if case["call"] == "batch":
        sizes, efs, _, _ = _batch_members(case)
        # every graph read once, about half of its arcs written
        return {"bytes": sum(16 * (n + 1) + 12 * n * ef for n, ef in zip(sizes, efs)), "flops": 0}
    n, arcs = case["n"], 2 * case["ef"] * case["n"]
    read = 8 * (n + 1) + 4 * arcs
    if case["call"] == "pagerank":
        return {"bytes": 50 * read + 4 * n, "flops": 50 * 2 * arcs}
    if case["call"] == "divergence":
        return {"bytes": 50 * read + 25 * read, "flops": 50 * 2 * arcs * 1.5}
    if case["call"] == "vertex_triangles":
        return {"bytes": read + 8 * n, "flops": 0}
    kept = case["p"] if case["kernel"] == "uniform" else 0.6
    weights = 4 * arcs if case.get("weighted") else 0
    out_weights = 4 * kept * arcs if case.get("weighted") or case.get("want_weights") else 0
    return {"bytes": read + weights + 8 * (n + 1) + 4 * kept * arcs + out_weights, "flops": 0}


# -------------------------------------------------------------------- 64 bits
def _pagerank64(n, off, col, damping=0.85, iters=50):
    deg = (off[1:] - off[:-1]).double()
    A = torch.sparse_csr_tensor(off, col.long(), torch.ones(col.numel(), dtype=torch.float64, device=DEV), (n, n))
    x = torch.full((n,), 1.0 / n, dtype=torch.float64, device=DEV)
    for _ in range(iters):
        y = torch.where(deg > 0, x / deg.clamp(min=1), torch.zeros_like(x))
        dangling = x[deg == 0].sum()
        x = (1.0 - damping) / n + damping * ((A @ y) + dangling / n)
    return x


def _philox(c0, c1, c2, c3, k0, k1):
    """First word of Philox4x32-10 (Salmon et al., SC'11) on int64 tensors of 32-bit words."""
    mask = 0xFFFFFFFF

    def mul(m, v):  # 32 x 32 -> 64 bits, in halves so that no product is negative
        lo, hi = m * (v & 0xFFFF), m * (v >> 16)
        t = hi + (lo >> 16)
        return (t >> 16) & mask, ((t & 0xFFFF) << 16 | (lo & 0xFFFF)) & mask

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c0


def _spectral64(case, seed):
    """The weights 1 / p_uv of the kept arcs, p_uv = min(1, Y / min(d_u, d_v))."""
    n = case["n"]
    off, col, _ = _graph(case, seed)
    deg = off[1:] - off[:-1]
    m = col.numel() // 2
    y = case["p"] * math.log(n) if case["kernel"] == "spectral_logn" else case["p"] * m / n
    ty = math.floor(y * 4294967296.0)
    key, out = _key(seed), []
    rows = torch.repeat_interleave(torch.arange(n, device=DEV, dtype=torch.int32), deg)
    for s in range(0, col.numel(), 1 << 24):
        a, b = rows[s:s + (1 << 24)].long(), col[s:s + (1 << 24)].long()
        zero = torch.zeros_like(a)
        r = _philox(torch.minimum(a, b), torch.maximum(a, b), zero, zero + 0x45444745, key & 0xFFFFFFFF, key >> 32)
        dmin = torch.minimum(deg[a], deg[b])
        dmin = dmin[r * dmin < ty]
        out.append(torch.where(dmin * 4294967296 <= ty, torch.ones_like(dmin, dtype=torch.float64), dmin.double() / y))
    weights = torch.zeros(_most_arcs(case), dtype=torch.float64, device=DEV)
    kept = torch.cat(out)
    weights[:kept.numel()] = kept
    return weights


def exact(case, seed):
    call = case["call"]
    if call == "compress" and case.get("want_weights") and case["kernel"].startswith("spectral"):
        return [None, None, _spectral64(case, seed)]
    if call == "pagerank":
        off, col, _ = _graph(case, seed)
        # the residual of 50 updates is of the size of rounding: no value
        return {"x": _pagerank64(case["n"], off, col), "residual": None}
    if call == "divergence":
        state = prepare(case, seed)
        h_off, h_col, _ = state["H"].tensors()  # the given second graph
        off, col, _ = _graph(case, seed)
        p, q = _pagerank64(case["n"], off, col), _pagerank64(case["n"], h_off.clone(), h_col.clone())
        p, q = p / p.sum(), q / q.sum()
        return {"kl_bits": float((p * torch.log2(p / q)).sum()), "cc_g": None, "cc_h": None, "m_g": None, "m_h": None,
                "pr_residual_g": None, "pr_residual_h": None}
    return None
