"""What is measured of this framework: whole calls through its public entry points.

Every case is work that a program using the package does: an exact count of one hypergraph
(load, step one, step two, clustering coefficient, free), a batch of hypergraphs, the two
sampling estimates, the listing of one pattern, and a burst of queries to the server.  The
hypergraphs are the shapes of this repository's own workloads (``hgen``): co-authorship
(power-law sizes, degree cap 100), tags (log-normal sizes, degree cap 1,000), the dense
uniform ``tiny_plain``, and the members of the batched and served workloads, at sizes from
a hundred hyperedges to half a million.

``listed()``, ``draw(rng)``, ``prepare(case, seed)``, ``run(state)``, ``work(case)`` and
``exact(case, seed)`` are independent of how the counting is done.
"""
from __future__ import annotations

import math
from dataclasses import replace
from functools import lru_cache

import numpy as np
import torch

import hgen
import paper_2504_02271_gb300 as hg

hg.use_torch_allocator()

EPS = [1.0] * 20   # weights of the clustering coefficient (every pattern alike)
EXACT_EDGES = 3000   # exact() answers counts of hypergraphs up to this many hyperedges


def listed() -> list[dict]:
    return [
        # the smallest resident hypergraph of the serving workload, asked from host arrays:
        # a query whose time is launches, copies and waits
        {"name": "count_small", "kind": "count", "shape": "coauthor", "edges": 1000,
         "vertices": 200, "host": True},
        # the configuration `tiny_plain`: 2,000 hyperedges over a popular core, so that most
        # hyperedges meet and the line graph is dense
        {"name": "count_tiny_plain", "kind": "count", "shape": "tiny_plain", "edges": 2000,
         "vertices": 1000, "host": True},
        # an ordinary co-authorship hypergraph of odd size, read from host arrays
        {"name": "count_medium", "kind": "count", "shape": "coauthor", "edges": 31007,
         "vertices": 6201, "host": True},
        # the co-authorship configuration in full, on the device: the benchmark's default step
        {"name": "count_coauthor", "kind": "count", "shape": "coauthor", "edges": 500000,
         "vertices": 100000, "host": False},
        # a prefix of the tag-shaped configuration: hyperedges of up to 200 vertices, large
        # out-degrees, and the largest hyperedges through the tensor-core tiles
        {"name": "count_tag", "kind": "count", "shape": "tag", "edges": 40009,
         "vertices": 20000, "host": False},
        # hyperedges of 256 vertices and more (mailing lists, tag sets of long threads):
        # rows whose intersection sizes need more than one byte
        {"name": "count_long_edges", "kind": "count", "shape": "long", "edges": 20011,
         "vertices": 30011, "host": False},
        # members of the batched workload, 100 to 200,000 hyperedges each, counted together
        {"name": "batch_64", "kind": "batch", "members": 64},
        # Algorithm 6 on a resident hypergraph (the sampler line's hypergraph)
        {"name": "sample", "kind": "sample", "edges": 500000, "vertices": 100000,
         "draws": 4000000},
        # Algorithm 7 on a resident hypergraph
        {"name": "sample_adv", "kind": "sample_adv", "edges": 500000, "vertices": 100000,
         "draws": 2000000},
        # a hypergraph that is only estimated: load, step one, the sampled sub-hypergraph
        # (sigma < 1) and its sorted rows, draws, free
        {"name": "estimate_sub", "kind": "estimate_sub", "edges": 150001, "vertices": 30000,
         "draws": 300000, "sigma": 0.5},
        # the hyper-triangles of one pattern of a resident hypergraph, listed in id order
        {"name": "list_pattern", "kind": "list", "edges": 50021, "vertices": 10004,
         "pattern": 17},
        # a burst of queries of every kind to a server that holds a dozen hypergraphs
        {"name": "serve_burst", "kind": "serve", "graphs": 12, "most_edges": 50000,
         "queries": 36, "draws": 1000000},
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng) -> dict:
    kind = rng.choice(["count"] * 5 + ["batch", "sample", "sample_adv", "estimate_sub", "list",
                                       "serve"])
    if kind == "count":
        shape = rng.choice(["coauthor", "coauthor", "tiny_plain", "tag", "long"])
        lo, hi = {"coauthor": (150, 500000), "tiny_plain": (150, 2500), "tag": (300, 40000),
                  "long": (3000, 20000)}[shape]
        edges = _log_int(rng, lo, hi)
        vertices = {"coauthor": max(edges // 5, 40), "tiny_plain": 1000, "tag": 20000,
                    "long": 30011}[shape]
        return {"kind": kind, "shape": shape, "edges": edges, "vertices": vertices,
                "host": rng.random() < 0.5}
    if kind == "batch":
        return {"kind": kind, "members": _log_int(rng, 2, 64)}
    edges = _log_int(rng, 1000, 500000)
    if kind in ("sample", "sample_adv"):
        return {"kind": kind, "edges": edges, "vertices": edges // 5,
                "draws": _log_int(rng, 10000, 4000000 if kind == "sample" else 2000000)}
    if kind == "estimate_sub":
        edges = min(edges, 150000)
        return {"kind": kind, "edges": edges, "vertices": edges // 5,
                "draws": _log_int(rng, 10000, 300000), "sigma": round(rng.uniform(0.2, 0.9), 3)}
    if kind == "list":
        edges = _log_int(rng, 1000, 50000)
        return {"kind": kind, "edges": edges, "vertices": edges // 5,
                "pattern": rng.choice([5, 12, 17])}
    return {"kind": "serve", "graphs": rng.randint(2, 12), "most_edges": _log_int(rng, 2000, 50000),
            "queries": rng.randint(6, 36), "draws": _log_int(rng, 10000, 1000000)}


# ------------------------------------------------------------------ inputs

def _spec(shape: str, edges: int, vertices: int, seed: int) -> hgen.HypergraphSpec:
    if shape == "tiny_plain":
        base = hgen.TINY_PLAIN
    elif shape == "tag":
        base = hgen.TAG_HEAVY
    elif shape == "long":   # log-normal sizes of mean 20, up to 600
        base = replace(hgen.TAG_HEAVY, size_p1=2.5, size_hi=600, degree_cap=100)
    else:
        base = hgen.COAUTHOR
    return replace(base, num_edges=edges, num_vertices=vertices, seed=seed, name=shape)


def _draw_csr(spec: hgen.HypergraphSpec):
    """The spec's hypergraph; a seed that runs out of fresh hyperedges is drawn again."""
    for r in range(65):
        try:
            return hgen.generate(replace(spec, seed=spec.seed + (r << 32)))
        except hgen.DedupExhausted:
            continue
    raise RuntimeError(f"no hypergraph for {spec}")


def _members(case: dict, seed: int) -> list[hgen.HypergraphSpec]:
    """Members of a batch: one of each of `members` equal parts of the size range [100,
    200,000] on its logarithm, so that seeds differ in the hypergraphs and not in their bulk."""
    out = []
    for m in range(case["members"]):
        lo, hi = (round(100 * 2000 ** ((m + k) / case["members"])) for k in (0, 1))
        s = seed * 1000 + m
        ne = hgen.loguniform_int(s, 0, lo, max(hi, lo + 1))
        out.append(replace(hgen.batched(s), num_edges=ne, num_vertices=max(ne // 4, 2)))
    order = np.random.default_rng(seed).permutation(len(out))
    return [out[k] for k in order]


def _served(case: dict, seed: int) -> list[hgen.HypergraphSpec]:
    out, top = [], case["most_edges"]
    for m in range(case["graphs"]):
        lo, hi = (round(1000 * (top / 1000) ** ((m + k) / case["graphs"])) for k in (0, 1))
        ne = hgen.loguniform_int(seed * 1000 + m, 0, lo, max(hi, lo + 1))
        out.append(_spec("coauthor", ne, ne // 5, seed * 1000 + m))
    return out


def _csr(case: dict, seed: int):
    return _draw_csr(_spec(case.get("shape", "coauthor"), case["edges"], case["vertices"], seed))


def prepare(case: dict, seed: int) -> dict:
    st = {"case": case, "seed": seed}
    kind = case["kind"]
    if kind == "batch":
        nv, eo, ep, ev, _ = hgen.generate_batch(_members(case, seed), redraw=hgen.batched_redraw)
        st.update(nv=nv, eo=eo, ptr=torch.from_numpy(ep).cuda(), idx=torch.from_numpy(ev).cuda())
    elif kind == "serve":
        srv = hg.Server(workers=4)
        ids = [srv.add_graph(sp.num_vertices, *_draw_csr(sp)) for sp in _served(case, seed)]
        rng = np.random.default_rng(seed)
        kinds = [hg.HG_Q_COUNTS, hg.HG_Q_CLUSTERING, hg.HG_Q_ESTIMATE]
        asks = [(kinds[k % 3], ids[int(rng.integers(len(ids)))]) for k in range(case["queries"])]
        st.update(server=srv, asks=asks)
    else:
        ptr, idx = _csr(case, seed)
        if not case.get("host", False):
            ptr, idx = torch.from_numpy(ptr).cuda(), torch.from_numpy(idx).cuda()
        st.update(ptr=ptr, idx=idx)
        if kind in ("sample", "sample_adv", "list"):   # resident: loaded, step one done
            g = hg.hg_load_csr(case["vertices"], case["edges"], ptr, idx)
            hg.hg_build_wedges(g)
            st["graph"] = g
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------ one pass

def _stats(s: dict) -> np.ndarray:
    return np.array([s[k] for k in ("W", "W_t", "W_c", "connected", "max_deg", "max_out_deg",
                                    "dense_edges")], dtype=np.int64)


def _count(st: dict):
    c = st["case"]
    g = hg.hg_load_csr(c["vertices"], c["edges"], st["ptr"], st["idx"])
    stats = hg.hg_build_wedges(g)
    counts = hg.hg_count_patterns(g)
    masks = hg.hg_mask_histogram(g)
    cc, open_, connected = hg.hg_clustering_coeff(g, EPS)
    hg.hg_free(g)
    return {"counts": counts.view(np.int64), "masks": masks.view(np.int64), "cc": cc,
            "open": open_, "connected": connected, "stats": _stats(stats)}


def _batch(st: dict):
    b = hg.hg_load_batch(st["nv"], st["eo"], st["ptr"], st["idx"])
    hg.hg_batch_build_wedges(b)
    counts, stats = hg.hg_batch_count_patterns(b)
    masks = hg.hg_batch_mask_histogram(b)
    cc, open_, connected = hg.hg_batch_clustering_coeff(b, EPS)
    hg.hg_batch_free(b)
    return {"counts": counts.view(np.int64), "masks": masks.view(np.int64), "cc": cc,
            "open": open_.view(np.int64), "connected": connected.view(np.int64),
            "W": stats["W"].view(np.int64), "W_c": stats["W_c"].view(np.int64),
            "max_deg": stats["max_deg"].view(np.int64)}


def _listing(st: dict):
    """The triples of one pattern as a program lists them: into a buffer with room for
    more than there are (the rest stays -1), then put in id order."""
    c, n = st["case"], st["case"]["edges"]
    out = torch.full((24 * n, 3), -1, dtype=torch.int32, device="cuda")
    _, total = hg.hg_enumerate_pattern(st["graph"], c["pattern"], out=out)
    key = (out[:, 0].long() * n + out[:, 1]) * n + out[:, 2]
    order = torch.argsort(torch.where(out[:, 0] < 0, n ** 3, key))
    return {"total": total, "triples": out[order]}


def _serve(st: dict):
    srv, draws = st["server"], st["case"]["draws"]
    tickets = [srv.submit(kind, gid, seed=2024, first_sample=k * draws, num_samples=draws, eps=EPS)
               for k, (kind, gid) in enumerate(st["asks"])]
    got = [srv.wait(t) for t in tickets]
    return {"counts": np.array([r["counts"].view(np.int64) for r in got]),
            "est": np.array([r["est"] for r in got]), "cc": np.array([r["cc"] for r in got]),
            "open": np.array([r["open"] for r in got]),
            "connected": np.array([r["connected"] for r in got]),
            "status": np.array([r["status"] for r in got])}


def run(st: dict):
    c = st["case"]
    kind = c["kind"]
    if kind == "count":
        return _count(st)
    if kind == "batch":
        return _batch(st)
    if kind == "sample":
        raw, est = hg.hg_sample_estimate(st["graph"], st["seed"], 0, c["draws"])
        return {"raw": raw.view(np.int64), "est": est}
    if kind == "sample_adv":
        raw, est, info = hg.hg_sample_estimate_adv(st["graph"], st["seed"], 0, c["draws"])
        return {"raw": raw.view(np.int64), "est": est, "alpha": [info[f"alpha_{k}"] for k in (1, 2, 3, 4)]}
    if kind == "estimate_sub":
        g = hg.hg_load_csr(c["vertices"], c["edges"], st["ptr"], st["idx"])
        hg.hg_build_wedges(g)
        raw, est = hg.hg_sample_estimate(g, st["seed"], 0, c["draws"], sigma=c["sigma"])
        hg.hg_free(g)
        return {"raw": raw.view(np.int64), "est": est}
    if kind == "list":
        return _listing(st)
    return _serve(st)


# ------------------------------------------------------------------ what a pass cannot do without

@lru_cache(maxsize=None)
def _bulk(kind: str, shape: str, edges: int, vertices: int, members: int, most: int
          ) -> tuple[int, int, int]:
    """(hyperedges, incidences, pairs of hyperedges that meet in a vertex, summed over the
    vertices) of the case's hypergraphs, drawn from one seed."""
    if kind == "batch":
        specs = _members({"members": members}, 1)
    elif kind == "serve":
        specs = _served({"graphs": members, "most_edges": most}, 1)
    else:
        specs = [_spec(shape, edges, vertices, 1)]
    ne = nnz = pairs = 0
    for sp in specs:
        ptr, idx = _draw_csr(sp)
        d = np.bincount(idx).astype(np.int64)
        ne, nnz, pairs = ne + len(ptr) - 1, nnz + len(idx), pairs + int((d * (d - 1) // 2).sum())
    return ne, nnz, pairs


def work(case: dict) -> dict:
    """Bytes: the CSR read once (8 per offset, 4 per vertex id) and the answers written.
    Operations: one for every pair of hyperedges and vertex that they share (step one's sum)
    where the pass does step one; of a draw, 10 Philox rounds of 8."""
    kind = case["kind"]
    ne, nnz, pairs = _bulk(kind, case.get("shape", "coauthor"), case.get("edges", 0),
                           case.get("vertices", 0), case.get("members", case.get("graphs", 0)),
                           case.get("most_edges", 0))
    csr = 8 * (ne + 1) + 4 * nnz
    if kind in ("sample", "sample_adv"):   # a drawn hyperwedge, and the sizes it leads to
        return {"bytes": 16 * case["draws"] + 2 * 21 * 8, "flops": 80 * case["draws"]}
    if kind == "list":                     # every hyperwedge once
        return {"bytes": csr + 4 * pairs, "flops": pairs}
    if kind == "estimate_sub":
        return {"bytes": csr + 2 * 21 * 8, "flops": pairs * case["sigma"] ** 2 + 80 * case["draws"]}
    if kind == "serve":
        ests = case["queries"] // 3
        return {"bytes": csr + case["queries"] * (2 * 21 * 8 + 24),
                "flops": pairs + 80 * case["draws"] * ests}
    return {"bytes": csr + (21 + 128 + 10) * 8 * max(1, case.get("members", 1)), "flops": pairs}


# ------------------------------------------------------------------ the answers in 64 bits

def _pattern(m: int) -> int:
    """Pattern 1..20 of a region mask (bits a b c d e f g; d = first and second only, e =
    second and third, f = first and third): 1 three inclusions, 2-5 two, 6-8 one, 9-16 none
    with a common region, 17-20 none without.  0: no hyper-triangle of distinct hyperedges."""
    sets = [m & r for r in (0b1101001, 0b1011010, 0b1110100)]
    pairs = [(0, 1, 2), (1, 2, 0), (0, 2, 1)]
    if any(not sets[x] & sets[y] or sets[x] == sets[y] for x, y, _ in pairs):
        return 0
    inside = [p for p in pairs if sets[p[0]] & sets[p[1]] in (sets[p[0]], sets[p[1]])]
    across = [p for p in pairs if p not in inside]
    if len(inside) == 3:
        return 1
    if len(inside) == 2:
        x, y, z = (sets[k] for k in across[0])
        if z & x & y == z:
            return 2 if z == x & y else 3
        return 4 if z == x | y else 5
    if len(inside) == 1:
        x, y, z = (sets[k] for k in inside[0])
        big, small = x | y, x & y
        return 6 if big & z == small & z else (7 if big == small | (big & z) else 8)
    two, single = bin(m >> 3 & 7).count("1"), bin(m & 7).count("1")
    if m >> 6:
        return {0: 9, 1: 10, 2: 9 + single, 3: 13 + single}[two]
    return 17 + single


def _canonical(m: int) -> int:
    """The smallest mask among the six orders of the three hyperedges."""
    code = [1, 2, 4, 3, 6, 5, 7]   # hyperedges holding each region
    best = 127
    for o in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        got = 0
        for r in range(7):
            if m >> r & 1:
                got |= 1 << code.index(sum((code[r] >> o[q] & 1) << q for q in range(3)))
        best = min(best, got)
    return best


def exact(case: dict, seed: int):
    """Counts of hypergraphs of at most EXACT_EDGES hyperedges, from dense matrices in 64
    bits.  A sampled estimate, a listing and the server's answers to estimates have no value
    apart from the draws; larger hypergraphs take too long this way."""
    if case["kind"] != "count" or case["edges"] > EXACT_EDGES:
        return None
    ptr, idx = _csr(case, seed)
    ne = case["edges"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    rows = np.repeat(np.arange(ne), np.diff(ptr))
    used, cols = np.unique(idx, return_inverse=True)
    h = torch.zeros((ne, len(used)), dtype=torch.float64, device=dev)
    h[torch.from_numpy(rows).to(dev), torch.from_numpy(cols).to(dev)] = 1
    w = h @ h.T
    size = w.diagonal().clone()
    w.fill_diagonal_(0)
    adj = w > 0
    labelled = torch.zeros(128, dtype=torch.int64, device=dev)
    for i in range(ne):
        nb = torch.nonzero(adj[i, i + 1:]).flatten() + i + 1
        if len(nb) < 2:
            continue
        hi = h[nb][:, h[i] > 0]
        g = hi @ hi.T
        x, y = torch.nonzero(torch.triu(adj[nb][:, nb], 1), as_tuple=True)
        j, k, g = nb[x], nb[y], g[x, y]
        ij, ik, jk = w[i, j], w[i, k], w[j, k]
        regions = (size[i] - ij - ik + g, size[j] - ij - jk + g, size[k] - ik - jk + g,
                   ij - g, jk - g, ik - g, g)
        m = sum((r > 0).long() << b for b, r in enumerate(regions))
        labelled += torch.bincount(m, minlength=128)
    counts, masks = np.zeros(21, dtype=np.int64), np.zeros(128, dtype=np.int64)
    for m, n in enumerate(labelled.tolist()):
        if n:
            counts[0] += n
            counts[_pattern(m)] += n
            masks[_canonical(m)] += n
    deg = adj.sum(1)
    connected = int((deg * (deg - 1) // 2).sum())
    open_ = connected - 3 * int(counts[0])
    return {"counts": counts, "masks": masks,
            "cc": 3.0 * float(counts[0]) / open_ if open_ else math.nan, "open": open_,
            "connected": connected, "stats": None}
