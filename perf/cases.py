"""The measured workloads of the k-clique library, each through its public calls.

Graphs are made on the GPU from a seed: R-MAT graphs (the benchmark's family, a = 0.57,
b = c = 0.19, 16 edges per vertex, any number of vertices) and Chung-Lu graphs with planted
groups (the small, batched and community workloads).  A user holds a loaded graph (and a
ring or a batch handle) and makes calls on it; ``load`` starts from host arrays instead.
"""
import math

import numpy as np
import torch

import paper_2203_13512_gb300 as kcl

RING_BYTES = 1 << 30  # wrapping listing ring
RECORDS = 1 << 18  # room of a ring that holds every record of a small graph


def listed():
    cl = dict(graph="chung_lu", gamma=2.5, cap=0.0, density=1.0)
    rmat = dict(graph="rmat", factor=16)
    return [
        # a smallest query on a resident graph: launches and host round trips
        dict(cl, name="count_2k_k5_color", call="count", n=2000, edges=9000, groups=4, lo=10, hi=14, k=5,
             order="color"),
        # every clique of a small graph, as records
        dict(cl, name="records_10k_k4_degree", call="records", n=10000, edges=50000, groups=20, lo=12, hi=12,
             k=4, order="degree"),
        # a one-shot query: host arrays in, count out, graph released
        dict(cl, name="load_10k_k5_degree", call="load", n=10000, edges=50000, groups=20, lo=12, hi=12, k=5,
             order="degree"),
        # many small graphs with their own k in one batched call
        dict(name="batch_64", call="batch", graphs=64, lo_n=50, hi_n=20000, max_k=6),
        # a degeneracy ordering for a caller that must not allocate
        dict(rmat, name="rounds_262k", call="rounds", n=1 << 18),
        # triangles of every vertex in a mid-size graph of odd size
        dict(rmat, name="triangles_300k_degree", call="per_root", n=300001, k=3, order="degree"),
        # deep counting on a mid-size skewed graph
        dict(rmat, name="count_131k_k6_degree", call="count", n=1 << 17, k=6, order="degree"),
        # dense communities on a social graph (most of the graph falls to Pre-Core)
        dict(graph="chung_lu", name="communities_400k_k6_color", call="count", n=400000, edges=4000000, gamma=2.1,
             cap=300.0, groups=200, lo=60, hi=120, density=0.8, k=6, order="color"),
        # the benchmark's graph: counting in both orderings, listing in both
        dict(rmat, name="count_1m_k5_color", call="count", n=1 << 20, k=5, order="color"),
        dict(rmat, name="count_524k_k5_degree", call="count", n=1 << 19, k=5, order="degree"),
        dict(rmat, name="list_1m_k4_color", call="list", n=1 << 20, k=4, order="color"),
        dict(rmat, name="list_500k_k4_degree", call="list", n=500003, k=4, order="degree"),
    ]


def draw(rng):
    order = rng.choice(["color", "degree"])
    kind = rng.choice(["count", "count", "small", "list", "records", "load", "batch", "rounds", "per_root",
                       "communities"])

    def log_uniform(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "count":
        n = log_uniform(1 << 12, 1 << 20)
        return dict(graph="rmat", call="count", n=n, factor=rng.randint(8, 16),
                    k=rng.randint(3, 6 if n <= 1 << 17 else 5), order=order)
    if kind == "list":
        return dict(graph="rmat", call="list", n=log_uniform(1 << 13, 1 << 20), factor=rng.randint(8, 16),
                    k=rng.randint(3, 4), order=order)
    if kind == "per_root":
        return dict(graph="rmat", call="per_root", n=log_uniform(1 << 12, 1 << 20), factor=rng.randint(8, 16),
                    k=rng.randint(3, 4), order=order)
    if kind == "rounds":
        return dict(graph="rmat", call="rounds", n=log_uniform(1 << 12, 1 << 20), factor=rng.randint(8, 16))
    if kind == "batch":
        return dict(call="batch", graphs=rng.randint(8, 96), lo_n=50, hi_n=log_uniform(1000, 20000), max_k=6)
    if kind == "communities":
        lo = rng.randint(30, 60)
        return dict(graph="chung_lu", call="count", n=log_uniform(20000, 400000), edges=log_uniform(200000, 4000000),
                    gamma=2.1, cap=300.0, groups=rng.randint(10, 200), lo=lo, hi=lo + rng.randint(0, 60),
                    density=0.8, k=rng.randint(4, 6), order=order)
    n = log_uniform(1000, 20000)
    return dict(graph="chung_lu", call={"small": "count"}.get(kind, kind), n=n,
                edges=n * rng.randint(3, 4 if kind == "records" else 8), gamma=rng.choice([2.3, 2.5]), cap=0.0, groups=rng.randint(0, 20), lo=8, hi=rng.randint(8, 16),
                density=1.0, k=rng.randint(3, 4 if kind == "records" else 7), order=order)


# ----------------------------------------------------------------- graphs
def _rmat_pairs(n, count, gen):
    """count R-MAT endpoint pairs on [0, n), as keys u * n + v with u < v (self-loops dropped)."""
    u = torch.zeros(count, dtype=torch.int64, device="cuda")
    v = torch.zeros_like(u)
    for _ in range(max(1, (n - 1).bit_length())):
        r = torch.rand(count, device="cuda", generator=gen)
        u = u * 2 + (r >= 0.76)
        v = v * 2 + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    a, b = torch.minimum(u, v), torch.maximum(u, v)
    return (a * n + b)[(a != b) & (b < n)]


def _csr(n, keys, gen):
    """Symmetric CSR (int64 row offsets, int32 ids) of the edge keys u * n + v, vertices relabelled at random."""
    perm = torch.randperm(n, device="cuda", generator=gen)
    u, v = perm[keys // n], perm[keys % n]
    both = torch.cat([u * n + v, v * n + u]).sort().values
    row = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row[1:] = torch.bincount(both // n, minlength=n).cumsum(0)
    return row, (both % n).to(torch.int32)


def _rmat(n, edges, gen):
    keys = torch.unique(_rmat_pairs(n, edges, gen))
    while keys.numel() < edges:  # sampled until that many distinct edges exist
        keys = torch.unique(torch.cat([keys, _rmat_pairs(n, (edges - keys.numel()) * 5 // 4 + 64, gen)]))
    pick = torch.randperm(keys.numel(), device="cuda", generator=gen)[:edges]
    return _csr(n, keys[pick], gen)


def _chung_lu(case, seed, gen):
    """edges endpoint pairs drawn by weight (i + 1)^(-1 / (gamma - 1)), plus planted groups."""
    n, rng = case["n"], np.random.default_rng(seed)
    w = np.arange(1, n + 1, dtype=np.float64) ** (-1.0 / (case["gamma"] - 1.0))
    w *= 2.0 * case["edges"] / w.sum()
    if case["cap"]:
        w = np.minimum(w, case["cap"])
    cum = np.cumsum(w)
    cum = torch.from_numpy(cum / cum[-1]).cuda()
    r = torch.rand(2, case["edges"], device="cuda", generator=gen, dtype=torch.float64)
    a, b = torch.searchsorted(cum, r).clamp_(max=n - 1)
    for _ in range(case["groups"]):
        m = torch.from_numpy(rng.choice(n, size=int(rng.integers(case["lo"], case["hi"] + 1)), replace=False)).cuda()
        i, j = torch.triu_indices(m.numel(), m.numel(), 1, device="cuda")
        keep = torch.rand(i.numel(), device="cuda", generator=gen) < case["density"]
        a, b = torch.cat([a, m[i[keep]]]), torch.cat([b, m[j[keep]]])
    lo, hi = torch.minimum(a, b), torch.maximum(a, b)
    return _csr(n, torch.unique((lo * n + hi)[lo != hi]), gen)


def _graph(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["graph"] == "rmat":
        n = case["n"]
        return _rmat(n, min(case["factor"] * n, n * (n - 1) // 8), gen)
    return _chung_lu(case, seed, gen)


def _batch_members(case, seed):
    """The batched workload: log-uniform sizes, mean degree 4 to 40, 0-5 planted cliques, each its own k."""
    rng = np.random.default_rng(seed)
    out = []
    for i in range(case["graphs"]):
        n = int(math.exp(rng.uniform(math.log(case["lo_n"]), math.log(case["hi_n"]))))
        out.append((dict(graph="chung_lu", n=n, edges=int(n * rng.uniform(2.0, 20.0)), gamma=2.3, cap=0.0,
                         groups=int(rng.integers(0, 6)), lo=8, hi=16, density=1.0),
                    int(rng.integers(3, case["max_k"] + 1)), "color" if i % 2 else "degree", seed * 1009 + i))
    return out


# ------------------------------------------------------------------ calls
def prepare(case, seed):
    s = {"case": case}
    if case["call"] == "batch":
        members = _batch_members(case, seed)
        s["graphs"] = [kcl.kcl_load_csr(*_graph(c, sd)) for c, _, _, sd in members]
        s["ks"], s["orders"] = [m[1] for m in members], [m[2] for m in members]
        s["batch"] = kcl.kcl_batch_create()
        return s
    row, col = _graph(case, seed)
    if case["call"] == "load":
        s["row"] = row.cpu().numpy().astype(np.uint64)
        s["col"] = col.cpu().numpy().astype(np.uint32)
        return s
    if case["call"] == "rounds":
        n = case["n"]
        s.update(row=row, col=col, alive=torch.ones(n, dtype=torch.uint8, device="cuda"),
                 degree=(row[1:] - row[:-1]).to(torch.int32), out=torch.empty(n, dtype=torch.int32, device="cuda"))
        return s
    s["g"] = kcl.kcl_load_csr(row, col)
    if case["call"] == "per_root":
        s["out"] = torch.empty(case["n"], dtype=torch.int64, device="cuda")
    if case["call"] in ("list", "records"):
        room = RING_BYTES // (4 * case["k"]) if case["call"] == "list" else RECORDS
        s["ring"] = torch.full((room * case["k"],), -1, dtype=torch.int32, device="cuda")
    return s


def run(s):
    case = s["case"]
    call = case["call"]
    if call == "count":
        return {"count": kcl.kcl_count(s["g"], case["k"], case["order"])}
    if call == "per_root":
        total, pre = kcl.kcl_count_per_root(s["g"], case["k"], case["order"], s["out"])
        return {"count": total, "prelist": pre, "per_root": s["out"]}
    if call == "list":
        # the ring wraps and keeps an arbitrary subset of the records: what a
        # caller can rely on is the count and the checksum over every record
        count, checksum, written, _ = kcl.kcl_list(s["g"], case["k"], case["order"], s["ring"], wrap=True)
        return {"count": count, "checksum": _halves(checksum), "written": written}
    if call == "records":
        count, checksum, written, _ = kcl.kcl_list(s["g"], case["k"], case["order"], s["ring"])
        # record order is unspecified: the ring's records, packed 15 bits an id and sorted (unused ones, -1, first)
        rec = s["ring"].view(-1, case["k"]).long()
        key = rec[:, 0]
        for i in range(1, case["k"]):
            key = (key << 15) | rec[:, i]
        return {"count": count, "checksum": _halves(checksum), "written": written,
                "records": key.sort().values}
    if call == "load":
        g = kcl.kcl_load_csr(s["row"], s["col"])
        count = kcl.kcl_count(g, case["k"], case["order"])
        g.free()
        return {"count": count}
    if call == "batch":
        counts, _ = kcl.kcl_count_batch(s["batch"], s["graphs"], s["ks"], s["orders"])
        return {"counts": np.array(counts, dtype=np.int64)}
    kcl.kcl_degeneracy_order_noalloc(s["row"], s["col"], s["alive"], s["degree"], s["out"])
    return {"round": s["out"]}


def _halves(x):
    return [x >> 32, x & 0xFFFFFFFF]


def work(case):
    """Bytes: the graph read once and the outputs written once (listing: about 80 n^1.4 4-cliques on
    an R-MAT graph of 16 edges a vertex).  No floating-point work."""
    if case["call"] == "batch":
        mean_n = (case["hi_n"] - case["lo_n"]) / math.log(case["hi_n"] / case["lo_n"])
        return {"bytes": case["graphs"] * (8 * mean_n + 8 * 11 * mean_n), "flops": 0}
    n = case["n"]
    edges = case["factor"] * n if case["graph"] == "rmat" else (
        case["edges"] + case["groups"] * case["density"] * ((case["lo"] + case["hi"]) / 2) ** 2 / 2)
    b = 8 * n + 8 * edges
    if case["call"] == "per_root":
        b += 8 * n
    if case["call"] == "rounds":
        b += 9 * n
    if case["call"] == "list":
        b += 4 * case["k"] * (80 * n ** 1.4 if case["k"] == 4 else 8 * n ** 1.3)
    return {"bytes": b, "flops": 0}


# ------------------------------------------------- the same, computed plainly
_M = (1 << 64) - 1


def _mix(z):
    z = z ^ (z >> np.uint64(30))
    z = z * np.uint64(0xBF58476D1CE4E5B9)
    z = z ^ (z >> np.uint64(27))
    z = z * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _cliques(row, col, k):
    """All k-cliques with ids ascending, grown level by level from adjacency sets."""
    adj = [set(col[row[u]:row[u + 1]].tolist()) for u in range(len(row) - 1)]
    out = []

    def grow(r, cand):
        if len(r) == k:
            out.append(r)
            return
        for v in sorted(cand):
            rest = {w for w in cand & adj[v] if w > v}
            if len(r) + 1 + len(rest) >= k:
                grow(r + (v,), rest)

    for u in range(len(adj)):
        grow((u,), {w for w in adj[u] if w > u})
    return np.array(out, dtype=np.uint64).reshape(-1, k)


def exact(case, seed):
    small = case["call"] in ("count", "records", "load") and case["graph"] == "chung_lu" and case["n"] <= 20000 \
        and case["edges"] <= 100000
    if not small or case["k"] > 5:
        return None
    row, col = _graph(case, seed)
    c = _cliques(row.cpu().numpy(), col.cpu().numpy(), case["k"])
    if case["call"] != "records":
        return {"count": len(c)}
    with np.errstate(over="ignore"):
        h = _mix(np.full(len(c), 0x9E3779B97F4A7C15 ^ case["k"], dtype=np.uint64))
        for i in range(case["k"]):
            h = _mix(h ^ c[:, i])
        total = int(h.sum(dtype=np.uint64)) & _M
    key = c[:, 0].astype(np.int64)
    for i in range(1, case["k"]):
        key = (key << 15) | c[:, i].astype(np.int64)
    key = np.concatenate([np.full(RECORDS - len(key), -1, dtype=np.int64), np.sort(key)])
    return {"count": len(c), "checksum": _halves(total), "written": len(c), "records": torch.from_numpy(key)}
