"""Performance cases: the calls that programs make of the library, over the
sizes it is used at, timed through the public entry points.

Graph families (the ones the benchmark, the tests and the server's workload
use, generated here with torch on the GPU from the seed alone):

* ``er``       a random Hamiltonian cycle plus random pairs (connected), average
               degree and weight range as given;
* ``rmat``     R-MAT (.57, .19, .19) with unit weights, ids permuted, its k-core,
               the largest component of that (web and social graphs);
* ``planted``  two random blocks of average degree 42, each reduced to its
               30-core, joined by 25 unit edges: a minimum cut that no vertex
               degree shows, the hard case of the exact rounds.

A solve returns the cut value and the side bitmap.  Batches and served requests
return the values alone, as a program that wants connectivities asks for them.
"""
import ctypes
import math

import numpy as np
import torch

import paper_2609_07204_gb300 as mc

DEV = "cuda"


# ------------------------------------------------------------------ generators
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1_000_003 + salt * 7919 + 12345) % (1 << 62))
    return g


def _unique_pairs(a, b, n):
    """Distinct undirected pairs without self-loops, as (lo, hi)."""
    lo, hi = torch.minimum(a, b), torch.maximum(a, b)
    key = torch.unique((lo * n + hi)[lo != hi])
    return key // n, key % n


def _csr(n, lo, hi, w):
    """Symmetric CSR with sorted rows of distinct undirected edges."""
    key = torch.cat([lo * n + hi, hi * n + lo])
    key, order = torch.sort(key)
    src = key // n
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return rp, (key - src * n).to(torch.int32), torch.cat([w, w])[order].to(torch.int32)


def _weights(m, wlo, whi, g):
    if wlo == whi:
        return torch.full((m,), wlo, dtype=torch.int32, device=DEV)
    return torch.randint(wlo, whi + 1, (m,), generator=g, device=DEV, dtype=torch.int32)


def _core(n, lo, hi, k):
    """Edges of the k-core (repeated removal of vertices of degree below k)."""
    while lo.numel():
        keep = torch.bincount(torch.cat([lo, hi]), minlength=n) >= k
        e = keep[lo] & keep[hi]
        if bool(e.all()):
            break
        lo, hi = lo[e], hi[e]
    return lo, hi


def _largest_component(n, lo, hi):
    lab = torch.arange(n, device=DEV)
    while True:
        new = lab.clone()
        new.scatter_reduce_(0, lo, lab[hi], "amin")
        new.scatter_reduce_(0, hi, lab[lo], "amin")
        new = new[new]
        if torch.equal(new, lab):
            break
        lab = new
    top = torch.bincount(lab[torch.cat([lo, hi])], minlength=n).argmax()
    e = lab[lo] == top
    return lo[e], hi[e]


def _compact(n, lo, hi, g=None):
    """Renumber the vertices that have edges to 0.., optionally permuted."""
    has = torch.zeros(n, dtype=torch.bool, device=DEV)
    has[lo] = True
    has[hi] = True
    ids = torch.cumsum(has.to(torch.int64), 0) - 1
    n2 = int(has.sum())
    lo, hi = ids[lo], ids[hi]
    if g is not None:
        p = torch.randperm(n2, generator=g, device=DEV)
        lo, hi = p[lo], p[hi]
    return n2, torch.minimum(lo, hi), torch.maximum(lo, hi)


def _er(n, deg, wlo, whi, seed, salt=1):
    g = _gen(seed, salt)
    p = torch.randperm(n, generator=g, device=DEV)
    m = max(0, int(n * deg / 2) - n)
    a = torch.cat([p, torch.randint(0, n, (m,), generator=g, device=DEV)])
    b = torch.cat([p.roll(-1), torch.randint(0, n, (m,), generator=g, device=DEV)])
    lo, hi = _unique_pairs(a, b, n)
    return (n, *_csr(n, lo, hi, _weights(lo.numel(), wlo, whi, g)))


def _rmat(scale, edge_factor, core, wlo, whi, seed, keep=0, salt=2):
    g = _gen(seed, salt)
    n, m = 1 << scale, int(edge_factor * (1 << scale))
    u = torch.zeros(m, dtype=torch.int64, device=DEV)
    v = torch.zeros(m, dtype=torch.int64, device=DEV)
    for _ in range(scale):
        r = torch.rand(m, generator=g, device=DEV)
        u = u * 2 + (r >= 0.76)
        v = v * 2 + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    p = torch.randperm(n, generator=g, device=DEV)
    lo, hi = _unique_pairs(p[u], p[v], n)
    if keep:  # the first `keep` vertices only (a graph of any size)
        e = hi < keep
        lo, hi = lo[e], hi[e]
    lo, hi = _largest_component(n, *_core(n, lo, hi, core))
    n2, lo, hi = _compact(n, lo, hi)
    return (n2, *_csr(n2, lo, hi, _weights(lo.numel(), wlo, whi, g)))


def _planted(nb, seed, salt=3):
    g = _gen(seed, salt)
    m = 21 * nb
    a = torch.randint(0, nb, (2 * m,), generator=g, device=DEV)
    b = torch.randint(0, nb, (2 * m,), generator=g, device=DEV)
    a[m:] += nb
    b[m:] += nb
    n = 2 * nb
    lo, hi = _core(n, *_unique_pairs(a, b, n), 30)
    n2, lo, hi = _compact(n, lo, hi)
    split = _block_split(n2, lo, hi)
    c = 25
    while True:  # 25 distinct cross pairs
        x = torch.randint(0, split, (c,), generator=g, device=DEV)
        y = torch.randint(split, n2, (c,), generator=g, device=DEV)
        if torch.unique(x * n2 + y).numel() == c:
            break
    p = torch.randperm(n2, generator=g, device=DEV)
    lo, hi = _unique_pairs(p[torch.cat([lo, x])], p[torch.cat([hi, y])], n2)
    return (n2, *_csr(n2, lo, hi, _weights(lo.numel(), 1, 1, g)))


def _block_split(n, lo, hi):
    """Vertices 0..split-1 and split..n-1 are joined by no edge: the split."""
    reach = torch.zeros(n, dtype=torch.int64, device=DEV)
    reach.scatter_reduce_(0, lo, hi, "amax")
    far = torch.cummax(torch.maximum(reach, torch.arange(n, device=DEV)), 0).values
    return int((far == torch.arange(n, device=DEV)).nonzero()[0]) + 1


def _graph(case, seed, salt=0):
    kind = case["graph"]
    if kind == "er":
        return _er(case["n"], case["deg"], case["wlo"], case["whi"], seed, 1 + salt)
    if kind == "rmat":
        return _rmat(case["scale"], case["edge_factor"], case["core"], 1, 1, seed, salt=2 + salt)
    return _planted(case["nb"], seed, 3 + salt)


def _host(arrays, pinned):
    out = []
    for t in arrays:
        h = torch.empty(t.shape, dtype=t.dtype, pin_memory=pinned)
        h.copy_(t)
        out.append(h.numpy())
    return out


# ----------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest whole call: a small graph from host arrays, solved once
        {"name": "call_er_256", "call": "host", "graph": "er", "n": 256, "deg": 8.0, "wlo": 1,
         "whi": 100, "pinned": False},
        # the smallest configuration: one dense little graph, resident
        {"name": "solve_er_2000", "call": "solve", "graph": "er", "n": 2000, "deg": 16.0,
         "wlo": 1, "whi": 10},
        # an ordinary social-network core, resident
        {"name": "solve_rmat_16", "call": "solve", "graph": "rmat", "scale": 16,
         "edge_factor": 16, "core": 10},
        # the benchmark's R-MAT core, resident
        {"name": "solve_rmat_20", "call": "solve", "graph": "rmat", "scale": 20,
         "edge_factor": 16, "core": 10},
        # the same from pinned host arrays: create, solve, read the side, release
        {"name": "call_rmat_20", "call": "host", "graph": "rmat", "scale": 20,
         "edge_factor": 16, "core": 10, "pinned": True},
        # planted cuts, resident: a small one and a large one
        {"name": "solve_planted_15", "call": "solve", "graph": "planted", "nb": 1 << 15},
        {"name": "solve_planted_19", "call": "solve", "graph": "planted", "nb": 1 << 19},
        # a weighted random graph handed over on the device, solved once
        {"name": "call_er_weighted", "call": "device", "graph": "er", "n": 150_001, "deg": 16.0,
         "wlo": 1, "whi": 100},
        # the batched workload: 4,096 graphs of 20 to 2,000 vertices, solved repeatedly
        {"name": "batch_4096", "call": "batch", "count": 4096, "nlo": 20, "nhi": 2000},
        # the server: requests of mixed sizes arriving together, until all are answered
        {"name": "serve_64", "call": "serve", "count": 64, "nlo": 100, "nhi": 65536},
        # one round driven by the caller: contraction to given clusters, result read back
        {"name": "contract_rmat_18", "call": "contract", "graph": "rmat", "scale": 18,
         "edge_factor": 16, "core": 10, "clusters": 300},
        # the allocation-free contraction of a device CSR
        {"name": "noalloc_er", "call": "noalloc", "graph": "er", "n": 15_001, "deg": 16.0,
         "wlo": 1, "whi": 10, "clusters": 3750},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["solve", "solve", "solve", "host", "device", "batch", "serve", "contract",
                       "noalloc"])
    if call == "batch":
        return {"call": "batch", "count": _log(rng, 200, 4096), "nlo": rng.randint(8, 60),
                "nhi": _log(rng, 300, 2000)}
    if call == "serve":
        return {"call": "serve", "count": _log(rng, 8, 64), "nlo": rng.randint(50, 400),
                "nhi": _log(rng, 4000, 65536)}
    if call == "noalloc":
        n = _log(rng, 300, 16000)
        return {"call": "noalloc", "graph": "er", "n": n, "deg": rng.uniform(4.0, 16.0), "wlo": 1,
                "whi": rng.choice([1, 10, 100]), "clusters": max(2, n // _log(rng, 2, 100))}
    kind = rng.choice(["er", "rmat"] if call == "contract" else ["er", "rmat", "planted"])
    case = {"call": call, "graph": kind}
    if kind == "er":
        case.update(n=_log(rng, 100, 300_000), deg=rng.uniform(6.0, 32.0), wlo=1,
                    whi=rng.choice([1, 10, 100]))
    elif kind == "rmat":
        case.update(scale=rng.randint(13, 19), edge_factor=rng.randint(12, 20),
                    core=rng.choice([5, 8, 10, 12]))
    else:
        case.update(nb=_log(rng, 4000, 400_000))
    if call == "host":
        case["pinned"] = rng.random() < 0.5
    if call == "contract":
        case["clusters"] = _log(rng, 4, max(5, math.sqrt(_size(case)[1] / 40)))
    return case


def _requests(case, seed):
    """Host graphs of log-uniform sizes, R-MAT and random ones in turn."""
    out = []
    steps = max(1, case["count"] - 1)
    g = torch.Generator().manual_seed(int(seed) * 31 + 7)
    jitter = torch.rand(case["count"], generator=g).tolist()
    for i in range(case["count"]):
        x = (i + jitter[i]) / (steps + 1)
        n = int(round(case["nlo"] * (case["nhi"] / case["nlo"]) ** x))
        if i % 2:
            scale = max(4, math.ceil(math.log2(n)) + 1)
            gr = _rmat(scale, 16, 1, 1, 100, seed, keep=n, salt=100 + i)
        else:
            gr = _er(n, 16.0, 1, 100, seed, salt=100 + i)
        out.append((gr[0], *_host(gr[1:], True)))
    return out


def _batch_graphs(case, seed):
    """`count` graphs packed in one CSR (sizes log-uniform in [nlo, nhi],
    average degree 3 to 12, weights 1 to 100), generated together."""
    g = _gen(seed, 50)
    G = case["count"]
    u = torch.rand(G, generator=g, device=DEV, dtype=torch.float64)
    n = (case["nlo"] * (case["nhi"] / case["nlo"]) ** u).floor().to(torch.int64)
    d = 3.0 + 9.0 * torch.rand(G, generator=g, device=DEV, dtype=torch.float64)
    vo = torch.zeros(G + 1, dtype=torch.int64, device=DEV)
    vo[1:] = torch.cumsum(n, 0)
    total = int(vo[-1])
    gid = torch.repeat_interleave(torch.arange(G, device=DEV), n)
    # a random Hamiltonian cycle of each graph
    key = gid.to(torch.float64) + torch.rand(total, generator=g, device=DEV, dtype=torch.float64)
    order = torch.argsort(key)
    nxt = torch.arange(1, total + 1, device=DEV)
    nxt[vo[1:] - 1] = vo[:-1]
    a, b = order, order[nxt]
    # and random pairs within it
    extra = torch.clamp((n * d / 2).floor().to(torch.int64) - n, min=0)
    eg = torch.repeat_interleave(torch.arange(G, device=DEV), extra)
    m = eg.numel()
    r = torch.rand(2, m, generator=g, device=DEV, dtype=torch.float64)
    ne = n[eg].to(torch.float64)
    ea = vo[eg] + torch.minimum((r[0] * ne).to(torch.int64), n[eg] - 1)
    eb = vo[eg] + torch.minimum((r[1] * ne).to(torch.int64), n[eg] - 1)
    lo, hi = _unique_pairs(torch.cat([a, ea]), torch.cat([b, eb]), total)
    rp, col, w = _csr(total, lo, hi, _weights(lo.numel(), 1, 100, g))
    return [t.cpu().numpy() for t in (vo, rp, col, w)]


def _labels(n, n2, seed):
    """A random label in [0, n2) per vertex, every label in use."""
    g = _gen(seed, 60)
    lab = torch.randint(0, n2, (n,), generator=g, device=DEV, dtype=torch.int32)
    lab[torch.randperm(n, generator=g, device=DEV)[:n2]] = torch.arange(n2, dtype=torch.int32,
                                                                         device=DEV)
    return lab


def prepare(case, seed):
    call = case["call"]
    st = {"call": call}
    if call == "batch":
        st["graph"] = mc.mincut_batch_from_csr(*_batch_graphs(case, seed))
        return st
    if call == "serve":
        st["requests"] = _requests(case, seed)
        st["server"] = mc.Server(mc.server_default_options(workers=16, want_bitmap=0))
        return st
    n, rp, col, w = _graph(case, seed)
    st["n"] = n
    # the program's buffers hold the largest graph of the family
    st["bitmap"] = np.zeros((_capacity(case) + 63) // 64, np.uint64)
    if call == "host":
        st["csr"] = _host((rp, col, w), case["pinned"])
    elif call == "device":
        st["csr"] = (rp, col, w)
    elif call == "noalloc":
        n2 = case["clusters"]
        cap = int(n * case["deg"]) + 2 * n
        st.update(csr=(rp, col, w), n2=n2, labels=_labels(n, n2, seed), m=col.numel(),
                  out=(torch.zeros(n2 + 1, dtype=torch.int64, device=DEV),
                       torch.zeros(cap, dtype=torch.int32, device=DEV),
                       torch.zeros(cap, dtype=torch.int32, device=DEV)))
    else:
        st["graph"] = mc.mincut_graph_from_csr(n, rp, col, w)
        if call == "contract":
            st["groups"] = _labels(n, case["clusters"], seed).cpu().numpy()
    return st


def _solve(g, bitmap):
    value, bitmap, _ = mc.mincut_solve(g, side_bitmap_out=bitmap)
    return [value, bitmap.view(np.int64)]


def run(st):
    call = st["call"]
    if call == "solve":
        return _solve(st["graph"], st["bitmap"])
    if call in ("host", "device"):
        g = mc.mincut_graph_from_csr(st["n"], *st["csr"])
        out = _solve(g, st["bitmap"])
        mc.mincut_graph_destroy(g)
        return out
    if call == "batch":
        return mc.mincut_batch_solve(st["graph"], bitmap=False)[0]
    if call == "serve":
        sv = st["server"]
        ids = [sv.submit(*r, borrow=True) for r in st["requests"]]
        return np.array([sv.wait(i, bitmap=False)[0] for i in ids], np.int64)
    if call == "contract":
        g = st["graph"]
        mc.mincut_graph_reset(g)
        ro = mc.default_round_options()
        ro.groups = ctypes.c_void_p(st["groups"].ctypes.data)
        mc.mincut_contract_round(g, ro)
        return list(mc.mincut_graph_export_csr(g))
    rp, col, w = st["out"]
    m = mc.mincut_contract_csr_noalloc(st["n"], *st["csr"], st["labels"], st["n2"], rp, col, w,
                                       m_directed=st["m"])
    return [m, rp, col, w]


# ------------------------------------------------------------- what it must do
def _capacity(case):
    """Vertices the family can have before its reductions."""
    return {"er": case.get("n"), "rmat": 1 << case.get("scale", 0),
            "planted": 2 * case.get("nb", 0)}[case["graph"]]


def _size(case):
    """(vertices, directed entries), the families' expected sizes."""
    kind = case["graph"]
    if kind == "er":
        return case["n"], int(case["n"] * case["deg"])
    if kind == "planted":
        return int(1.94 * case["nb"]), int(2 * 40.4 * case["nb"])
    s = case["scale"]
    share = min(0.95, 0.772 + 0.0234 * (s - 16)) * (case["edge_factor"] / 16) ** 0.9
    return int(2 ** s * 0.25), int(32 * 2 ** s * share)


def work(case):
    """Bytes: the CSR read once (row offsets, columns, weights) and the result
    written once."""
    call = case["call"]
    if call in ("batch", "serve"):
        mean = (case["nhi"] - case["nlo"]) / math.log(case["nhi"] / case["nlo"])
        deg = 7.5 if call == "batch" else 16.0
        return {"bytes": case["count"] * (mean * (8 + 8 * deg) + 8), "flops": 0}
    n, M = _size(case)
    read = 8 * n + 8 * M
    if call in ("contract", "noalloc"):
        n2 = case["clusters"]
        m2 = n2 * n2 * -math.expm1(-M / (n2 * n2))
        return {"bytes": read + 4 * n + 8 * n2 + (8 if call == "noalloc" else 12) * m2,
                "flops": 0}
    return {"bytes": read + n / 8, "flops": 0}


def _contracted(lab, n2, rp, col, w):
    """Contraction by labels in 64-bit integers: (row_ptr, col, w)."""
    src = np.repeat(np.arange(len(rp) - 1), np.diff(rp))
    a, b = lab[src].astype(np.int64), lab[col].astype(np.int64)
    keep = (a != b) & (w > 0)
    key, inv = np.unique(a[keep] * n2 + b[keep], return_inverse=True)
    s = np.zeros(len(key), np.int64)
    np.add.at(s, inv, w[keep].astype(np.int64))
    out = np.zeros(n2 + 1, np.int64)
    out[1:] = np.cumsum(np.bincount(key // n2, minlength=n2))
    return out, key % n2, s


def _stoer_wagner(n, rp, col, w):
    a = np.zeros((n, n), np.int64)
    a[np.repeat(np.arange(n), np.diff(rp)), col] += w
    best, alive = None, np.ones(n, bool)
    for left in range(n, 1, -1):
        r = np.where(alive, 0, -1)
        s = t = -1
        for _ in range(left):
            s, t = t, int(r.argmax())
            cut = int(r[t])
            r = np.where(r >= 0, r + a[t], r)
            r[t] = -1
        best = cut if best is None else min(best, cut)
        a[s] += a[t]
        a[:, s] += a[:, t]
        a[s, s] = 0
        a[t] = 0
        a[:, t] = 0
        alive[t] = False
    return best


def exact(case, seed):
    call = case["call"]
    if call in ("batch", "serve") or case["graph"] == "planted":
        return None
    n, M = _size(case)
    if call == "noalloc" or (call == "contract" and M <= 8_000_000):
        n, rp, col, w = _graph(case, seed)
        n2 = case["clusters"]
        lab = _labels(n, n2, seed).cpu().numpy()
        rp, col, w = (t.cpu().numpy() for t in (rp, col, w))
        if call == "contract":  # vertices are numbered by their smallest member
            first = np.full(n2, n, np.int64)
            np.minimum.at(first, lab, np.arange(n))
            rank = np.empty(n2, np.int64)
            rank[np.argsort(first)] = np.arange(n2)
            lab = rank[lab]
        out = list(_contracted(lab, n2, rp, col, w))
        if call == "noalloc":
            cap, m2 = int(n * case["deg"]) + 2 * n, len(out[1])
            out = [m2, out[0], *(np.pad(x, (0, cap - m2)) for x in out[1:])]
        return out
    if case["graph"] == "er" and n <= 512:
        n, rp, col, w = _graph(case, seed)
        return [_stoer_wagner(n, *(t.cpu().numpy() for t in (rp, col, w))), None]
    return None
