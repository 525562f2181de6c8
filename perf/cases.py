"""The calls whose time matters to a user of this library, over the sizes and options it is used with.

A case is one call (or one chain of calls) of the public interface on a seeded synthetic input: the whole
method from an edge list, the CSR build alone, a clustering with its quotient graph and estimate on a built
CSR, the Delta-stepping baseline, a many-graph batch, and the diameter of a small dense graph.  Graph
families, weights, edge factors and tau follow the workloads of the tests and the benchmark: square meshes,
road-like meshes (10 % of the edges deleted, 0.1 % chords) and R-MAT (.57, .19, .19) graphs.

Every output is a whole number and is compared for equality.  Arrays come back in device memory through the
C ABI's copy calls (``include/cldiam.h``), which take device pointers, in buffers sized by the input (its node
and edge counts bound every output): what the graph at hand does not fill stays zero.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_1506_03265_gb300 as cd

_RMAT = (0.57, 0.19, 0.19)


def listed():
    return [
        # the smallest call: a 64 x 64 mesh in host memory, the smoke test's graph; latency counts
        {"name": "run_mesh64", "call": "run", "family": "mesh", "side": 64, "wmax": 100, "tau": 0.3, "host": True},
        # the benchmark's second configuration end to end: a pinned host edge list through the one-call form
        {"name": "run_rmat20_host", "call": "run", "family": "rmat", "n": 1 << 20, "ef": 16, "wmax": 1 << 20,
         "tau": 4.65, "host": True},
        # a road-like network of 16.8M nodes: long growth of many small steps
        {"name": "run_road4096", "call": "run", "family": "road", "side": 4096, "wmax": 1000, "tau": 5.4,
         "host": False},
        # the benchmark's headline configuration: R-MAT scale 24, 268M edges resident on the device
        {"name": "run_rmat24", "call": "run", "family": "rmat", "n": 1 << 24, "ef": 16, "wmax": 1000, "tau": 21.0,
         "host": False},
        # the CSR of the whole graph (no component selection), node count no power of two, copied out
        {"name": "build_rmat_odd", "call": "build", "family": "rmat", "n": 700001, "ef": 16, "wmax": 1000,
         "lcc": False},
        # 31-bit weights: ids and weight do not fit one 64-bit word (the paper's real weights scaled to integers)
        {"name": "build_rmat20_wide", "call": "build", "family": "rmat", "n": 1 << 20, "ef": 16, "wmax": (1 << 31) - 1,
         "lcc": True},
        # tuning tau on a built graph: clustering + quotient + estimate at the middle size
        {"name": "cluster_rmat22", "call": "cluster", "family": "rmat", "n": 1 << 22, "ef": 16, "wmax": 1000,
         "tau": 10.5, "algorithm": 1, "cumulative": False, "delta0_min": False},
        # the options of Section 3 (initial Delta = minimum weight, bounds within Delta) on an odd-sided mesh
        {"name": "cluster_mesh1001", "call": "cluster", "family": "mesh", "side": 1001, "wmax": 1000, "tau": 1.4,
         "algorithm": 1, "cumulative": True, "delta0_min": True},
        # Algorithm 2 on a built graph
        {"name": "cluster2_rmat20", "call": "cluster", "family": "rmat", "n": 1 << 20, "ef": 16, "wmax": 1 << 20,
         "tau": 4.65, "algorithm": 2, "cumulative": False, "delta0_min": False},
        # the shortest-path baseline the paper compares with, on the headline graph
        {"name": "sssp_rmat24", "call": "sssp", "family": "rmat", "n": 1 << 24, "ef": 16, "wmax": 1000},
        # many small graphs (R-MAT 2^8 .. 2^16 nodes and meshes) in one batch
        {"name": "batch_200", "call": "batch", "graphs": 200, "wmax": 1000},
        # diameter of a dense quotient-like graph given by the caller
        {"name": "apsp_dense2048", "call": "apsp", "k": 2048, "density": 0.25, "wmax": 1000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the call, the family and the options at random, sizes over their logarithm."""
    call = rng.choice(["run", "run", "build", "cluster", "cluster", "sssp", "batch", "apsp"])
    if call == "batch":
        return {"call": "batch", "graphs": _log(rng, 8, 200), "wmax": 1000}
    if call == "apsp":
        return {"call": "apsp", "k": _log(rng, 65, 2047), "density": rng.choice([0.02, 0.25, 0.6]), "wmax": 1000}
    c = {"call": call, "family": rng.choice(["rmat", "rmat", "mesh", "road"]), "wmax": rng.choice([100, 1000])}
    top = {"run": 1 << 24, "build": 1 << 20, "cluster": 1 << 22, "sssp": 1 << 24}[call]
    if c["family"] == "rmat":
        c.update(n=_log(rng, 1 << 10, top - 1), ef=rng.choice([8, 16]))
        if rng.random() < 0.3:
            c["wmax"] = 1 << 20  # (long mesh paths over such weights would leave the exact 32-bit range)
        n, tau = c["n"], 0.005 * math.sqrt(c["n"])
    else:
        # Delta-stepping on a mesh takes a round per bucket: its sizes end where a pass is still short
        c["side"] = _log(rng, 33, 400 if call == "sssp" else math.isqrt(top) - 1)
        n = c["side"] ** 2
        tau = _tau(n)
    if call == "run":
        c.update(tau=round(max(tau, 0.05), 3), host=rng.random() < 0.3 and n <= 1 << 20)
    elif call == "build":
        c.update(lcc=rng.random() < 0.5)
        if rng.random() < 0.3:
            c["wmax"] = (1 << 31) - 1
    elif call == "cluster":
        c.update(tau=round(max(tau, 0.05), 3), algorithm=rng.choice([1, 1, 1, 2]), cumulative=rng.random() < 0.3,
                 delta0_min=rng.random() < 0.2)
    return c


def _tau(n):
    """tau for about sqrt(n) clusters on a mesh of n nodes."""
    L = max(1.0, math.log2(max(n, 2)))
    return max(0.05, math.sqrt(n) / (4 * math.log(2) * L * max(1.0, L / 2)))


# ---------------------------------------------------------------- inputs, on the GPU
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)


def _weights(m, wmax, g):
    return torch.randint(1, wmax + 1, (m,), generator=g, device="cuda", dtype=torch.int32)


def _rmat(n, ef, wmax, seed):
    """R-MAT on the next power of two, scaled down to n ids and relabelled at random."""
    a, b, c = _RMAT
    g = _gen(seed)
    scale, m = max(1, (n - 1).bit_length()), ef * n
    perm = torch.randperm(n, generator=g, device="cuda").to(torch.int32)
    src = torch.empty(m, dtype=torch.int32, device="cuda")
    dst = torch.empty_like(src)
    step = 1 << 25
    for lo in range(0, m, step):
        k = min(step, m - lo)
        u = torch.zeros(k, dtype=torch.int32, device="cuda")
        v = torch.zeros_like(u)
        r = torch.empty(k, dtype=torch.float32, device="cuda")
        for _ in range(scale):
            r.uniform_(generator=g)
            u.mul_(2).add_(r >= a + b)
            v.mul_(2).add_(((r >= a) & (r < a + b)) | (r >= a + b + c))
        for ids, out in ((u, src), (v, dst)):
            out[lo:lo + k] = perm[(ids.long() * n) >> scale]
    return n, src, dst, _weights(m, wmax, g)


def _mesh(side, wmax, seed, road):
    g = _gen(seed)
    ids = torch.arange(side * side, dtype=torch.int32, device="cuda").view(side, side)
    src = torch.cat([ids[:, :-1].reshape(-1), ids[:-1].reshape(-1)])
    dst = torch.cat([ids[:, 1:].reshape(-1), ids[1:].reshape(-1)])
    if road:
        keep = torch.rand(src.numel(), generator=g, device="cuda") >= 0.1
        chords = src.numel() // 1000
        ends = torch.randint(0, side * side, (2, chords), generator=g, device="cuda", dtype=torch.int32)
        src, dst = torch.cat([src[keep], ends[0]]), torch.cat([dst[keep], ends[1]])
    return side * side, src.contiguous(), dst.contiguous(), _weights(src.numel(), wmax, g)


def _edges(c, seed):
    if c["family"] == "rmat":
        return _rmat(c["n"], c["ef"], c["wmax"], seed)
    return _mesh(c["side"], c["wmax"], seed, c["family"] == "road")


def _dense(c, seed):
    """A connected symmetric CSR; an edge joins a pair when drawn in either direction with probability density."""
    k, g = c["k"], _gen(seed)
    full = torch.zeros(k, k, dtype=torch.bool, device="cuda")
    full |= torch.rand(k, k, generator=g, device="cuda") < c["density"]
    ring = torch.arange(k, device="cuda")
    full[ring, (ring + 1) % k] = True  # connected
    full = torch.triu(full | full.t(), 1)
    w = torch.where(full, torch.randint(1, c["wmax"] + 1, (k, k), generator=g, device="cuda", dtype=torch.int32), 0)
    w = w + w.t()
    at = w.nonzero()
    off = torch.zeros(k + 1, dtype=torch.int64, device="cuda")
    off[1:] = (w > 0).sum(1).cumsum(0)
    return k, off, at[:, 1].to(torch.int32).contiguous(), w[at[:, 0], at[:, 1]].contiguous()


def _mixture(c, seed):
    """(n, src, dst, w) of every graph of a batch: half R-MAT (2^8 .. 2^16 nodes, edge factor 8), half meshes."""
    pick = np.random.default_rng(int(seed))
    for i in range(c["graphs"]):
        sub = int(pick.integers(1 << 62))
        if pick.random() < 0.5:
            yield _rmat(1 << int(pick.integers(8, 17)), 8, c["wmax"], sub)
        else:
            yield _mesh(int(round(2 ** pick.uniform(5, 9))), c["wmax"], sub, False)


def _out(n, dtype=torch.int32):
    return torch.zeros(max(int(n), 1), dtype=dtype, device="cuda")


def prepare(case, seed):
    c = dict(case)
    s = {"case": c, "seed": int(seed)}
    if c["call"] == "apsp":
        s["csr"] = _dense(c, seed)
    elif c["call"] == "batch":
        s["arena"] = cd.arena_create()
        ns = []
        for n, src, dst, w in _mixture(c, seed):
            torch.cuda.synchronize()
            s["arena"].add(src, dst, w, n)
            ns.append(n)
        s["ids"] = np.arange(len(ns), dtype=np.uint32)
        s["taus"] = np.array([_tau(n) for n in ns])
        s["seeds"] = np.arange(len(ns), dtype=np.uint64) + np.uint64(seed)
    else:
        n, src, dst, w = _edges(c, seed)
        if c.get("host"):
            src, dst, w = (t.cpu().pin_memory() for t in (src, dst, w))
        torch.cuda.synchronize()
        if c["call"] in ("run", "build"):
            s["edges"] = (n, src, dst, w)
        else:
            s["graph"] = cd.build_csr(src, dst, w, n)
        cap = 2 * int(src.numel())
        if c["call"] == "build":
            s["out"] = (_out(n + 1, torch.int64), _out(cap), _out(cap), _out(n))
        elif c["call"] == "cluster":
            s["out"] = (_out(n), _out(n), _out(n), _out(n + 1, torch.int64), _out(cap), _out(cap))
        elif c["call"] == "sssp":
            s["out"] = _out(n)
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------- one pass
def _ptrs(*tensors):
    return [t.data_ptr() for t in tensors]


def _ok(status, where):
    if status != cd.OK:
        raise RuntimeError(f"{where}: status {status}")


def _run_build(s):
    c, (n, src, dst, w) = s["case"], s["edges"]
    g = cd.build_csr(src, dst, w, n, lcc=c["lcc"])
    _ok(cd.load().cldiam_graph_copy(g.handle, *_ptrs(*s["out"])), "cldiam_graph_copy")
    r = {"n": g.n, "nnz": g.nnz, "delta0": g.delta0()}
    g.free()
    return {**dict(zip(("off", "col", "w", "orig"), s["out"])), **r}


def _run_cluster(s):
    c, lib = s["case"], cd.load()
    opts = {"contract_mode": cd.CONTRACT_CUMULATIVE if c["cumulative"] else cd.CONTRACT_RESET,
            "delta0_mode": cd.DELTA0_MIN if c["delta0_min"] else cd.DELTA0_AVG}
    cl = (cd.cluster if c["algorithm"] == 1 else cd.cluster2)(s["graph"], c["tau"], s["seed"], **opts)
    _ok(lib.cldiam_clustering_copy(cl.handle, *_ptrs(*s["out"][:3])), "cldiam_clustering_copy")
    q = cd.quotient_build(cl)
    _ok(lib.cldiam_quotient_copy(q.handle, *_ptrs(*s["out"][3:])), "cldiam_quotient_copy")
    est = cd.estimate(q)
    if c["algorithm"] == 2:
        # Algorithm 2's growth rounds and updates are those of its asynchronous relaxation, no fixed counts
        est = {f: est[f] for f in ("phi_gc", "radius", "phi_approx", "k", "stages", "delta_end", "centers_drawn")}
    q.free()
    cl.free()
    return {**dict(zip(("center", "D", "cid", "qoff", "qcol", "qw"), s["out"])), "estimate": est}


def _run_sssp(s):
    lib, g = cd.load(), s["graph"]
    ecc = ctypes.c_uint64()
    _ok(lib.cldiam_sssp_delta(g.handle, cd.sssp_source(g, s["seed"]), 0, s["out"].data_ptr(), ctypes.byref(ecc), None,
                              None), "cldiam_sssp_delta")
    return {"dist": s["out"], "ecc": ecc.value}


def run(state):
    c = state["case"]
    if c["call"] == "run":
        n, src, dst, w = state["edges"]
        return cd.run(src, dst, w, n, c["tau"], state["seed"])
    if c["call"] == "build":
        return _run_build(state)
    if c["call"] == "cluster":
        return _run_cluster(state)
    if c["call"] == "sssp":
        return _run_sssp(state)
    if c["call"] == "batch":
        res, sts = state["arena"].run(state["ids"], state["taus"], state["seeds"])
        out = {f: np.array([r[f] for r in res], dtype=np.int64) for f in res[0]}
        out["status"] = np.array(sts, dtype=np.int64)
        return out
    return {"phi": cd.apsp_max(*state["csr"])}


# ---------------------------------------------------------------- what a pass cannot do without
def _size(c):
    """(nodes, input edges)"""
    if c["family"] == "rmat":
        return c["n"], c["ef"] * c["n"]
    n = c["side"] ** 2
    m = 2 * c["side"] * (c["side"] - 1)
    return n, m - m // 10 + m // 1000 if c["family"] == "road" else m


def work(case):
    """Bytes of the inputs read once and the outputs written once; operations: one per edge of a growth or
    shortest-path pass, two (add, minimum) per relaxation of the dense closure."""
    c = case
    if c["call"] == "apsp":
        z = (1 - (1 - c["density"]) ** 2) * c["k"] ** 2
        return {"bytes": 8.0 * z + 8.0 * c["k"], "flops": 2.0 * c["k"] ** 3}
    if c["call"] == "batch":
        # expected sizes of the mixture: R-MAT 8 * 2^s edges, meshes 2 * 4^u
        rm = 8 * sum(2 ** s for s in range(8, 17)) / 9
        me = 2 * (4.0 ** 9 - 4.0 ** 5) / (4 * math.log(4))
        entries = c["graphs"] * (rm + me)  # two directed entries per edge, half of the graphs each
        return {"bytes": 8.0 * entries, "flops": entries}
    n, m = _size(c)
    if c["call"] == "run":
        return {"bytes": 12.0 * m, "flops": 2.0 * m}
    if c["call"] == "build":
        return {"bytes": 12.0 * m + 16.0 * m + 12.0 * n, "flops": 2.0 * m}
    if c["call"] == "sssp":
        return {"bytes": 16.0 * m + 12.0 * n, "flops": 2.0 * m}
    return {"bytes": 16.0 * m + 20.0 * n, "flops": 2.0 * m}


# ---------------------------------------------------------------- the same values by plain torch, in 64 bits
def _largest_component(n, src, dst):
    """Nodes of the largest component (ties: the one holding the smallest id), by label minima."""
    label = torch.arange(n, device="cuda")
    src, dst = src.long(), dst.long()
    while True:
        old = label.clone()
        low = torch.minimum(label[src], label[dst])
        label.scatter_reduce_(0, label[src], low, "amin")
        label.scatter_reduce_(0, label[dst], low, "amin")
        for _ in range(3):
            label = label[label]
        if torch.equal(label, old):
            break
    size = torch.bincount(label, minlength=n)
    return label == int(size.argmax())


def _plain_csr(n, src, dst, w, lcc):
    """off, col, w, orig by sorting (row, col, weight) keys: parallel edges keep their smallest weight."""
    src, dst, w = src.cuda().long(), dst.cuda().long(), w.cuda().long()
    ok = src != dst
    key = torch.cat([(src * n + dst)[ok], (dst * n + src)[ok]])
    w = torch.cat([w[ok], w[ok]])
    w, order = w.sort()
    key, by = key[order].sort(stable=True)
    w = w[by]
    first = torch.ones_like(key, dtype=torch.bool)
    first[1:] = key[1:] != key[:-1]
    row, col, w = key[first] // n, key[first] % n, w[first]
    orig = torch.arange(n, device="cuda")
    if lcc:
        keep = _largest_component(n, src, dst)
        new = keep.long().cumsum(0) - 1
        at = keep[row]
        row, col, w, orig = new[row[at]], new[col[at]], w[at], orig[keep]
    off = torch.zeros(orig.numel() + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.bincount(row, minlength=orig.numel()).cumsum(0)
    return off, col, w, orig


def exact(case, seed):
    """The outputs by plain torch where they have a short definition: the CSR and the dense closure; else None."""
    c = case
    if c["call"] == "apsp":
        k, off, col, w = _dense(c, seed)
        d = torch.full((k, k), 1 << 40, dtype=torch.int64, device="cuda")
        d[torch.repeat_interleave(torch.arange(k, device="cuda"), off.diff()), col.long()] = w.long()
        d.fill_diagonal_(0)
        for p in range(k):
            torch.minimum(d, d[:, p:p + 1] + d[p:p + 1], out=d)
        return {"phi": int(d.max())}
    if c["call"] == "build":
        n, src, dst, w = _edges(c, seed)
        off, col, w, orig = _plain_csr(n, src, dst, w, c["lcc"])
        nnz, cap = int(col.numel()), 2 * int(src.numel())
        d0 = max(1, int(w.sum()) // 2 // (nnz // 2)) if nnz else 1
        pad = lambda t, to: torch.nn.functional.pad(t, (0, to - t.numel()))  # noqa: E731
        return {"off": pad(off, n + 1), "col": pad(col, cap), "w": pad(w, cap), "orig": pad(orig, n),
                "n": int(orig.numel()), "nnz": nnz, "delta0": d0}
    return None
