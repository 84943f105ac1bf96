"""Performance cases of the library: what its users have it do, from the
smallest call to the largest, each through the public binding.

Graphs are seeded R-MAT graphs (a/b/c/d = 0.57/0.19/0.19/0.05, symmetrised,
self-loops and duplicates dropped; n need not be a power of two, edges to ids
past n are left out) and 4-neighbour grids with symmetric weights on the 1/16
lattice in [1, 100).  They are generated on the device.  The conversions, whose
results are as long as the graph has entries and tiles, take one graph whose
vertices the seed rotates by whole blocks of 32, so that every seed gives other
arrays of the same lengths.

A case names an operation (`op`) and its sizes and options:
  spmv      one B2SR SpMV over a semiring, the unit every driver repeats
  pagerank  fp32 PageRank, d = 0.85
  from_csr  CSR -> B2SR, with the three arrays read back (encode)
  to_csr    B2SR -> CSR (decode)
  bfs       single-source BFS
  bfs_multi up to 64 BFS searches in one call
  tc        triangle count by masked SpGEMM
  sssp      push SSSP with delta-stepping buckets on a weighted grid
  serve     mixed BFS and personalised-PageRank queries to a running server
"""
import functools

import numpy as np
import torch

from paper_2201_08560_gb300 import binding as B

AUTO, DIRECT = B.SCHED_AUTO, B.SCHED_DIRECT
L2_BYTES = 129 << 20


def listed():
    return [
        # one Boolean SpMV on the smallest graph a user would put on a GPU: launches and latency
        {"name": "spmv_bool_r12_k8", "op": "spmv", "semiring": "bool", "n": 1 << 12, "ef": 16, "k": 8,
         "perm": False, "schedule": AUTO, "mask": "none"},
        # the Boolean SpMV of the benchmark graph, one byte per tile row (the paper's uint8 packing)
        {"name": "spmv_bool_r20_k8", "op": "spmv", "semiring": "bool", "n": 1 << 20, "ef": 16, "k": 8,
         "perm": False, "schedule": AUTO, "mask": "none"},
        # the float SpMV under PageRank at the benchmark's tile size and schedule
        {"name": "spmv_plus_r20_k4", "op": "spmv", "semiring": "plus", "n": 1 << 20, "ef": 16, "k": 4,
         "perm": False, "schedule": DIRECT, "mask": "none"},
        # a whole driver as the quick start calls it (default schedule), on vertices in no order
        {"name": "pagerank_r20_k4_perm", "op": "pagerank", "n": 1 << 20, "ef": 16, "k": 4, "perm": True,
         "schedule": AUTO, "iters": 20},
        # loading a graph: every user pays it once per graph, the benchmark step once per step
        {"name": "from_csr_r20_k4", "op": "from_csr", "n": 1 << 20, "ef": 16, "k": 4, "perm": False},
        # reading a graph back, ragged size
        {"name": "to_csr_n700001_k8", "op": "to_csr", "n": 700001, "ef": 16, "k": 8, "perm": False},
        # one small query: the cost of a driver call
        {"name": "bfs_r12_k8", "op": "bfs", "n": 1 << 12, "ef": 16, "k": 8, "perm": False, "schedule": AUTO},
        # the benchmark step's 16 searches
        {"name": "bfs16_r20_k4", "op": "bfs_multi", "n": 1 << 20, "ef": 16, "k": 4, "perm": False,
         "schedule": DIRECT, "nsrc": 16},
        # a full 64-lane batch on the largest graph
        {"name": "bfs64_r22_k4", "op": "bfs_multi", "n": 1 << 22, "ef": 16, "k": 4, "perm": False,
         "schedule": DIRECT, "nsrc": 64},
        # triangle counting on the denser graph
        {"name": "tc_r18_ef32_k8", "op": "tc", "n": 1 << 18, "ef": 32, "k": 8, "perm": False},
        # shortest paths on a mesh: a long chain of small rounds
        {"name": "sssp_grid4096_k8", "op": "sssp", "rows": 4096, "cols": 4096, "k": 8, "delta": 400.0},
        # a burst of queries at a server with resident graphs
        {"name": "serve_8graphs", "op": "serve", "graphs": 8, "lo": 14, "hi": 17, "ef": 16, "k": 4,
         "schedule": DIRECT, "queries": 128, "iters": 20},
    ]


def _log_size(rng, lo, hi):
    """A size between 2^lo and 2^hi, spread over the logarithm, mostly ragged."""
    return int(round(2.0 ** rng.uniform(lo, hi)))


def draw(rng):
    op = rng.choice(["spmv", "spmv", "spmv", "pagerank", "from_csr", "to_csr", "bfs", "bfs_multi", "bfs_multi", "tc",
                     "sssp", "serve"])
    c = {"op": op, "ef": rng.choice([8, 16, 16, 32]), "k": rng.choice([4, 8, 16, 32]), "perm": rng.random() < 0.4,
         "schedule": rng.choice([AUTO, DIRECT])}
    if op == "spmv":
        c["n"] = _log_size(rng, 10, 20)
        c["semiring"] = rng.choice(["bool", "bool", "count", "plus", "plus", "min", "max", "minplus"])
        c["mask"] = rng.choice(["none", "none", "keep", "complement"])
    elif op == "pagerank":
        c["n"], c["iters"] = _log_size(rng, 12, 19), rng.choice([5, 20, 50])
    elif op in ("from_csr", "to_csr"):
        c["n"] = _log_size(rng, 12, 19.8)
        del c["schedule"]
    elif op == "bfs":
        c["n"] = _log_size(rng, 10, 20)
    elif op == "bfs_multi":
        c["n"], c["nsrc"] = _log_size(rng, 12, 20), rng.randint(2, 64)
    elif op == "tc":
        c["n"], c["k"] = _log_size(rng, 12, 17.5), rng.choice([4, 8, 16])
        del c["schedule"]
    elif op == "sssp":
        c = {"op": op, "rows": _log_size(rng, 6, 11), "cols": _log_size(rng, 6, 11), "k": rng.choice([4, 8, 16, 32]),
             "delta": rng.choice([100.0, 400.0, 1600.0])}
    else:
        lo = rng.randint(11, 14)
        c = {"op": op, "graphs": rng.randint(2, 10), "lo": lo, "hi": lo + rng.randint(0, 3), "ef": 16,
             "k": rng.choice([4, 8]), "schedule": rng.choice([AUTO, DIRECT]), "queries": rng.randint(16, 128),
             "iters": 20}
    return c


# ---------------------------------------------------------------------------
# graphs
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _generator(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed))
    return g


def _rmat(n, ef, perm, seed, rotate=0):
    """(rowptr, colind) of a symmetric R-MAT graph on ids [0, n), int32 on the
    device; `rotate` blocks of 32 ids move round (the last, short block stays)."""
    dev, gen = _device(), _generator(seed)
    scale = max(1, (n - 1).bit_length())
    m = ef * n
    src = torch.zeros(m, dtype=torch.int64, device=dev)
    dst = torch.zeros(m, dtype=torch.int64, device=dev)
    for _ in range(scale):
        u = torch.rand(m, generator=gen, device=dev)
        src.mul_(2).add_(u >= 0.76)
        dst.mul_(2).add_(((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
    keep = (src < n) & (dst < n) & (src != dst)
    src, dst = src[keep], dst[keep]
    if perm:
        p = torch.randperm(n, generator=gen, device=dev)
        src, dst = p[src], p[dst]
    if rotate:
        full = n // 32 * 32
        src, dst = (torch.where(v < full, (v + 32 * rotate) % full, v) for v in (src, dst))
    key = torch.unique(torch.cat([src * n + dst, dst * n + src]))
    rowptr = torch.searchsorted(key, torch.arange(n + 1, device=dev) * n).to(torch.int32)
    return rowptr, (key % n).to(torch.int32)


def _graph(case, seed):
    if case["op"] in ("from_csr", "to_csr"):
        return _rmat(case["n"], case["ef"], case["perm"], 1, rotate=37 * seed % (case["n"] // 32))
    return _rmat(case["n"], case["ef"], case["perm"], seed)


def _grid_slots(rows, cols):
    """(columns, present) of the 4-neighbour grid as (n, 4) arrays: up, left, right, down."""
    dev = _device()
    ids = torch.arange(rows * cols, device=dev).reshape(rows, cols)
    cols4 = torch.stack([ids - cols, ids - 1, ids + 1, ids + cols], dim=2)
    ok = torch.ones(rows, cols, 4, dtype=torch.bool, device=dev)
    ok[0, :, 0] = ok[:, 0, 1] = ok[:, -1, 2] = ok[-1, :, 3] = False
    return cols4, ok


def _grid_weights(rows, cols, seed):
    """Weights of the edges to the right and downwards, fp32 on the 1/16 lattice in [1, 100)."""
    dev, gen = _device(), _generator(seed)
    right = 1.0 + torch.randint(0, 99 * 16, (rows, cols - 1), generator=gen, device=dev) / 16.0
    down = 1.0 + torch.randint(0, 99 * 16, (rows - 1, cols), generator=gen, device=dev) / 16.0
    return right.float(), down.float()


def _grid(rows, cols, seed):
    """(rowptr, colind, weights) of the grid, CSR order."""
    cols4, ok = _grid_slots(rows, cols)
    right, down = _grid_weights(rows, cols, seed)
    w4 = torch.zeros(rows, cols, 4, device=cols4.device)
    w4[1:, :, 0], w4[:, 1:, 1], w4[:, :-1, 2], w4[:-1, :, 3] = down, right, right, down
    rowptr = torch.zeros(rows * cols + 1, dtype=torch.int32, device=cols4.device)
    rowptr[1:] = ok.reshape(-1, 4).sum(1).cumsum(0)
    return rowptr, cols4[ok].to(torch.int32), w4[ok].contiguous()


def _edges(rowptr, colind):
    """(row, column) of every entry, int64."""
    n = rowptr.numel() - 1
    rows = torch.repeat_interleave(torch.arange(n, device=rowptr.device), (rowptr[1:] - rowptr[:-1]).long())
    return rows, colind.long()


def _pack(bits):
    """A bool vector as LSB-first 32-bit words."""
    pad = torch.zeros(-(-bits.numel() // 32) * 32, dtype=torch.int64, device=bits.device)
    pad[:bits.numel()] = bits
    words = (pad.reshape(-1, 32) << torch.arange(32, device=bits.device)).sum(1)
    return torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32)


def _sources(rowptr, count, seed):
    """Vertices with at least one edge (vertex 0 where there is none)."""
    deg = (rowptr[1:] - rowptr[:-1]).cpu().numpy()
    cand = np.flatnonzero(deg > 0)
    rng = np.random.default_rng(seed)
    return [int(v) for v in rng.choice(cand, size=count)] if cand.size else [0] * count


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
KINDS = {"bool": (B.BOOL_OR_AND, B.VEC_BITS, B.VEC_BITS), "count": (B.PLUS_TIMES, B.VEC_BITS, B.VEC_I32),
         "plus": (B.PLUS_TIMES, B.VEC_F32, B.VEC_F32), "min": (B.MIN_PLUS, B.VEC_I32, B.VEC_I32),
         "max": (B.MAX_TIMES, B.VEC_F32, B.VEC_F32), "minplus": (B.MIN_PLUS, B.VEC_F32, B.VEC_F32)}


def _spmv_vectors(case, nnz, seed):
    """(x, mask as bool or None, weights in CSR order or None); x is a bool vector for the bit schemes."""
    dev, gen, n, sr = _device(), _generator(seed + 1), case["n"], case["semiring"]
    if sr in ("bool", "count"):
        x = torch.rand(n, generator=gen, device=dev) < 0.1
    elif sr == "min":
        x = torch.randperm(n, generator=gen, device=dev).to(torch.int32)
    else:
        x = torch.rand(n, generator=gen, device=dev)
    mask = None if case["mask"] == "none" else torch.rand(n, generator=gen, device=dev) < 0.5
    w = torch.rand(nnz, generator=gen, device=dev) * 99.0 + 1.0 if sr == "minplus" else None
    return x, mask, w


def prepare(case, seed):
    op, dev = case["op"], _device()
    if op == "sssp":
        rowptr, colind, w = _grid(case["rows"], case["cols"], seed)
        n = rowptr.numel() - 1
        m = B.b2sr_from_csr(n, rowptr, colind, case["k"])
        return {"case": case, "m": m, "w": B.b2sr_weights_from_csr(m, rowptr, colind, w)}
    if op == "serve":
        server = B.Server(64 << 30, 64, 2)
        mats, srcs = [], []
        for i in range(case["graphs"]):
            n = 1 << (case["lo"] + i % (case["hi"] - case["lo"] + 1))
            rowptr, colind = _rmat(n, case["ef"], False, 1000 * seed + i)
            mats.append(B.b2sr_from_csr(n, rowptr, colind, case["k"]))
            B.b2sr_set_schedule(mats[-1], case["schedule"])
            server.add_graph(mats[-1])
            srcs.append(_sources(rowptr, case["queries"], seed + i))
        queries, outs = [], []
        for q in range(case["queries"]):
            gid = q // 2 % case["graphs"]  # a BFS and a PageRank query per graph, round and round
            queries.append((gid, q % 2 == 0, srcs[gid][q]))
        # one result matrix per graph and kind, a row per query
        for gid in range(case["graphs"]):
            n = mats[gid].n
            outs.append([torch.empty((sum(1 for x in queries if x[0] == gid and x[1] == bfs), n), device=dev,
                                     dtype=torch.int32 if bfs else torch.float32) for bfs in (True, False)])
        return {"case": case, "server": server, "mats": mats, "queries": queries, "outs": outs}
    rowptr, colind = _graph(case, seed)
    if op == "from_csr":
        return {"case": case, "rowptr": rowptr, "colind": colind}
    m = B.b2sr_from_csr(case["n"], rowptr, colind, case["k"])
    st = {"case": case, "m": m}
    if "schedule" in case:
        B.b2sr_set_schedule(m, case["schedule"])
    if op == "spmv":
        x, mask, w = _spmv_vectors(case, colind.numel(), seed)
        bits = case["semiring"] in ("bool", "count")
        st["x"] = _pack(x) if bits else x
        st["mask"] = None if mask is None else _pack(mask)
        st["w"] = None if w is None else B.b2sr_weights_from_csr(m, rowptr, colind, w)
        kind = {"bool": torch.int32, "count": torch.int32, "min": torch.int32}.get(case["semiring"], torch.float32)
        size = B.bitset_words(case["n"]) if case["semiring"] == "bool" else case["n"]
        st["y"] = torch.empty(size, dtype=kind, device=dev)
    elif op == "bfs":
        st["src"] = _sources(rowptr, 1, seed)[0]
    elif op == "bfs_multi":
        st["srcs"] = _sources(rowptr, case["nsrc"], seed)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(st):
    case = st["case"]
    op = case["op"]
    if op == "spmv":
        semiring, kin, kout = KINDS[case["semiring"]]
        return B.b2sr_spmv(st["m"], semiring, kin, st["x"], kout, st["y"], st["mask"], case["mask"] == "complement",
                           st["w"])
    if op == "pagerank":
        return B.b2sr_pagerank(st["m"], 0.85, case["iters"])
    if op == "from_csr":
        with B.b2sr_from_csr(case["n"], st["rowptr"], st["colind"], case["k"]) as m:
            return B.b2sr_export(m)
    if op == "to_csr":
        return B.b2sr_to_csr(st["m"])
    if op == "bfs":
        return B.b2sr_bfs(st["m"], st["src"])
    if op == "bfs_multi":
        return B.b2sr_bfs_multi(st["m"], st["srcs"])
    if op == "tc":
        return B.b2sr_tc(st["m"])
    if op == "sssp":
        return B.b2sr_sssp_push(st["m"], 0, st["w"], delta=case["delta"])
    server, used, ids = st["server"], {}, []
    for gid, bfs, src in st["queries"]:
        row = used.get((gid, bfs), 0)
        used[(gid, bfs)] = row + 1
        if bfs:
            ids.append(server.submit_bfs(gid, src, st["outs"][gid][0][row])[0])
        else:
            ids.append(server.submit_pagerank(gid, src, 0.85, case["iters"], st["outs"][gid][1][row])[0])
    for qid in ids:
        server.wait(qid)
    return st["outs"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=64)
def _matrix_bytes(n, ef, perm, k):
    """(CSR bytes, B2SR bytes, entries) of the graph of one seed; other seeds differ by a fraction of a percent."""
    rowptr, colind = _rmat(n, ef, perm, 1)
    rows, cols = _edges(rowptr, colind)
    ntr = -(-n // k)
    tiles = int(torch.unique((rows // k) * ntr + cols // k).numel())
    word = {4: 1, 8: 1, 16: 2, 32: 4}[k]
    return 4.0 * (n + 1 + colind.numel()), 4.0 * (ntr + 1) + tiles * (4.0 + k * word), float(colind.numel())


def work(case):
    """Bytes: the matrix once (once an iteration where it is larger than the
    last-level cache), inputs and results once.  Flops: additions, minima or
    ANDs of one bit each with one value, where the count is known in advance."""
    op = case["op"]
    if op == "sssp":
        n, k = case["rows"] * case["cols"], case["k"]
        nnz = 4.0 * n - 2 * case["rows"] - 2 * case["cols"]
        word = {4: 1, 8: 1, 16: 2, 32: 4}[k]
        tiles = 5.0 * n / k  # the diagonal tile and its four neighbours
        return {"bytes": 4.0 * n / k + tiles * (4 + k * word) + 4 * nnz + 4.0 * n, "flops": nnz}
    if op == "serve":
        total = flops = 0.0
        for i in range(case["graphs"]):
            n = 1 << (case["lo"] + i % (case["hi"] - case["lo"] + 1))
            _, mat, nnz = _matrix_bytes(n, case["ef"], False, case["k"])
            each = case["queries"] / case["graphs"]
            total += mat + each * 4.0 * n
            flops += each / 2 * nnz * case["iters"]
        return {"bytes": total, "flops": flops}
    n = case["n"]
    csr, mat, nnz = _matrix_bytes(n, case["ef"], case["perm"], case["k"])
    if op in ("from_csr", "to_csr"):
        return {"bytes": csr + mat, "flops": 0.0}
    if op == "spmv":
        bits = {"bool": (1 / 8, 1 / 8), "count": (1 / 8, 4)}.get(case["semiring"], (4, 4))
        mask = 0.0 if case["mask"] == "none" else n / 8
        w = 4.0 * nnz if case["semiring"] == "minplus" else 0.0
        return {"bytes": mat + n * sum(bits) + mask + w, "flops": nnz}
    if op == "pagerank":
        passes = case["iters"] if mat > L2_BYTES else 1
        return {"bytes": mat * passes + 4.0 * n, "flops": nnz * case["iters"]}
    if op == "tc":
        return {"bytes": mat, "flops": nnz}
    return {"bytes": mat + 4.0 * n * case.get("nsrc", 1), "flops": nnz}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------
def _exact_pagerank(rowptr, colind, iters, teleport=None):
    n = rowptr.numel() - 1
    rows, cols = _edges(rowptr, colind)
    out = torch.zeros(n, dtype=torch.float64, device=rowptr.device).index_add_(
        0, cols, torch.ones_like(cols, dtype=torch.float64))
    t = torch.full_like(out, 1.0 / n) if teleport is None else teleport
    x = torch.full_like(out, 1.0 / n)
    for _ in range(iters):
        c = torch.where(out > 0, x / out.clamp(min=1.0), torch.zeros_like(x))
        x = 0.15 * t + 0.85 * torch.zeros_like(x).index_add_(0, rows, c[cols])
    return x


def _exact_sssp(rows, cols, right, down):
    right, down = right.double(), down.double()
    d = torch.full((rows, cols), float("inf"), dtype=torch.float64, device=right.device)
    d[0, 0] = 0.0
    while True:
        before = d.clone()
        for _ in range(64):
            torch.minimum(d[:, 1:], d[:, :-1] + right, out=d[:, 1:])
            torch.minimum(d[:, :-1], d[:, 1:] + right, out=d[:, :-1])
            torch.minimum(d[1:], d[:-1] + down, out=d[1:])
            torch.minimum(d[:-1], d[1:] + down, out=d[:-1])
        if torch.equal(before, d):
            return d.reshape(-1)


def exact(case, seed):
    """fp32 results in 64 bits, and the arrays that plain tensor code gives
    at once; levels, decoded arrays and the triangle count are whole numbers,
    equal to another run's or wrong, and have None here."""
    op = case["op"]
    if op == "sssp":
        return _exact_sssp(case["rows"], case["cols"], *_grid_weights(case["rows"], case["cols"], seed))
    if op == "serve":
        csrs, srcs, outs = [], [], []
        for i in range(case["graphs"]):
            n = 1 << (case["lo"] + i % (case["hi"] - case["lo"] + 1))
            csrs.append(_rmat(n, case["ef"], False, 1000 * seed + i))
            srcs.append(_sources(csrs[-1][0], case["queries"], seed + i))
            outs.append([None, []])
        for q in range(case["queries"]):
            gid = q // 2 % case["graphs"]
            if q % 2 == 0:
                continue
            t = torch.zeros(csrs[gid][0].numel() - 1, dtype=torch.float64, device=_device())
            t[srcs[gid][q]] = 1.0
            outs[gid][1].append(_exact_pagerank(*csrs[gid], case["iters"], t))
        for gid, o in enumerate(outs):
            o[1] = torch.stack(o[1]) if o[1] else torch.empty((0, csrs[gid][0].numel() - 1), dtype=torch.float64)
        return outs
    if op not in ("spmv", "pagerank", "to_csr"):
        return None
    rowptr, colind = _graph(case, seed)
    if op == "to_csr":
        return rowptr, colind
    if op == "pagerank":
        return _exact_pagerank(rowptr, colind, case["iters"])
    n, sr = case["n"], case["semiring"]
    x, mask, w = _spmv_vectors(case, colind.numel(), seed)
    rows, cols = _edges(rowptr, colind)
    if sr in ("bool", "count", "plus"):
        fill = 0.0
        y = torch.zeros(n, dtype=torch.float64, device=x.device).index_add_(0, rows, x.double()[cols])
    else:
        fill = -float("inf") if sr == "max" else float(2**31 - 1) if sr == "min" else float("inf")
        y = torch.full((n,), fill, dtype=torch.float64, device=x.device) if sr == "max" else x.double()
        v = x.double()[cols] if w is None else x.double()[cols] + w.double()
        y = y.scatter_reduce(0, rows, v, "amax" if sr == "max" else "amin")
    if mask is not None:
        y = torch.where(mask != (case["mask"] == "complement"), y, torch.full_like(y, fill))
    if sr == "bool":
        return _pack(y > 0)
    return y.to(torch.int32) if sr in ("count", "min") else y
