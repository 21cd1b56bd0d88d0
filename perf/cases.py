"""The work that users of this library have it do, as cases that can be timed.

Each case is one call (or one short exchange with the server) through the
public entry points, on synthetic data with the types, dimensions and index
parameters of the repository's configurations: SIFT-like uint8 d = 128,
Deep-like float32 d = 96, MSSPACEV-like int8 d = 100, PQ with 32 to 74
subspaces, graphs of degree 32 to 68.

A search case's index is made from the case alone (a user keeps one index and
sends it ever new queries); the seed gives the queries and, in the batched form,
their k and L (served: their L).  The build and ground-truth cases take all
their inputs from the seed.  The arrays of an index (vectors, PQ, graph) are
kept by this module once built; every state loads its own handle from them.
"""
import math
import random

import numpy as np
import torch

import paper_2401_11324_gb300 as bang

DTYPES = {"u8": torch.uint8, "i8": torch.int8, "f32": torch.float32}
NP = {"u8": np.uint8, "i8": np.int8, "f32": np.float32}
SIZE = {"u8": 1, "i8": 1, "f32": 4}
PLACEMENTS = {
    "host": 0,
    "host-packed": bang.BANG_GRAPH_PACKED,
    "host-records": bang.BANG_GRAPH_PACKED | bang.BANG_NODE_RECORDS,
    "hbm-vectors": bang.BANG_VECTORS_IN_HBM,
    "hbm": bang.BANG_GRAPH_IN_HBM | bang.BANG_VECTORS_IN_HBM,
    "hbm-packed": bang.BANG_GRAPH_IN_HBM | bang.BANG_VECTORS_IN_HBM | bang.BANG_GRAPH_PACKED,
}
MODES = {"f32": bang.BANG_MODE_PQ_F32, "bf16": bang.BANG_MODE_PQ_BF16,
         "exact": bang.BANG_MODE_EXACT, "q8": bang.BANG_MODE_PQ_Q8}


def _search(name, n, dtype, d, M, R, nq, k, L, mode="f32", place="hbm", bloom=16, early=0,
            rerank=0, source=0, buffers="device"):
    return dict(name=name, kind="search", n=n, dtype=dtype, d=d, M=M, R=R, nq=nq, k=k, L=L,
                mode=mode, place=place, bloom=bloom, early=early, rerank=rerank, source=source,
                buffers=buffers)


def listed():
    return [
        # one lookup of an online service, every setting left at its default
        _search("one query", 1_000_000, "u8", 128, 32, 64, nq=1, k=10, L=64),
        # the plain method at its smallest: 10,000 float points read in place
        # from host memory, 100 queries, host arrays in and out
        _search("small float, host arrays", 10_000, "f32", 128, 32, 32, nq=100, k=10, L=64,
                place="host", buffers="host"),
        # the benchmark's headline: a 10,000-query batch, FP32 table, graph and
        # vectors in HBM, early code rows, staged re-rank, L = 224
        _search("batch fp32 staged", 1_000_000, "u8", 128, 32, 64, nq=10_000, k=10, L=224,
                early=1, rerank=1),
        # the paper's placement with what the autotuner picks there: graph
        # (packed rows) and vectors in host memory, 8-bit table, 2^15-bit filter
        _search("batch q8 host packed", 1_000_000, "u8", 128, 32, 64, nq=10_000, k=10, L=160,
                mode="q8", place="host-packed", bloom=15),
        # the Exact-distance variant (no PQ in the loop) from HBM
        _search("batch exact", 1_000_000, "u8", 128, 32, 64, nq=10_000, k=10, L=48, mode="exact"),
        # float vectors of 96 dimensions, 48 subspaces, rows of 68 neighbours
        _search("batch float d=96", 300_000, "f32", 96, 48, 68, nq=3_000, k=10, L=128),
        # uneven k and L in one persistent launch: int8, d = 100, M = 50, 8-bit table
        dict(name="batched mix int8", kind="batched", n=500_000, dtype="i8", d=100, M=50, R=64,
             nq=10_000, kmax=100, Lmin=32, Lmax=256, mode="q8", place="hbm", bloom=16, early=0),
        # the server: BF16 table, requests of 1 to 1,024 queries, k = 10, L = 64 to 256
        dict(name="served bf16", kind="serve", n=1_000_000, dtype="u8", d=128, M=32, R=64,
             requests=24, most=1024, k=10, Lmin=64, Lmax=256, mode="bf16", place="hbm", bloom=16,
             early=1),
        # PQ tables of a batch on the tensor cores, FP32 out
        dict(name="pq tables", kind="tables", n=20_000, dtype="u8", d=128, M=32, nq=10_000, form=0),
        # exact 100 nearest neighbours of a query set, to measure recall against
        dict(name="ground truth", kind="truth", n=1_000_000, dtype="u8", d=128, nq=10_000, k=100),
        # index build, first half: PQ training and encoding
        dict(name="build pq", kind="pq", n=400_000, dtype="u8", d=128, M=32, ns=100_000, iters=10),
        # index build, second half: the overlapping-shard graph
        dict(name="build graph", kind="graph", n=200_000, dtype="u8", d=128, R=64, Lb=64, shards=8,
             ell=2),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng):
    """An element type with a dimension and subspace count that goes with it."""
    return rng.choice([("u8", 128, 32), ("u8", 128, 32), ("u8", 128, 64), ("u8", 130, 32),
                       ("u8", 128, 74), ("u8", 97, 30), ("i8", 100, 50), ("i8", 100, 30),
                       ("f32", 96, 48), ("f32", 128, 32), ("f32", 200, 50)])


def draw(rng):
    kind = rng.choice(["search"] * 6 + ["batched", "serve", "tables", "truth", "pq", "graph"])
    dtype, d, M = _shape(rng)
    if kind == "truth":
        n = _logint(rng, 10_000, 600_000)
        # float distances are FP64 sums, bytes without a 16-byte row are read one by one
        pairs = 1.5e8 if dtype == "f32" else 5e9 if d % 16 == 0 else 8e8
        return dict(kind=kind, n=n, dtype=dtype, d=d, nq=_logint(rng, 10, min(10_000, pairs / n)),
                    k=rng.choice([1, 10, 37, 100]))
    if kind == "pq":
        if dtype == "f32":
            d, M = 96, 48
        return dict(kind=kind, n=_logint(rng, 20_000, 400_000), dtype=dtype, d=d, M=M,
                    ns=_logint(rng, 1_000, 20_000 if M > 32 else 50_000), iters=rng.randint(2, 10))
    if kind == "graph":
        d = min(d, 130)
        ell = rng.choice([1, 2])
        return dict(kind=kind, n=_logint(rng, 5_000, 100_000 if dtype != "f32" else 15_000),
                    dtype=dtype, d=d, R=rng.choice([32, 48, 64]), Lb=rng.choice([32, 64, 100]),
                    shards=rng.choice([2, 4, 9, 16]), ell=ell)
    if kind == "tables":
        return dict(kind=kind, n=rng.randint(5_000, 30_000), dtype=dtype, d=d, M=M,
                    nq=_logint(rng, 1, 6_000), form=rng.choice([0, 0, 1, 2]))
    n = _logint(rng, 10_000, 200_000)
    R = rng.choice([32, 64, 64, 68])
    place = rng.choice(["host", "host-packed", "host-records", "hbm", "hbm", "hbm", "hbm-packed",
                        "hbm-vectors"])
    mode = rng.choice(["f32", "f32", "bf16", "q8", "exact"])
    early = rng.choice([0, 1])
    bloom = rng.choice([14, 15, 16, 16, 17]) if M <= 50 else 15
    if kind == "serve":
        return dict(kind=kind, n=n, dtype=dtype, d=d, M=M, R=R, requests=rng.randint(3, 24),
                    most=rng.randint(16, 512), k=rng.choice([1, 10, 20]), Lmin=32,
                    Lmax=rng.randint(40, 200), mode=mode, place=place, bloom=bloom, early=early)
    if kind == "batched":
        return dict(kind=kind, n=n, dtype=dtype, d=d, M=M, R=R, nq=_logint(rng, 5, 6_000),
                    kmax=rng.choice([10, 100]), Lmin=rng.choice([16, 32]),
                    Lmax=rng.randint(100, 256), mode=mode, place=place, bloom=bloom, early=early)
    k = rng.choice([1, 5, 10, 10, 10, 40, 100])
    L = max(k, _logint(rng, 16, 400))
    nq = _logint(rng, 1, min(10_000, 600_000 / L))
    rerank = 0 if mode == "exact" else rng.choice([0, 0, 1, 2])
    source = rng.choice([0, 0, 0, 1]) if mode in ("f32", "bf16") and nq <= 3000 else 0
    c = _search("", n, dtype, d, M, R, nq, k, L, mode, place, bloom, early, rerank, source,
                rng.choice(["device", "device", "host"]))
    del c["name"]
    return c


# ---- data: low-rank mixture components like SIFT descriptors (the uint8 and
# int8 configurations), unit vectors around unit centres (the float one)

def _data(seed, n, nq, dtype, d):
    """n points and nq queries of one mixture."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    ncomp, rank = max(4, n // 4000), 12

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda")

    if dtype == "f32":
        cen = torch.nn.functional.normalize(normal(ncomp, d), dim=1)
    else:
        u = torch.rand(ncomp, d, generator=g, device="cuda")
        cen = u * 255.0 if dtype == "u8" else u * 200.0 - 100.0
        fac = normal(ncomp, rank, d) * ((20.0 if dtype == "u8" else 16.0) / rank ** 0.5)

    def points(m):
        out = torch.empty(m, d, dtype=DTYPES[dtype], device="cuda")
        for i in range(0, m, 65536):
            c = min(m, i + 65536) - i
            lab = torch.randint(0, ncomp, (c,), generator=g, device="cuda")
            if dtype == "f32":
                x = torch.nn.functional.normalize(cen[lab] + 0.1 * normal(c, d), dim=1)
            else:
                x = cen[lab] + 4.0 * normal(c, d)
                # sorted by component, so that a component's factors are read once
                z, order = normal(c, rank), torch.argsort(lab)
                x[order] += torch.bmm(z[order].unsqueeze(1), fac[lab[order]]).squeeze(1)
                x = x.round().clamp(*((0, 255) if dtype == "u8" else (-128, 127)))
            out[i:i + c] = x.to(DTYPES[dtype])
        return out

    return points(n), points(nq) if nq else None


def _queries(seed, like, nq):
    """Queries around points of the index: a point moved by a little noise."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = like[torch.randint(0, like.shape[0], (nq,), generator=g, device="cuda")].float()
    noise = torch.randn(x.shape, generator=g, device="cuda")
    if like.dtype == torch.float32:
        return torch.nn.functional.normalize(x + 0.03 * noise, dim=1)
    lo, hi = (0, 255) if like.dtype == torch.uint8 else (-128, 127)
    return (x + 6.0 * noise).round().clamp(lo, hi).to(like.dtype)


def _pq_choices(seed, n, M, ns):
    rng = np.random.default_rng(seed)
    sample = np.sort(rng.choice(n, size=min(n, ns), replace=False)).astype(np.uint64)
    init = np.stack([sample[rng.choice(len(sample), size=256, replace=False)] for _ in range(M)])
    return sample, np.ascontiguousarray(init.astype(np.uint64))


def _centres(seed, base, S):
    g = torch.Generator(device="cuda").manual_seed(seed)
    at = torch.randperm(base.shape[0], generator=g, device="cuda")[:S]
    return base[at].float().cpu().numpy()


_INDEXES = {}          # index arrays by what they are made from; the last three


def _index_arrays(c):
    R = c.get("R", 0)
    key = (c["n"], c["dtype"], c["d"], c["M"], R)
    if key not in _INDEXES:
        while len(_INDEXES) >= 3:
            del _INDEXES[next(iter(_INDEXES))]
        base, _ = _data(1000 + c["d"], c["n"], 0, c["dtype"], c["d"])
        sample, init = _pq_choices(3000, c["n"], c["M"], 20_000)
        codebook, codes = bang.bang_build_pq(base, c["M"], sample, init, 8)
        if R:
            # two shards for each point, as the large configurations have
            S = max(2, c["n"] // 50_000)
            adj, _ = bang.bang_build_shard_graph(base, _centres(4000, base, S), 2, R, 64, 1.2)
        else:
            adj = None
        mean = base.float().mean(dim=0)
        medoid = int((base.float() - mean).square().sum(dim=1).argmin())
        _INDEXES[key] = dict(base=base.cpu().numpy(), codebook=codebook, codes=codes, adj=adj,
                             medoid=medoid)
    return _INDEXES[key]


class _State:
    """A user's objects around one case: the index handle and the buffers."""

    def __init__(self, case):
        self.case = case
        self.index = self.server = self.handle = None

    def load(self, arrays, place):
        c = self.case
        base = bang.host_empty(arrays["base"].shape, NP[c["dtype"]])
        base[:] = arrays["base"]
        adj = bang.host_empty(arrays["adj"].shape, np.uint32)
        adj[:] = arrays["adj"]
        self.index = bang.Index(base, arrays["codebook"], arrays["codes"], adj, arrays["medoid"],
                                c["M"])
        if PLACEMENTS[place]:
            self.index.set_placement(PLACEMENTS[place])

    def __del__(self):
        if self.server is not None:
            self.server.stop()
        if self.index is not None:
            self.index.close()
        if self.handle is not None:
            bang.bang_destroy(self.handle)


def _request_sizes(case):
    """The requests' query counts, small and large ones alike: the same for every seed."""
    r = random.Random(case["requests"] * 10_000 + case["most"])
    return [_logint(r, 1, case["most"]) for _ in range(case["requests"])]


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    if kind == "truth":
        s.base, s.queries = _data(seed, case["n"], case["nq"], case["dtype"], case["d"])
        return s
    if kind == "pq":
        s.base, _ = _data(seed, case["n"], 0, case["dtype"], case["d"])
        s.sample, s.init = _pq_choices(seed, case["n"], case["M"], case["ns"])
        return s
    if kind == "graph":
        s.base, _ = _data(seed, case["n"], 0, case["dtype"], case["d"])
        s.centres = _centres(seed, s.base, case["shards"])
        s.adj = torch.empty(case["n"], case["R"], dtype=torch.int32, device="cuda")
        return s
    a = _index_arrays(case)
    like = torch.from_numpy(a["base"]).cuda()
    if kind == "tables":
        # the tables need the PQ data and the element type: no graph
        s.queries = _queries(seed, like, case["nq"])
        s.handle = bang.bang_create(0)
        bang.bang_load_pq(s.handle, case["d"], case["M"], a["codebook"], a["codes"], case["n"])
        s.keep = bang.host_empty(a["base"].shape, NP[case["dtype"]])
        s.keep[:] = a["base"]
        bang.bang_register_vectors(s.handle, s.keep, bang._DTYPES[np.dtype(NP[case["dtype"]])])
        out = torch.bfloat16 if case["form"] & 1 else torch.float32
        s.out = torch.empty(case["nq"], case["M"], 256, dtype=out, device="cuda")
        return s
    s.load(a, case["place"])
    rng = np.random.default_rng(seed)
    if kind == "serve":
        s.server = bang.Server(s.index, case["k"], case["Lmax"], max_batch=1024, streams=8,
                               mode=MODES[case["mode"]], bloom_log2=case["bloom"],
                               early_codes=case["early"])
        s.requests = []
        for nq in _request_sizes(case):
            q = _queries(int(rng.integers(1 << 30)), like, nq).cpu().numpy()
            k = np.full(nq, case["k"], np.uint32)
            L = rng.integers(max(case["Lmin"], case["k"]), case["Lmax"] + 1, nq).astype(np.uint32)
            s.requests.append((q, k, L))
        return s
    s.queries = _queries(seed, like, case["nq"])
    k = case["kmax"] if kind == "batched" else case["k"]
    s.ids = torch.empty(case["nq"], k, dtype=torch.int32, device="cuda")
    s.dist = torch.empty(case["nq"], k, dtype=torch.float32, device="cuda")
    if kind == "batched":
        ks = rng.choice([x for x in (1, 10, 100) if x <= case["kmax"]], case["nq"])
        Ls = np.maximum(rng.integers(case["Lmin"], case["Lmax"] + 1, case["nq"]), ks)
        s.k = torch.from_numpy(ks.astype(np.int32)).cuda()
        s.L = torch.from_numpy(Ls.astype(np.int32)).cuda()
        s.params = bang.make_params(mode=MODES[case["mode"]], bloom_log2=case["bloom"],
                                    early_codes=case["early"])
        return s
    if case["buffers"] == "host":
        s.queries = s.queries.cpu().numpy()
        s.ids = np.empty((case["nq"], k), np.uint32)
        s.dist = np.empty((case["nq"], k), np.float32)
    s.params = bang.make_params(mode=MODES[case["mode"]], bloom_log2=case["bloom"],
                                early_codes=case["early"], rerank=case["rerank"],
                                table_source=case["source"])
    return s


def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "search":
        s.index.search(s.queries, c["k"], c["L"], s.ids, s.dist, s.params)
        return {"ids": s.ids, "dist": s.dist}
    if kind == "batched":
        s.index.search_batched(s.queries, s.k, s.L, c["kmax"], c["Lmax"], s.ids, s.dist, s.params)
        return {"ids": s.ids, "dist": s.dist}
    if kind == "serve":
        tickets = [s.server.submit(*r) for r in s.requests]
        got = [s.server.wait(t) for t in tickets]
        return {"ids": np.concatenate([g[0] for g in got]).view(np.int32),
                "dist": np.concatenate([g[1] for g in got])}
    if kind == "tables":
        bang.bang_pq_tables(s.handle, s.queries, c["nq"], s.out, c["form"])
        return {"tables": s.out}
    if kind == "truth":
        ids, dist = bang.bang_ground_truth(s.base, s.queries, c["k"])
        return {"ids": ids.view(np.int32), "dist": dist}
    if kind == "pq":
        codebook, codes = bang.bang_build_pq(s.base, c["M"], s.sample, s.init, c["iters"])
        return {"codebook": codebook, "codes": codes}
    adj, shard_of = bang.bang_build_shard_graph(s.base, s.centres, c["ell"], c["R"], c["Lb"], 1.2,
                                                adj=s.adj)
    return {"adj": adj, "shard_of": shard_of.view(np.int32)}


def work(case):
    n, d, e = case["n"], case["d"], SIZE[case["dtype"]]
    kind = case["kind"]
    if kind == "truth":
        # a product and a sum for each dimension of each pair
        return {"bytes": (n + case["nq"]) * d * e + 12 * case["nq"] * case["k"],
                "flops": 2.0 * n * case["nq"] * d}
    if kind == "pq":
        # every point against the 256 centroids of each subspace (the encoding),
        # and the sample in each iteration
        return {"bytes": n * d * e + case["ns"] * d * e + 1024 * d + n * case["M"],
                "flops": 2.0 * 256 * d * (n + case["ns"] * case["iters"])}
    if kind == "graph":
        # each member is searched and pruned once in each of two passes: about
        # 1.3 Lb expansions of which some 15 neighbours are new
        m = n * case["ell"]
        return {"bytes": n * d * e + 4.0 * n * (case["R"] + case["ell"]),
                "flops": 2 * m * 1.3 * case["Lb"] * 15 * 2.0 * d}
    if kind == "tables":
        return {"bytes": case["nq"] * (d * e + case["M"] * 256 * (2 if case["form"] & 1 else 4)) +
                1024 * d, "flops": 2.0 * 256 * d * case["nq"]}
    if kind == "serve":
        nq = sum(_request_sizes(case))
        L, k = 0.5 * (max(case["Lmin"], case["k"]) + case["Lmax"]), case["k"]
    elif kind == "batched":
        nq, L, k = case["nq"], 0.5 * (case["Lmin"] + case["Lmax"]), case["kmax"]
    else:
        nq, L, k = case["nq"], case["L"], case["k"]
    # every worklist entry is expanded: its row and vector are read, and some 18
    # of its neighbours are new and measured; no more than the index is read
    new = nq * L * 18.0
    per = nq * L * (4 * case["R"] + d * e) + new * (d * e if case["mode"] == "exact" else case["M"])
    whole = n * (4.0 * case["R"] + d * e + case["M"])
    flops = new * (3 * d if case["mode"] == "exact" else case["M"]) + nq * 3.0 * d * (
        L + (0 if case["mode"] == "exact" else 256))
    return {"bytes": nq * (d * e + 8.0 * k) + min(per, whole), "flops": flops}


def exact(case, seed):
    kind = case["kind"]
    if kind == "tables":
        s = prepare(case, seed)
        a = _index_arrays(case)
        q = s.queries.double()
        cb = torch.from_numpy(a["codebook"]).cuda().double()
        out = torch.empty(case["nq"], case["M"], 256, dtype=torch.float64, device="cuda")
        for m, o, w in _subspaces(case["d"], case["M"]):
            cent = cb[256 * o:256 * (o + w)].view(256, w)
            out[:, m] = (q[:, None, o:o + w] - cent[None]).square().sum(dim=2)
        return {"tables": out}
    if kind == "truth":
        s = prepare(case, seed)
        x, q, k = s.base.double(), s.queries.double(), min(case["k"], case["n"])
        xx = x.square().sum(dim=1)
        dist = torch.full((case["nq"], case["k"]), float("inf"), dtype=torch.float64, device="cuda")
        step = max(1, 200_000_000 // case["n"])
        for i in range(0, case["nq"], step):
            p = q[i:i + step]
            near = (xx[None] - 2.0 * (p @ x.T)).topk(min(k + 16, case["n"]), largest=False).indices
            full = (x[near] - p[:, None]).square().sum(dim=2)
            dist[i:i + step, :k] = full.sort(dim=1).values[:, :k]
        return {"ids": None, "dist": dist}
    if kind == "pq":
        s = prepare(case, seed)
        at = torch.from_numpy(s.sample.astype(np.int64)).cuda()
        x = s.base[at].double()
        out = torch.empty(256 * case["d"], dtype=torch.float64, device="cuda")
        init = torch.from_numpy(s.init.astype(np.int64)).cuda()
        for m, o, w in _subspaces(case["d"], case["M"]):
            y = x[:, o:o + w].contiguous()
            cent = s.base[init[m], o:o + w].double()
            for _ in range(case["iters"]):
                lab = torch.cat([(p[:, None] - cent[None]).square().sum(dim=2).argmin(dim=1)
                                 for p in y.split(16384)])
                count = torch.bincount(lab, minlength=256).double()
                total = torch.zeros_like(cent).index_add_(0, lab, y)
                cent = torch.where(count[:, None] > 0, total / count.clamp(min=1)[:, None], cent)
            out[256 * o:256 * (o + w)] = cent.reshape(-1)
        return {"codebook": out, "codes": None}
    # a search's result depends on the order of its own visits, a graph is ids only
    return None


def _subspaces(d, M):
    o = 0
    for m in range(M):
        w = d // M + (1 if m < d % M else 0)
        yield m, o, w
        o += w
