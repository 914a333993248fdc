"""Timed cases: what a program that mines frequent itemsets, joins set families
or answers set queries with this library asks of it, over the range of sizes
that the repository's workloads (datagen), tests and benchmark span.

Every case goes through the public entry points with tidlists resident in HBM
(the host case: in pinned host memory) and the library's computed permutations.
Output buffers are the caller's and are reused from pass to pass, as the
benchmark does; a list of frequent itemsets comes back as the whole buffer, whose
rows past the number found keep the zeros it was made with.  A mining pass is
build + supports + free: a new instance needs all three.  Serving and itemset
queries run on a pool or set that stays.
"""
import math

import numpy as np
import torch

import paper_1102_1003_gb300 as pkg

# Limits of a drawn case: no dearer than the dearest listed one, in expected
# element-pair incidences and in BatMap words compared.
_MAX_WORDS = 4096 * 4095 / 2 * 3 * 2.0 ** 19 / 4
_MAX_TIDS = 4096 * 0.05 * 4_194_304


def listed():
    return [
        # A small instance mined on demand (the m = 10,000, n = 200 workload of
        # the tests): latency and launches count.
        _mine("mine-bern-m10k-n200", 10_000, 200, 0.05, "bernoulli", 25),
        # Retail-like skew (the Zipf workload): nine width classes, 40 M tids.
        _mine("mine-zipf-m1m-n2000", 1_000_000, 2_000, 0.02, "zipf", 1_000),
        # The density sweep at 5% (the benchmark's default line) with half its items:
        # one width class, 8.6e8 tids, the largest case.
        _mine("mine-bern-m4m-n4096-p5", 4_194_304, 4_096, 0.05, "bernoulli", 4_195),
        # Many items, few transactions (the n-sweep: 10^7 items in all at 5%):
        # the output, n^2 supports, is the largest part of the traffic.
        _mine("mine-nsweep-n8000", 25_000, 8_000, 0.05, "bernoulli", 25),
        # Two families (sparse boolean matrix product, join-project).
        {"name": "cross-m1m-2000x4000", "kind": "cross", "m": 1_000_000, "n_a": 2_000, "n_b": 4_000,
         "density": 0.01, "p_b": 0.002, "s": 1},
        # Many instances kept built, their supports in one batched pass.
        {"name": "batch-16", "kind": "batch", "k": 16, "spec_seed": 1000},
        # The dense-bitmap call on the Zipf workload.
        {"name": "dense-zipf-m1m-n2000", "kind": "dense", "m": 1_000_000, "n": 2_000, "density": 0.02,
         "shape": "zipf", "s": 1_000},
        # Frequent itemsets of size 3: pairs, then triples on a 3-of-4 set.
        {"name": "triples-m100k-n1000", "kind": "triples", "m": 100_000, "n": 1_000, "density": 0.02,
         "shape": "zipf", "s": 100},
        # ... and of size 4, on a 4-of-5 set, from the frequent pairs.
        {"name": "quads-m100k-n1000", "kind": "quads", "m": 100_000, "n": 1_000, "density": 0.02,
         "shape": "zipf", "s": 100},
        # Supports of given itemsets on a set that is kept (rule checking).
        {"name": "itemsets-k3-q20001", "kind": "itemsets", "m": 100_000, "n": 1_000, "density": 0.02,
         "shape": "zipf", "d": 3, "k": 3, "n_q": 20_001},
        # Conjunctive queries on a resident pool: counts of all, elements of some.
        {"name": "queries-u64m-q4096", "kind": "queries", "m": 1 << 26, "n": 4_000, "lo": 10, "hi": 1_000_000,
         "n_q": 4_096, "n_list": 256},
        # One call from host buffers, copies inside (a program with no device data).
        {"name": "host-zipf-m1m-n2000", "kind": "host", "m": 1_000_000, "n": 2_000, "density": 0.02,
         "shape": "zipf", "s": 1_000},
    ]


def _mine(name, m, n, density, shape, s):
    return {"name": name, "kind": "mine", "m": m, "n": n, "density": density, "shape": shape, "s": s}


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["mine", "mine", "mine", "cross", "batch", "dense", "triples", "quads", "itemsets", "queries",
                       "host"])
    if kind == "queries":
        return {"kind": kind, "m": log_int(1 << 20, 1 << 26), "n": log_int(100, 4_000), "lo": 10,
                "hi": log_int(10_000, 1_000_000), "n_q": log_int(1, 16_384), "n_list": log_int(1, 300)}
    if kind == "batch":
        return {"kind": kind, "k": rng.randint(2, 16), "spec_seed": rng.randint(1, 10 ** 6)}
    if kind in ("triples", "quads", "itemsets"):
        c = {"kind": kind, "m": log_int(10_000, 150_000), "n": log_int(100, 1_000), "density": rng.uniform(0.005, 0.02),
             "shape": "zipf"}
        if kind == "itemsets":
            c["d"] = rng.choice([3, 4])
            c["k"] = rng.randint(2, c["d"])
            c["n_q"] = log_int(10, 40_000)
        else:
            c["s"] = max(10, int(math.ceil(0.001 * c["m"])))
        return c
    if kind == "cross":
        m = log_int(10_000, 1_000_000)
        return {"kind": kind, "m": m, "n_a": log_int(50, 2_000), "n_b": log_int(50, 4_000),
                "density": rng.uniform(0.002, 0.02), "p_b": math.exp(rng.uniform(math.log(0.001), math.log(0.02))),
                "s": 1}
    m = log_int(5_000, 4_194_304 if kind == "mine" else 1_000_000)
    n = log_int(150, 8_192 if kind == "mine" else 3_000)
    density = math.exp(rng.uniform(math.log(0.001), math.log(0.05)))
    shape = rng.choice(["bernoulli", "zipf"])
    while _words(m, n, density, shape) > _MAX_WORDS or n * density * m > _MAX_TIDS:
        n = int(n * 0.8)
    return {"kind": kind, "m": m, "n": n, "density": density, "shape": shape, "s": int(math.ceil(0.001 * m))}


def _words(m, n, density, shape):
    """BatMap words of all pairs, from above (every pair at the widest of its class)."""
    p = np.sort(_probabilities(n, density, shape))
    r = 2.0 ** np.ceil(np.log2(np.maximum(2 * p * m, max(128, m / 127))))
    return float((np.arange(n) * 3 * r / 4).sum())


# ---- inputs -------------------------------------------------------------------


def _probabilities(n, density, shape):
    """Inclusion probability per rank: uniform, or min(1, c / rank) of the given mean."""
    if shape == "bernoulli":
        return np.full(n, float(density))
    base = 1.0 / np.arange(1, n + 1)
    lo, hi = 0.0, float(n) * n
    for _ in range(200):
        c = 0.5 * (lo + hi)
        lo, hi = (c, hi) if np.minimum(1.0, c * base).sum() < density * n else (lo, c)
    return np.minimum(1.0, 0.5 * (lo + hi) * base)


def _tidlists(m, probs, gen):
    """CSR tidlists on the GPU: item i holds each transaction with probability probs[i]
    (geometric gaps, so the cost is the number of tids)."""
    dev = torch.device("cuda")
    n = len(probs)
    mean = m * probs
    cnt = np.minimum(m + 1, (mean + 6 * np.sqrt(mean) + 16).astype(np.int64))
    offs, parts, start = [np.zeros(1, np.int64)], [], 0
    while start < n:  # blocks of items, to bound the temporaries
        end = start + 1
        while end < n and cnt[start:end + 1].sum() <= 100_000_000:
            end += 1
        c = torch.from_numpy(cnt[start:end]).to(dev)
        lq = np.where(probs[start:end] >= 1.0, -np.inf, np.log1p(-np.minimum(probs[start:end], 1 - 1e-16)))
        lq = torch.repeat_interleave(torch.from_numpy(lq).to(dev), c)
        gaps = torch.rand(lq.numel(), generator=gen, device=dev, dtype=torch.float64).clamp_(min=1e-300).log_()
        gaps = gaps.div_(lq).ceil_().clamp_(min=1.0, max=float(m + 1)).to(torch.int64)
        del lq
        pos = torch.cumsum(gaps, 0)
        ends = torch.cumsum(c, 0)
        before = torch.cat([torch.zeros(1, dtype=torch.int64, device=dev), pos[ends[:-1] - 1]])
        pos -= torch.repeat_interleave(before, c) + 1
        keep = pos < m
        kept = torch.cumsum(keep, 0)[ends - 1]
        parts.append(pos[keep].to(torch.int32))
        offs.append(kept.cpu().numpy() + offs[-1][-1])
        start = end
    off = torch.from_numpy(np.concatenate(offs)).to(dev)
    return off, torch.cat(parts) if len(parts) > 1 else parts[0]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _instance(case, seed):
    """(offsets, tids) of a case's items, ranks shuffled onto item ids."""
    probs = _probabilities(case["n"], case["density"], case["shape"])
    probs = probs[np.random.default_rng([seed, 0x5A1F]).permutation(case["n"])]
    return _tidlists(case["m"], probs, _gen(seed))


def _specs(case):
    """Instances of the batched workload: m log-uniform, n and density uniform."""
    g = np.random.default_rng(case["spec_seed"])
    return [{"m": int(round(10 ** g.uniform(4, 6))), "n": int(g.integers(100, 4001)),
             "density": float(g.uniform(0.01, 0.10)), "shape": "zipf"} for _ in range(case["k"])]


def _cross_probs(case, seed):
    a = _probabilities(case["n_a"], case["density"], "zipf")
    a = a[np.random.default_rng([seed, 0x5A1F]).permutation(case["n_a"])]
    return np.concatenate([a, np.full(case["n_b"], case["p_b"])])


def _pool_sizes(case, seed):
    u = np.random.default_rng([seed, 0x9001]).random(case["n"])
    return np.minimum(case["hi"], np.floor(case["lo"] * np.exp(u * math.log((case["hi"] + 1) / case["lo"]))))


def _query_ids(case, seed):
    """80% pairs, 20% of 3 to 8 sets, uniform ids."""
    g = np.random.default_rng([seed, 0x0E])
    k = np.where(g.random(case["n_q"]) < 0.8, 2, g.integers(3, 9, case["n_q"]))
    return [g.choice(case["n"], size=int(x), replace=False).astype(np.uint32) for x in k]


def _items(case, seed):
    return np.random.default_rng([seed, 0x17]).integers(0, case["n"], (case["n_q"], case["k"])).astype(np.int32)


def _buf(rows, cols=1):
    return torch.zeros((max(int(rows), 1), cols) if cols > 1 else max(int(rows), 1), dtype=torch.int32, device="cuda")


def _answer_cap(case):
    """Room for the elements that the listed queries' sets have in common."""
    return min(case["hi"] * min(case["n_list"], case["n_q"]), 20_000_000)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("mine", "dense"):
        st["off"], st["tids"] = _instance(case, seed)
        np_ = case["n"] * (case["n"] - 1) // 2
        st["full"], st["pairs"] = _buf(np_), _buf(np_, 3)
    elif kind == "cross":
        st["off"], st["tids"] = _tidlists(case["m"], _cross_probs(case, seed), _gen(seed))
        st["full"], st["pairs"] = _buf(case["n_a"] * case["n_b"]), _buf(case["n_a"] * case["n_b"], 3)
    elif kind == "batch":
        specs = _specs(case)
        st["sets"], st["s"], st["full"], st["pairs"] = [], [], [], []
        for q, sp in enumerate(specs):
            off, tids = _instance(sp, seed * 1000 + q)
            st["sets"].append(pkg.batmap_build(sp["m"], off, tids))
            st["s"].append(int(math.ceil(0.001 * sp["m"])))
            np_ = sp["n"] * (sp["n"] - 1) // 2
            st["full"].append(_buf(np_))
            st["pairs"].append(_buf(np_, 3))
    elif kind in ("triples", "quads"):
        st["off"], st["tids"] = _instance(case, seed)
        st["pairs"] = _buf(case["n"] * (case["n"] - 1) // 2, 3)
        # room for the answer, as a program that mines again and again keeps it
        st["out3"], st["out4"] = _buf(4_000_000, 4), _buf(4_000_000, 5)
        if kind == "quads":
            b = pkg.batmap_build(case["m"], st["off"], st["tids"])
            _, st["pairs"] = pkg.pair_support_all(b, case["s"], pairs=st["pairs"])
            b.free()
    elif kind == "itemsets":
        off, tids = _instance(case, seed)
        st["set"] = pkg.batmap_build_d(case["d"], case["m"], off, tids)
        st["items"] = torch.from_numpy(_items(case, seed)).cuda()
    elif kind == "queries":
        off, tids = _tidlists(case["m"], _pool_sizes(case, seed) / case["m"], _gen(seed))
        st["pool"] = pkg.batmap_pool_create(case["m"], off, tids)
        st["queries"] = _query_ids(case, seed)
        st["elems"] = _buf(_answer_cap(case))
    elif kind == "host":
        off, tids = _instance(case, seed)
        st["h_off"] = torch.empty(off.shape, dtype=torch.int64, pin_memory=True).copy_(off)
        st["h_tids"] = torch.empty(tids.shape, dtype=torch.int32, pin_memory=True).copy_(tids)
        st["h_pairs"] = torch.zeros((case["n"] * (case["n"] - 1) // 2, 3), dtype=torch.int32, pin_memory=True)
    return st


# ---- one pass -------------------------------------------------------------------


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "mine":
        b = pkg.batmap_build(c["m"], state["off"], state["tids"])
        n_out, _ = pkg.pair_support_all(b, c["s"], pairs=state["pairs"], full=state["full"])
        b.free()
        return [n_out, state["full"], state["pairs"]]
    if kind == "dense":
        n_out, _, _ = pkg.pair_support_dense(c["m"], state["off"], state["tids"], c["s"], pairs=state["pairs"],
                                                 full=state["full"])
        return [n_out, state["full"], state["pairs"]]
    if kind == "cross":
        b = pkg.batmap_build_cross(c["m"], c["n_a"], state["off"], state["tids"])
        n_out, _ = pkg.pair_support_all(b, c["s"], pairs=state["pairs"], full=state["full"])
        b.free()
        return [n_out, state["full"], state["pairs"]]
    if kind == "batch":
        n_out = pkg.pair_support_batch(state["sets"], state["s"], state["pairs"], state["full"])
        return [np.array(n_out, np.int64)] + state["full"] + state["pairs"]
    if kind == "triples":
        a = pkg.batmap_build(c["m"], state["off"], state["tids"])
        k2, pairs = pkg.pair_support_all(a, c["s"], pairs=state["pairs"])
        a.free()
        b = pkg.batmap_build_d(3, c["m"], state["off"], state["tids"])
        k3, _, n_cand = pkg.frequent_triples(b, c["s"], pairs, out=state["out3"])
        b.free()
        return [k2, k3, n_cand, state["pairs"], state["out3"]]
    if kind == "quads":
        b = pkg.batmap_build_d(4, c["m"], state["off"], state["tids"])
        k3, triples, n3 = pkg.frequent_triples(b, c["s"], state["pairs"], out=state["out3"])
        k4, _, n4 = pkg.frequent_quadruples(b, c["s"], triples, out=state["out4"])
        b.free()
        return [k3, k4, n3, n4, state["out3"], state["out4"]]
    if kind == "itemsets":
        return [pkg.itemset_support(state["set"], state["items"])]
    if kind == "queries":
        counts = pkg.intersect_query(state["pool"], state["queries"])
        off, elems = pkg.intersect_query_list(state["pool"], state["queries"][:c["n_list"]])
        state["elems"][:elems.numel()].copy_(elems)  # the caller's own list of answers
        return [counts, off, state["elems"]]
    n_out = pkg.pair_support_host(c["m"], state["h_off"].numpy(), state["h_tids"].numpy(), None, c["s"],
                                  state["h_pairs"].numpy())
    return [n_out, state["h_pairs"].numpy()]


# ---- what a pass cannot do without ------------------------------------------------


def _pair_work(m, p, s):
    """(common elements over all pairs, frequent pairs), expected."""
    p = np.sort(p)
    common = m * (p.sum() ** 2 - (p ** 2).sum()) / 2
    need = s / m
    # pairs (i, j) with p_i p_j >= s / m
    j = np.searchsorted(p, need / np.maximum(p, 1e-300))
    freq = max(0.0, ((len(p) - j).sum() - (p * p >= need).sum()) / 2)
    return common, freq


def work(case):
    """Bytes: the tidlists once, the answers once.  Operations: a multiply-add per
    element that two (or k) sets have in common, which is what an answer counts."""
    kind, m = case["kind"], case.get("m", 0)
    if kind in ("mine", "dense", "host"):
        n = case["n"]
        p = _probabilities(n, case["density"], case["shape"])
        common, freq = _pair_work(m, p, case["s"])
        full = 0 if kind == "host" else n * (n - 1) // 2
        return {"bytes": 4 * m * p.sum() + 8 * (n + 1) + 4 * full + 12 * freq, "flops": 2 * common}
    if kind == "cross":
        p = _cross_probs(case, 0)
        a, b = p[:case["n_a"]], p[case["n_a"]:]
        return {"bytes": 4 * m * p.sum() + 16 * a.size * b.size, "flops": 2 * m * a.sum() * b.sum()}
    if kind == "batch":
        # the tidlists' information is in the kept sets: a bit per element and its place, a byte
        by = fl = 0.0
        for sp in _specs(case):
            p = _probabilities(sp["n"], sp["density"], sp["shape"])
            common, freq = _pair_work(sp["m"], p, math.ceil(0.001 * sp["m"]))
            by += sp["m"] * p.sum() + 4 * (sp["n"] * (sp["n"] - 1) // 2) + 12 * freq
            fl += 2 * common
        return {"bytes": by, "flops": fl}
    if kind in ("triples", "quads"):
        p = _probabilities(case["n"], case["density"], case["shape"])
        common, freq = _pair_work(m, p, case["s"])
        # itemsets of size 3 and more: about six (ten) times the frequent pairs here
        up = 6 * freq if kind == "triples" else 16 * freq
        return {"bytes": 4 * m * p.sum() + 12 * freq + 16 * up, "flops": 2 * common + 2 * case["s"] * up}
    if kind == "itemsets":
        mean = m * float(_probabilities(case["n"], case["density"], case["shape"]).mean())
        return {"bytes": case["n"] * mean + 4 * case["n_q"] * (case["k"] + 1),
                "flops": 2.0 * case["n_q"] * case["k"] * mean / 10}
    # queries: the smallest set of each, and a look into each other set per element
    sizes = _pool_sizes(case, 0)
    small = float(np.minimum(np.roll(sizes, 1), sizes).mean())
    return {"bytes": case["n_q"] * small * (4 + 1.9), "flops": case["n_q"] * small * 1.9}


# ---- the same in plain 64-bit torch -------------------------------------------------


def _rows(off, tids, n, m):
    """n x m matrix of 0 and 1 (bool)."""
    x = torch.zeros((n, m), dtype=torch.bool, device=off.device)
    item = torch.repeat_interleave(torch.arange(n, device=off.device), off[1:] - off[:-1])
    x[item, tids.long()] = True
    return x


def _gram(x, y):
    c = torch.zeros((x.shape[0], y.shape[0]), dtype=torch.float64, device=x.device)
    for k in range(0, x.shape[1], 20_000):
        c += x[:, k:k + 20_000].double() @ y[:, k:k + 20_000].double().T
    return c.round().long()


def _pairs_of(full, i, j, s):
    """(number, rows (i, j, support) with zeros behind them) of the frequent pairs."""
    keep = full >= s
    rows = torch.zeros((max(full.numel(), 1), 3), dtype=torch.int64, device=full.device)
    k = int(keep.sum())
    rows[:k] = torch.stack([i[keep], j[keep], full[keep]], 1)
    return k, rows


def exact(case, seed):
    kind, m = case["kind"], case.get("m", 0)
    if kind in ("mine", "dense", "host"):
        n = case["n"]
        if 2.0 * n * n * m > 2e12 or n * m > 2e10:  # more than a few seconds in 64 bits
            return None
        off, tids = _instance(case, seed)
        x = _rows(off, tids, n, m)
        i, j = torch.triu_indices(n, n, 1, device=off.device)
        full = _gram(x, x)[i, j]
        k, pairs = _pairs_of(full, i, j, case["s"])
        if kind == "host":
            return [k, pairs.cpu().numpy()]
        return [k, full, pairs]
    if kind == "cross":
        na, nb = case["n_a"], case["n_b"]
        if 2.0 * na * nb * m > 2e12 or (na + nb) * m > 2e10:
            return None
        off, tids = _tidlists(m, _cross_probs(case, seed), _gen(seed))
        x = _rows(off, tids, na + nb, m)
        i = torch.arange(na, device=off.device).repeat_interleave(nb)
        j = torch.arange(nb, device=off.device).repeat(na)
        full = _gram(x[:na], x[na:]).reshape(-1)
        k, pairs = _pairs_of(full, i, j, case["s"])
        return [k, full, pairs]
    if kind == "itemsets":
        off, tids = _instance(case, seed)
        x = _rows(off, tids, case["n"], m)
        items = torch.from_numpy(_items(case, seed)).to(off.device).long()
        out = []
        for q in range(0, items.shape[0], 1_000):
            y = x[items[q:q + 1_000, 0]]
            for t in range(1, items.shape[1]):
                y &= x[items[q:q + 1_000, t]]
            out.append(y.sum(1))
        return [torch.cat(out)]
    if kind == "queries":
        if case["n_q"] > 5_000:
            return None
        off, tids = _tidlists(m, _pool_sizes(case, seed) / m, _gen(seed))
        h = off.tolist()
        counts, lists = [], []
        for q, ids in enumerate(_query_ids(case, seed)):
            ids = sorted((int(i) for i in ids), key=lambda i: h[i + 1] - h[i])
            x = tids[h[ids[0]]:h[ids[0] + 1]]
            for i in ids[1:]:
                y = tids[h[i]:h[i + 1]]
                if not y.numel() or not x.numel():
                    x = x[:0]
                    break
                at = torch.searchsorted(y, x).clamp_(max=y.numel() - 1)
                x = x[y[at] == x]
            counts.append(x.numel())
            if q < case["n_list"]:
                lists.append(x)
        o = np.concatenate([[0], np.cumsum([x.numel() for x in lists])])
        elems = torch.zeros(_answer_cap(case), dtype=torch.int64, device=off.device)
        elems[:int(o[-1])] = torch.cat(lists)
        return [np.array(counts, np.int64), o, elems]
    # a batch of large instances, and itemsets joined level by level: minutes in 64 bits
    return None
