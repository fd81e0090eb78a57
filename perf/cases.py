"""Performance cases of the library: what its users have it compute, through the public entry points.

The cases cover each entry point that computes something: the all-pairs identity-by-state matrix (plain, square and
allocation-free), the batched subsets of a pool, the served queries against a resident panel, linkage
disequilibrium, the relationship matrix and complete-linkage clustering.  Sizes run from the smallest calls, where
launches and latency count, to the 20,000 x 500,000 cohort; some are odd in both directions (samples not a
multiple of 4, markers not a multiple of any chunk).  Inputs are the seeded synthetic genotypes that the package's
generator draws on the device.

A program keeps one library context and its outputs' buffers; prepare() does the same (a served panel belongs to a
context of its own, which the state releases).
"""
import math

import numpy as np
import torch

from paper_1410_4803_gb300 import ibs, synth

DEV = "cuda:0"


def listed():
    return [
        # A quick look at a small study (the smallest configuration): latency of the call and its launches.
        {"name": "ibs_small", "kind": "ibs", "n": 256, "m": 4096, "dist": True, "square": False, "pops": 1},
        # A mid-size study after filtering: sizes that divide by nothing.
        {"name": "ibs_ragged", "kind": "ibs", "n": 1501, "m": 30011, "dist": True, "square": False, "pops": 1},
        # A genotyping-array cohort.
        {"name": "ibs_plain", "kind": "ibs", "n": 4096, "m": 100000, "dist": True, "square": False, "pops": 1},
        # The large structured cohort: subpopulations, relatives, duplicates.
        {"name": "ibs_structured", "kind": "ibs", "n": 20000, "m": 500000, "dist": True, "square": False, "pops": 5},
        # The paper's own command: the full square matrix.
        {"name": "ibs_square", "kind": "ibs", "n": 3001, "m": 60000, "dist": True, "square": True, "pops": 1},
        # The same counts for a caller that may not allocate (the integer kernels).
        {"name": "ibs_noalloc", "kind": "noalloc", "n": 1000, "m": 20000, "dist": True},
        # Many cohort subsets over marker windows of one pool (permutation and cross-validation work).
        {"name": "batch_pool", "kind": "batch", "pool_n": 10000, "pool_m": 200000, "subsets": 24, "n_lo": 100,
         "n_hi": 3000, "m_lo": 5000, "m_hi": 80000, "shape": 3},
        # One new sample's nearest relatives in a resident reference panel: latency.
        {"name": "query_one", "kind": "query", "panel_n": 20000, "m": 100000, "requests": 1, "q_max": 1, "k": 16,
         "counts": False, "shape": 4},
        # Twenty requests of log-uniform sizes at once, counts kept on the device for what follows: throughput.
        {"name": "query_burst", "kind": "query", "panel_n": 20000, "m": 100000, "requests": 20, "q_max": 512, "k": 16,
         "counts": True, "shape": 4},
        # Linkage disequilibrium of an array cohort within 1,000 markers.
        {"name": "ld_window", "kind": "ld", "n": 4096, "m": 100000, "window": 1000},
        # Relationship matrix of the array cohort.
        {"name": "grm_plain", "kind": "grm", "n": 4096, "m": 100000},
        # Clustering of the array cohort's finished distance matrix.
        {"name": "cluster", "kind": "cluster", "n": 4096, "m": 4000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ibs", "ibs", "ibs", "square", "noalloc", "batch", "query", "ld", "grm", "cluster"])
    if kind in ("ibs", "square"):
        square = kind == "square"
        n = _log(rng, 40, 6000 if square else 12000)
        m = min(_log(rng, 700, 400000), int(1.5e13 / (n * n)) + 700)
        return {"kind": "ibs", "n": n, "m": m, "dist": rng.random() < 0.85, "square": square,
                "pops": rng.choice([1, 5])}
    if kind == "noalloc":
        n = _log(rng, 40, 3000)
        return {"kind": "noalloc", "n": n, "m": min(_log(rng, 500, 60000), 80_000_000 // (n + 64)),
                "dist": rng.random() < 0.85}
    if kind == "batch":
        return {"kind": "batch", "pool_n": _log(rng, 3500, 20000), "pool_m": _log(rng, 90000, 300000),
                "subsets": rng.randint(2, 28), "n_lo": 50, "n_hi": _log(rng, 300, 3000), "m_lo": 2000,
                "m_hi": _log(rng, 5000, 80000), "shape": rng.randint(0, 1 << 30)}
    if kind == "query":
        return {"kind": "query", "panel_n": _log(rng, 3000, 40000), "m": _log(rng, 5000, 120000),
                "requests": rng.choice([1, 1, 2, 5, 12, 20]), "q_max": _log(rng, 1, 512), "k": rng.choice([0, 1, 16, 64]),
                "counts": True, "shape": rng.randint(0, 1 << 30)}
    if kind == "ld":
        m = _log(rng, 1000, 100000)
        return {"kind": "ld", "n": _log(rng, 100, 6000), "m": m, "window": min(_log(rng, 10, 1500), m - 1)}
    if kind == "grm":
        n = _log(rng, 50, 4500)
        return {"kind": "grm", "n": n, "m": min(_log(rng, 500, 200000), int(2e12 / (n * n)) + 500)}
    return {"kind": "cluster", "n": _log(rng, 60, 4096), "m": 4000}


# ---------------------------------------------------------------------------
# Inputs and state.

_CTX = {}


def _ctx(flags=0):
    """The program's one context per set of flags."""
    if flags not in _CTX:
        _CTX[flags] = ibs.ibs_init(0, flags=flags)
    return _CTX[flags]


class _PanelContext:
    """A context with a resident panel, shut down when the state that holds it goes."""

    def __init__(self):
        self.ctx = ibs.ibs_init(0)

    def __del__(self):
        try:
            ibs.ibs_shutdown(self.ctx)
        except Exception:
            pass


def _genotypes(n, m, seed, pops=1):
    """Packed genotypes uint8 [m][ceil(n/4)] on the device: one population with uneven missingness, or five
    subpopulations with relatives and duplicates where the cohort is large enough for them."""
    if pops == 1:
        model = synth.plain_model(m, seed, maf=(0.01, 0.5), miss=0.02, hi_miss_frac=0.005, hi_miss_rate=0.3)
        samples = synth.Samples.base(n)
    else:
        model = synth.balding_nichols_model(m, seed, n_pop=pops, fst=0.05, anc=(0.02, 0.5), miss=0.01)
        off, dup = n // 100, n // 400
        samples = synth.structured_samples(n - off - dup, pops, off, dup, seed)
    return synth.generate_device(model, samples, pad_garbage=True)


def _pairs(n):
    return n * (n + 1) // 2


def _subset_shapes(case):
    """Sizes and window lengths of a batch: the case's own, whatever the inputs' seed."""
    rng = np.random.default_rng(case["shape"])
    k = case["subsets"]
    n = rng.integers(case["n_lo"], min(case["n_hi"], case["pool_n"]) + 1, k)
    m = rng.integers(case["m_lo"], min(case["m_hi"], case["pool_m"]) + 1, k)
    return [(int(a), int(b)) for a, b in zip(n, m)]


def _query_sizes(case):
    rng = np.random.default_rng(case["shape"])
    q = np.floor(np.exp(rng.uniform(0.0, math.log(case["q_max"]) if case["q_max"] > 1 else 0.0, case["requests"])))
    return [int(min(case["q_max"], max(1, v))) for v in q]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("ibs", "noalloc"):
        n, m = case["n"], case["m"]
        square = kind == "ibs" and case["square"]
        P = n * n if square else _pairs(n)
        return {"kind": kind, "n": n, "m": m, "packed": _genotypes(n, m, seed, case.get("pops", 1)),
                "ctx": None if kind == "noalloc" else _ctx(ibs.IBS_OUT_SQUARE if square else 0),
                "counts": torch.empty((P, 4), dtype=torch.int32, device=DEV),
                "dist": torch.empty(P, dtype=torch.float64, device=DEV) if case["dist"] else None}
    if kind == "batch":
        pool = _genotypes(case["pool_n"], case["pool_m"], seed)
        rng = np.random.default_rng(seed + 17)
        subs = []
        for n, m in _subset_shapes(case):
            idx = np.sort(rng.choice(case["pool_n"], size=n, replace=False)).astype(np.int64)
            begin = int(rng.integers(0, case["pool_m"] - m + 1))
            subs.append((torch.from_numpy(idx).to(DEV), begin, m,
                         torch.empty((_pairs(n), 4), dtype=torch.int32, device=DEV),
                         torch.empty(_pairs(n), dtype=torch.float64, device=DEV)))
        return {"kind": kind, "ctx": _ctx(), "pool": pool, "pool_n": case["pool_n"], "pool_m": case["pool_m"],
                "subs": subs}
    if kind == "query":
        n, m, k = case["panel_n"], case["m"], case["k"]
        panel = synth.balding_nichols_model(m, seed, n_pop=5, fst=0.05, anc=(0.02, 0.5), miss=0.01)
        samples = synth.structured_samples(n - n // 80, 5, n // 100, n // 80 - n // 100, seed)
        packed = synth.generate_device(panel, samples)
        holder = _PanelContext()
        ibs.ibs_panel_load(holder.ctx, packed, n, m)
        rng = np.random.default_rng(seed + 23)
        reqs = []
        for r, q in enumerate(_query_sizes(case)):
            # fresh samples of the panel's populations, about a tenth of them relatives of panel samples
            gid = (1 << 40) + r * 4096 + np.arange(q, dtype=np.int64)
            s = synth.Samples(gid, rng.integers(0, 5, q).astype(np.int32), np.zeros(q, np.int32), gid.copy(),
                              np.zeros(q, np.int32))
            for t in np.flatnonzero(rng.random(q) < 0.1):
                b = int(rng.integers(0, n - n // 80))
                s.kind[t] = synth.OFFSPRING if rng.random() < 0.5 else synth.DUPLICATE
                s.src_gid[t] = samples.gid[b]
                s.pop[t] = samples.pop[b]
            s.src_pop[:] = s.pop
            reqs.append({"q": q, "packed": synth.generate_device(panel, s).cpu().pin_memory(),
                         "counts": torch.empty((q, n, 4), dtype=torch.int32, device=DEV) if case["counts"] else None,
                         "idx": torch.empty((q, k), dtype=torch.int32).pin_memory() if k else None,
                         "dist": torch.empty((q, k), dtype=torch.float64).pin_memory() if k else None})
        torch.cuda.synchronize()
        return {"kind": kind, "holder": holder, "k": k, "reqs": reqs}
    if kind == "ld":
        n, m, w = case["n"], case["m"], case["window"]
        return {"kind": kind, "ctx": _ctx(), "n": n, "m": m, "window": w, "packed": _genotypes(n, m, seed),
                "r": torch.empty((m, w), dtype=torch.float64, device=DEV),
                "cnt": torch.empty((m, w), dtype=torch.int32, device=DEV)}
    if kind == "grm":
        n, m = case["n"], case["m"]
        return {"kind": kind, "ctx": _ctx(), "n": n, "m": m, "packed": _genotypes(n, m, seed),
                "out": torch.empty(_pairs(n), dtype=torch.float64, device=DEV)}
    n = case["n"]
    return {"kind": kind, "ctx": _ctx(), "n": n, "dist": _ibs_exact(_genotypes(n, case["m"], seed), n, case["m"])[1],
            "link": torch.empty((n - 1, 4), dtype=torch.float64, device=DEV)}


def run(state):
    kind = state["kind"]
    if kind == "ibs":
        ibs.ibs_compute(state["ctx"], state["packed"], state["n"], state["m"], state["counts"], state["dist"])
        return [state["counts"], state["dist"]]
    if kind == "noalloc":
        ibs.ibs_compute_noalloc(state["packed"], state["n"], state["m"], state["counts"], state["dist"])
        return [state["counts"], state["dist"]]
    if kind == "batch":
        ibs.ibs_compute_batch(state["ctx"], state["pool"], state["pool_n"], state["pool_m"], state["subs"])
        return [[s[3], s[4]] for s in state["subs"]]
    if kind == "query":
        ctx, k = state["holder"].ctx, state["k"]
        ids = [ibs.ibs_query(ctx, r["packed"], r["q"], k, r["counts"], r["idx"], r["dist"]) for r in state["reqs"]]
        for i in ids:
            ibs.ibs_wait(ctx, i)
        return [[r["counts"], r["idx"], r["dist"]] for r in state["reqs"]]
    if kind == "ld":
        ibs.ibs_ld_r(state["ctx"], state["packed"], state["n"], state["m"], state["window"], state["r"], state["cnt"])
        return [state["r"], state["cnt"]]
    if kind == "grm":
        ibs.ibs_grm(state["ctx"], state["packed"], state["n"], state["m"], state["out"])
        return [state["out"]]
    ibs.ibs_cluster_complete(state["ctx"], state["dist"], state["n"], state["link"])
    return [state["link"]]


# ---------------------------------------------------------------------------
# Work and tolerances.


def work(case):
    """Input genotypes read once (2 bits each), outputs written once; four multiply-adds per pair and marker for the
    pair counts and for the relationship matrix, six per marker pair and sample for r."""
    kind = case["kind"]
    if kind in ("ibs", "noalloc"):
        n, m = case["n"], case["m"]
        pairs = n * n if case.get("square") else _pairs(n)
        return {"bytes": m * ((n + 3) // 4) + pairs * (24 if case["dist"] else 16), "flops": 8.0 * _pairs(n) * m}
    if kind == "batch":
        b = f = 0.0
        for n, m in _subset_shapes(case):
            b += m * ((n + 3) // 4) + 24 * _pairs(n)
            f += 8.0 * _pairs(n) * m
        return {"bytes": b, "flops": f}
    if kind == "query":
        q, n, m = sum(_query_sizes(case)), case["panel_n"], case["m"]
        # the resident panel is read once, as packed genotypes, however many requests are in flight
        return {"bytes": m * ((n + 3) // 4) + m * ((q + 3) // 4) + (16.0 * q * n if case["counts"] else 0)
                + 12.0 * q * case["k"], "flops": 8.0 * q * n * m}
    if kind == "ld":
        n, m, w = case["n"], case["m"], case["window"]
        return {"bytes": m * ((n + 3) // 4) + 12.0 * m * w, "flops": 12.0 * n * (m * w - w * (w + 1) / 2)}
    if kind == "grm":
        n, m = case["n"], case["m"]
        return {"bytes": m * ((n + 3) // 4) + 8.0 * _pairs(n), "flops": 8.0 * _pairs(n) * m}
    n = case["n"]
    return {"bytes": 8.0 * _pairs(n) + 32.0 * (n - 1), "flops": 2.0 * n * n}


def tolerance(case):
    kind = case["kind"]
    if kind in ("ibs", "noalloc", "batch"):
        # counts are whole numbers and equal; the distance is a quotient of whole numbers in FP64 within its stated
        # few ulps (measured against FP64 division: 2e-15 and less)
        return {"rel": 8e-15, "max": 6e-14}
    if kind == "query":
        return "exact"  # whole counts and indices; the k distances are correctly rounded quotients
    if kind == "ld":
        # six exact sums, then a correlation within its stated 1e-12 (measured against FP64: 3.8e-15)
        return {"rel": 1.6e-14, "max": 1e-12}
    if kind == "grm":
        # products of FP16 pairs in FP32 segments (measured against FP64: 1.1e-6 of the result's norm)
        return {"rel": 4.5e-6, "max": 9e-5}
    return "exact"  # heights are input distances, ids and sizes whole numbers


# ---------------------------------------------------------------------------
# The same results in plain torch.


def _codes(packed, n):
    """2-bit codes [rows][n] of packed rows."""
    sh = torch.tensor([0, 2, 4, 6], dtype=torch.uint8, device=packed.device)
    return ((packed[:, :, None] >> sh) & 3).reshape(packed.shape[0], -1)[:, :n]


def _ibs_counts(a_packed, na, b_packed, nb, m):
    """IBS0, IBS1, N of every pair as float64 [na][nb] (whole numbers: exact)."""
    i0 = torch.zeros((na, nb), dtype=torch.float64, device=DEV)
    i1, nn = torch.zeros_like(i0), torch.zeros_like(i0)
    step = max(1, min(8192, int(4e8 / max(na, nb))))
    for k in range(0, m, step):
        ca, cb = _codes(a_packed[k:k + step], na), _codes(b_packed[k:k + step], nb)
        f = lambda x: x.to(torch.float32)  # noqa: E731
        va, vb = f(ca != 1), f(cb != 1)
        ha, hb = f(ca == 2), f(cb == 2)
        qa, qb, ra, rb = f(ca == 3), f(cb == 3), f(ca == 0), f(cb == 0)
        nn += va.T @ vb
        i0 += qa.T @ rb + ra.T @ qb
        i1 += ha.T @ (qb + rb) + (qa + ra).T @ hb
    return i0, i1, nn


def _ibs_exact(packed, n, m, square=False):
    i0, i1, nn = _ibs_counts(packed, n, packed, n, m)
    if not square:
        i, j = torch.triu_indices(n, n, device=DEV)
        i0, i1, nn = i0[i, j], i1[i, j], nn[i, j]
    else:
        i0, i1, nn = i0.reshape(-1), i1.reshape(-1), nn.reshape(-1)
    counts = torch.stack([i0, i1, nn - i0 - i1, nn], 1).to(torch.int32)
    return counts, (i1 + 2 * i0) / (2 * nn)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("ibs", "noalloc"):
        n, m = case["n"], case["m"]
        if float(n) * n * m > 2e14 or n > 8000:
            return None
        counts, dist = _ibs_exact(_genotypes(n, m, seed, case.get("pops", 1)), n, m, case.get("square", False))
        return [counts, dist if case["dist"] else None]
    if kind == "batch":
        s = prepare(case, seed)
        out = []
        for idx, begin, m, _, _ in s["subs"]:
            n = idx.numel()
            c = _codes(s["pool"][begin:begin + m], s["pool_n"])[:, idx]
            if n % 4:
                c = torch.cat([c, torch.ones((m, 4 - n % 4), dtype=torch.uint8, device=DEV)], 1)
            c = c.reshape(m, -1, 4)
            packed = c[:, :, 0] | (c[:, :, 1] << 2) | (c[:, :, 2] << 4) | (c[:, :, 3] << 6)
            out.append(list(_ibs_exact(packed, n, m)))
        return out
    if kind == "query":
        n, m, k = case["panel_n"], case["m"], case["k"]
        if float(sum(_query_sizes(case))) * n * m > 1e14:
            return None
        panel = synth.balding_nichols_model(m, seed, n_pop=5, fst=0.05, anc=(0.02, 0.5), miss=0.01)
        samples = synth.structured_samples(n - n // 80, 5, n // 100, n // 80 - n // 100, seed)
        packed = synth.generate_device(panel, samples)
        s = prepare(case, seed)
        out = []
        for r in s["reqs"]:
            i0, i1, nn = _ibs_counts(r["packed"].to(DEV), r["q"], packed, n, m)
            counts = torch.stack([i0, i1, nn - i0 - i1, nn], 2).to(torch.int32) if case["counts"] else None
            top = idx = None
            if k:
                d, order = torch.sort((i1 + 2 * i0) / (2 * nn), dim=1, stable=True)
                kk = min(k, n)
                top, idx = d[:, :kk], order[:, :kk].to(torch.int32)
            out.append([counts, idx, top])
        return out
    if kind == "ld":
        n, m, w = case["n"], case["m"], case["window"]
        packed = _genotypes(n, m, seed)
        r = torch.full((m, w), float("nan"), dtype=torch.float64, device=DEV)
        cnt = torch.zeros((m, w), dtype=torch.int32, device=DEV)
        B = 512
        for a0 in range(0, m, B):
            a1, b1 = min(m, a0 + B), min(m, a0 + B + w)
            c = _codes(packed[a0:b1], n)
            v = (c != 1).to(torch.float32)
            x = (c == 0).to(torch.float32) - (c == 3).to(torch.float32)
            h = x * x
            sign = torch.where(x.sum(1) >= 0, 1.0, -1.0).double()
            na = a1 - a0
            va, xa, ha = v[:na], x[:na], h[:na]
            N, sx, sy = (va @ v.T).double(), (xa @ v.T).double(), (va @ x.T).double()
            sxx, syy, sxy = (ha @ v.T).double(), (va @ h.T).double(), (xa @ x.T).double()
            den = (N * sxx - sx * sx) * (N * syy - sy * sy)
            R = (N * sxy - sx * sy) / den.sqrt() * sign[:na, None] * sign[None, :]
            R = torch.where(den > 0, R, torch.nan)
            col = torch.arange(na, device=DEV)[:, None] + 1 + torch.arange(w, device=DEV)[None, :]
            ok = col < b1 - a0
            col = col.clamp(max=b1 - a0 - 1)
            r[a0:a1] = torch.where(ok, R.gather(1, col), torch.nan)
            cnt[a0:a1] = torch.where(ok, N.gather(1, col), 0.0).to(torch.int32)
        return [r, cnt]
    if kind == "grm":
        n, m = case["n"], case["m"]
        packed = _genotypes(n, m, seed)
        num = torch.zeros((n, n), dtype=torch.float64, device=DEV)
        cnt = torch.zeros((n, n), dtype=torch.float64, device=DEV)
        for k in range(0, m, 8192):
            c = _codes(packed[k:k + 8192], n)
            v = (c != 1).double()
            x = 2.0 * (c == 0).double() + (c == 2).double()
            p = (x * v).sum(1) / (2.0 * v.sum(1))
            used = (p > 0) & (p < 1)
            v, x, p = v[used], x[used], p[used][:, None]
            z = (x - 2 * p) / (2 * p * (1 - p)).sqrt() * v
            num += z.T @ z
            cnt += (v.float().T @ v.float()).double()
        i, j = torch.triu_indices(n, n, device=DEV)
        return [(num / cnt)[i, j]]
    return [_cluster_exact(prepare(case, seed)["dist"], case["n"])]


def _cluster_exact(dist, n):
    """Greedy complete linkage: the smallest distance first, ties by the smallest (row, column)."""
    D = torch.full((n, n), float("inf"), dtype=torch.float64, device=DEV)
    i, j = torch.triu_indices(n, n, device=DEV)
    D[i, j] = dist
    full = torch.minimum(D, D.T).contiguous()
    full.fill_diagonal_(float("inf"))
    upper = torch.triu(torch.ones((n, n), dtype=torch.bool, device=DEV), 1)
    rowmin = torch.where(upper, full, torch.inf).min(1).values
    ids, size = list(range(n)), [1] * n
    out = np.empty((n - 1, 4))
    pos = torch.arange(n, device=DEV)
    gone = torch.zeros(n, dtype=torch.bool, device=DEV)
    for step in range(n - 1):
        low = rowmin.min()
        a = int((rowmin == low).nonzero()[0, 0])
        b = int(((full[a] == low) & (pos > a)).nonzero()[0, 0])
        out[step] = (min(ids[a], ids[b]), max(ids[a], ids[b]), float(low), size[a] + size[b])
        ids[a], size[a] = n + step, size[a] + size[b]
        gone[b] = True
        new = torch.maximum(full[a], full[b])
        new[gone] = torch.inf
        new[a] = torch.inf
        full[a] = new
        full[:, a] = new
        full[b] = torch.inf
        full[:, b] = torch.inf
        rowmin = torch.where(upper, full, torch.inf).min(1).values
    return torch.from_numpy(out).to(DEV)
