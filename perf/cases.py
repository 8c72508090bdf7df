"""The work a user of this library has it do, as cases that can be timed.

Every case is one kind of call through the public Python layer
(paper_2407_20205_gb300.binding) at one size:

  device   one n x n matrix already on the device, all 2^n Gray indices
           (perm_f3_range_counts_async)
  host     one n x n host matrix, exact counts of all 2^n terms
           (perm_f3_counts: copied in, result copied out, synchronous)
  window   one range of Gray indices, ragged at both ends, of a matrix too
           large to walk in one call (a rank's or a job's share of the sum)
  rankone  a device matrix with entries d_i * e_j (d, e in {1, -1}): two terms
           in three are nonzero, where a uniform matrix has (2/3)^n of them
  pooled   a host matrix whose columns are multiples of a few vectors
  batch    many device matrices in one call, sizes lo..hi
           (perm_f3_batch_async, with the histogram)
  mc       many small host matrices in one call, sizes lo..hi (perm_f3_batch
           with the histogram, as the Monte Carlo estimate calls it)
  serve    a burst of requests to a serving context, every result waited for

work(): bytes are the matrices and results, each once; flops are the terms of
Ryser's sum, one operation per Gray index (2^n for a whole matrix).  Nothing
shorter than that is known to be needed, and less may be possible.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2407_20205_gb300 import binding as pf3
from paper_2407_20205_gb300 import inputs


def listed():
    return [
        # the paper's smallest timing size, one launch per permanent: latency
        {"name": "device_n20", "kind": "device", "n": 20},
        # one plane word, odd size, through the host-pointer call: a user's
        # single mid-sized permanent
        {"name": "host_n31", "kind": "host", "n": 31},
        # the two headline sizes (two plane words per state)
        {"name": "device_n36", "kind": "device", "n": 36},
        {"name": "device_n40", "kind": "device", "n": 40},
        # one job's share of a long sum: a ragged range of the middle of a
        # 47 x 47 matrix's 2^47 indices
        {"name": "window_n47", "kind": "window", "n": 47, "first": 70368744177000 // 3 + 77,
         "count": (1 << 36) + 12345},
        # rank-one matrices (J_n and its scalings appear among the known
        # answers of the serving mix): most terms nonzero
        {"name": "rankone_n33", "kind": "rankone", "n": 33},
        # few distinct columns, through the host call
        {"name": "pooled_n40", "kind": "pooled", "n": 40, "pool": 7},
        # the Monte Carlo headline: 200,000 permanents of 24 x 24
        {"name": "batch_n24", "kind": "batch", "lo": 24, "hi": 24, "count": 200000},
        # a device batch of uneven sizes around the one/two word boundary
        {"name": "batch_n19_34", "kind": "batch", "lo": 19, "hi": 34, "count": 300},
        # the small sizes of the Monte Carlo table, host buffers
        {"name": "mc_n6_16", "kind": "mc", "lo": 6, "hi": 16, "count": 40000},
        # a burst of the serving mix (uniform, sparse, known answers)
        {"name": "serve_n12_36", "kind": "serve", "lo": 12, "hi": 36, "jobs": 64},
    ]


def draw(rng):
    kind = rng.choice(["device", "host", "window", "rankone", "pooled", "batch", "batch", "mc", "serve"])
    if kind == "device":
        return {"kind": kind, "n": rng.randint(12, 40)}
    if kind == "host":
        return {"kind": kind, "n": rng.randint(8, 38)}
    if kind == "window":
        n = rng.randint(41, 64)
        count = int(2.0 ** rng.uniform(20, 37))
        return {"kind": kind, "n": n, "first": rng.randrange((1 << min(n, 62)) - count), "count": count}
    if kind == "rankone":
        return {"kind": kind, "n": rng.randint(16, 35)}
    if kind == "pooled":
        return {"kind": kind, "n": rng.randint(33, 64), "pool": rng.randint(1, 7)}
    if kind == "batch":
        lo = rng.randint(17, 34)
        hi = min(34, lo + rng.choice([0, 0, 1, 3, 8]))
        top = min(200000, int(2.0 ** (41 - hi)))
        return {"kind": kind, "lo": lo, "hi": hi, "count": max(1, int(top ** rng.uniform(0.25, 1.0)))}
    if kind == "mc":
        lo = rng.randint(4, 14)
        hi = min(18, lo + rng.choice([0, 2, 4]))
        return {"kind": kind, "lo": lo, "hi": hi, "count": int(2.0 ** rng.uniform(7, 15.5))}
    hi = rng.randint(24, 37)
    return {"kind": kind, "lo": 12, "hi": hi, "jobs": int(2.0 ** rng.uniform(2, 6.5))}


def _uniform(seed, shape):
    g = torch.Generator().manual_seed(seed)
    return torch.randint(0, 3, shape, generator=g, dtype=torch.uint8)


def _sizes(case, seed):
    """Sizes of a batch, spread evenly over lo..hi in a seeded order."""
    lo, hi, count = case["lo"], case["hi"], case["count"]
    ns = (lo + np.arange(count) % (hi - lo + 1)).astype(np.int32)
    np.random.default_rng(seed).shuffle(ns)
    return ns


def _rank_one(seed, n):
    g = torch.Generator().manual_seed(seed)
    d = torch.randint(1, 3, (n,), generator=g)
    e = torch.randint(1, 3, (n,), generator=g)
    return d, e, ((d[:, None] * e[None, :]) % 3).to(torch.uint8)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("device", "window", "rankone"):
        n = case["n"]
        A = _rank_one(seed, n)[2] if kind == "rankone" else _uniform(seed, (n, n))
        st["A"] = A.cuda()
        st["out"] = torch.zeros(3, dtype=torch.int64, device="cuda")
        st["first"] = case.get("first", 0)
        st["last"] = st["first"] + case.get("count", 1 << n) - 1
    elif kind == "host":
        st["A"] = _uniform(seed, (case["n"], case["n"])).numpy()
    elif kind == "pooled":
        st["A"] = _pooled(seed, case["n"], case["pool"])
    elif kind == "batch":
        ns = _sizes(case, seed)
        total = int((ns.astype(np.int64) ** 2).sum())
        g = torch.Generator(device="cuda").manual_seed(seed)
        st["ns"] = ns
        st["As"] = torch.randint(0, 3, (total,), generator=g, dtype=torch.uint8, device="cuda")
        st["res"] = torch.zeros(len(ns), dtype=torch.uint8, device="cuda")
        st["hist"] = torch.zeros(3, dtype=torch.int64, device="cuda")
    elif kind == "mc":
        st["ns"] = _sizes(case, seed)
        st["flat"] = _uniform(seed, (int((st["ns"].astype(np.int64) ** 2).sum()),)).numpy()
    else:
        st["mats"] = [inputs.serve_job(seed, j, case["lo"], case["hi"])[2] for j in range(case["jobs"])]
        st["ctx"] = pf3.ServeContext()
    return st


def _pooled(seed, n, pool):
    """n columns, each +-1 times one of `pool` uniform vectors, every vector
    used an odd number of times but one where n - pool is odd (the merge keeps
    an odd multiplicity once, an even one twice)."""
    g = np.random.default_rng(seed)
    vecs = g.integers(0, 3, (pool, n))
    mult = [1] * pool
    mult[0] += (n - pool) % 2
    for _ in range((n - pool) // 2):
        mult[g.integers(pool)] += 2
    cols = np.repeat(np.arange(pool), mult)
    g.shuffle(cols)
    return (vecs[cols].T * g.integers(1, 3, n)[None, :] % 3).astype(np.uint8)


def run(st):
    kind = st["case"]["kind"]
    if kind in ("device", "window", "rankone"):
        pf3.perm_f3_range_counts_async(st["A"], st["case"]["n"], st["first"], st["last"], st["out"],
                                       torch.cuda.current_stream())
        return st["out"]
    if kind in ("host", "pooled"):
        return np.array(pf3.perm_f3_counts(st["A"]), dtype=np.uint64)
    if kind == "batch":
        pf3.perm_f3_batch_async(st["As"], st["ns"], st["res"], st["hist"], torch.cuda.current_stream())
        return st["res"], st["hist"]
    if kind == "mc":
        return pf3.perm_f3_batch(flat=st["flat"], ns=st["ns"], with_hist=True)
    tickets = [st["ctx"].submit(A) for A in st["mats"]]
    return np.array([st["ctx"].wait(t) for t in tickets], dtype=np.uint8)


def work(case):
    kind = case["kind"]
    if kind in ("device", "host", "window", "rankone", "pooled"):
        n = case["n"]
        b = n * n + 24
        if kind == "window":
            return {"bytes": b, "flops": case["count"]}
        if kind == "pooled":
            # the terms fall on 3^m column-sum vectors of two parities; each
            # row moves every one of them once
            m = case["pool"] + (n - case["pool"]) % 2
            return {"bytes": b, "flops": n * 2 * 3 ** m}
        return {"bytes": b, "flops": 1 << n}
    if kind == "serve":
        ns = range(case["lo"], case["hi"] + 1)
        return {"bytes": int(case["jobs"] * sum(n * n for n in ns) / len(ns)),
                "flops": int(case["jobs"] * sum(1 << n for n in ns) / len(ns))}
    ns = _sizes(case, 0).astype(np.int64)
    return {"bytes": int((ns ** 2).sum() + len(ns)), "flops": float((2.0 ** ns).sum())}


# ---------------------------------------------------------------- references
# Eq. (2) written out: for every row subset S the column sums over S, the sign
# (-1)^{|S|} and the product over the columns, in 64-bit floating point (sums
# of at most 64 entries, exact).

def _where():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _terms(A, dev):
    """+1/-1 term counts (two int64 tensors [b]) of the matrices A[b, n, n]."""
    b, n = A.shape[0], A.shape[1]
    A = A.to(dev, torch.float64)
    plus = torch.zeros(b, dtype=torch.int64, device=dev)
    minus = torch.zeros(b, dtype=torch.int64, device=dev)
    step = max(1, min(1 << n, (1 << 25) // (n * b)))
    for s0 in range(0, 1 << n, step):
        s = torch.arange(s0, min(s0 + step, 1 << n), device=dev)
        bits = ((s[:, None] >> torch.arange(n, device=dev)) & 1).to(torch.float64)
        sums = torch.remainder(torch.matmul(bits, A), 3.0)
        nonzero = (sums != 0).all(dim=2)
        odd = ((sums == 2).sum(dim=2) + bits.sum(dim=1).to(torch.int64)) & 1
        plus += (nonzero & (odd == 0)).sum(dim=1)
        minus += (nonzero & (odd == 1)).sum(dim=1)
    return plus, minus


def _residue(n, plus, minus):
    return ((-1) ** n * (int(plus) - int(minus))) % 3


def _rank_one_counts(d, e):
    """Counts of a matrix d_i * e_j: the column sums over S are e_j * t with
    t = (#d=1 in S) - (#d=-1 in S), so a term is nonzero unless 3 divides t."""
    n = len(d)
    p = int((d == 1).sum())
    neg_e = int((e == 2).sum())
    cnt = [0, 0]
    for a in range(p + 1):
        for b in range(n - p + 1):
            t = (a - b) % 3
            if t:
                negs = neg_e if t == 1 else n - neg_e
                cnt[(a + b + negs) & 1] += math.comb(p, a) * math.comb(n - p, b)
    return cnt


def _few_column_counts(A):
    """Counts of a matrix whose columns are multiples of a few vectors, by the
    number of row subsets on every (column-sum vector, parity) pair."""
    n = A.shape[0]
    reps, mult, neg = [], [], 0
    for j in range(n):
        c = A[:, j].astype(np.int64)
        nz = np.flatnonzero(c)
        if len(nz) and c[nz[0]] == 2:
            c = (2 * c) % 3
            neg ^= 1
        for k, r in enumerate(reps):
            if (r == c).all():
                mult[k] += 1
                break
        else:
            reps.append(c)
            mult.append(1)
    m = len(reps)
    tab = np.zeros((2,) + (3,) * m, dtype=np.uint64)
    tab[(0,) + (0,) * m] = 1
    for i in range(n):
        moved = tab
        for k in range(m):
            moved = np.roll(moved, int(reps[k][i]), axis=k + 1)
        tab = tab + moved[::-1]
    digits = np.indices((3,) * m)
    ok = (digits != 0).all(axis=0)
    odd = np.zeros((3,) * m, dtype=np.int64)
    for k in range(m):
        odd ^= (digits[k] == 2).astype(np.int64) * (mult[k] & 1)
    plus = tab[0][ok & (odd == 0)].sum() + tab[1][ok & (odd == 1)].sum()
    minus = tab[0][ok & (odd == 1)].sum() + tab[1][ok & (odd == 0)].sum()
    return [plus, minus] if not neg else [minus, plus]


def exact(case, seed):
    kind = case["kind"]
    if kind == "rankone":
        d, e, _ = _rank_one(seed, case["n"])
        p, m = _rank_one_counts(d.numpy(), e.numpy())
        return torch.tensor([p, m, _residue(case["n"], p, m)], dtype=torch.int64)
    if kind == "pooled":
        return np.array(_few_column_counts(_pooled(seed, case["n"], case["pool"])), dtype=np.uint64)
    if kind in ("device", "host"):
        n = case["n"]
        if n > 22:
            return None
        p, m = (int(x[0]) for x in _terms(_uniform(seed, (1, n, n)), _where()))
        if kind == "host":
            return np.array([p, m], dtype=np.uint64)
        return torch.tensor([p, m, _residue(n, p, m)], dtype=torch.int64)
    if kind == "mc":
        ns = _sizes(case, seed)
        if (2.0 ** ns.astype(np.int64)).sum() > 2.0 ** 29:
            return None
        flat = _uniform(seed, (int((ns.astype(np.int64) ** 2).sum()),))
        off = np.concatenate([[0], np.cumsum(ns.astype(np.int64) ** 2)])
        res = np.zeros(len(ns), dtype=np.uint8)
        for n in range(case["lo"], case["hi"] + 1):
            idx = np.flatnonzero(ns == n)
            per = max(1, (1 << 25) // (n << n))
            for i0 in range(0, len(idx), per):
                part = idx[i0:i0 + per]
                A = torch.stack([flat[off[k]:off[k] + n * n].view(n, n) for k in part])
                p, m = _terms(A, _where())
                res[part] = (((-1) ** n * (p - m)) % 3).cpu().numpy()
        return res, np.bincount(res, minlength=3).astype(np.uint64)
    return None
