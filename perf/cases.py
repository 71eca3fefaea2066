"""Performance cases of the level-line Newton splitter: the calls its users make.

A user splits a polynomial of one of the three families in one of the three
precision tiers, certifies a list of roots, or takes its separation
statistics.  The polynomial is an integer or a pair of integers; what a user
sets besides is the level lambda0 of the line the descents start from (or,
in the double-double tier, the separation of the root set), which the seed
moves by up to 2 % here: the roots are the same, their last digits are not.  The list operations take their points from such a split, and the
certificate a radius cap.

Sizes are those of the benchmark, the README and the tests; the drawn cases
cover the orders that each tier is made for.
"""
from __future__ import annotations

import random

import numpy as np
import torch

import paper_2402_06083_gb300 as mt

LEVEL = {"hyp": 5.0, "mis": 100.0, "q": 100.0, "batch": 100.0}  # the library's lambda0 of each family


def _split(name, kind, l, n, prec, **kw):
    c = {"op": "split", "kind": kind, "l": l, "n": n, "prec": prec, "level": LEVEL[kind], "lo": False, "dd_all": 0}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def _list(name, op, kind, l, n, count, lo=False, mask=False):
    c = {"op": op, "kind": kind, "l": l, "n": n, "count": count, "lo": lo, "mask": mask}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest configuration: a few thousand roots, an interactive call
        _split("hyp12_fp64", "hyp", 0, 12, "fp64"),
        # the plain binary64 tier at its usual size (README's first example)
        _split("hyp20_fp64", "hyp", 0, 20, "fp64"),
        # the same polynomial in the mixed tier, the benchmark's comparison
        _split("hyp20_mixed", "hyp", 0, 20, "mixed"),
        # the mixed tier at its largest usual size
        _split("hyp24_mixed", "hyp", 0, 24, "mixed"),
        # the benchmark's headline: 134 M roots, double-double zones at the tip
        _split("hyp28_dd", "hyp", 0, 28, "dd"),
        # a whole split in double-double, high and low parts returned
        _split("hyp14_dd_all", "hyp", 0, 14, "dd", lo=True, dd_all=1),
        # every s_{l,n} with l + n <= 16 in one pass
        _split("mis16_batch", "batch", 0, 16, "fp64"),
        # a Misiurewicz polynomial past FP80: s_{4,22}, tip roots 4.86e-20 apart
        _split("mis_4_22_dd", "mis", 4, 22, "dd"),
        # q_{9,9} with its multiple roots, types and multiplicities
        _split("q_9_9_fp64", "q", 9, 9, "fp64"),
        # the disk certificate of a whole root list (README's example)
        _list("certify_hyp20", "certify", "hyp", 0, 20, 1 << 19),
        # the Newton-basin certificate of the same list
        _list("basin_hyp20", "basin", "hyp", 0, 20, 1 << 19),
        # nearest-neighbour distances of the centres of exact period 22
        _list("separation_hyp22", "separation", "hyp", 0, 22, 1 << 21, mask=True),
    ]


def draw(rng: random.Random):
    """One more case of the same ranges: the order (the logarithm of the
    work) is uniform over the range of its tier, the level within 20 % above
    the default, list lengths odd as well as even."""
    op = rng.choice(["split"] * 8 + ["certify", "basin", "separation", "separation"])
    if op == "split":
        kind, prec = rng.choice([("hyp", "fp64"), ("hyp", "fp64"), ("hyp", "mixed"), ("hyp", "mixed"), ("hyp", "dd"),
                                 ("mis", "fp64"), ("mis", "mixed"), ("mis", "dd"), ("batch", "fp64"), ("q", "fp64")])
        lo, dd_all = False, 0
        l = 0
        if kind == "hyp":
            n = rng.randint(*{"fp64": (8, 21), "mixed": (13, 25), "dd": (25, 28)}[prec])
            if prec == "dd" and rng.random() < 0.4:
                n, lo, dd_all = rng.randint(8, 14), True, 1
        elif kind == "mis":
            order = rng.randint(*{"fp64": (8, 18), "mixed": (12, 18), "dd": (18, 23)}[prec])
            l = rng.randint(2, order - 1)
            n = order - l
        elif kind == "batch":
            n = rng.randint(6, 16)
        else:
            order = rng.randint(8, 17)
            l = rng.randint(1, order - 1)
            n = order - l
        level = round(LEVEL[kind] * rng.uniform(1.0, 1.2), 3)
        return _split(None, kind, l, n, prec, level=level, lo=lo, dd_all=dd_all)
    n = rng.randint(12, 22)
    count = int(round(2 ** rng.uniform(9.0, n - 1)))
    lo = n <= 14 and rng.random() < 0.5
    return _list(None, op, "hyp", 0, n, count, lo=lo, mask=op == "separation" and rng.random() < 0.5)


# ---------------------------------------------------------------------------
def _level(case, seed):
    return case["level"] * (1.0 + 0.02 * random.Random(seed).random())


def _cap(case, seed):
    """The radius cap of a certificate: up to a fifth below the library's."""
    return (1e-20 if case["lo"] else 1e-12) * (1.0 - 0.2 * random.Random(seed + 2).random())


def _roots(case, seed):
    """The first 'count' roots (in the list's order) of a split."""
    kw = {"lambda0": LEVEL[case["kind"]] * (1.0 + 0.02 * random.Random(seed).random())}
    if case["lo"]:
        kw["dd_all"] = 1
    r = mt.split_hyperbolic(case["n"], "dd" if case["lo"] else "mixed", want_lo=case["lo"], **kw)
    # a window of the sorted list that the seed places
    first = random.Random(seed + 1).randint(0, r.roots.numel() - case["count"])
    z = r.roots[first:first + case["count"]].clone()
    return z, (r.roots_lo[first:first + case["count"]].clone() if case["lo"] else None)


def prepare(case, seed):
    """What a program has in hand: a workspace and the output buffers of a
    split, or the points of a list operation (with the proven radii for the
    basin certificate, the exact-period mask for the separation)."""
    s = {"case": case}
    if case["op"] == "split":
        s["level"] = _level(case, seed)
        s["work"] = mt.Workspace()
        kw = {"lambda0": s["level"]}
        if case["dd_all"]:
            kw["dd_all"] = 1
        elif case["prec"] == "dd":
            # p_n past n = 24 and s_{l,n} past order 17 are split at the library's level; what
            # varies is the separation of the root set, from the library's 64 ulp(2) up
            kw = {"eps_dup": 2.0 ** -45 * s["level"] / LEVEL[case["kind"]]}
        s["kw"] = kw
        if case["kind"] in ("hyp", "mis"):
            s["work"].ensure(mt.workspace_bytes(case["kind"], case["n"], case["l"], mt.options(case["prec"], **kw)))
            d = mt.degree(case["kind"], case["n"], case["l"])
            s["out"] = torch.empty((d, 2), dtype=torch.float64, device="cuda")
            s["out_lo"] = torch.empty((d, 2), dtype=torch.float64, device="cuda") if case["lo"] else None
        return s
    z, zl = _roots(case, seed)
    s["z"], s["zl"] = z, zl
    s["tol"] = _cap(case, seed)
    s["work"] = mt.Workspace()
    if case["op"] == "basin":
        s["radius"] = mt.certify(case["kind"], case["n"], z, l=case["l"], roots_lo=zl)[1]
    s["mask"] = None
    if case["mask"]:
        s["mask"] = (mt.classify(case["kind"], case["n"], z, l=case["l"]) == case["n"]).to(torch.uint8)
    return s


def run(s):
    c = s["case"]
    if c["op"] == "certify":
        ok, rad, n_pass = mt.certify(c["kind"], c["n"], s["z"], l=c["l"], tol=s["tol"], work=s["work"],
                                     roots_lo=s["zl"])
        return {"pass": ok, "radius": rad, "n_pass": n_pass}
    if c["op"] == "basin":
        basin, n_pass = mt.certify_basin(c["kind"], c["n"], s["z"], s["radius"], l=c["l"], work=s["work"],
                                         roots_lo=s["zl"])
        return {"basin": basin, "n_pass": n_pass}
    if c["op"] == "separation":
        nn, bands, least = mt.separation(s["z"], roots_lo=s["zl"], mask=s["mask"], work=s["work"])
        return {"nn": nn, "bands": np.asarray(bands), "least": least}
    if c["kind"] == "batch":
        roots, is_mis, offsets, stats, _ = mt.split_misiurewicz_batch(c["n"], c["prec"], work=s["work"], **s["kw"])
        return {"roots": roots, "is_mis": is_mis, "offsets": np.asarray(offsets),
                "certified": np.asarray([x["n_cert_pass"] for x in stats])}
    if c["kind"] == "q":
        r = mt.split_misiurewicz_q(c["l"], c["n"], c["prec"], work=s["work"], **s["kw"])
        return {"roots": r.roots, "mult": r.mult, "pre": r.pre, "per": r.per, "certified": r.stats["n_cert_pass"]}
    if c["kind"] == "hyp":
        r = mt.split_hyperbolic(c["n"], c["prec"], work=s["work"], want_lo=c["lo"], out=s["out"], out_lo=s["out_lo"],
                                **s["kw"])
    else:
        r = mt.split_misiurewicz(c["l"], c["n"], c["prec"], work=s["work"], want_lo=c["lo"], out=s["out"],
                                 out_lo=s["out_lo"], **s["kw"])
    out = {"roots": r.roots, "certified": r.stats["n_cert_pass"], "types": np.asarray(r.stats["count_by_type"])}
    if r.roots_lo is not None:
        out["roots_lo"] = r.roots_lo
    if r.is_mis is not None:
        out["is_mis"] = r.is_mis
    return out


# ---------------------------------------------------------------------------
def _orbit_len(kind, l, n):
    return n if kind == "hyp" else l + n - 1 if kind == "mis" else l + n


def work(case):
    """Bytes: each given point read once, each result written once.  Flops:
    an orbit step of P and P' is 13, and per root of the upper half the
    method evaluates at least the 8 points of a turn of the level line, about
    8 Newton steps for each of the 4 descents and one certificate (26 a
    step); a list operation one certificate, or a handful of distances."""
    k, l, n = case["kind"], case["l"], case["n"]
    if case["op"] == "split":
        pairs = [(l, n)] if k != "batch" else mt.misiurewicz_pairs(n)
        flops = d = 0
        for a, b in pairs:
            kk = "mis" if k == "batch" else k
            m = _orbit_len(kk, a, b)
            deg = 2 ** (m if kk == "q" else m) // 2
            d += deg
            flops += deg // 2 * m * (13 * (8 + 4 * 8) + 26)
        return {"bytes": 16.0 * d * (2 if case["lo"] else 1), "flops": float(flops)}
    c, m = case["count"], _orbit_len(k, l, n)
    pts = 32 if case["lo"] else 16
    if case["op"] == "certify":
        return {"bytes": float(c * (pts + 9)), "flops": float(c * 26 * m)}
    if case["op"] == "basin":
        return {"bytes": float(c * (pts + 16)), "flops": float(c * 2 * 26 * m)}
    return {"bytes": float(c * (pts + 8 + (1 if case["mask"] else 0))), "flops": float(c * 8 * 6)}


# ---------------------------------------------------------------------------
# Plain torch in 64 bits: every root of p_n and s_{l,n} by the same theory
# (lift of a circle through the nested family, Newton), every step on all
# points at once.
def _eval(m, lcap, alpha, c):
    """P and P' at c for P = p_m + alpha p_lcap (lcap: None or one per point)."""
    z = torch.zeros_like(c)
    d = torch.zeros_like(c)
    zc, dc = torch.zeros_like(c), torch.zeros_like(c)
    for k in range(1, m + 1):
        d = 2.0 * z * d + 1.0
        z = z * z + c
        if lcap is not None:
            at = lcap == k
            zc = torch.where(at, z, zc)
            dc = torch.where(at, d, dc)
    return (z, d) if lcap is None else (z + alpha * zc, d + alpha * dc)


def _unique(z, d, eps):
    """The distinct points of z folded into the upper half, conjugates added,
    in (Re, Im) order; None unless there are d of them."""
    x, y = z.real.clone(), z.imag.abs()
    y = torch.where(y < 0.5 * eps, torch.zeros_like(y), y)
    order = torch.argsort(x, stable=True)
    x, y = x[order], y[order]
    new = torch.ones(x.numel(), dtype=torch.bool, device=x.device)
    for k in range(1, min(x.numel(), 4096)):
        near = x[k:] - x[:-k] < eps
        if not bool(near.any()):
            break
        new[k:] &= ~(near & ((y[k:] - y[:-k]).abs() < eps))
    x, y = x[new], y[new]
    up = y > 0
    x, y = torch.cat([x, x[up]]), torch.cat([y, -y[up]])
    if d is not None and x.numel() != d:
        return None
    o = torch.argsort(y, stable=True)
    o = o[torch.argsort(x[o], stable=True)]
    return torch.complex(x[o], y[o])


def _all_roots(m, lcaps, level):
    """Converged Newton limits from 4 d starts of the upper half of |P| =
    level, one row per polynomial p_m + p_lcap (lcaps: None for p_m alone)."""
    d = 1 << (m - 1)
    s = torch.arange(2 * d + 1, device="cuda", dtype=torch.int64)
    rows = 1 if lcaps is None else len(lcaps)
    s = s.repeat(rows)
    cap = None if lcaps is None else torch.tensor(lcaps, device="cuda").repeat_interleave(2 * d + 1)
    full = 4 * d

    def unit(k):  # e^{2 i pi 2^k s / (4 d)}
        t = ((s << k) % full).to(torch.float64) * (2.0 * np.pi / full)
        return torch.polar(torch.ones_like(t), t)

    z = level * unit(0)
    for k in range(1, m):
        u = unit(k)
        for q in range(1, 5):
            t = level ** (2.0 - q / 4.0) * u
            for _ in range(6):
                v, dv = _eval(k + 1, None, 0.0, z)
                z = z - (v - t) / dv
    if cap is not None:
        t = level * unit(m - 1)
        for a in range(1, 9):
            for _ in range(5):
                v, dv = _eval(m, cap, a / 8.0, z)
                z = z - (v - t) / dv
    for it in range(2 * m + 24):
        v, dv = _eval(m, cap, 1.0, z)
        q = v / dv
        z = torch.where(torch.isfinite(q.real) & torch.isfinite(q.imag) & (z.abs() < 1e3), z - q, z)
    # every root lies in |c| <= 2 (an escaped point's quotient can underflow to 0)
    z = torch.where((q.abs() <= 1e-14) & (z.abs() < 2.1), z, torch.full_like(z, float("nan")))
    return [r[torch.isfinite(r.real) & torch.isfinite(r.imag)] for r in z.view(rows, -1)]


def _nearest(x, y):
    """Distance from each point to the nearest other: along the list sorted
    by Re until the gap in Re exceeds the best on both sides."""
    o = torch.argsort(x)
    x, y = x[o], y[o]
    n = x.numel()
    best = torch.full_like(x, float("inf"))
    i = torch.arange(n, device=x.device)
    k = 0
    while i.numel() and k < n:
        more = torch.zeros_like(i, dtype=torch.bool)
        for k in range(k + 1, k + 17):
            b = best[i]
            more.zero_()
            for j in (i + k, i - k):
                ok = (j >= 0) & (j < n)
                j = j.clamp(0, n - 1)
                gap = (x[j] - x[i]).abs()
                ok &= gap <= b
                h = torch.hypot(gap, y[j] - y[i])
                b = torch.where(ok & (h < b), h, b)
                more |= ok
            best[i] = b
        i = i[more]
    out = torch.empty_like(best)
    out[o] = best
    return out


def exact(case, seed):
    k, n = case["kind"], case["n"]
    if case["op"] == "split":
        level = _level(case, seed)
        if k == "hyp" and n <= 20:
            r = _unique(_all_roots(n, None, level)[0], 1 << (n - 1), 1e-12 if n > 8 else 1e-9)
            return None if r is None else {"roots": r, "certified": None, "types": None}
        if k == "mis" and case["l"] + n <= 17:
            m = case["l"] + n - 1
            r = _unique(_all_roots(m, [case["l"] - 1], level)[0], 1 << (m - 1), 1e-12)
            return None if r is None else {"roots": r, "certified": None, "types": None}
        if k == "batch":
            got = {}
            for order in range(3, n + 1):
                pairs = [(l, order - l) for l in range(2, order)]
                for (l, b), z in zip(pairs, _all_roots(order - 1, [l - 1 for l, _ in pairs], level)):
                    got[l, b] = _unique(z, 1 << (order - 2), 1e-11)
            # pairs ordered by l, then n
            rows = [got[l, b] for l in range(2, n) for b in range(1, n - l + 1)]
            return None if any(r is None for r in rows) else {"roots": torch.cat(rows), "certified": None}
        return None
    if case["lo"] or case["op"] == "basin":
        return None
    z, _ = _roots(case, seed)
    if case["op"] == "certify":
        nn = _nearest(z.real.contiguous(), z.imag.contiguous())
        # the radius cap, where no neighbour is near enough to lower it
        if float(nn.min()) < 1e-11:
            return None
        return {"pass": None, "radius": torch.full((z.numel(),), _cap(case, seed), dtype=torch.float64, device="cuda")}
    on = None
    if case["mask"]:
        on = mt.classify(k, n, z, l=case["l"]) == n  # the given mask, an input
        z = z[on]
    nn = _nearest(z.real.contiguous(), z.imag.contiguous())
    if on is not None:
        full = torch.zeros(on.numel(), dtype=torch.float64, device="cuda")
        full[on] = nn
        return {"nn": full, "bands": None, "least": float(nn.min())}
    return {"nn": nn, "bands": None, "least": float(nn.min())}
