"""The scans that users of this package run, as timing cases.

Each case is one whole pass through the public Python entry points on inputs that
are already where a user has them (on the GPU; in page-locked host memory for the
end-to-end entry).  Hit lists come back in unspecified order, so a pass puts them
into a result table of a fixed number of rows, in (SNP, trait) order, as a program
that reports them does (rows past the last hit stay zero).

`exact` evaluates the same statistics in 64 bits with plain torch, from the
definitions: average ranks, tie-corrected Kruskal-Wallis H, chi-square tails,
one-way ANOVA F and dosage-regression t.
"""
from __future__ import annotations

import math

import torch

import paper_1307_3519_gb300 as krux

DEV = "cuda"
CAUSAL_BLOCK = 1000  # SNPs of one linkage-disequilibrium block
BIN_WIDTH, BINS = 0.1, 40  # histogram of the empirical FDR
COHORT_NS = (48, 75, 102, 150, 200, 300, 400, 500)
CHROMS, CHROM_LEN, CIS_WINDOW = 22, 150_000_000, 1_000_000


def listed():
    return [
        # a candidate panel with rounded expression values (many ties): the smallest
        # call, dominated by launches and host work
        dict(name="panel", kind="scan", T=500, S=2_000, N=60, p=1e-3, geno="hwe", expr="rounded", causal=0),
        # the same kind of panel kept as a captured graph and replayed per request
        dict(name="panel_graph", kind="graph", T=2_000, S=10_000, N=102, p=1e-4, geno="ld", expr="log", causal=2),
        # the full table of H and p of a candidate region (every pair is written)
        dict(name="region_dense", kind="dense", T=1_000, S=20_003, N=102, p=1e-4, geno="ld", expr="log", causal=2),
        # a genome-wide scan of one tissue with planted associations: the largest
        # plain scan
        dict(name="genome", kind="scan", T=20_000, S=500_000, N=102, p=1e-5, geno="ld", expr="log", causal=1),
        # a biobank-sized cohort: many samples, odd sizes, independent SNPs
        dict(name="many_samples", kind="scan", T=9_973, S=100_003, N=301, p=1e-6, geno="hwe", expr="log", causal=0),
        # the whole analysis from host arrays (copies in and out included)
        dict(name="genome_host", kind="host", T=20_000, S=500_000, N=102, p=1e-7, geno="hwe", expr="log", causal=0),
        # missing genotypes (200 sample patterns) and 1 % missing expression values
        dict(name="missing", kind="scan", T=5_000, S=100_000, N=102, p=1e-4, geno="ld", expr="nan", causal=0, patterns=200),
        # permutation null with the empirical-FDR histogram
        dict(name="permutations", kind="permute", T=20_000, S=200_000, N=102, p=1e-5, geno="ld", expr="log", causal=1, P=16),
        # eight cohorts of uneven sample counts in one call
        dict(name="cohorts", kind="cohorts", T=15_000, S=300_000, N=500, p=1e-5, cohorts=8),
        # local associations: pairs within 1 Mbp of each other
        dict(name="cis", kind="cis", T=20_000, S=500_000, N=102, p=1e-4, geno="ld", expr="log", causal=1),
        # markers with two to five genotype groups
        dict(name="multiallelic", kind="multi", T=20_000, S=100_000, N=102, p=1e-5, geno="multi", expr="log", causal=0),
        # the parametric comparison, on expression that is normal already
        dict(name="anova", kind="anova", T=20_000, S=100_000, N=102, p=1e-5, geno="ld", expr="normal", causal=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["scan"] * 6 + ["nan"] * 2 + ["graph", "dense", "host", "permute", "permute", "cohorts",
                                                  "cis", "multi", "anova", "linear"])
    N = rng.choice([rng.randint(24, 128), rng.randint(24, 128), rng.randint(129, 512)])
    T = _log(rng, 300, 20_000)
    S = _log(rng, 2_000, 500_000)
    geno = rng.choice(["ld", "ld", "hwe"])
    c = dict(kind=kind, T=T, S=S, N=N, geno=geno, expr="log", causal=rng.choice([0, 1, 3]))
    if kind == "scan":
        c["expr"] = rng.choice(["log", "log", "rounded"])
    elif kind == "nan":
        c.update(kind="scan", expr="nan", causal=0, T=min(T, 8_000), S=min(S, 200_000), N=min(N, 160),
                 patterns=rng.choice([0, rng.randint(1, 300)]))
    elif kind == "graph":
        c.update(T=min(T, 5_000), S=min(S, 50_000))
    elif kind == "dense":
        c.update(T=min(T, 2_000), S=min(S, 40_000))
    elif kind == "permute":
        c.update(P=rng.randint(2, 16), S=min(S, 100_000), N=min(N, 200))
    elif kind == "cohorts":
        c = dict(kind=kind, T=T, S=min(S, 100_000), N=500, cohorts=rng.randint(2, 8))
    elif kind == "cis":
        c.update(S=max(S, 20_000))
    elif kind == "multi":
        c.update(geno="multi", causal=0, S=min(S, 100_000), N=min(N, 200))
    elif kind in ("anova", "linear"):
        c.update(S=min(S, 100_000), N=min(N, 250), expr="normal")
    if c.get("geno") == "hwe":  # associations are planted through the founders of LD blocks
        c["causal"] = 0
    pairs = c["T"] * c["S"]
    c["p"] = rng.choice([1e-3, 1e-4] if pairs < 2e7 else [1e-4, 1e-5] if pairs < 1e9 else [1e-5, 1e-6])
    return c


# ---- inputs -------------------------------------------------------------------

def _hwe(g, maf, rows, N):
    u = torch.rand((rows, N), generator=g, device=DEV)
    q = maf[:, None]
    return (u >= (1 - q) ** 2).to(torch.int8) + (u >= 1 - q * q).to(torch.int8)


def _genotypes(g, c, N):
    """(codes int8 [S, N], founders or None)."""
    S = c["S"]
    if c.get("geno", "hwe") == "hwe":
        return _hwe(g, 0.05 + 0.45 * torch.rand(S, generator=g, device=DEV), S, N), None
    if c["geno"] == "multi":  # codes 0..k with k in 1..4 and uneven frequencies
        k = torch.randint(2, 6, (S,), generator=g, device=DEV)
        f = torch.rand((S, 5), generator=g, device=DEV).neg().log1p().neg() ** 0.7 + 1e-3
        f = f * (torch.arange(5, device=DEV)[None] < k[:, None])
        edge = (f / f.sum(1, keepdim=True)).cumsum(1)[:, :4].contiguous()
        u = torch.rand((S, N), generator=g, device=DEV)
        code = torch.zeros((S, N), dtype=torch.int8, device=DEV)
        for i in range(4):
            code += (u >= edge[:, i:i + 1]).to(torch.int8)
        return torch.minimum(code, (k - 1)[:, None].to(torch.int8)), None
    nb = -(-S // CAUSAL_BLOCK)
    maf = (0.01 if c["causal"] else 0.05) + 0.49 * torch.rand(nb, generator=g, device=DEV).clamp(max=0.9)
    founders = _hwe(g, maf, nb, N)
    blk = torch.arange(S, device=DEV) // CAUSAL_BLOCK
    codes = founders[blk]
    fresh = _hwe(g, maf[blk], S, N)
    redraw = torch.rand((S, N), generator=g, device=DEV) < 0.02
    return torch.where(redraw, fresh, codes), founders


def _expression(g, c, N, founders):
    T = c["T"]
    z = torch.randn((T, N), generator=g, device=DEV)
    kind = c.get("expr", "log")
    if kind == "rounded":
        return (z * 100).round() / 100
    if founders is not None:  # one standard deviation on the log scale in one genotype
        for _ in range(c.get("causal", 0)):  # group, for about every third trait
            b = torch.randint(0, founders.shape[0], (T,), generator=g, device=DEV)
            k = torch.randint(0, N, (T,), generator=g, device=DEV)
            f = founders[b]
            has = torch.rand((T, 1), generator=g, device=DEV) < 0.3
            z = z + ((f == f.gather(1, k[:, None])) & has).float()
    if kind == "normal":
        return z
    x = z.exp()
    x = torch.where(torch.rand((T, N), generator=g, device=DEV) < 0.01, x * 10, x)
    if kind == "nan":
        x = torch.where(torch.rand((T, N), generator=g, device=DEV) < 0.01, torch.full_like(x, math.nan), x)
    return x.contiguous()


def _missing_patterns(g, c, codes):
    """10 % of the SNPs miss the two samples of one of `patterns` patterns."""
    n = c.get("patterns", 0)
    if not n:
        return codes
    S, N = codes.shape
    first = torch.randint(0, N, (n,), generator=g, device=DEV)
    second = (first + torch.randint(1, N, (n,), generator=g, device=DEV)) % N
    rows = torch.randperm(S, generator=g, device=DEV)[: S // 10]
    which = torch.randint(0, n, (rows.numel(),), generator=g, device=DEV)
    codes[rows, first[which]] = -1
    codes[rows, second[which]] = -1
    return codes


def _positions(g, c):
    """Sorted global coordinates (chromosome * 2^40 + base) of SNPs and traits."""
    out = []
    for n in (c["S"], c["T"]):
        chrom = torch.randint(0, CHROMS, (n,), generator=g, device=DEV)
        pos = torch.randint(0, CHROM_LEN, (n,), generator=g, device=DEV)
        out.append(((chrom << 40) + pos).sort().values)
    return out


def _inputs(case, seed):
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    c = dict(case)
    if c["kind"] == "cohorts":
        ns = COHORT_NS[-c["cohorts"]:]
        both = []
        for n in ns:
            both.append((_expression(g, c, n, None), _genotypes(g, c, n)[0]))
        return dict(cohorts=both)
    codes, founders = _genotypes(g, c, c["N"])
    d = dict(geno=_missing_patterns(g, c, codes), expr=_expression(g, c, c["N"], founders))
    if c["kind"] == "cis":
        d["snp_pos"], d["trait_pos"] = _positions(g, c)
    if c["kind"] == "permute":
        d["perms"] = torch.rand((c["P"], c["N"]), generator=g, device=DEV).argsort(1).to(torch.int32)
    return d


def _rows(c):
    """Rows of the result table: room for the expected hits twice over (a planted
    association's block is up to 1000 correlated SNPs)."""
    pairs = c["T"] * c["S"]
    planted = 0.25 * c["T"] * min(c.get("causal", 0) * CAUSAL_BLOCK, c["S"])
    return int(min(pairs, 2 * c["p"] * pairs + planted + 4096))


def _table(rows, stat, **how):
    return {"hits": torch.zeros((rows, 4), dtype=torch.int32, **how), stat: torch.zeros(rows, dtype=torch.float64, **how),
            "p": torch.zeros(rows, dtype=torch.float64, **how)}


_context = None


def prepare(case, seed):
    global _context
    if _context is None:  # one library context per process, as in a user's program
        _context = krux.Krux(torch.cuda.current_device())
    kind, rows = case["kind"], _rows(case)
    stat = "stat" if kind in ("anova", "linear") else "H"
    s = dict(case=dict(case), ctx=_context, cap=rows, stat=stat, **_inputs(case, seed))
    how = dict(device="cpu" if kind == "host" else DEV)
    s["table"] = [_table(rows, stat, **how) for _ in s.get("cohorts", [0])]
    if kind == "host":
        s["expr"] = s["expr"].cpu().pin_memory()
        s["geno"] = s["geno"].cpu().pin_memory()
        s["out"] = tuple(v.pin_memory() for v in _table(rows, stat).values())
    elif kind == "graph":
        s["rs"] = s["ctx"].krux_rank(s["expr"])
        s["graph"] = s["ctx"].graph_scan(s["rs"], s["geno"], case["p"], s["cap"])
    return s


# ---- one pass --------------------------------------------------------------------

def _report(r, table, stat="H"):
    """The hit list into the result table, in (SNP, trait) order."""
    hits = torch.as_tensor(r["hits"])
    if hits.shape[0] == 0:
        return dict(table, n_hits=r["n_hits"])
    order = hits.view(torch.int64)[:, 0].argsort()  # snp << 32 | trait
    record = torch.complex128  # a hit record moves as one 16-byte element
    for v, to in ((hits.view(record)[:, 0], table["hits"].view(record)[:, 0]),
                  (torch.as_tensor(r[stat]), table[stat]), (torch.as_tensor(r["p"]), table["p"])):
        torch.index_select(v, 0, order, out=to[: order.numel()])
    return dict(table, n_hits=r["n_hits"])


def run(state):
    c, kx, table = state["case"], state["ctx"], state["table"][0]
    kind, p, cap = c["kind"], c["p"], state["cap"]
    if kind == "graph":
        state["graph"].launch()
        return _report(state["graph"].wait()[0], table)
    if kind == "host":
        return _report(kx.krux_scan_host(state["expr"], state["geno"], p, cap, out=state["out"]), table)
    if kind in ("anova", "linear"):
        return _report(kx.krux_scan_parametric(state["expr"], state["geno"], kind, p, cap), table, "stat")
    if kind == "cohorts":
        group = [dict(rs=kx.krux_rank(e), geno=g, capacity=cap) for e, g in state["cohorts"]]
        out = [_report(r, t) for r, t in zip(kx.krux_scan_grouped(group, p), state["table"])]
        for x in group:
            x["rs"].free()
        return out
    rs = kx.krux_rank(state["expr"])
    if kind == "dense":
        r = kx.krux_scan(rs, state["geno"], p, cap, dense=True)
        out = dict(_report(r, table), dense_H=r["dense_H"], dense_p=r["dense_p"])
    elif kind == "cis":
        r = kx.krux_scan_cis(rs, state["geno"], state["snp_pos"], state["trait_pos"], CIS_WINDOW, p, cap)
        out = _report(r, table)
    elif kind == "permute":
        r = kx.krux_permute(rs, state["geno"], state["perms"], p, cap, fdr_bins=BINS, fdr_bin_width=BIN_WIDTH)
        out = dict(_report(r, table), minp=r["minp"], fdr_hist=r["fdr_hist"])
    else:
        out = _report(kx.krux_scan(rs, state["geno"], p, cap, multiallelic=kind == "multi"), table)
    rs.free()
    return out


def work(case):
    c = case
    T, S, N, kind = c["T"], c["S"], c["N"], c["kind"]
    if kind == "cohorts":
        ns = COHORT_NS[-c["cohorts"]:]
        return {"bytes": float(sum(4 * T * n + S * n + 32 * c["p"] * T * S for n in ns)),
                "flops": float(sum(4.0 * T * S * n for n in ns))}
    pairs = float(T) * S
    if kind == "cis":
        pairs *= 2.0 * CIS_WINDOW / (CHROMS * float(CHROM_LEN))
    # two indicator columns per three-group marker (four per marker of up to five
    # groups, one dosage column for the regression), a multiply and an add each
    flops = {"multi": 8.0, "linear": 2.0}.get(kind, 4.0) * N * pairs * (1 + c.get("P", 0))
    # a few per cent of a planted trait's block are hits
    hits = c["p"] * pairs + 0.03 * T * min(c.get("causal", 0) * CAUSAL_BLOCK, S) * (kind != "cis")
    size = 4 * T * N + S * N + 32 * hits
    if kind == "dense":
        size += 16 * pairs
    if kind == "permute":
        size += 8 * c["P"] * T
    return {"bytes": float(size), "flops": float(flops)}


# ---- 64-bit values -----------------------------------------------------------------

BLOCK = 1 << 27  # pairs evaluated at a time


def _ranks(x):
    """Centred ranks 2 * rank - (K + 1) (0 at NaN), K and sum(t^3 - t) of every row."""
    nan = torch.isnan(x)
    K = (~nan).sum(1)
    s = torch.where(nan, torch.full_like(x, math.inf), x).sort(1).values.contiguous()
    v = torch.where(nan, torch.full_like(x, math.inf), x).contiguous()
    lo = torch.searchsorted(s, v)
    hi = torch.minimum(torch.searchsorted(s, v, right=True), K[:, None])
    eq = torch.where(nan, torch.ones_like(lo), hi - lo)
    a = torch.where(nan, torch.zeros_like(lo), lo + hi - K[:, None])
    return a, K, (eq * eq - 1).sum(1)


def _tail(H, df):
    """Upper chi-square tail for df 1..4."""
    x = 0.5 * H
    one, two = torch.erfc(x.sqrt()), torch.exp(-x)
    three = one + 2 / math.sqrt(math.pi) * x.sqrt() * two
    p = torch.where(df == 1, one, torch.where(df == 2, two, torch.where(df == 3, three, two * (1 + x))))
    return torch.where((df > 0) & (H > 0), p, torch.ones_like(p))


def _threshold(p, df):
    """h with _tail(h, df) = p, by bisection, for df 1..4."""
    lo, hi = 0.0, 2000.0
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        t = float(_tail(torch.tensor([mid], dtype=torch.float64), torch.tensor([df]))[0])
        lo, hi = (mid, hi) if t > p else (lo, mid)
    return lo


def _pairs(rank, codes, present=None, groups=3):
    """H and df of every (trait, SNP) pair of a block.
    The sums are whole numbers below 2^24, which 32-bit products and sums hold exactly;
    everything after them is in 64 bits."""
    a, K, tie = rank
    af = a.float()
    pf = None if present is None else present.float()
    Q, df = 0.0, -1
    for i in range(groups):
        I = (codes == i).float()
        D = (af @ I.t()).double()
        n = I.sum(1).double()[None] if pf is None else (pf @ I.t()).double()
        Q = Q + torch.where(n > 0, D * D / n.clamp(min=1), torch.zeros_like(D))
        df = df + (n > 0).long()
    k = K.double()[:, None]
    denom = k * (k + 1) * (1 - tie.double()[:, None] / (k ** 3 - k).clamp(min=1))
    ok = (denom > 0) & (K[:, None] > 1)
    H = torch.where(ok, 3 * Q / torch.where(ok, denom, torch.ones_like(denom)), torch.zeros_like(Q))
    return H, df.expand_as(H)


def _sorted(found, case, stat="H"):
    t, s, H, p = (torch.cat(x) for x in zip(*found)) if found else [torch.zeros(0, device=DEV)] * 4
    o = ((s.long() << 32) | t.long()).argsort()[: _rows(case)]
    table = _table(_rows(case), stat, device=DEV)
    table[stat][: o.numel()] = H[o]
    table["p"][: o.numel()] = p[o]
    return dict(table, hits=None, n_hits=None)


def _kw_hits(expr, geno, pth, groups=3, rows=None, window=None, dense=None):
    """Hits of one expression matrix against SNP rows (`rows`: their indices)."""
    nan = torch.isnan(expr)
    rank = _ranks(expr)
    present = ~nan if bool(nan.any()) else None
    h = torch.tensor([math.inf] + [_threshold(pth, k) for k in range(1, 5)], dtype=torch.float64, device=DEV)
    T, S = expr.shape[0], geno.shape[0]
    st = min(T, 4096)
    step = max(256, BLOCK // st)
    found = []
    for t0 in range(0, T, st):
        r = [x[t0:t0 + st] for x in rank]
        lo, hi = 0, S
        if window is not None:
            sp, tp = window[0], window[1][t0:t0 + st]
            lo = int(torch.searchsorted(sp, tp[:1] - CIS_WINDOW))
            hi = int(torch.searchsorted(sp, tp[-1:] + CIS_WINDOW, right=True))
        for s0 in range(lo, hi, step):
            s1 = min(hi, s0 + step)
            H, df = _pairs(r, geno[s0:s1], None if present is None else present[t0:t0 + st], groups)
            if dense is not None:
                dense[0][t0:t0 + st, s0:s1] = H
                dense[1][t0:t0 + st, s0:s1] = _tail(H, df)
            maybe = H > h[df.clamp(0, 4)] * (1 - 1e-9)
            if window is not None:
                maybe &= (sp[None, s0:s1] - tp[:, None]).abs() <= CIS_WINDOW
            at = maybe.nonzero(as_tuple=True)
            Hh = H[at]
            ph = _tail(Hh, df[at])
            k = ph < pth
            t, s = at[0][k] + t0, at[1][k] + s0
            found.append((t, s if rows is None else rows[s], Hh[k], ph[k]))
    return found


def _exact_permute(d, c):
    real = _kw_hits(d["expr"], d["geno"], c["p"])
    rank = _ranks(d["expr"])
    T, S = d["expr"].shape[0], d["geno"].shape[0]
    st, step = min(T, 4096), max(256, BLOCK // min(T, 4096))
    minp = torch.ones((c["P"], T), dtype=torch.float64, device=DEV)
    for q in range(c["P"]):
        a = rank[0][:, d["perms"][q].long()]
        for t0 in range(0, T, st):
            best = [torch.zeros(min(st, T - t0), dtype=torch.float64, device=DEV) for _ in range(2)]
            for s0 in range(0, S, step):
                H, df = _pairs((a[t0:t0 + st], rank[1][t0:t0 + st], rank[2][t0:t0 + st]), d["geno"][s0:s0 + step])
                for k in (0, 1):
                    best[k] = torch.maximum(best[k], torch.where(df == k + 1, H, torch.zeros_like(H)).amax(1))
            for k in (0, 1):
                m = _tail(best[k], torch.full_like(best[k], k + 1).long())
                minp[q, t0:t0 + st] = torch.minimum(minp[q, t0:t0 + st], m)
    return dict(_sorted(real, c), minp=minp, fdr_hist=None)


def _half_beta(x, a):
    """I_x(a, 1/2) by the hypergeometric series (x well below 1 for small tails)."""
    term, total = torch.ones_like(x), torch.ones_like(x)
    for k in range(1, 600):
        term = term * x * (k - 0.5) / k
        total = total + term * a / (a + k)
    lb = math.lgamma(a) + math.lgamma(0.5) - math.lgamma(a + 0.5)
    return (a * x.log() - math.log(a) - lb).exp() * total


def _exact_parametric(d, c):
    x = d["expr"].double()
    x = x - x.mean(1, keepdim=True)
    sst = (x * x).sum(1)
    N, T, S = c["N"], c["T"], c["S"]
    found = []
    st, step = min(T, 4096), max(256, BLOCK // min(T, 4096))
    for t0 in range(0, T, st):
        xt, v = x[t0:t0 + st], sst[t0:t0 + st, None]
        for s0 in range(0, S, step):
            codes = d["geno"][s0:s0 + step]
            if c["kind"] == "linear":
                g = codes.double()
                g = g - g.mean(1, keepdim=True)
                sxx = (g * g).sum(1)[None]
                r2 = torch.where((sxx > 0) & (v > 0), (xt @ g.t()) / (sxx * v).clamp(min=1e-300).sqrt(), 0.0)
                d2 = torch.full_like(r2, N - 2.0)
                stat = r2 * (d2 / (1 - r2 * r2).clamp(min=1e-300)).sqrt()
                f, d1 = stat * stat, torch.ones_like(stat)
            else:
                ssb, groups = 0.0, 0
                for i in range(3):
                    I = (codes == i).double()
                    n = I.sum(1)[None]
                    D = xt @ I.t()
                    ssb = ssb + torch.where(n > 0, D * D / n.clamp(min=1), torch.zeros_like(D))
                    groups = groups + (n > 0).double()
                d1 = (groups - 1).expand_as(ssb)
                d2 = N - groups.expand_as(ssb)
                ok = (d1 > 0) & (v > 0)
                stat = torch.where(ok, (ssb / d1.clamp(min=1)) / ((v - ssb).clamp(min=1e-300) / d2), 0.0)
                f = stat
            at = (f > 6.0).nonzero(as_tuple=True)  # below it p is above every threshold used here
            F, a1, a2 = f[at], d1[at], d2[at]
            p = torch.where(a1 == 2, (1 + 2 * F / a2) ** (-a2 / 2), torch.zeros_like(F))
            one = a1 == 1
            if bool(one.any()):
                nu = float(a2[one][0])
                p[one] = _half_beta(nu / (nu + F[one]), nu / 2)
            k = p < c["p"]
            found.append((at[0][k] + t0, at[1][k] + s0, stat[at][k], p[k]))
    return _sorted(found, c, "stat")


def exact(case, seed):
    d, kind, pth = _inputs(case, seed), case["kind"], case["p"]
    if kind == "cohorts":
        return [_sorted(_kw_hits(e, g, pth), case) for e, g in d["cohorts"]]
    if kind in ("anova", "linear"):
        return _exact_parametric(d, case)
    if kind == "permute":
        return _exact_permute(d, case)
    geno, expr = d["geno"], d["expr"]
    extra = {}
    dense = None
    if kind == "dense":
        dense = [torch.empty((case["T"], case["S"]), dtype=torch.float64, device=DEV) for _ in range(2)]
        extra = dict(dense_H=dense[0], dense_p=dense[1])
    window = (d["snp_pos"], d["trait_pos"]) if kind == "cis" else None
    if case.get("patterns", 0):
        miss = geno < 0
        complete = (~miss.any(1)).nonzero()[:, 0]
        found = _kw_hits(expr, geno[complete], pth, rows=complete)
        rest = miss.any(1).nonzero()[:, 0]
        masks, of = torch.unique(miss[rest], dim=0, return_inverse=True)
        for b in range(masks.shape[0]):
            rows = rest[of == b]
            x = torch.where(masks[b][None], torch.full_like(expr, math.nan), expr)
            found += _kw_hits(x, geno[rows], pth, rows=rows)
    else:
        found = _kw_hits(expr, geno, pth, groups=5 if kind == "multi" else 3, window=window, dense=dense)
    return dict(_sorted(found, case), **extra)
