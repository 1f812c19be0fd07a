"""The work that a user of this framework has it do, as measurable cases.

Kinds (all through the package's public entry points):

  cycles     ``REWL.run_cycles`` on a run in progress: the sampling of every
             walker, the exchanges, the flatness checks; then the walkers'
             state and the tables (whole where they are small, else through
             ``REWL.digest``, the call for tables too large to copy out).
  batch      ``Batch.run_cycles`` over runs of different lattice sizes.
  whole      a run from creation to its final ln f and its joined ln g.
  join       ``REWL.lng``: merge, join and normalisation of sampled tables.
  jackknife  ``REWL.jackknife``: the join once per left-out walker.
  eq5        ``relative_difference`` of two joined tables (Eq. 5).

Sizes are those of ``paper_1508_02748_gb300.workloads`` and of the tests, with
the library's automatic choice of sampler tiling (a default ``Config``).
"""
import math

import numpy as np
import torch

import paper_1508_02748_gb300 as P
from paper_1508_02748_gb300 import rewl as R
from paper_1508_02748_gb300 import workloads as W

WHOLE_TABLES = 1_000_000    # table entries up to which a run's tables are returned whole


def _cycles(name, w, precision, cycles, warm=0, **kw):
    c = dict(kind="cycles", name=name, L=w.L, nE=w.n_win_E, nM=w.n_win_M, oE=w.overlap_E, oM=w.overlap_M,
             walkers=w.walkers_per_window, precision=precision, interval=w.exchange_interval,
             check_every=w.check_every, cycles=cycles, warm=warm)
    c.update(kw)
    return c


def listed():
    return [
        # Eq. 5 between two runs at the paper's smallest lattice: the smallest call, launch latency alone
        dict(kind="eq5", name="eq5_L8", L=8),
        # and at the largest lattice the library takes: 16.8 million bins
        dict(kind="eq5", name="eq5_L64", L=64),
        # the joined ln g(E, M) a user reads while the L = 8 workload runs
        dict(kind="join", name="join_L8", L=8, nE=3, nM=3, oE=0.75, oM=0.75, walkers=4, marginal=False, per_slice=False),
        # the E marginal of the paper's own split (E only, 50% overlap), by the per-slice rescaling rule
        dict(kind="join", name="join_L16_paper_slices", L=16, nE=3, nM=1, oE=0.5, oM=0.5, walkers=3, marginal=True,
             per_slice=True),
        # the join of the batched workload, L = 32: 2048 walkers, 3.1 GB of tables
        dict(kind="join", name="join_L32", L=32, nE=16, nM=4, oE=0.75, oM=0.75, walkers=32, marginal=False,
             per_slice=False),
        # error bars of the uneven batch's L = 16 member: 32 leave-one-out joins
        dict(kind="jackknife", name="jackknife_L16", L=16, nE=4, nM=2, oE=0.75, oM=0.75, walkers=32, marginal=False,
             per_slice=False),
        # a whole run at the L = 4 check workload's size, with the walkers that meet the error gate: creation, 21
        # iterations polled every 64 cycles, the joined table
        dict(kind="whole", name="whole_L4_w16", L=4, nE=1, nM=1, walkers=16, lnf_final=1e-6, flatness=0.8,
             interval=10_000),
        # the L = 8 workload in mid-run, polled every 64 cycles: few walkers, each one's chain is the time
        _cycles("cycles_L8", W.REWL_L8, P.FP64, 64, warm=500),
        # an odd lattice (two words a row) with a ragged number of walkers, intervals and checks
        dict(kind="cycles", name="cycles_L33_ragged", L=33, nE=7, nM=3, oE=0.75, oM=0.75, walkers=5, precision=P.F32X2,
             interval=3001, check_every=3, cycles=7, warm=0),
        # the batched workload: L = 32, 2048 walkers, one check block
        _cycles("cycles_L32", W.REWL_L32, P.FP64, 8),
        # the precision study's geometry: L = 64, 4096 walkers, 46 GB of tables, one check block
        _cycles("cycles_L64_f32x2", W.REWL_L64, P.F32X2, 16),
        # the uneven batch: 24 runs, L = 16, 24, 32 and 48, 10,752 walkers, advanced by one graph
        dict(kind="batch", name="batch_24_mixed", runs=24, big=True, precision=P.F32X2, interval=10_000, cycles=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(bins, n, o):
    return bins if n == 1 else min(bins, math.ceil(bins / (1.0 + (n - 1) * (1.0 - o))))


def _entries(c):
    B = c["L"] * c["L"] + 1
    return c["nE"] * c["nM"] * c["walkers"] * _width(B, c["nE"], c["oE"]) * _width(B, c["nM"], c["oM"])


def draw(rng):
    kind = rng.choice(["eq5", "join", "jackknife", "whole", "cycles", "cycles", "cycles", "batch"])
    if kind == "eq5":
        return dict(kind=kind, L=_log_int(rng, 4, 64))
    if kind == "whole":
        return dict(kind=kind, L=4, nE=1, nM=1, walkers=rng.randint(1, 24), lnf_final=0.5 ** rng.randint(10, 20),
                    flatness=rng.randint(60, 80) / 100.0, interval=_log_int(rng, 5000, 20000))
    if kind == "batch":
        return dict(kind=kind, runs=rng.randint(2, 23), big=rng.random() < 0.5, precision=rng.choice([P.FP64, P.F32X2]),
                    interval=_log_int(rng, 1000, 10000), cycles=8)
    o = rng.choice([0.5, 0.6, 0.7, 0.75])
    if kind == "cycles":
        L = _log_int(rng, 8, 64)
        c = dict(kind=kind, L=L, nE=rng.randint(1, max(3, L // 2)), nM=rng.randint(1, max(2, L // 8)), oE=o, oM=0.75,
                 walkers=_log_int(rng, 1, 32), precision=rng.choice([P.FP64, P.F32X2]),
                 interval=_log_int(rng, 1000, 20000), check_every=rng.randint(1, 16), cycles=_log_int(rng, 2, 64), warm=0)
        # no more tables than the listed L = 64 case, no more trials than the listed batch
        while _entries(c) > 2_000_000_000 or c["nE"] * c["nM"] * c["walkers"] > 4096:
            c["walkers"] = c["walkers"] // 2
        while c["nE"] * c["nM"] * c["walkers"] * c["interval"] * c["cycles"] > 400_000_000 and c["cycles"] > 1:
            c["cycles"] //= 2
        c["cycles"] = max(1, min(c["cycles"], 600_000 // c["interval"]))
        return c
    L = _log_int(rng, 5, 32)
    c = dict(kind=kind, L=L, nE=rng.randint(1, max(2, L // 2)), nM=rng.randint(1, max(2, L // 8)), oE=o, oM=o,
             walkers=rng.randint(1, 12), marginal=rng.random() < 0.3, per_slice=rng.random() < 0.3)
    most = 250_000_000
    if kind == "jackknife":
        c["walkers"] = rng.randint(2, 24)
        most = 7_000_000
    while _entries(c) > most and c["walkers"] > 2:
        c["walkers"] -= 1
    while _entries(c) > most and c["nE"] > 1:
        c["nE"] -= 1
    return c


# ------------------------------------------------------------------ inputs --

def _config(case, seed, **kw):
    return P.Config(L=case["L"], n_win_E=case["nE"], n_win_M=case["nM"], walkers_per_window=case["walkers"],
                    overlap_E=case.get("oE", 0.75), overlap_M=case.get("oM", 0.75), seed=1 + int(seed), **kw)


def _starts(bins, n, o):
    w = _width(bins, n, o)
    s = bins - w
    return [(2 * k * s + (n - 1)) // (2 * (n - 1)) if n > 1 else 0 for k in range(n)], w


def _possible(L):
    """(N+1) x (N+1) mask of the bins [e][m] that a configuration can have (the
    compact-droplet or stripe lower edge, the upper edge of isolated spins)."""
    N = L * L
    m = np.arange(N + 1)
    k = np.minimum(m, N - m)
    drop = np.array([2 * (math.isqrt(4 * x - 1) + 1) if x else 0 for x in k])
    low = np.where(k == 0, 0, np.minimum(drop, 2 * L + 2 * (k % L != 0)))
    high = np.where(k == 0, 0, 2 * N - 2 * np.abs(2 * m - N))
    b = 2 * np.arange(N + 1)[:, None]
    return (b >= low[None, :]) & (b <= high[None, :])


def _surface(L):
    """A smooth stand-in for ln g(e, m): the entropy of the magnetisation and a
    parabola in e around the uncorrelated mean."""
    N = L * L
    x = np.clip(np.arange(N + 1) / N, 1e-9, 1 - 1e-9)
    s = -N * (x * np.log(x) + (1 - x) * np.log(1 - x))
    mid = 2 * N * x * (1 - x)
    e = np.arange(N + 1)[:, None]
    return s[None, :] - (e - mid[None, :]) ** 2 / (0.5 * N)


def _tables(case, seed, device):
    """What a sampled run holds: per walker the surface of its window plus an
    offset (the ln g it piled up) and the sampling noise, and the visits H
    (-1 where no configuration exists or the walker has not been)."""
    L, B = case["L"], case["L"] ** 2 + 1
    g = torch.Generator(device=device).manual_seed(77_000 + int(seed))
    surf = torch.from_numpy(_surface(L)).to(device)
    can = torch.from_numpy(_possible(L)).to(device)
    es, wE = _starts(B, case["nE"], case["oE"])
    ms, wM = _starts(B, case["nM"], case["oM"])
    n = case["walkers"]
    lng, H, rects = [], [], []
    for mb in ms:
        for ea in es:
            s, c = surf[ea:ea + wE, mb:mb + wM], can[ea:ea + wE, mb:mb + wM]
            off = torch.rand(n, 1, 1, generator=g, device=device, dtype=torch.float64) * 1e4
            noise = torch.randn(n, wE, wM, generator=g, device=device, dtype=torch.float32).double() * 0.01
            visits = torch.randint(400, 1200, (n, wE, wM), generator=g, device=device, dtype=torch.int32)
            seen = c & (torch.rand(n, wE, wM, generator=g, device=device) < 0.995)
            lng.append(torch.where(seen, s + off + noise, 0.0))
            H.append(torch.where(seen, visits, -1))
            rects.append((ea, mb, wE, wM, bool(c.any())))
    return lng, H, rects


def _batch_runs(case):
    """The workloads of a batch: the uneven batch's members in turn, or (not
    big) its L = 16 and 24 members with fewer walkers."""
    all_ = W.mixed_batch()
    if case["runs"] == len(all_):
        return all_
    order = [all_[6 * (i % 4) + (i // 4) % 6] for i in range(case["runs"])]
    if not case["big"]:
        order = [all_[6 * (i % 2) + (i // 2) % 6].with_(walkers_per_window=3 + i % 5) for i in range(case["runs"])]
    return order


def prepare(case, seed):
    kind = case["kind"]
    if kind == "eq5":
        # two joined tables of one system: their difference is the sampling error
        B = case["L"] ** 2 + 1
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        s = torch.from_numpy(_surface(case["L"])).cuda()
        can = torch.from_numpy(_possible(case["L"])).cuda()
        out = []
        for _ in range(2):
            t = s + torch.randn(B, B, generator=g, device="cuda", dtype=torch.float64) * 0.02
            hole = torch.rand(B, B, generator=g, device="cuda") < 0.001
            out.append(torch.where(can & ~hole, t, -math.inf))
        return dict(kind=kind, a=out[0], b=out[1])
    if kind == "whole":
        return dict(kind=kind, cfg=_config(case, seed, lnf_final=case["lnf_final"], flatness=case["flatness"],
                                            exchange_interval=case["interval"]))
    if kind in ("join", "jackknife"):
        run = P.REWL(_config(case, seed))
        lng, H, _ = _tables(case, seed, "cuda")
        run.set_tables(torch.cat([t.reshape(-1) for t in lng]).cpu().numpy(),
                       torch.cat([t.reshape(-1) for t in H]).cpu().numpy())
        return dict(kind=kind, run=run, what=R.LNG_MARGINAL_E if case["marginal"] else R.LNG_JOINED,
                    rule=R.JOIN_PER_SLICE if case["per_slice"] else R.JOIN_MARGINAL)
    if kind == "batch":
        runs = [P.REWL(P.Config.from_workload(w, replicate=37 * int(seed) + i, precision=case["precision"],
                                               exchange_interval=case["interval"]))
                for i, w in enumerate(_batch_runs(case))]
        return dict(kind=kind, batch=P.Batch(runs), cycles=case["cycles"])
    # lnf_final far below: a run in progress stays in progress however many passes are taken
    run = P.REWL(_config(case, seed, lnf_final=1e-8, precision=case["precision"], exchange_interval=case["interval"],
                         check_every=case["check_every"]))
    if case["warm"]:
        run.run_cycles(case["warm"])
    return dict(kind=kind, run=run, cycles=case["cycles"], whole=_entries(case) <= WHOLE_TABLES)


# --------------------------------------------------------------------- run --

def _halves(digest):
    return [digest & 0xFFFFFFFF, digest >> 32]


def run(state):
    kind = state["kind"]
    if kind == "eq5":
        return P.relative_difference(state["a"], state["b"])
    if kind == "whole":
        r = P.REWL(state["cfg"])
        while not r.run_cycles(64)["done"]:
            pass
        st, spins = r.walkers()
        out = dict(lng=r.lng(), walkers=st, spins=spins, cycles=r.status()["cycles"])
        r.close()
        return out
    if kind == "join":
        return state["run"].lng(state["what"], matches=True, rule=state["rule"])
    if kind == "jackknife":
        return state["run"].jackknife(state["what"], rule=state["rule"])
    if kind == "batch":
        b = state["batch"]
        b.run_cycles(state["cycles"])
        return dict(walkers=np.concatenate([r.walkers(spins=False)[0] for r in b.runs]),
                    digests=np.array([_halves(r.digest()) for r in b.runs], dtype=np.int64))
    r = state["run"]
    status = r.run_cycles(state["cycles"])
    if state["whole"]:
        st, spins = r.walkers()
        lng, H = r.tables()
        return dict(status=status, walkers=st, spins=spins, lng=lng, H=H)
    return dict(status=status, walkers=r.walkers(spins=False)[0], digest=_halves(r.digest()))


# -------------------------------------------------------------------- work --

# One trial: half a Philox4x32-10 call (50 integer operations), ln u (15), the site and its five spins (25), the
# move, the window test and the bin (12), the acceptance (10), the bookkeeping (8).
OPS_PER_TRIAL = 120


def _run_work(L, nwalk, trials):
    # each walker's lattice, position and counters in and out; the tables' touched bins: at most two 8-byte
    # entries (screen, visits) read and one count written per trial, and no more than the tables hold
    return dict(bytes=2.0 * nwalk * (L * L / 8 + 24) + 20.0 * trials, flops=float(OPS_PER_TRIAL) * trials)


def work(case):
    kind = case["kind"]
    if kind == "eq5":
        n = (case["L"] ** 2 + 1) ** 2
        return dict(bytes=24.0 * n, flops=20.0 * n)
    if kind == "whole":
        # about 2.5e5 trials per walker and iteration
        its = math.ceil(-math.log2(case["lnf_final"])) + 1
        return _run_work(4, case["walkers"], 2.5e5 * its * case["walkers"])
    if kind == "batch":
        ws = _batch_runs(case)
        parts = [_run_work(w.L, w.n_walkers, w.n_walkers * case["interval"] * case["cycles"]) for w in ws]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    B = case["L"] ** 2 + 1
    out = B if case.get("marginal") else B * B
    if kind == "join":
        return dict(bytes=12.0 * _entries(case) + 8.0 * out, flops=6.0 * _entries(case) + 30.0 * B * B)
    if kind == "jackknife":
        return dict(bytes=12.0 * _entries(case) + 16.0 * out,
                    flops=6.0 * _entries(case) + 30.0 * B * B * case["walkers"])
    nwalk = case["nE"] * case["nM"] * case["walkers"]
    w = _run_work(case["L"], nwalk, nwalk * case["interval"] * case["cycles"])
    tables = _entries(case)
    w["bytes"] += 12.0 * tables        # the tables handed out, or read for their digest
    return w


# ------------------------------------------------------------------- exact --

def _lse(v, dim):
    return torch.logsumexp(v, dim=dim)


def _match(a, b, lo, hi, floor, step):
    """Lowest bin q in [max(lo, floor), hi) with the least |slope difference| of two marginals."""
    q = torch.arange(max(lo, floor), hi, device=a.device)
    fin = torch.isfinite(a[q]) & torch.isfinite(a[q + 1]) & torch.isfinite(b[q]) & torch.isfinite(b[q + 1])
    if bool(fin.any()):
        q = q[fin]
        d = ((a[q + 1] - a[q]) / step - (b[q + 1] - b[q]) / step).abs()
        return int(q[torch.argmin(d)])
    q = torch.arange(max(lo, floor), hi + 1, device=a.device)
    q = q[torch.isfinite(a[q]) & torch.isfinite(b[q])]
    return int(q[0])


def _exact_join(case, lng, H, rects, skip):
    """Merge, join (E then M) and normalisation in 64 bits of the walkers but `skip`."""
    L, nE, nM, n = case["L"], case["nE"], case["nM"], case["walkers"]
    N, B = L * L, L * L + 1
    dev = lng[0].device
    inf = math.inf
    keep = [k for k in range(n) if k != skip]
    em = np.full(max(1, nM * max(1, nE - 1)), -1, dtype=np.int32)
    mm = np.full(max(1, nM - 1), -1, dtype=np.int32)
    slices = case["per_slice"]
    rows = []
    for b in range(nM):
        pieces = []
        for a in range(nE):
            ea, mb, wE, wM, some = rects[b * nE + a]
            t = torch.full((B, B), -inf, dtype=torch.float64, device=dev)
            if some:
                g, seen = lng[b * nE + a][keep], H[b * nE + a][keep] >= 0
                both = seen.all(dim=0)
                off = ((g - g[:1]) * both).sum(dim=(1, 2)) / both.sum()
                cnt = seen.sum(dim=0)
                mean = torch.where(seen, g - off[:, None, None], 0.0).sum(dim=0) / cnt
                t[ea:ea + wE, mb:mb + wM] = torch.where(cnt > 0, mean, -inf)
            pieces.append((ea, ea + wE - 1, some, t))
        live = [a for a in range(nE) if pieces[a][2]]
        row = torch.full((B, B), -inf, dtype=torch.float64, device=dev)
        shift = torch.zeros(B, dtype=torch.float64, device=dev)
        start = pieces[live[0]][0]
        for a in live:
            t = pieces[a][3]
            if a != live[-1]:
                u = pieces[a + 1][3]
                ga, gb = _lse(t, 1), _lse(u, 1)
                q = _match(ga, gb, pieces[a + 1][0], pieces[a][1], start, 4.0)
                em[b * (nE - 1) + a] = q
                end = q
                step = (ga[q] - gb[q]).expand(B)
                if slices:
                    step = torch.where(torch.isfinite(t[q]) & torch.isfinite(u[q]), t[q] - u[q], step)
            else:
                end, step = pieces[a][1] + 1, torch.zeros(B, dtype=torch.float64, device=dev)
            row[start:end] = t[start:end] + shift[None, :]
            shift, start = shift + step, end
        mb, wM = rects[b * nE][1], rects[b * nE][3]
        rows.append((mb, mb + wM - 1, row))
    out = torch.full((B, B), -inf, dtype=torch.float64, device=dev)
    shift = torch.zeros(B, dtype=torch.float64, device=dev)
    start = rows[0][0]
    for b in range(nM):
        t = rows[b][2]
        if b < nM - 1:
            u = rows[b + 1][2]
            fa, fb = _lse(t, 0), _lse(u, 0)
            q = _match(fa, fb, rows[b + 1][0], rows[b][1], start, 2.0)
            mm[b] = q
            end = q
            step = (fa[q] - fb[q]).expand(B)
            if slices:
                step = torch.where(torch.isfinite(t[:, q]) & torch.isfinite(u[:, q]), t[:, q] - u[:, q], step)
        else:
            end, step = rows[b][1] + 1, torch.zeros(B, dtype=torch.float64, device=dev)
        out[:, start:end] = t[:, start:end] + shift[:, None]
        shift, start = shift + step, end
    out = out + (N * math.log(2.0) - torch.logsumexp(out.reshape(-1), 0))
    if case["marginal"]:
        out = _lse(out, 1)
    return out, em, mm


def exact(case, seed):
    kind = case["kind"]
    if kind == "eq5":
        s = prepare(case, seed)
        a, b = s["a"], s["b"]
        d = 2.0 * torch.tanh(0.5 * (a - b).abs())
        ea, eb = torch.isinf(a), torch.isinf(b)
        return torch.where(ea & eb, math.nan, torch.where(ea | eb, 2.0, d))
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if kind == "join":
        out, em, mm = _exact_join(case, *_tables(case, seed, dev), skip=-1)
        return (out, em, mm)
    if kind == "jackknife":
        t = _tables(case, seed, dev)
        n = case["walkers"]
        first, s1, s2 = None, 0.0, 0.0
        for k in range(n):
            v = _exact_join(case, *t, skip=k)[0]
            first = v if first is None else torch.where(torch.isfinite(v), first, math.nan)
            d = v - first
            s1, s2 = s1 + d, s2 + d * d
        mean = first + s1 / n
        err = torch.sqrt(torch.clamp((n - 1) / n * (s2 - s1 * s1 / n), min=0.0))
        hole = ~torch.isfinite(mean)
        return (torch.where(hole, -math.inf, mean), torch.where(hole, math.nan, err))
    return None     # the chain itself: whole numbers and exact sums, which stay equal
