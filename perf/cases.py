"""What the framework is measured by: flatPERM runs as its users make them.

Every case goes through the package's own entry points (`Run`, `Batch`, the
serving engine).  There are two groups:

- Runs whose result follows from the seed alone: one sequence with fresh
  thresholds, Algorithm 1 (a private table per sequence) and the original PERM
  with cut-offs.  They return their estimates or tables whole; `exact` grows the
  same trees in 64-bit torch arithmetic.
- Interacting sequences (Algorithm 2, snapshot thresholds), the framework's main
  use: what a node sees of the shared table depends on the GPU's scheduling, so
  two runs of one seed give two estimates.  They return log(c_{n+1}/c_n) for
  every n, the ratios that the growth-constant analysis fits, whose statistical
  errors are nearly independent over n (those of log c_n accumulate), and the
  tours finished.  `exact` gives them no value.
"""
import math

import numpy as np
import torch

from paper_2002_03000_gb300 import PERM_ALG1, PERM_THRESH_FRESH, Run
from paper_2002_03000_gb300 import batch as pbatch
from paper_2002_03000_gb300 import serve as pserve

SEED0 = 0x5EED0000


def listed():
    return [
        # the build's first check: one sequence, fresh thresholds, as a user tries the
        # library out; one walk on the whole GPU, latency only
        dict(name="first_check", kind="fresh", d=2, n_max=16, n_seq=1, tours=400),
        # Algorithm 1 against Algorithm 2 on the exact-count lattice (the paper's T_M
        # comparison): the Algorithm 1 side
        dict(name="alg1_t16", kind="alg1", d=2, n_max=16, n_seq=12, tours=400),
        # Algorithm 1 with many sequences, one private table each
        dict(name="alg1_many", kind="alg1", d=3, n_max=100, n_seq=1500, tours=8),
        # 12 interacting sequences to n = 16, chunk after chunk until c_n is known to
        # 1e-4 (the exact-count workload): few walks, short tours
        dict(name="exact_count", kind="interacting", d=2, n_max=16, n_seq=12, warm=2000, tours=2000, observables=0),
        # a medium cubic run with the squared end-to-end distance summed as well
        dict(name="cubic_r2", kind="interacting", d=3, n_max=255, n_seq=1024, warm=64, tours=32, observables=1),
        # the square benchmark workload continued: the steady state of a long run
        dict(name="square_continued", kind="interacting", d=2, n_max=512, n_seq=4096, warm=128, tours=96, observables=0),
        # the square benchmark workload: one complete run from empty tables, start-up included
        dict(name="square_complete", kind="complete", d=2, n_max=512, n_seq=4096, tours=256),
        # the cubic benchmark workload, from empty tables; more sequences than walks
        dict(name="cubic_complete", kind="complete", d=3, n_max=512, n_seq=8192, tours=128),
        # one round of the serving loop: a chunk of tours for each of 16 resident requests
        dict(name="served_round", kind="served", requests=16, n_lo=64, n_hi=256, n_seq=1024, tours=8),
        # a batch of independent runs of mixed sizes, regrown by one persistent launch
        dict(name="batch_mixed", kind="batch", runs=24, n_lo=64, n_hi=256, seq_lo=256, seq_hi=2048, tours=8),
        # original PERM with cut-offs around c_n
        dict(name="cutoffs_square", kind="cutoffs", d=2, n_max=257, n_seq=2000, tours=8, copies=2, q=2.0, f=1.5, observables=1),
        # long cubic walks, no cut-off active (Rosenbluth chains): 64-bit site keys, walks
        # in the global arena
        dict(name="chains_long", kind="cutoffs", d=3, n_max=10000, n_seq=608, tours=4, copies=2, q=2.0, f=0.0, observables=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges, its work below the largest listed one's."""
    kind = rng.choice(["fresh", "alg1", "interacting", "interacting", "complete", "served", "batch", "cutoffs", "cutoffs"])
    d = rng.choice([2, 3])
    if kind == "fresh":
        n_max = _log_int(rng, 8, 96)
        return dict(kind=kind, d=d, n_max=n_max, n_seq=1, tours=max(8, 6000 // n_max))
    if kind == "alg1":
        n_max = _log_int(rng, 12, 128)
        return dict(kind=kind, d=d, n_max=n_max, n_seq=_log_int(rng, 12, 4096), tours=max(8, 800 // n_max))
    if kind == "interacting":
        n_max, n_seq = _log_int(rng, 16, 512), _log_int(rng, 12, 8192)
        # about 2e7 nodes a pass, fewer when few walks grow them
        tours = max(16, int(min(2e7, 4e4 * n_seq) / (n_seq * n_max)))
        return dict(kind=kind, d=d, n_max=n_max, n_seq=n_seq, warm=max(64, tours), tours=tours,
                    observables=rng.choice([0, 0, 1]))
    if kind == "complete":
        n_max, n_seq = _log_int(rng, 64, 512), _log_int(rng, 512, 8192)
        return dict(kind=kind, d=d, n_max=n_max, n_seq=n_seq, tours=_log_int(rng, 32, 128))
    if kind == "served":
        return dict(kind=kind, requests=rng.randint(3, 16), n_lo=rng.randint(48, 96), n_hi=rng.randint(128, 256),
                    n_seq=_log_int(rng, 256, 1024), tours=rng.randint(4, 12))
    if kind == "batch":
        return dict(kind=kind, runs=rng.randint(4, 24), n_lo=64, n_hi=rng.randint(128, 256), seq_lo=256,
                    seq_hi=rng.randint(512, 2048), tours=rng.randint(4, 10))
    n_max = _log_int(rng, 64, 12000)
    n_seq = _log_int(rng, 32, max(64, min(4096, 3000000 // n_max)))
    # cut-offs make a tour's tree as large as n_max^2 nodes on one walk: longer walks are chains
    if n_max > 600:
        return dict(kind=kind, d=3, n_max=n_max, n_seq=n_seq, tours=max(1, int(6e6 / (n_max * n_seq))), copies=2, q=2.0, f=0.0,
                    observables=rng.choice([0, 1]))
    return dict(kind=kind, d=d, n_max=n_max, n_seq=n_seq, tours=max(1, min(32, int(4e6 / (n_max * n_seq)))),
                copies=rng.choice([2, 3]), q=rng.choice([2.0, 3.0]), f=rng.choice([1.3, 1.5]), observables=rng.choice([0, 1]))


# ---------------------------------------------------------------------------
# What a user's program has in hand before the call.
# ---------------------------------------------------------------------------
def _scale_exp(d, n):
    return (11 * n) >> 3 if d == 2 else (9 * n) >> 2


def _cutoffs(case):
    """T_n = f a_n and t_n = a_n / f around c_n ~ A mu^n n^(gamma-1), at the stored
    scale; f = 0: no cut-off active."""
    if case["f"] == 0.0:
        return np.full(case["n_max"] + 1, np.inf), np.zeros(case["n_max"] + 1)
    mu, gamma, amp = {2: (2.63815853, 43.0 / 32.0, 1.18), 3: (4.6840386, 1.1570, 1.21)}[case["d"]]
    a = np.array([math.exp(math.log(amp) + n * math.log(mu) + (gamma - 1.0) * math.log(max(n, 1))
                           - _scale_exp(case["d"], n) * math.log(2.0)) for n in range(case["n_max"] + 1)])
    return case["f"] * a, a / case["f"]


def _served_sizes(case, seed):
    """(d, n_max) of each resident request: d alternates, n_max log-uniform."""
    R, rng = case["requests"], np.random.Generator(np.random.PCG64(seed))
    return [(2 + r % 2, int(round(math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))) for r in range(R)]


def _batch_sizes(case):
    """(d, n_max, sequences) of each run, spread over the case's ranges."""
    R, out = case["runs"], []
    for r in range(R):
        u, v = (r + 0.5) / R, ((r * 7) % R + 0.5) / R
        n_max = int(round(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** u))
        n_seq = int(round(case["seq_lo"] * (case["seq_hi"] / case["seq_lo"]) ** v))
        out.append((2 + r % 2, n_max, n_seq))
    return out


def prepare(case, seed):
    kind, key = case["kind"], SEED0 + int(seed)
    if kind == "served":
        engine = pserve.GpuEngine()
        jobs = [engine.start(pserve.Request(rid=r, d=d, n_max=n, target=1e-2, arrival=0.0, n_seq=case["n_seq"], seed=key))
                for r, (d, n) in enumerate(_served_sizes(case, 1))]
        # each request has had its first chunks
        for job in jobs:
            engine.queue_chunk(job, 2 * case["tours"])
        torch.cuda.synchronize()
        return dict(case=case, engine=engine, jobs=jobs)
    if kind == "batch":
        cfgs = [pbatch.make_config(d, n, N, key, run_id=r, max_seconds=60.0) for r, (d, n, N) in enumerate(_batch_sizes(case))]
        return dict(case=case, batch=pbatch.Batch(cfgs, [case["tours"]] * case["runs"], persistent=True))
    kw = dict(max_seconds=60.0)
    if kind == "alg1":
        kw["alg"] = PERM_ALG1
    elif kind == "fresh":
        kw["threshold"] = PERM_THRESH_FRESH
    elif kind == "cutoffs":
        kw.update(share_copies=-1, observables=case["observables"])
    elif kind == "interacting":
        kw["observables"] = case["observables"]
    run = Run(case["d"], case["n_max"], case["n_seq"], key, **kw)
    if kind == "cutoffs":
        hi, lo = _cutoffs(case)
        run.set_cutoffs(hi, lo, case["copies"], case["q"])
    elif kind == "interacting":
        run.run(case["warm"])
    return dict(case=case, run=run)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "served":
        # as the server's loop: a chunk for every resident request, each read when done
        engine, jobs = state["engine"], state["jobs"]
        for job in jobs:
            engine.queue_chunk(job, case["tours"])
        ratios, waiting = [None] * len(jobs), set(range(len(jobs)))
        while waiting:
            for r in list(waiting):
                if engine.chunk_done(jobs[r]):
                    ratios[r] = np.diff(engine.read(jobs[r])[0])
                    waiting.discard(r)
        return dict(log_ratios=np.concatenate(ratios))
    if kind == "batch":
        b = state["batch"]
        b.run()
        return dict(log_ratios=np.concatenate([np.diff(b.estimates(r)[0]) for r in range(case["runs"])]))
    h = state["run"]
    if kind == "interacting":
        h.run(case["tours"])
        out = dict(log_ratios=np.diff(h.estimates()[0]), tours=h.stats()["tours_finished"])
        if case["observables"]:
            out["mean_r2"] = h.mean_r2()[0]
        return out
    h.reset()
    h.run(case["tours"])
    if kind == "complete":
        return dict(log_ratios=np.diff(h.estimates()[0]), tours=h.stats()["tours_finished"])
    if kind == "cutoffs":
        out = h.tables()
        if case["observables"]:
            out["mean_r2"] = h.mean_r2()[0]
        return out
    lc, S, rv = h.estimates()
    return dict(log_cn=lc, S=S, relvar=rv)


def _nodes(case):
    """Nodes of a pass: flatPERM's histogram is flat, about one node per length and tour."""
    kind = case["kind"]
    if kind == "served":
        return sum((n + 1) * case["n_seq"] * case["tours"] for _, n in _served_sizes(case, 1))
    if kind == "batch":
        return sum((n + 1) * N * case["tours"] for _, n, N in _batch_sizes(case))
    return (case["n_max"] + 1) * case["n_seq"] * case["tours"]


def work(case):
    """Bytes a growth step cannot do without (probes, insert and delete, coordinates,
    W_n, S_n and tour-sum updates, the read of W_n; a fifth of a copy's record), and
    its arithmetic (the weight's product, three sums, the ratio, the decision)."""
    d = case.get("d", 3)
    per_node = (72 if d == 2 else 84) + 6
    return dict(bytes=per_node * _nodes(case), flops=10 * _nodes(case))


# ---------------------------------------------------------------------------
# The same runs in 64 bits: all sequences (Algorithm 1, one sequence) or all tours
# (cut-offs) grow in lockstep, one node of each per step, depth first.
# ---------------------------------------------------------------------------
MAX_STEPS = 18000          # nodes of one lane (about a millisecond each); past it: no value


def _mul(a, b):
    """(high, low) words of the product of two 32-bit words, in int64 tensors."""
    t = a * (b & 0xFFFF)
    u = a * (b >> 16) + (t >> 16)
    return u >> 16, ((u & 0xFFFF) << 16) | (t & 0xFFFF)


def _philox(ordinal, tour, seq, k0, k1):
    c0, c1, c2, c3 = ordinal & 0xFFFFFFFF, ordinal >> 32, tour, seq
    for _ in range(10):
        h0, l0 = _mul(0xD2511F53, c0)
        h1, l1 = _mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1


def _grow(case, key):
    """Tables (W, S, Q, R2: one row per sequence for Algorithm 1, else one row)."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    d, n_max, N, tours = case["d"], case["n_max"], case["n_seq"], case["tours"]
    cut = case["kind"] == "cutoffs"
    L = n_max + 1
    i64, f64 = dict(dtype=torch.int64, device=dev), dict(dtype=torch.float64, device=dev)
    lanes = N * tours if cut else N                # a lane: one tour, or one sequence's tours
    if lanes * L > 1 << 28:
        return None
    seq, tour = torch.arange(lanes, **i64) % N, torch.arange(lanes, **i64) // N
    last = tour + 1 if cut else torch.full((lanes,), tours, **i64)
    rows = 1 if cut else N
    row = torch.zeros(lanes, **i64) if cut else torch.arange(lanes, **i64)
    W_t, Q_t, R_t = (torch.zeros(rows * L, **f64) for _ in range(3))
    S_t = torch.zeros(rows * L, **i64)
    if cut:
        hi, lo = (torch.tensor(a, **f64) for a in _cutoffs(case))
    scale = torch.tensor([0.5 ** (_scale_exp(d, n + 1) - _scale_exp(d, n)) for n in range(L)], **f64)
    unit = [1 << (21 * (j // 2)) if j % 2 == 0 else -(1 << (21 * (j // 2))) for j in range(2 * d)]
    unit = torch.tensor(unit, **i64)
    origin = sum((1 << 20) << (21 * k) for k in range(d))
    s = dict(seq=seq, tour=tour, last=last, row=row, n=torch.zeros(lanes, **i64), at=torch.full((lanes,), origin, **i64),
             w=torch.ones(lanes, **f64), ordinal=torch.zeros(lanes, **i64), top=torch.zeros(lanes, **i64),
             X=torch.zeros(lanes, L, **f64), sites=torch.full((lanes, L), origin, **i64),
             sdepth=torch.zeros(lanes, L, **i64), sdirs=torch.zeros(lanes, L, **i64), scount=torch.zeros(lanes, L, **i64),
             sw=torch.zeros(lanes, L, **f64), live=torch.ones(lanes, dtype=torch.bool, device=dev))
    mask21 = (1 << 21) - 1
    for step in range(MAX_STEPS):
        if step % 64 == 0:
            left = int(s["live"].sum())
            if left == 0:
                return [t.cpu().numpy().reshape(rows, L) for t in (W_t, S_t, Q_t, R_t)]
            if left < 0.8 * s["live"].numel():
                keep = s["live"]
                s = {k: v[keep] for k, v in s.items()}
        B = s["n"].numel()
        lane = torch.arange(B, **i64)
        live, n, at, w, row = s["live"], s["n"], s["at"], s["w"], s["row"]
        s["sites"][lane, n] = torch.where(live, at, s["sites"][lane, n])
        wl = torch.where(live, w, torch.zeros_like(w))
        idx = row * L + n
        before = W_t[idx]
        r2 = sum(((at >> (21 * k)) & mask21).sub(1 << 20).square() for k in range(d))
        W_t.index_add_(0, idx, wl)
        R_t.index_add_(0, idx, wl * r2)
        S_t.index_add_(0, idx, live.long())
        s["X"][lane, n] += wl
        # free neighbours
        top_n = int(n.max()) + 1
        valid = torch.arange(top_n, **i64)[None, :] <= n[:, None]
        nb = at[:, None] + unit[None, :]
        occ = torch.stack([((s["sites"][:, :top_n] == nb[:, j:j + 1]) & valid).any(1) for j in range(2 * d)], 1)
        free = ~occ
        a = free.sum(1)
        lst = torch.argsort(occ.long() * 8 + torch.arange(2 * d, **i64)[None, :], dim=1)
        w0, w1 = _philox(s["ordinal"], s["tour"], s["seq"], key & 0xFFFFFFFF, key >> 32)
        u0 = w0.double() * 2.0 ** -32
        one = torch.ones_like(n)
        if cut:
            nc = n.clamp(max=n_max)
            above, below = (w > hi[nc]) & (n > 0), (w < lo[nc]) & (n > 0)
            c = torch.where(above, torch.minimum(one * case["copies"], a),
                            torch.where(below, (u0 < 1.0 / case["q"]).long(), one))
            base = torch.where(above, w / c.clamp(min=1), torch.where(below, w * case["q"], w))
        else:
            r = torch.where(n == 0, torch.ones_like(w), w / ((before + w) / (s["tour"] + 1).double()))
            up = r >= 1.0
            craw = torch.where(u0 < torch.ceil(r) - r, torch.floor(r), torch.ceil(r))
            c = torch.where(up, torch.minimum(craw, a.double()).long(), (u0 < r).long())
            base = torch.where(up, w / c.clamp(min=1), w * (1.0 / r))
        grows = live & (n < n_max) & (a > 0) & (c > 0)
        c = torch.where(grows, c, torch.zeros_like(c))
        x = w1
        for i in range(int(c.max())):
            pick = i < c
            h, l = _mul((a - i).clamp(min=1), x)
            j = torch.where(pick, i + h, one * i)
            x = torch.where(pick, l, x)
            vi, vj = lst[:, i].clone(), lst.gather(1, j[:, None])[:, 0]
            lst[lane, j] = vi
            lst[:, i] = vj
        child = base * a.double() * scale[n.clamp(max=n_max)]
        # copies 1 .. c-1 wait (3 bits a step), the first one grows
        wait = grows & (c > 1)
        dirs = sum(lst[:, i + 1] << (3 * i) for i in range(2 * d - 1))
        tp = s["top"].clamp(max=n_max)
        for name, v in (("sdepth", n), ("sdirs", dirs), ("scount", c - 1), ("sw", child)):
            s[name][lane, tp] = torch.where(wait, v, s[name][lane, tp])
        s["top"] = s["top"] + wait.long()
        # a leaf: the most recent waiting copy, or the end of the tour
        leaf = live & ~grows
        ends = leaf & (s["top"] == 0)
        pop = leaf & ~ends
        tp = (s["top"] - 1).clamp(min=0)
        pd, pdir, pcnt, pw = (s[k][lane, tp] for k in ("sdepth", "sdirs", "scount", "sw"))
        s["sdirs"][lane, tp] = torch.where(pop, pdir >> 3, pdir)
        s["scount"][lane, tp] = torch.where(pop, pcnt - 1, pcnt)
        s["top"] = s["top"] - (pop & (pcnt == 1)).long()
        if bool(ends.any()):
            e = ends.nonzero()[:, 0]
            X = s["X"][e]
            Q_t.view(rows, L).index_add_(0, row[e], X * X)
            s["X"][e] = 0.0
        step_dir = torch.where(grows, lst[:, 0], pdir & 7)
        origin_at = torch.where(grows, at, s["sites"][lane, pd])
        s["n"] = torch.where(ends, 0 * n, torch.where(grows, n + 1, torch.where(pop, pd + 1, n)))
        s["at"] = torch.where(ends, 0 * at + origin, torch.where(grows | pop, origin_at + unit[step_dir], at))
        s["w"] = torch.where(ends, torch.ones_like(w), torch.where(grows, child, torch.where(pop, pw, w)))
        s["ordinal"] = torch.where(ends, 0 * n, s["ordinal"] + 1)
        s["tour"] = s["tour"] + ends.long()
        s["live"] = live & (s["tour"] < s["last"])
        s["tour"] = torch.where(s["live"], s["tour"], s["tour"] - ends.long())
    return None


def exact(case, seed):
    if case["kind"] not in ("fresh", "alg1", "cutoffs") or case["n_max"] > 2048:
        return None
    got = _grow(case, SEED0 + int(seed))
    if got is None:
        return None
    W, S, Q, R = got
    if case["kind"] == "cutoffs":
        out = dict(W=W[0], S=S[0].astype(np.float64), Q=Q[0], M=np.array([case["n_seq"] * case["tours"]]))
        if case["observables"]:
            with np.errstate(divide="ignore", invalid="ignore"):
                out["mean_r2"] = np.where(W[0] > 0, R[0] / W[0], np.nan)
        return out
    M = float(case["tours"])
    c = W / M
    mean = c.mean(0)
    var = np.maximum((Q / M - c * c) / (M - 1.0), 0.0).sum(0) / W.shape[0] ** 2
    shift = np.array([_scale_exp(case["d"], n) for n in range(case["n_max"] + 1)]) * math.log(2.0)
    with np.errstate(divide="ignore", invalid="ignore"):
        return dict(log_cn=np.log(mean) + shift, S=S.sum(0).astype(np.float64),
                    relvar=np.where(mean > 0, var / (mean * mean), np.inf))
