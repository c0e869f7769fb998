"""What is timed of this engine: the calls its users make, over the range of sizes they make them at.

Every case is a dict of plain values with a "kind":

  anneal   one-shot nmc_anneal through host buffers, instance and schedule resident
  sweep    a resident replica set: reset, sweeps, results into device buffers
  batch    uneven k-SAT sets in one batched launch
  pt       replica exchange on a ladder of temperatures
  chain    the two-chain schedule (held units), a collective flip and whitening
  qap      uneven QAP sets in one batched call
  lbp      the learning stage: loopy belief propagation around seeds, then backbones
  fresh    a new formula: load, schedule, anneal, unload, all through host buffers
  serve    a burst of requests through the anneal server

Inputs are the generators' (random k-SAT near the paper's densities, symmetric QAP matrices),
with inhomogeneous inverse-temperature profiles, all from the seed; the sizes inside an uneven set
of instances are the case's own ("mix"). States, permutations and energies are whole numbers; only
the learning stage computes in floating point.
"""
import math

import numpy as np
import torch

import nmc_inputs as W
import paper_2111_13628_gb300 as nmc

LAMBDAS = (0.4, 0.2, 0.1, 0.05, 0.025)  # continuation list of the learning stage
LBP_BETA, LBP_TOL, LBP_ITER = 1.0, 1e-8, 100
ALPHA = {3: 4.2, 4: 9.6, 6: 12.0}  # clause densities of the workloads by k


def listed():
    return [
        # the smallest one-shot call: the 200-variable formula, bound by latency and launches
        dict(name="anneal_n200", kind="anneal", n=200, k=4, alpha=9.6, R=64, T=200),
        # the headline: one large formula over 1,024 replicas, sweeps resident on the device
        dict(name="sweep_n50000", kind="sweep", n=50000, k=4, alpha=9.6, R=1024, T=200),
        # many uneven formulas at once, 3-SAT and 4-SAT mixed
        dict(name="batch_3_4sat", kind="batch", sets=24, k0=3, k1=4, n_lo=1000, n_hi=20000,
             r_lo=32, r_hi=256, T=100, mix=1),
        # the same with clauses of six literals (two list entries per occurrence)
        dict(name="batch_3_6sat", kind="batch", sets=12, k0=3, k1=6, n_lo=1000, n_hi=20000,
             r_lo=32, r_hi=256, T=100, mix=2),
        # replica exchange at the paper's size: 32 ladders of 32 temperatures, rounds every 10
        dict(name="pt_n5000", kind="pt", n=5000, k=4, alpha=9.884, ladders=32, temps=32, T=100,
             per=10),
        # two-chain sampling with a held backbone, ragged sizes, the collective move, whitening
        dict(name="chain_n20001", kind="chain", n=20001, k=4, alpha=9.6, R=500, cycles=2),
        # uneven QAP sets, the int16 permutations of 4,096 replicas each
        dict(name="qap_batch", kind="qap", sets=12, n_lo=32, n_hi=256, R=4096, T=20, mix=3),
        # one small QAP through host buffers
        dict(name="qap_n33", kind="anneal", n=33, k=0, alpha=0.0, R=256, T=100),
        # the learning stage at the paper's size, 64 seeds at once
        dict(name="lbp_n5000", kind="lbp", n=5000, k=4, alpha=9.884, S=64),
        # and for a few seeds of a small formula, where each iteration's launches count
        dict(name="lbp_n500", kind="lbp", n=500, k=4, alpha=9.884, S=5),
        # a formula seen for the first time: host preparation, upload, schedule, anneal, results
        dict(name="fresh_n10007", kind="fresh", n=10007, k=4, alpha=9.6, R=256, T=100),
        # the server: a burst of k-SAT and QAP requests of mixed sizes, 32 / 256 replicas each
        dict(name="serve_16", kind="serve", requests=16, n_lo=500, n_hi=20000, t_lo=100, t_hi=400,
             mix=4),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["anneal", "anneal", "sweep", "sweep", "batch", "pt", "chain", "qap", "qap",
                       "lbp", "fresh", "serve"])
    k = rng.choice([3, 4, 4, 6])
    alpha = round(ALPHA[k] * rng.uniform(0.94, 1.03), 3)
    if kind == "anneal":
        if rng.random() < 0.4:
            return dict(kind=kind, n=log(8, 256), k=0, alpha=0.0, R=log(32, 1024), T=log(10, 100))
        return dict(kind=kind, n=log(100, 4000), k=k, alpha=alpha, R=log(20, 256), T=log(20, 200))
    if kind == "sweep":
        n = log(1000, 50000)
        return dict(kind=kind, n=n, k=k if k == 4 or n <= 20000 else 4,
                    alpha=alpha if k == 4 or n <= 20000 else 9.6, R=log(32, 1024),
                    T=log(20, 200))
    if kind == "batch":
        lo = log(500, 4000)
        return dict(kind=kind, sets=rng.randint(5, 24), k0=3, k1=rng.choice([4, 6]), n_lo=lo,
                    n_hi=log(lo, 20000), r_lo=32, r_hi=log(33, 256), T=log(20, 100),
                    mix=rng.randint(5, 999))
    if kind == "pt":
        temps = rng.choice([7, 16, 32, 33])
        return dict(kind=kind, n=log(500, 10000), k=4, alpha=round(rng.uniform(9.0, 9.9), 3),
                    ladders=rng.randint(4, 32), temps=temps, T=log(20, 100), per=rng.randint(1, 10))
    if kind == "chain":
        return dict(kind=kind, n=log(1000, 25000), k=k if k != 3 else 4,
                    alpha=alpha if k != 3 else 9.6, R=log(64, 512), cycles=rng.randint(1, 2))
    if kind == "qap":
        lo = log(32, 200)
        return dict(kind=kind, sets=rng.randint(1, 12), n_lo=lo, n_hi=rng.randint(lo, 256),
                    R=log(256, 4096), T=log(5, 20), mix=rng.randint(5, 999))
    if kind == "lbp":
        return dict(kind=kind, n=log(300, 5000), k=4, alpha=round(rng.uniform(9.0, 9.884), 3),
                    S=log(1, 64))
    if kind == "fresh":
        return dict(kind=kind, n=log(500, 20000), k=k, alpha=alpha, R=log(32, 256), T=log(20, 100))
    lo = log(500, 2000)
    return dict(kind="serve", requests=rng.randint(6, 16), n_lo=lo, n_hi=log(2 * lo, 20000),
                t_lo=100, t_hi=log(150, 400), mix=rng.randint(5, 999))


# ---- inputs ------------------------------------------------------------------------------------

def _ksat(n, k, alpha, seed):
    return W.random_ksat(n, alpha, k, 7_000_003 * (seed + 1))


def _profile(n, T, seed):
    """Inhomogeneous profile in factored form: base linear 0.5 -> 4.0, a seeded 30% at 0.5x."""
    base = W.linear_profile(0.5, 4.0, T).astype(np.float32)
    factor = np.where(W.seeded_subset(n, 0.3, 7_000_013 * (seed + 1)), 0.5, 1.0).astype(np.float32)
    return base, factor


def _qap_beta(n, T, seed):
    return W.beta_scaled_linear(n, T, 0.01, 1.0, 0.5, 1.5, 7_000_031 * (seed + 1))


def _philox(seed):
    return 1_000_003 * (seed + 1)


def _buffers(sizes, state_dtype):
    """Device result buffers of several sets ((R, n) each): one flat tensor per result, and the
    sets' views into it."""
    ns, nr = sum(R * n for R, n in sizes), sum(R for R, _ in sizes)
    flat = dict(states=torch.empty(ns, dtype=state_dtype, device="cuda"),
                energies=torch.empty(nr, dtype=torch.int64, device="cuda"),
                best_energies=torch.empty(nr, dtype=torch.int64, device="cuda"),
                best_states=torch.empty(ns, dtype=state_dtype, device="cuda"))
    views, a, b = [], 0, 0
    for R, n in sizes:
        views.append(dict(states=flat["states"][a:a + R * n],
                          energies=flat["energies"][b:b + R],
                          best_energies=flat["best_energies"][b:b + R],
                          best_states=flat["best_states"][a:a + R * n]))
        a, b = a + R * n, b + R
    return flat, views


def _lbp_inputs(case, seed):
    """Formula and seeds x* [S, n]: random states after a parallel greedy descent (every variable
    whose flip lowers the number of violated clauses flips with probability 0.3, 60 rounds)."""
    n, k, S = case["n"], case["k"], case["S"]
    lits = _ksat(n, k, case["alpha"], seed)
    g = torch.Generator().manual_seed(99_991 * (seed + 1))
    x = torch.randint(0, 2, (S, n), generator=g).cuda().bool()
    var = torch.from_numpy(np.abs(lits).astype(np.int64) - 1).cuda()
    pos = torch.from_numpy(lits > 0).cuda()
    for _ in range(60):
        true = (x[:, var.reshape(-1)].reshape(S, -1, k) == pos)
        cnt = true.sum(2, keepdim=True, dtype=torch.int32)
        gain = (cnt == 0).int() - (true & (cnt == 1)).int()  # flipping this literal mends / breaks
        d = torch.zeros(S, n, dtype=torch.int32, device="cuda")
        d.index_add_(1, var.reshape(-1), gain.reshape(S, -1).int())
        go = torch.rand(S, n, generator=g) < 0.3
        x = x ^ ((d > 0) & go.cuda())
    return lits, x.to(torch.uint8).cpu().numpy()


def _requests(case, seed):
    s = W.Stream(7_000_057 * case["mix"])  # the sizes; everything else is from the seed
    out = []
    for i in range(case["requests"]):
        T = case["t_lo"] + int(s.below(case["t_hi"] - case["t_lo"] + 1, 1)[0])
        if i % 3 == 2:
            n = 32 + int(s.below(161, 1)[0])
            F, D = W.random_qap(n, 7_000_061 * (seed + 1) + i)
            base = W.linear_profile(0.01, 1.0, T).astype(np.float32)
            out.append(("qap", F, D, base, (0.5 + W.Stream(100 * seed + i).unit(n)).astype(np.float32)))
        else:
            u = float(s.unit(1)[0])
            n = int(round(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** u))
            lits = _ksat(n, 4, 9.0 + 0.8 * float(s.unit(1)[0]), 100 * seed + i)
            out.append(("ksat", lits, n) + _profile(n, T, 100 * seed + i))
    return out


# ---- what a user has in hand ---------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, seed=seed)
    if kind == "serve":
        st["requests"] = _requests(case, seed)
        st["server"] = nmc.Server(0)
        return st
    ctx = st["ctx"] = nmc.Context(0)
    n, T = case.get("n"), case.get("T")
    if kind == "anneal" and case["k"] == 0:
        F, D = W.random_qap(n, 7_000_037 * (seed + 1))
        st["inst"] = ctx.load_qap(F, D)
        ctx.set_schedule(st["inst"], _qap_beta(n, T, seed))
    elif kind == "anneal":
        st["inst"] = ctx.load_ksat(_ksat(n, case["k"], case["alpha"], seed), n)
        ctx.set_schedule_factored(st["inst"], *_profile(n, T, seed))
    elif kind == "sweep":
        st["inst"] = ctx.load_ksat(_ksat(n, case["k"], case["alpha"], seed), n)
        beta = W.beta_frozen_ramp(n, T, 0.3, 6.0, 0.20, 0.4, 7_000_019 * (seed + 1))
        ctx.set_schedule(st["inst"], torch.from_numpy(beta).cuda())
        st["rs"] = ctx.replicas_create(st["inst"], case["R"], _philox(seed))
        st["out"], st["views"] = _buffers([(case["R"], n)], torch.uint8)
    elif kind == "batch":
        s = W.Stream(7_000_043 * case["mix"])
        pick = s.below(2, case["sets"])
        ns = case["n_lo"] + s.below(case["n_hi"] - case["n_lo"] + 1, case["sets"])
        rs = case["r_lo"] + s.below(case["r_hi"] - case["r_lo"] + 1, case["sets"])
        st["rs"], sizes = [], []
        for i in range(case["sets"]):
            k, m, R = case["k1"] if pick[i] else case["k0"], int(ns[i]), int(rs[i])
            inst = ctx.load_ksat(_ksat(m, k, ALPHA[k], 1000 * seed + i), m)
            ctx.set_schedule_factored(inst, *_profile(m, T, 1000 * seed + i))
            st["rs"].append(ctx.replicas_create(inst, R, _philox(seed) + i))
            sizes.append((R, m))
        st["out"], st["views"] = _buffers(sizes, torch.uint8)
    elif kind == "pt":
        R = case["ladders"] * case["temps"]
        st["inst"] = ctx.load_ksat(_ksat(n, 4, case["alpha"], seed), n)
        ctx.set_schedule_factored(st["inst"], np.ones(T, np.float32), np.ones(n, np.float32))
        st["rs"] = ctx.replicas_create(st["inst"], R, _philox(seed))
        st["ladder"] = W.geometric_profile(0.3, 6.0, case["temps"]).astype(np.float32)
        ctx.set_ladder(st["rs"], st["ladder"])
        st["out"], st["views"] = _buffers([(R, n)], torch.uint8)
    elif kind == "chain":
        st["inst"] = ctx.load_ksat(_ksat(n, case["k"], case["alpha"], seed), n)
        back = W.seeded_subset(n, 0.2, 7_000_049 * (seed + 1))
        ctx.set_schedule_backbone(st["inst"], np.where(back, 0, -1).astype(np.int32),
                                  case["cycles"], 20, 20, 10, 3.0, 4.0)
        st["mask"], st["beta"] = back.astype(np.uint8)[None, :], np.float32(0.75)
        st["rs"] = ctx.replicas_create(st["inst"], case["R"], _philox(seed))
        st["out"], st["views"] = _buffers([(case["R"], n)], torch.uint8)
    elif kind == "qap":
        ns = case["n_lo"] + W.Stream(7_000_069 * case["mix"]).below(
            case["n_hi"] - case["n_lo"] + 1, case["sets"])
        st["rs"], sizes = [], []
        for i, m in enumerate(int(v) for v in ns):
            F, D = W.random_qap(m, 7_000_037 * (seed + 1) + i)
            inst = ctx.load_qap(F, D)
            ctx.set_schedule(inst, _qap_beta(m, T, 1000 * seed + i))
            st["rs"].append(ctx.replicas_create(inst, case["R"], _philox(seed) + i))
            sizes.append((case["R"], m))
        st["out"], st["views"] = _buffers(sizes, torch.int16)
    elif kind == "lbp":
        lits, st["x"] = _lbp_inputs(case, seed)
        st["inst"] = ctx.load_ksat(lits, n)
    elif kind == "fresh":
        st["lits"] = _ksat(n, case["k"], case["alpha"], seed)
        base, factor = _profile(n, T, seed)
        st["sched"] = np.ascontiguousarray(factor[:, None] * base[None, :])
    else:
        raise ValueError(kind)
    return st


# ---- one pass --------------------------------------------------------------------------------------

def run(st):
    case, seed = st["case"], st["seed"]
    kind = case["kind"]
    if kind == "serve":
        srv, ids = st["server"], []
        for i, r in enumerate(st["requests"]):
            if r[0] == "qap":
                ids.append(srv.submit_qap(r[1], r[2], base=r[3], factor=r[4], replicas=256, seed=i))
            else:
                ids.append(srv.submit_ksat(r[1], r[2], base=r[3], factor=r[4], replicas=32, seed=i))
        out = []
        for i in ids:
            while srv.poll(i, wait_ms=500) in (0, 1):
                pass
            out.append(srv.result(i)[0])
        return out
    ctx = st["ctx"]
    if kind == "anneal":
        return ctx.anneal(st["inst"], case["R"], 0, case["T"], _philox(seed))
    if kind == "fresh":
        inst = ctx.load_ksat(st["lits"], case["n"])
        ctx.set_schedule(inst, st["sched"])
        out = ctx.anneal(inst, case["R"], 0, case["T"], _philox(seed))
        ctx.unload(inst)
        return out
    if kind == "lbp":
        # `deltas` is left out: the last change of the messages, a difference of nearly equal
        # numbers below the tolerance, which a user reads as a size at most
        r = ctx.cnf_lbp(st["inst"], st["x"], LBP_BETA, LAMBDAS, LBP_TOL, LBP_ITER)
        labels, clusters = ctx.cnf_backbone(st["inst"], r["corr"], LBP_BETA, 2.5, 2.0)
        return dict(marg=r["marg"], corr=r["corr"], p=r["p"], q1=r["q1"], iters=r["iters"],
                    n_done=r["n_done"], labels=labels, clusters=clusters)
    extra = {}
    if kind in ("batch", "qap"):
        for i, rs in enumerate(st["rs"]):
            ctx.replicas_reset(rs, _philox(seed) + i)
        (ctx.batch_run if kind == "batch" else ctx.qap_batch_run)(st["rs"], 0, case["T"])
        for rs, v in zip(st["rs"], st["views"]):
            ctx.replicas_read_device(rs, **v)
        return st["out"]
    rs = st["rs"]
    ctx.replicas_reset(rs, _philox(seed))
    if kind == "sweep":
        ctx.replicas_run(rs, 0, case["T"])
    elif kind == "pt":
        ctx.set_ladder(rs, st["ladder"])  # every replica back at its first slot
        ctx.run_pt(rs, 0, case["T"], case["per"])
        extra["slots"] = ctx.read_slots(rs)
    else:
        ctx.replicas_run(rs, 0, 50 * case["cycles"])
        extra["accepted"] = ctx.cluster_flip(rs, st["mask"], st["beta"], 3, accepted=True)
        extra["count"], extra["frozen"], _ = ctx.whitening(rs, use_best=True, masks=True)
    ctx.replicas_read_device(rs, **st["views"][0])
    return {**st["out"], **extra}


# ---- what a pass cannot do without -------------------------------------------------------------------

def _ksat_work(n, k, alpha, R, T, full_schedule):
    """Bytes: formula, schedule and results once. Operations: 32-bit integer ones with 32 replicas
    to a word: per attempted word its clauses' other literals, their counting, eight Philox blocks
    (ten rounds of two wide products and four xors) and five for each replica's acceptance."""
    words, deg = -(-R // 32), k * alpha
    sched = 4 * n * T if full_schedule else 4 * (n + T)
    return (4 * k * alpha * n + sched + 2 * R * n + 16 * R,
            n * words * T * (deg * (k - 1 + 1.5) + 8 * 10 * 8 + 32 * 5))


def _qap_work(n, R, T):
    """Bytes: matrices, schedule, int16 results. Operations: a swap's O(n) change (two
    differences, a product, a sum per facility), a Philox block and the acceptance."""
    return 8 * n * n + 4 * n * T + 4 * R * n + 16 * R, n * R * T * (4 * n + 80 + 10)


def work(case):
    kind = case["kind"]
    if kind == "anneal" and case["k"] == 0:
        b, f = _qap_work(case["n"], case["R"], case["T"])
    elif kind in ("anneal", "sweep", "fresh"):
        b, f = _ksat_work(case["n"], case["k"], case["alpha"], case["R"], case["T"],
                          kind != "anneal")
    elif kind == "batch":
        n, R = (case["n_lo"] + case["n_hi"]) / 2, (case["r_lo"] + case["r_hi"]) // 2
        w = [_ksat_work(n, k, ALPHA[k], R, case["T"], False) for k in (case["k0"], case["k1"])]
        b, f = (case["sets"] / 2 * (w[0][j] + w[1][j]) for j in (0, 1))
    elif kind == "pt":
        b, f = _ksat_work(case["n"], 4, case["alpha"], case["ladders"] * case["temps"], case["T"],
                          False)
    elif kind == "chain":
        # of 50 sweeps a cycle, 20 attempt a fifth of the variables, 20 the rest and 10 all
        n, words = case["n"], -(-case["R"] // 32)
        b, f = _ksat_work(n, case["k"], case["alpha"], case["R"], 30 * case["cycles"], False)
        b += 2 * n * case["R"]
        f += 4 * 2 * case["k"] * case["alpha"] * n * words
    elif kind == "qap":
        n = (case["n_lo"] + case["n_hi"]) / 2
        b, f = (case["sets"] * v for v in _qap_work(n, case["R"], case["T"]))
    elif kind == "lbp":
        # eight iterations at each lambda; per message a product of the others, one division, one
        # sum into the field and the size of its change, about 12 operations in 64 bits
        m, S = case["alpha"] * case["n"], case["S"]
        b = 4 * case["k"] * m + S * (case["n"] + 8 * case["n"] + 8 * m + 4 * case["n"])
        f = 8 * len(LAMBDAS) * S * m * case["k"] * 12
    else:
        n, T = math.sqrt(case["n_lo"] * case["n_hi"]), (case["t_lo"] + case["t_hi"]) / 2
        w, q = _ksat_work(n, 4, 9.4, 32, T, False), _qap_work(112, 256, T)
        b, f = (case["requests"] * (2 * w[j] + q[j]) / 3 for j in (0, 1))
    return {"bytes": float(b), "flops": float(f)}


# ---- the same in 64 bits -----------------------------------------------------------------------------

def exact(case, seed):
    """Belief propagation in plain torch, 64 bits, in fields and logarithms; the sweeps' results
    are whole numbers and have no such value."""
    if case["kind"] != "lbp":
        return None
    lits, x = _lbp_inputs(case, seed)
    n, k, S = case["n"], case["k"], case["S"]
    m = lits.shape[0]
    dev = torch.device("cuda")
    f64 = dict(dtype=torch.float64, device=dev)
    var = torch.from_numpy(np.abs(lits).astype(np.int64) - 1).to(dev)
    sig = torch.from_numpy(np.sign(lits).astype(np.float64)).to(dev)[:, :, None]
    flat = var.reshape(-1)
    eps = torch.bincount(flat, minlength=n).to(**f64)[:, None]
    spin = 2.0 * torch.from_numpy(x.T.astype(np.float64)).to(dev) - 1.0
    c = -math.expm1(-2.0 * LBP_BETA)

    def clause(h):
        # u_i = -1/2 log(1 - c prod_{j != i} (1 - tanh h_j) / 2)
        f = torch.sigmoid(-2.0 * h)
        u = torch.empty_like(f)
        for i in range(k):
            p = torch.ones_like(f[:, 0])
            for j in range(k):
                if j != i:
                    p = p * f[:, j]
            u[:, i] = -0.5 * torch.log1p(-c * p)
        return u

    def total(u, lam):
        t = lam * eps * spin
        return t.index_add(0, flat, (sig * u).reshape(m * k, S))

    h = sig * (LAMBDAS[0] * eps * spin)[flat].reshape(m, k, S)
    u = clause(h)
    run_, alive = torch.ones(S, dtype=torch.bool, device=dev), torch.ones(S, dtype=torch.bool, device=dev)
    done = torch.zeros(S, dtype=torch.long, device=dev)
    at = torch.zeros(S, dtype=torch.long, device=dev)
    hg, ug = h.clone(), u.clone()
    for q, lam in enumerate(LAMBDAS):
        run_ = alive.clone()
        for it in range(LBP_ITER):
            hn = sig * (total(u, lam)[flat].reshape(m, k, S) - sig * u)
            h = torch.where(run_, hn, h)
            un = torch.where(run_, clause(h), u)
            d = (un - u).abs().amax((0, 1))
            u = un
            ok = run_ & (d < LBP_TOL)
            done[ok], at[ok] = q + 1, q
            hg, ug = torch.where(ok, h, hg), torch.where(ok, u, ug)
            run_ = run_ & ~ok
            if it + 1 == LBP_ITER and bool(run_.any()):
                back = run_ & (done > 0)
                h, u = torch.where(back, hg, h), torch.where(back, ug, u)
                at[run_ & (done == 0)] = q
                alive = alive & ~run_
                run_ = torch.zeros_like(run_)
            if not bool(run_.any()):
                break
        if not bool(alive.any()):
            break
    lam = torch.tensor(LAMBDAS, **f64)[at]
    marg = torch.tanh(total(u, lam[None, :])).T
    t = torch.tanh(h)
    free, viol, sign = torch.ones(m, S, **f64), torch.ones(m, S, **f64), torch.ones(m, 1, **f64)
    for j in range(k):
        free, viol, sign = free * sig[:, j] * t[:, j], viol * (1 - t[:, j]) / 2, -sign * sig[:, j]
    corr = ((free - c * sign * viol) / (1.0 - c * viol)).T
    s = spin.T
    return dict(marg=marg.contiguous(), corr=corr.contiguous(), p=(s * marg).mean(1),
                q1=(marg * marg).mean(1), iters=None, n_done=None, labels=None, clusters=None)
