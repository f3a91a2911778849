"""The solves whose time is followed: what a user of the annealer calls, over
the range of sizes and options in use.

Every case goes through the package's public entry points (``moda.anneal``,
``anneal_batch``, ``Server``, ``sbda``, ``Qubo.anneal``, ``anneal_noalloc``)
on seeded instances of the repository's own generators, and ends where a
program that calls them ends: with the merged front on the host (the result
of Alg. 3), and for small runs also every replica's archive, final state and
counters.  All outputs are integers.
"""
import math
import time

import numpy as np
import torch

from paper_2205_13399_gb300 import inputs, moda

# Table 1's schedule, the default of every entry point.
DELTA0, DELTAF, XI = 1e9, 1e4, 1e-3
# Iterations until delta stops falling.
COOLING = math.ceil(math.log(DELTAF / DELTA0) / math.log(1.0 - XI))


def listed():
    return [
        # The smallest call: the 64-bit workload, 16 replicas; one warp's
        # worth of bits, so launch and per-iteration latency count.
        dict(name="p8", kind="anneal", flows="uniform", n=8, rho=0.0, replicas=16, I_max=10_000,
             accept="strict", archive="explore"),
        # The headline solve: n = 25, dense flows, 128 replicas at I_max =
        # 10^5, fewer replicas than SMs.
        dict(name="p25", kind="anneal", flows="dense", n=25, rho=0.5, replicas=128, I_max=100_000,
             accept="strict", archive="explore"),
        # The two large single-instance workloads with sparse real-like
        # flows at their full 10^6 iterations, most of them after the
        # schedule has cooled; 256 replicas, more than SMs.  n = 75 is the
        # one whose Delta E bound passes int32.
        dict(name="p50", kind="anneal", flows="sparse", n=50, rho=-0.5, replicas=256,
             I_max=1_000_000, accept="strict", archive="explore"),
        dict(name="p75", kind="anneal", flows="sparse", n=75, rho=-0.5, replicas=256,
             I_max=1_000_000, accept="strict", archive="explore"),
        # The other acceptance and archive rule (Eq. pacceptml, Alg. 5) on an
        # odd size, the paper's rule comparison.
        dict(name="lenient_exploit", kind="anneal", flows="dense", n=33, rho=-0.7, replicas=64,
             I_max=30_000, accept="lenient", archive="exploit"),
        # Near the largest instance the library takes, few replicas.
        dict(name="n100", kind="anneal", flows="dense", n=100, rho=0.0, replicas=32, I_max=20_000,
             accept="strict", archive="explore"),
        # The batched workload (uneven n in [10, 75], 32 replicas each, one
        # graph launch) with a sixteenth of its instances.
        dict(name="batch", kind="batch", instances=32, n_lo=10, n_hi=75, replicas=32,
             I_max=100_000),
        # The serving mix (n of 20, 30, 50, 75, budgets of 10^4 and 10^5),
        # requests already queued when the server starts.
        dict(name="serve", kind="serve", requests=16, replicas=32),
        # The paper's scalarisation baseline on normalised QUBOs (Alg. 1 and
        # 2): eleven weights in one batch launch, the offset escape.
        dict(name="sbda", kind="sbda", n=25, rho=0.5, replicas=16, I_max=24_414),
        # Hypervolume traces: archive snapshots every K iterations.
        dict(name="hvtrace", kind="hvtrace", n=25, rho=0.5, replicas=128, I_max=50_000,
             snapshot_every=5_000),
        # Explicit QUBO matrices with three objectives.
        dict(name="qubo", kind="qubo", K=3, m=1024, replicas=128, I_max=10_000),
        # A caller that owns all device memory.
        dict(name="noalloc", kind="noalloc", n=25, rho=0.5, replicas=16, I_max=20_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["anneal"] * 7 + ["batch", "batch", "serve", "sbda", "hvtrace", "qubo",
                                        "noalloc"])
    rho = round(rng.uniform(-0.75, 0.75), 2)
    if kind == "anneal":
        n = _log_int(rng, 8, 110)
        # at most a third of the largest listed case's cooling work
        most = max(1, min(256, int(256 * 75 ** 2 / (3 * n * n))))
        return dict(kind=kind, flows=rng.choice(["dense", "dense", "sparse", "uniform"]), n=n,
                    rho=rho, replicas=_log_int(rng, 1, most),
                    I_max=_log_int(rng, 5_000, 200_000),
                    accept=rng.choice(["strict", "strict", "lenient"]),
                    archive=rng.choice(["explore", "explore", "exploit"]))
    if kind == "batch":
        lo = rng.randint(8, 40)
        return dict(kind=kind, instances=_log_int(rng, 2, 24), n_lo=lo,
                    n_hi=rng.randint(lo, 70), replicas=rng.choice([4, 16, 32]),
                    I_max=_log_int(rng, 10_000, 100_000))
    if kind == "serve":
        return dict(kind=kind, requests=rng.randint(2, 16), replicas=rng.choice([8, 16, 32]))
    if kind == "sbda":
        n = rng.randint(8, 27)
        return dict(kind=kind, n=n, rho=rho, replicas=rng.randint(2, 16),
                    I_max=_log_int(rng, 2_000, 20_000))
    if kind == "hvtrace":
        I_max = _log_int(rng, 5_000, 50_000)
        return dict(kind=kind, n=rng.randint(8, 30), rho=rho, replicas=rng.randint(8, 128),
                    I_max=I_max, snapshot_every=max(1, I_max // rng.randint(2, 10)))
    if kind == "qubo":
        return dict(kind=kind, K=rng.randint(1, 3), m=_log_int(rng, 64, 1100),
                    replicas=rng.randint(8, 128), I_max=_log_int(rng, 1_000, 10_000))
    return dict(kind="noalloc", n=rng.randint(8, 25), rho=rho, replicas=rng.randint(1, 16),
                I_max=_log_int(rng, 1_000, 20_000))


def _instance(case, seed):
    flows = case.get("flows", "dense")
    if flows == "uniform":
        return inputs.uniform_instance(case["n"], index=seed, workload="P8")
    return inputs.euclid_instance(case["n"], case["rho"], flows == "sparse", index=seed,
                                  workload="P25")


def _mixed(case, seed):
    """The instances of a batch, or the requests of a served mix."""
    ss = np.random.SeedSequence([int(seed), 512])
    rng = np.random.Generator(np.random.PCG64(ss))
    out = []
    for k in range(case.get("instances", case.get("requests"))):
        if case["kind"] == "batch":
            n, I_max = int(rng.integers(case["n_lo"], case["n_hi"] + 1)), case["I_max"]
        else:
            n = int(rng.choice([20, 30, 50, 75]))
            I_max = int(rng.choice([10_000, 100_000]))
        rho = float(rng.choice([-0.7, 0.0, 0.7]))
        q = inputs.euclid_instance(n, rho, False, index=int(rng.integers(1 << 31)),
                                   workload="BATCH")
        out.append((q, I_max, int(rng.integers(1 << 31))))
    return out


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, stream=torch.cuda.current_stream())
    if kind in ("batch", "serve"):
        mix = _mixed(case, seed)
        st["insts"] = [moda.Instance(q.F1, q.F2, q.D) for q, _, _ in mix]
        st["params"] = [moda.make_params(replicas=case["replicas"], I_max=I, seed=s)
                        for _, I, s in mix]
        return st
    if kind == "qubo":
        st["qubo"] = moda.Qubo(inputs.random_qubo(case["K"], case["m"], index=seed))
        st["kw"] = dict(replicas=case["replicas"], I_max=case["I_max"], seed=int(seed))
        return st
    q = _instance(case, seed)
    kw = dict(replicas=case["replicas"], I_max=case["I_max"], seed=int(seed))
    if kind == "noalloc":
        st["qap"] = q
        R, m = case["replicas"], q.n * q.n
        W = (m + 31) // 32
        z = dict(device="cuda")
        st["out"] = dict(arch_E=torch.zeros(R, m, 2, dtype=torch.int64, **z),
                         arch_bits=torch.zeros(R * m * W + 8, dtype=torch.int32, **z),
                         arch_count=torch.zeros(R, dtype=torch.int32, **z),
                         x_final=torch.zeros(R, W, dtype=torch.int32, **z),
                         E_final=torch.zeros(R, 2, dtype=torch.int64, **z),
                         stats=torch.zeros(R, 8, dtype=torch.int64, **z),
                         error=torch.zeros(1, dtype=torch.int32, **z))
        st["params"] = moda.make_params(**kw)
        return st
    st["inst"] = moda.Instance(q.F1, q.F2, q.D)
    if kind == "anneal":
        kw.update(accept=case["accept"], archive=case["archive"])
    if kind == "hvtrace":
        kw.update(snapshot_every=case["snapshot_every"])
    if kind == "sbda":
        kw.update(normalize=True)
    st["kw"] = kw
    return st


# Fronts come back with a fixed number of rows (an output buffer's capacity,
# far above the fronts these runs reach), unused ones -1.
ROWS = 1024


def _front(points, n):
    """A front (list of dicts) as arrays: energies, costs, constraint, origin
    and permutations (rows of -1 for an infeasible point)."""
    vals = np.full((ROWS, 7), -1, dtype=np.int64)
    perm = np.full((ROWS, n), -1, dtype=np.int16)
    for k, p in enumerate(points[:ROWS]):
        vals[k] = (p["E1"], p["E2"], p["c1"], p["c2"], p["g"], p["replica"], p["slot"])
        if p["perm"]:
            perm[k, :len(p["perm"])] = p["perm"]
    return vals, perm


def _fronts(runs, n):
    """The merged fronts of several runs, stacked."""
    got = [_front(r.read_archive(-1), n) for r in runs]
    for r in runs:
        r.close()
    return dict(front=np.stack([g[0] for g in got]), perm=np.stack([g[1] for g in got]))


def _members(count, E, bits):
    """Archives with the slots past |A|, which hold nothing, cleared."""
    empty = np.arange(E.shape[1])[None, :] >= count[:, None]
    E[empty] = 0
    bits[empty] = 0
    return dict(count=count, E=E, bits=bits.view(np.int32))


# Runs of at most this many bits return every replica's archive, state and
# counters besides the front; larger ones the front, as a program that wants
# the solutions does (the raw archives of n = 75 are a gigabyte).
WHOLE_BITS = 33 * 33


def _result(run):
    out = {}
    out["front"], out["perm"] = _front(run.read_archive(-1), run.inst.n)
    if run.inst.m <= WHOLE_BITS:
        r = run.read()
        out.update(_members(r.count, r.E, r.bits), x=r.x.view(np.int32), E_final=r.E_final,
                   # flips, jumps, empty escapes, offset raises; the other
                   # four describe how a launch served the jumps
                   counters=r.stats[:, :4])
    run.close()
    return out


def run(state):
    case, stream = state["case"], state["stream"]
    kind = case["kind"]
    if kind == "anneal":
        return _result(moda.anneal(state["inst"], stream=stream, **state["kw"]).wait())
    if kind == "batch":
        runs = moda.anneal_batch(state["insts"], state["params"], stream=stream)
        for r in runs:
            r.wait()
        return _fronts(runs, case["n_hi"])
    if kind == "serve":
        srv = moda.Server()
        tickets = [srv.submit(i, params=p) for i, p in zip(state["insts"], state["params"])]
        done = [None] * len(tickets)
        while any(d is None for d in done):
            for k, t in enumerate(tickets):
                if done[k] is None:
                    r = srv.poll(t)
                    if r is not None:
                        done[k] = _fronts([r], 75)
            time.sleep(0.0002)
        srv.close()
        return {k: np.concatenate([d[k] for d in done]) for k in ("front", "perm")}
    if kind == "sbda":
        runs, front = moda.sbda(state["inst"], stream=stream, **state["kw"])
        res = []
        for q in runs:
            r = q.read()
            res.append(dict(_members(r.count, r.E, r.bits), x=r.x.view(np.int32),
                            E_final=r.E_final, counters=r.stats[:, :4]))
            q.close()
        vals = np.full((ROWS, 4), -1, dtype=np.int64)
        perm = np.full((ROWS, case["n"]), -1, dtype=np.int16)
        for k, p in enumerate(front[:ROWS]):
            vals[k] = (p["c1"], p["c2"], p["weight"], p["replica"])
            perm[k] = p["perm"]
        return dict({k: np.stack([r[k] for r in res]) for k in res[0]}, front=vals, perm=perm)
    if kind == "hvtrace":
        r = moda.anneal(state["inst"], stream=stream, **state["kw"]).wait()
        snaps = [_front(r.read_archive(snapshot=j), case["n"])
                 for j in range(case["I_max"] // case["snapshot_every"])]
        return dict(_result(r), snapshots=np.stack([s[0] for s in snaps]),
                    snapshot_perms=np.stack([s[1] for s in snaps]))
    if kind == "qubo":
        r = state["qubo"].anneal(stream=stream, **state["kw"]).wait()
        d = r.read()
        r.close()
        return dict(_members(d["count"], d["E"], d["bits"]), x=d["x"].view(np.int32),
                    E_final=d["E_final"], counters=d["stats"])
    q, o = state["qap"], state["out"]
    moda.anneal_noalloc(q.F1, q.F2, q.D, o, params=state["params"], stream=stream)
    return dict(arch_E=o["arch_E"], arch_bits=o["arch_bits"], arch_count=o["arch_count"],
                x_final=o["x_final"], E_final=o["E_final"], counters=o["stats"][:, :4],
                error=o["error"])


def _solve_work(m, n, replicas, I_max):
    """One run of Alg. 3: while the schedule cools nearly every iteration
    flips a bit, which changes every bit's Delta E (20 integer operations a
    bit-trial: field update 2, Delta E 10, acceptance 6, ballot 2); once it
    has, an iteration needs its restart draw (40 operations)."""
    cool = min(I_max, COOLING)
    ops = replicas * (cool * m * 20 + I_max * 40)
    W = (m + 31) // 32
    # matrices in; per replica a final state, energies and counters out
    return 3 * n * n * 2 + replicas * (4 * W + 16 + 64), ops


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        b = f = 0
        for q, I_max, _ in _mixed(case, 0):
            db, df = _solve_work(q.n * q.n, q.n, case["replicas"], I_max)
            b, f = b + db, f + df
        return dict(bytes=b, flops=f)
    if kind == "qubo":
        K, m, R, I_max = case["K"], case["m"], case["replicas"], case["I_max"]
        return dict(bytes=K * m * m * 4 + R * (m // 8 + 8 * K + 64),
                    flops=R * min(I_max, COOLING) * m * (8 + 6 * K))
    n, R, I_max = case["n"], case["replicas"], case["I_max"]
    b, f = _solve_work(n * n, n, R, I_max)
    if kind == "sbda":  # eleven runs with the offset escape: every iteration a trial
        f = 11 * R * I_max * n * n * 20
    return dict(bytes=b, flops=f)


# ---- the same solve in plain numpy ----------------------------------------

_M0, _M1 = np.uint64(0xD2511F53), np.uint64(0xCD9E8D57)
_LOW, _32 = np.uint64(0xFFFFFFFF), np.uint64(32)


def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 words of the given counters (Salmon et al., SC'11)."""
    c0, c1, c2, c3 = (np.broadcast_arrays(*[np.asarray(c, np.uint64) for c in (c0, c1, c2, c3)]))
    k0, k1 = key & 0xFFFFFFFF, key >> 32
    for _ in range(10):
        a, b = _M0 * c0, _M1 * c2
        c0, c1, c2, c3 = ((b >> _32) ^ c1 ^ np.uint64(k0), b & _LOW,
                          (a >> _32) ^ c3 ^ np.uint64(k1), a & _LOW)
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1, c2, c3


def _pick(u, count):
    return ((u * np.asarray(count).astype(np.uint64)) >> _32).astype(np.int64)


def exact(case, seed):
    """Alg. 3 with strict acceptance and the Alg. 4 archive in 64-bit numpy,
    all replicas side by side, for the cases small enough for it."""
    if (case["kind"] != "anneal" or case["n"] ** 2 * case["I_max"] > 64 * 10_000
            or case["replicas"] > 16 or case["accept"] != "strict"
            or case["archive"] != "explore"):
        return None
    q = _instance(case, seed)
    n, R, I_max, key = q.n, case["replicas"], case["I_max"], int(seed)
    m = n * n
    W = (m + 31) // 32
    D = q.D.astype(np.int64)
    F = [f.astype(np.int64) + f.astype(np.int64).T for f in (q.F1, q.F2)]
    w = [int(f.sum(1).max()) * int(D.sum(1).max()) for f in F]
    P = [np.kron(f, D) for f in F]  # P[(i,u),(j,v)] = Fs_ij d_uv
    T = np.array([-math.log((i + 0.5) / 65536.0) for i in range(65536)])
    rep = np.arange(R, dtype=np.uint64)
    rows = np.arange(R)
    bit = np.arange(m)
    # initial state: bit p is bit p % 32 of word (p / 32) % 4 of block p / 128
    wd = np.stack(_philox(np.arange((m + 127) // 128)[None, :], 0, rep[:, None], 4, key), 2)
    x = ((wd.reshape(R, -1)[:, bit // 32] >> (bit % 32).astype(np.uint64)) & np.uint64(1))
    x = x.astype(np.int64)
    L = [x @ p for p in P]
    X = x.reshape(R, n, n)
    Rc, Cc = X.sum(2), X.sum(1)
    g = ((1 - Rc) ** 2).sum(1) + ((1 - Cc) ** 2).sum(1)
    E = np.stack([(x * L[k]).sum(1) // 2 + w[k] * (g // 2) for k in (0, 1)], 1)
    AE = np.zeros((R, m, 2), np.int64)
    AX = np.zeros((R, m, m), np.int64)
    cnt = np.zeros(R, np.int64)
    stats = np.zeros((R, 4), np.int64)
    slot_no = np.arange(m)
    grp = np.arange((m + 3) // 4)
    delta = DELTA0
    for t in range(1, I_max + 1):
        if delta > DELTAF:
            delta = delta * (1.0 - XI)
        h = (Rc[:, :, None] + Cc[:, None, :]).reshape(R, m) - 1 - 2 * x
        dE = [(1 - 2 * x) * (L[k] + w[k] * h) for k in (0, 1)]
        a = np.maximum(dE[0], 0) + np.maximum(dE[1], 0)
        u = np.stack(_philox(grp[None, :], t, rep[:, None], 0, key), 2).reshape(R, -1)[:, :m]
        acc = a.astype(np.float64) <= delta * T[(u >> np.uint64(16)).astype(np.int64)]
        total = acc.sum(1)
        flip = total > 0
        r = _pick(_philox(0, t, rep, 1, key)[0], total)
        ps = np.argmax((acc.cumsum(1) == (r + 1)[:, None]) & acc, 1)
        fr = rows[flip]
        if fr.size:
            p = ps[fr]
            s = 1 - 2 * x[fr, p]
            for k in (0, 1):
                E[fr, k] += dE[k][fr, p]
                L[k][fr] += s[:, None] * P[k][p]
            x[fr, p] ^= 1
            Rc[fr, p // n] += s
            Cc[fr, p % n] += s
            e = E[fr][:, None, :]
            A = AE[fr]
            dom = ((e <= A).all(2) & (e != A).any(2) & (slot_no[None, :] < cnt[fr][:, None]))
            tgt = np.where(dom.any(1), dom.argmax(1), cnt[fr])
            ok = tgt < m
            AE[fr[ok], tgt[ok]] = E[fr[ok]]
            AX[fr[ok], tgt[ok]] = x[fr[ok]]
            cnt[fr[ok]] = np.maximum(cnt[fr[ok]], tgt[ok] + 1)
        jr = rows[~flip & (cnt > 0)]
        if jr.size:
            y = _pick(_philox(0, t, rep[jr], 2, key)[0], cnt[jr])
            x[jr] = AX[jr, y]
            E[jr] = AE[jr, y]
            for k in (0, 1):
                L[k][jr] = x[jr] @ P[k]
            X = x[jr].reshape(-1, n, n)
            Rc[jr], Cc[jr] = X.sum(2), X.sum(1)
        stats[:, 0] += flip
        stats[:, 1] += ~flip & (cnt > 0)
        stats[:, 2] += ~flip & (cnt == 0)

    def words(b):
        pad = np.zeros(b.shape[:-1] + (W * 32,), np.uint64)
        pad[..., :m] = b
        return (pad.reshape(b.shape[:-1] + (W, 32)) << np.arange(32, dtype=np.uint64)).sum(
            -1).astype(np.uint32)

    # the merged non-dominated members, lowest (replica, slot) among equals
    pts = sorted((int(AE[i, j, 0]), int(AE[i, j, 1]), i, j) for i in range(R)
                 for j in range(cnt[i]))
    points, best = [], None
    for e1, e2, i, j in pts:
        if best is not None and e2 >= best:
            continue
        best = e2
        Y = AX[i, j].reshape(n, n)
        gg = int(((1 - Y.sum(1)) ** 2).sum() + ((1 - Y.sum(0)) ** 2).sum())
        points.append(dict(E1=e1, E2=e2, c1=e1 - w[0] * (gg // 2), c2=e2 - w[1] * (gg // 2), g=gg,
                           replica=i, slot=j,
                           perm=[int(v) for v in Y.argmax(1)] if gg == 0 else None))
    front, perm = _front(points, n)
    return dict(front=front, perm=perm, **_members(cnt.astype(np.int32), AE, words(AX)),
                x=words(x).view(np.int32), E_final=E, counters=stats)
