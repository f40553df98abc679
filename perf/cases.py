"""The workloads whose speed is measured: growth and reduction through the public entry points.

Every growth case is what a user of the library does with an ensemble: grow
its chains, then reduce them to the ensemble statistics.  The sizes are those
of the repository's configurations (athermal lattice N = 16 with 10^5 chains;
interacting lattice and hard spheres at N = 64 with 10^7 chains; the mixed
batch of default_rng(4)'s recipe; PERM at N = 64 from 10^6 chains; the scaling
series' longest chains; the long-chain workloads) and ragged sizes between.
"""
import math

import numpy as np
import torch

from paper_1704_04381_gb300 import rosen

# (N - 1) N / 2 pair tests per chain (times k in real space) beyond which the
# 64-bit evaluation below would take longer than about 20 seconds.
LATTICE_PAIRS_MAX = 4e11
SPACE_PAIRS_MAX = 4e11


def listed():
    return [
        # The smallest everyday call: a quick correctness-size lattice ensemble.
        dict(name="lattice_small", kind="lattice", N=16, C=100_000, beta_eps=0.0, attempts=0),
        # The interacting lattice configuration at full size.
        dict(name="lattice_isaw", kind="lattice", N=64, C=10_000_000, beta_eps=0.4, attempts=0),
        # Restart mode (no chain is lost) at a ragged, mid-length size.
        dict(name="lattice_restart", kind="lattice", N=101, C=999_983, beta_eps=0.0, attempts=64),
        # The longest chains of the lattice scaling series.
        dict(name="lattice_512", kind="lattice", N=512, C=500_000, beta_eps=0.0, attempts=0),
        # Long lattice chains (caller-owned workspace).
        dict(name="lattice_long", kind="lattice_long", N=1000, C=200_000, beta_eps=0.0, attempts=0),
        # The hard-sphere configuration at full size.
        dict(name="hard_spheres", kind="space", N=64, C=10_000_000, k=32, potential=0,
             beta_eps=0.0, store=False),
        # The longest chains of the hard-sphere scaling series, conformations kept.
        dict(name="hard_spheres_256", kind="space", N=256, C=60_000, k=32, potential=0,
             beta_eps=0.0, store=True),
        # Lennard-Jones chains at the usual length and trial count.
        dict(name="lennard_jones", kind="space", N=64, C=500_000, k=32, potential=1,
             beta_eps=1.0, store=False),
        # A ragged Lennard-Jones ensemble with many trials, conformations kept.
        dict(name="lennard_jones_150", kind="space", N=150, C=30_011, k=64, potential=1,
             beta_eps=0.7, store=True),
        # Long hard-sphere chains (caller-owned workspace).
        dict(name="hard_spheres_long", kind="space_long", N=1000, C=20_000, k=32, potential=0,
             beta_eps=0.0, store=False),
        # PERM at its usual size.
        dict(name="perm", kind="perm", N=64, M0=1_000_000, cap=4_000_000, beta_eps=0.0),
        # Many mixed ensembles (interacting lattice, Lennard-Jones) in one graph launch.
        dict(name="batch", kind="batch", members=24, recipe=4, C_max=100_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice", "lattice", "space", "space", "space", "lattice_long",
                       "space_long", "perm", "batch"])
    if kind == "lattice":
        N = _log_int(rng, 8, 512)
        C = _log_int(rng, 1000, min(1e7, 6e10 / (N * N)))
        return dict(kind=kind, N=N, C=C, beta_eps=rng.choice([0.0, round(rng.uniform(0.05, 0.6), 3)]),
                    attempts=rng.choice([0, 0, 16]))
    if kind == "lattice_long":
        N = _log_int(rng, 513, 4000)
        return dict(kind=kind, N=N, C=_log_int(rng, 500, 2e8 / N),
                    beta_eps=rng.choice([0.0, round(rng.uniform(0.05, 0.4), 3)]), attempts=0)
    if kind == "space":
        lj = rng.randrange(2)
        k = rng.choice([8, 16, 32, 64, rng.randrange(5, 101)])
        N = _log_int(rng, 8, 320)
        most = (4e10 if lj else 2e11) / (k * N * (N + 60))
        C = _log_int(rng, 300, max(400, min(2e6, most)))
        return dict(kind=kind, N=N, C=C, k=k, potential=lj,
                    beta_eps=round(rng.uniform(0.1, 1.2), 3) if lj else 0.0,
                    store=rng.random() < 0.3 and N * C < 2e7)
    if kind == "space_long":
        lj = rng.randrange(2)
        N = _log_int(rng, 300, 3000)
        return dict(kind=kind, N=N, C=_log_int(rng, 200, (1e7 if lj else 2e7) / N),
                    k=rng.choice([16, 32, 64]), potential=lj,
                    beta_eps=round(rng.uniform(0.1, 1.0), 3) if lj else 0.0, store=False)
    if kind == "perm":
        N = _log_int(rng, 16, 256)
        M0 = _log_int(rng, 1000, min(1e6, 4e9 / (N * N)))
        return dict(kind=kind, N=N, M0=M0, cap=int(M0 * rng.uniform(1.3, 4.0)),
                    beta_eps=rng.choice([0.0, 0.3]))
    return dict(kind=kind, members=rng.randrange(4, 25), recipe=rng.randrange(10, 10_000),
                C_max=_log_int(rng, 2000, 100_000))


def _seed(seed):
    """A 64-bit generator seed of the inputs numbered `seed`."""
    return int(np.random.default_rng([1704, 4381, seed]).integers(1 << 62))


def _members(case):
    """The mixed batch: even members interacting lattice, odd ones Lennard-Jones."""
    g = np.random.default_rng(case["recipe"])
    rows = []
    for e in range(case["members"]):
        N = int(g.integers(8, 257))
        C = min(int(10 ** g.uniform(3, 6)), case["C_max"])
        if e % 2 == 0:
            rows.append(dict(kind="lattice", N=N, C=C, beta_eps=float(g.uniform(0, 0.5)), attempts=0))
        else:
            rows.append(dict(kind="space", N=N, C=C, beta_eps=float(g.uniform(0, 1)),
                             k=int(g.choice([16, 32, 64])), potential=1, store=False))
    return rows


PERM = dict(mu=4.684, c_hi=3.0, c_lo=1.0 / 3.0)


def prepare(case, seed):
    s = _seed(seed)
    kind = case["kind"]
    if kind == "batch":
        ens = [rosen.ensemble(rosen.ROSEN_MODEL_LATTICE, m["N"], m["C"], s + e, e,
                              beta_eps=m["beta_eps"]) if m["kind"] == "lattice" else
               rosen.ensemble(rosen.ROSEN_MODEL_OFFLATTICE, m["N"], m["C"], s + e, e, k=m["k"],
                              potential=m["potential"], beta_eps=m["beta_eps"])
               for e, m in enumerate(_members(case))]
        b = rosen.RosenBatch(ens)
        b.tune()
        return dict(kind=kind, batch=b, stats=torch.zeros(len(ens), len(rosen.STAT_KEYS),
                                                          dtype=torch.float64, device="cuda"))
    if kind == "perm":
        out = rosen.perm_outputs(case["N"], case["cap"])
        out["w_m"].zero_()      # the entries beyond the final population are not written
        out["w_e"].zero_()
        return dict(kind=kind, out=out, workspace=rosen.perm_workspace(case["N"], case["cap"]),
                    params=rosen.perm_params(s, case["N"], case["M0"], case["cap"],
                                             beta_eps=case["beta_eps"], **PERM))
    N, C = case["N"], case["C"]
    st = dict(kind=kind, stats=rosen.stats_tensor(), scratch=rosen.reduce_workspace(C))
    if kind.startswith("lattice"):
        st["params"] = rosen.lattice_params(s, N, C, beta_eps=case["beta_eps"],
                                            max_attempts=case["attempts"])
        st["out"] = rosen.lattice_outputs(N, C, attempts=case["attempts"] > 1)
        st["reduce"] = rosen.lattice_reduce_in(st["out"], N, case["beta_eps"] == 0.0)
        if kind == "lattice_long":
            st["workspace"] = rosen.lattice_long_workspace(N, C)
    else:
        flags = rosen.ROSEN_STORE_TRACE | rosen.ROSEN_STORE_COORDS if case["store"] else 0
        st["params"] = rosen.offlattice_params(s, N, C, case["k"], potential=case["potential"],
                                               beta_eps=case["beta_eps"], flags=flags)
        st["out"] = rosen.offlattice_outputs(N, C, trace=case["store"], coords=case["store"])
        st["reduce"] = rosen.offlattice_reduce_in(st["out"], N, case["k"])
        if kind == "space_long":
            st["workspace"] = rosen.offlattice_long_workspace(N, C)
    return st


def run(state):
    kind = state["kind"]
    if kind == "batch":
        b = state["batch"]
        b.run()
        return dict(stats=b.stats(state["stats"]),
                    chains=[_views(b.lattice_outputs(e) if b.ensembles[e].model == 0
                                   else b.offlattice_outputs(e)) for e in (0, 1)])
    if kind == "perm":
        rosen.rosen_perm_run(state["params"], state["out"], state["workspace"])
        return dict(state["out"])
    if kind == "lattice":
        rosen.rosen_lattice_grow(state["params"], state["out"])
    elif kind == "lattice_long":
        rosen.rosen_lattice_grow_long(state["params"], state["out"], state["workspace"])
    elif kind == "space":
        rosen.rosen_offlattice_grow(state["params"], state["out"])
    else:
        rosen.rosen_offlattice_grow_long(state["params"], state["out"], state["workspace"])
    rosen.rosen_reduce(state["reduce"], state["stats"], state["scratch"])
    return dict(state["out"], stats=state["stats"])


def _views(out):
    return [out[key] for key in sorted(out)]


# ---- what a pass cannot do without ------------------------------------------------
def work(case):
    """Bytes: every output written once (growth reads no inputs).  Operations:
    a Philox draw (about 80) and the observables (about 20) per step; on the
    lattice an occupancy test of the six neighbours (interacting: and their
    contacts); in real space half a draw, a direction (about 20) and the pair
    terms of the few near beads per trial (hard spheres about 3 beads of 8
    operations, Lennard-Jones about 10 of 20)."""
    kind = case["kind"]
    if kind == "batch":
        parts = [work(m) for m in _members(case)]
        return {q: sum(p[q] for p in parts) for q in ("bytes", "flops")}
    if kind == "perm":
        steps = case["M0"] * (case["N"] - 1)
        return {"bytes": 24.0 * case["N"] + 12.0 * case["M0"], "flops": 120.0 * steps}
    steps = float(case["C"]) * (case["N"] - 1)
    if kind.startswith("lattice"):
        out = 32 + (2 if case["attempts"] > 1 else 0)
        return {"bytes": float(out) * case["C"], "flops": steps * (106 if case["beta_eps"] == 0 else 160)}
    out = 13.0 * case["C"] + (13.0 * case["N"] * case["C"] if case["store"] else 0.0)
    return {"bytes": out, "flops": steps * case["k"] * (60 + (200 if case["potential"] else 24))}


# ---- the same results in 64 bits, in plain torch ------------------------------------
_M32 = 0xFFFFFFFF


def _philox(chain, ens, step, slot, seed):
    """Philox4x32-10 of the counters (chain, ens, step, slot); int64 tensors of 32-bit words."""
    x0, x1, x2, x3 = torch.broadcast_tensors(*(torch.as_tensor(v, dtype=torch.int64, device="cuda")
                                               for v in (chain, ens, step, slot)))
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for _ in range(10):
        p0, p1 = x0 * 0xD2511F53, x2 * 0xCD9E8D57
        x0, x1, x2, x3 = (((p1 >> 32) & _M32) ^ x1 ^ k0, p1 & _M32,
                          ((p0 >> 32) & _M32) ^ x3 ^ k1, p0 & _M32)
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return x0, x1, x2, x3


def _u24(word):
    return (word >> 8).double() * 2.0 ** -24


_DIRS = ((1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1))


def _pack(v):
    """Linear site key of a displacement (13 bits per axis, signed)."""
    return v[0] + (v[1] << 13) + (v[2] << 26)


def _lattice_step(keys, i, x, weights):
    """One Rosenbluth step of chains with site keys [i, C]: free flags, factor, slot taken."""
    end = keys[i - 1]
    seen = keys[i % 2:i - 1:2] if weights is None else keys[:i - 1]

    def occupied(d):
        return (seen == end + _pack(d)).any(0)

    occ = {d: occupied(d) for d in _DIRS}
    free = torch.stack([~occ[d] for d in _DIRS])
    if weights is None:
        m = free.sum(0)
        rank = free.long().cumsum(0) - 1
        hit = free & (rank == ((x * m) >> 32))
        return free, m.double(), hit.long().argmax(0)
    w = []
    for d in _DIRS:
        c = torch.zeros_like(end, dtype=torch.int64)
        for f in _DIRS:
            t = tuple(a + b for a, b in zip(d, f))
            if t != (0, 0, 0):
                if t not in occ:
                    occ[t] = occupied(t)
                c += occ[t]
        w.append(torch.where(occ[d], 0.0, weights[c]))
    w = torch.stack(w)
    prefix, P = [], torch.zeros_like(w[0])
    for d in range(6):
        P = P + w[d]
        prefix.append(P)
    above = torch.stack(prefix) > (_u24(x) * P)[None]
    last = (5 - (w > 0).flip(0).long().argmax(0))
    return free, P, torch.where(above.any(0), above.long().argmax(0), last)


def _axes(keys):
    """Coordinates of site keys."""
    x = ((keys + 4096) & 8191) - 4096
    r = (keys - x) >> 13
    y = ((r + 4096) & 8191) - 4096
    return x, y, (r - y) >> 13


def _lattice(case, seed, ens=0):
    N, C, beta = case["N"], case["C"], case["beta_eps"]
    weights = None
    if beta != 0:
        weights = torch.exp(beta * torch.arange(6, dtype=torch.float64, device="cuda"))
    step_key = torch.tensor([_pack(d) for d in _DIRS], device="cuda")
    out = dict(counts=torch.zeros(C, 8, dtype=torch.int16, device="cuda"),
               logw=torch.full((C,), -math.inf, dtype=torch.float64, device="cuda"),
               r2=torch.zeros(C, dtype=torch.int32, device="cuda"),
               n2rg2=torch.zeros(C, dtype=torch.int64, device="cuda"))
    tries = torch.zeros(C, dtype=torch.int16, device="cuda")
    chunk = max(1, int(2e8 / N))

    def grow(idx, att):
        n = idx.numel()
        keys = torch.zeros(N, n, dtype=torch.int64, device="cuda")
        counts = torch.zeros(n, 8, dtype=torch.int16, device="cuda")
        logw = torch.zeros(n, dtype=torch.float64, device="cuda")
        alive = torch.ones(n, dtype=torch.bool, device="cuda")
        for i in range(1, N):
            x = _philox(idx, ens, i | (att << 16), 0, seed)[0]
            free, S, sel = _lattice_step(keys, i, x, weights)
            m = free.sum(0)
            alive &= m > 0
            counts.scatter_add_(1, m[:, None], (alive & (m > 0))[:, None].to(torch.int16))
            logw += torch.where(alive, S, 1.0).log()
            keys[i] = keys[i - 1] + step_key[sel]
        counts[:, 0] = (~alive).to(torch.int16)
        pos = torch.stack(_axes(keys))
        r2 = pos[:, -1].square().sum(0)
        n2rg2 = N * pos.square().sum((0, 1)) - pos.sum(1).square().sum(0)
        out["counts"][idx] = counts
        out["logw"][idx] = torch.where(alive, logw, -math.inf)
        out["r2"][idx] = torch.where(alive, r2, 0).int()
        out["n2rg2"][idx] = torch.where(alive, n2rg2, 0)
        tries[idx] = att + 1
        return idx[~alive]

    for c0 in range(0, C, chunk):
        todo = torch.arange(c0, min(C, c0 + chunk), device="cuda")
        for att in range(max(1, case["attempts"])):
            todo = grow(todo, att)
            if not todo.numel():
                break
    growths = float(C)
    if case["attempts"] > 1:
        out["attempts"] = tries
        growths = float(tries.double().sum())
    out["stats"] = _stats(out["logw"], out["r2"].double(), out["n2rg2"].double() / N ** 2, growths,
                          N, 0)
    return out


def _stats(logw, a, b, growths, N, k):
    live = torch.isfinite(logw)
    alive, M = float(live.sum()), float(logw.max())
    if not alive:
        nan, inf = math.nan, math.inf
        v = [growths, 0.0, -inf] + [0.0] * 8 + [-inf, -inf, nan, nan, nan, nan, 0.0]
        return torch.tensor(v, dtype=torch.float64, device="cuda")
    w = torch.where(live, (logw - M).exp(), 0.0)
    S = [float((w * t).sum()) for t in (torch.ones_like(a), a, b)]
    Q = [float((w * w * t).sum()) for t in (torch.ones_like(a), a, a * a, b, b * b)]
    logZ = M + math.log(S[0] / growths)
    m1, m2 = S[1] / S[0], S[2] / S[0]
    se = [math.sqrt(float((w * (t - m)).square().sum())) / S[0] for t, m in ((a, m1), (b, m2))]
    v = [growths, alive, M] + S + Q + [logZ, logZ - (N - 1) * math.log(k) if k else logZ, m1, se[0],
                                       m2, se[1], S[0] ** 2 / Q[0]]
    return torch.tensor(v, dtype=torch.float64, device="cuda")


def _space(case, seed, ens=0):
    N, C, k, lj, beta = case["N"], case["C"], case["k"], case["potential"], case["beta_eps"]
    chunk = max(1, int(6e7 / (k * N)))
    parts = []
    slots = torch.arange(1, (k + 1) // 2 + 1, device="cuda")[:, None]
    for c0 in range(0, C, chunk):
        idx = torch.arange(c0, min(C, c0 + chunk), device="cuda")
        n = idx.numel()
        pos = torch.zeros(N, 3, n, dtype=torch.float64, device="cuda")
        logw = torch.zeros(n, dtype=torch.float64, device="cuda")
        dead = torch.zeros(n, dtype=torch.int64, device="cuda")     # the step that dead-ends
        trace = torch.full((N - 1, n), 0xFF, dtype=torch.uint8, device="cuda")
        for i in range(1, N):
            w0, w1, w2, w3 = _philox(idx[None], ens, i, slots, seed)
            word = ((w0[0] & 255) | (w1[0] & 255) << 8 | (w2[0] & 255) << 16 | (w3[0] & 255) << 24)
            a = torch.stack([w0, w2], 1).reshape(-1, n)[:k]
            b = torch.stack([w1, w3], 1).reshape(-1, n)[:k]
            z = 1.0 - 2.0 * _u24(a)
            s = ((1.0 - z) * (1.0 + z)).sqrt()
            phi = 2.0 * math.pi * _u24(b)
            u = torch.stack([s * phi.cos(), s * phi.sin(), z])      # [3, k, n]
            trial = pos[i - 1][:, None] + u
            if lj:
                e = torch.zeros(k, n, dtype=torch.float64, device="cuda")
            else:
                free = torch.ones(k, n, dtype=torch.bool, device="cuda")
            if i >= 2:
                d2 = torch.zeros(i - 1, k, n, dtype=torch.float64, device="cuda")
                for q in range(3):
                    d2 += (trial[q][None] - pos[:i - 1, q][:, None]).square()
                if lj:
                    s3 = (1.0 / d2) ** 3
                    e = beta * torch.where(d2 < 6.25, 4.0 * s3 * (s3 - 1.0), 0.0).sum(0)
                else:
                    free = ~(d2 < 1.0).any(0)
            if lj:
                low = e.min(0).values
                w = (low - e).exp()
                P = w.cumsum(0)
                S = P[-1]
                above = P > _u24(word) * S
                last = k - 1 - (w > 0).flip(0).long().argmax(0)
                sel = torch.where(above.any(0), above.long().argmax(0), last)
                gain, ok = S.log() - low, torch.ones(n, dtype=torch.bool, device="cuda")
            else:
                m = free.sum(0)
                rank = free.long().cumsum(0) - 1
                sel = (free & (rank == ((word * m) >> 32))).long().argmax(0)
                gain, ok = m.clamp(min=1).double().log(), m > 0
            now = dead == 0
            trace[i - 1] = torch.where(now, torch.where(ok, sel, 0xFE), 0xFF).to(torch.uint8)
            dead = torch.where(now & ~ok, i, dead)
            logw += torch.where(dead == 0, gain, 0.0)
            pos[i] = pos[i - 1] + u.gather(1, sel[None, None].expand(3, 1, n))[:, 0]
        alive = dead == 0
        c = pos - pos.mean(0)
        kept = alive[None] | (torch.arange(N, device="cuda")[:, None] < dead[None])
        parts.append(dict(logw=torch.where(alive, logw, -math.inf),
                          r2=torch.where(alive, pos[-1].square().sum(0), 0.0),
                          rg2=torch.where(alive, c.square().sum((0, 1)) / N, 0.0),
                          alive=alive.to(torch.uint8)))
        if case["store"]:
            parts[-1].update(trace=trace, coords=torch.where(kept[:, None], pos, 0.0))
    out = {q: torch.cat([p[q] for p in parts], -1) for q in parts[0]}
    out["stats"] = _stats(out["logw"], out["r2"], out["rg2"], float(C), N, k)
    return out


def _split(x):
    """x = m 2^e with m in [1, 2)."""
    m, e = torch.frexp(x)
    return 2.0 * m, e.long() - 1


def _perm(case, seed):
    N, M0, cap, beta = case["N"], case["M0"], case["cap"], case["beta_eps"]
    dev = dict(device="cuda")
    weights = None
    if beta != 0:
        weights = torch.exp(beta * torch.arange(6, dtype=torch.float64, **dev))
    step_key = torch.tensor([_pack(d) for d in _DIRS], **dev)
    keys = torch.zeros(1, M0, dtype=torch.int64, **dev)
    wm = torch.ones(M0, dtype=torch.float64, **dev)
    we = torch.zeros(M0, dtype=torch.int64, **dev)
    pop, logz, mean = [M0], [0.0], [0.0]
    tm, te = 1.0, 0
    for i in range(1, N):
        tm, te = math.frexp(tm * PERM["mu"])[0] * 2.0, te + math.frexp(tm * PERM["mu"])[1] - 1
        j = torch.arange(wm.numel(), **dev)
        x = _philox(j, 0, i, 0, seed)[0]
        free, S, sel = _lattice_step(keys, i, x, weights)
        grew = free.any(0)
        keys = torch.cat([keys, (keys[-1] + step_key[sel])[None]])
        m, e = _split(wm * torch.where(grew, S, 1.0))
        wm, we = torch.where(grew, m, wm), torch.where(grew, we + e, we)
        if not bool(grew.any()):
            pop += [0] * (N - i)
            logz += [-math.inf] * (N - i)
            mean += [math.nan] * (N - i)
            wm, we, keys = wm[:0], we[:0], keys[:, :0]
            break
        top = int(we[grew].max())
        w = torch.where(grew, torch.ldexp(wm, (we - top).clamp(min=-1000)), 0.0)
        r2 = torch.stack(_axes(keys[-1])).square().sum(0).double()
        logz.append(math.log(float(w.sum())) + top * math.log(2.0) - math.log(M0))
        mean.append(float((w * r2).sum()) / float(w.sum()))

        def limit(c):
            f, q = math.frexp(c * tm)
            return 2.0 * f, te + q - 1

        hm, he = limit(PERM["c_hi"])
        lm, le = limit(PERM["c_lo"])
        rich = grew & ((we > he) | ((we == he) & (wm > hm)))
        poor = grew & ~rich & ((we < le) | ((we == le) & (wm < lm)))
        coin = (_philox(j, 0, i, 1, seed)[0] >> 31) == 1
        kept = grew & (~poor | coin)
        granted = rich & (rich.long().cumsum(0) - 1 < cap - int(kept.sum()))
        we = we + poor.long() - granted.long()
        take = torch.repeat_interleave(j, kept.long() + granted.long())
        keys, wm, we = keys[:, take], wm[take], we[take]
        pop.append(take.numel())
    n = wm.numel()
    full_m = torch.zeros(cap, dtype=torch.float64, **dev)
    full_e = torch.zeros(cap, dtype=torch.int32, **dev)
    full_m[:n], full_e[:n] = wm, we.int()
    f64 = dict(dtype=torch.float64, **dev)
    return dict(population=torch.tensor(pop, **dev), logz=torch.tensor(logz, **f64),
                mean_r2=torch.tensor(mean, **f64), final_n=torch.tensor([n], **dev),
                w_m=full_m, w_e=full_e)


def exact(case, seed):
    s = _seed(seed)
    kind = case["kind"]
    if kind == "perm":
        return _perm(case, s) if 2.0 * case["M0"] * case["N"] ** 2 < 3e10 else None
    if kind == "batch":
        return None       # hours of 64-bit pair terms; its members are the cases above
    pairs = case["C"] * (case["N"] - 1.0) * case["N"] / 2
    if kind.startswith("lattice"):
        pairs *= 1 if case["beta_eps"] == 0 else 6
        return _lattice(case, s) if pairs < LATTICE_PAIRS_MAX else None
    return _space(case, s) if pairs * case["k"] < SPACE_PAIRS_MAX else None
