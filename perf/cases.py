"""The workloads this library is measured on, through its Python binding.

A case is a dict of plain values: a "kind" (what the pass calls), the precision, and
the sizes o (occupied), v (virtual), X (auxiliary) and R (CP rank).  The kinds:

* sweep        one ALS sweep of a handle that a program keeps and sweeps on
* cpd          one CPD: `solve` with a fixed number of sweeps, from the same guess each time
* cc           two iterations of a coupled-cluster loop, each with amplitudes of its own
               (a program that keeps its amplitudes for extrapolation): `set_tau`, then a
               short `solve`
* mttkrp       the matrix-free MTTKRP of one mode
* batch        one sweep of many uneven instances from one graph
* energy       the CP energy of the current factors
* exact        the exact contraction on the tensor cores, with R itself
* exact64      the exact contraction in FP64, with R itself
* reconstruct  the CP model in canonical form, symmetrised

Inputs follow the library's synthetic recipe (decaying auxiliary spectrum, MP2-like
amplitudes plus a singles product), drawn on the GPU from the seed.
"""

import math
import random

import torch

from paper_2503_10380_gb300 import binding

MODES = ("a", "b", "i", "j")


def listed():
    return [
        # the smallest molecule of the tests: every step is launch latency
        {"name": "sweep_tiny", "kind": "sweep", "prec": "tf32x3", "o": 5, "v": 24, "X": 72, "R": 48, "fit": True},
        # the benchmark's smaller secondary size: an ordinary molecule, one sweep
        {"name": "sweep_mid", "kind": "sweep", "prec": "tf32x3", "o": 20, "v": 200, "X": 600, "R": 800},
        # the benchmark's larger secondary size: a big fit, two sweeps from a fixed guess
        {"name": "cpd_large", "kind": "cpd", "prec": "tf32x3", "o": 40, "v": 400, "X": 1200, "R": 1600, "sweeps": 2},
        # a CC loop on odd extents, eta on (the stopping rule the method proposes)
        {"name": "cc_ragged", "kind": "cc", "prec": "tf32x3", "o": 13, "v": 117, "X": 355, "R": 331, "sweeps": 3},
        # the t1-dressed tensor in the cheapest tensor-core precision, several r-chunks
        {"name": "sweep_dressed_tf32", "kind": "sweep", "prec": "tf32", "o": 10, "v": 90, "X": 270, "R": 250,
         "dressed": True, "r_chunk": 96},
        # one virtual mode alone, odd extents (a program with its own update step)
        {"name": "mttkrp_a_ragged", "kind": "mttkrp", "prec": "tf32x3", "o": 27, "v": 251, "X": 773, "R": 605, "mode": "a"},
        # one occupied mode alone, in the other split precision
        {"name": "mttkrp_i_bf16", "kind": "mttkrp", "prec": "bf16x3", "o": 20, "v": 200, "X": 600, "R": 800, "mode": "i"},
        # many fragments at once: a part of the 64-instance batch of the benchmark
        {"name": "batch_uneven_bf16", "kind": "batch", "prec": "bf16x3", "count": 16, "shapes": 0},
        # the plain FP64 form, which the mixed forms are judged against
        {"name": "sweep_fp64", "kind": "sweep", "prec": "fp64", "o": 12, "v": 100, "X": 300, "R": 320},
        # the energy after a fit, once per CC iteration
        {"name": "energy_mid", "kind": "energy", "prec": "tf32x3", "o": 20, "v": 200, "X": 600, "R": 800},
        # ||R||^2, E and R on the tensor cores: what a |fit| stopping rule needs for each tau
        {"name": "exact_mixed", "kind": "exact", "prec": "tf32x3", "o": 14, "v": 120, "X": 360, "R": 160},
        # the fitted tensor handed back to a CC program
        {"name": "reconstruct_mid", "kind": "reconstruct", "prec": "bf16x3", "o": 16, "v": 150, "X": 450, "R": 500},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# largest v drawn for a kind, so that no drawn case costs more than the largest listed one
_VMAX = {"sweep": 320, "cpd": 280, "cc": 220, "mttkrp": 380, "energy": 260, "exact": 160, "exact64": 72,
         "reconstruct": 200}


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "cpd", "cc", "mttkrp", "mttkrp", "batch", "energy", "exact", "exact64",
                       "reconstruct"])
    prec = rng.choice(["tf32x3", "tf32x3", "tf32x3", "bf16x3", "tf32", "fp64"])
    if kind == "batch":
        return {"kind": "batch", "prec": rng.choice(["bf16x3", "tf32x3"]), "count": rng.randint(3, 12),
                "shapes": rng.randint(1, 10 ** 6)}
    if kind == "exact" and prec == "fp64":
        prec = "tf32x3"
    if kind == "exact64":
        prec = "fp64"
    vmax = _VMAX[kind]
    if prec == "fp64":
        vmax = min(vmax, 110)
    v = _log_int(rng, 16, vmax)
    o = max(4, min(40, int(v * rng.uniform(0.06, 0.25))))
    X = int(v * rng.uniform(2.0, 4.0))
    R = max(8, int(v * rng.uniform(1.0, 4.0)))
    c = {"kind": kind, "prec": prec, "o": o, "v": v, "X": X, "R": R}
    if kind == "mttkrp":
        c["mode"] = rng.choice(MODES)
    if kind in ("cpd", "cc"):
        c["sweeps"] = rng.randint(2, 4)
    if kind in ("sweep", "mttkrp"):
        c["dressed"] = rng.random() < 0.3
        if rng.random() < 0.3:
            c["r_chunk"] = max(16, R // rng.randint(2, 5))
    return c


# ---- inputs ------------------------------------------------------------------


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, dtype=torch.float64, device="cuda")


def _inputs(o, v, X, R, seed, extra_taus=0):
    """B [X][n][n], tau [o][o][v][v] (and further ones), t1 [o][v], the initial factors."""
    g = _generator(seed)
    n = o + v
    e_occ = -1.5 + 1.2 * torch.rand(o, generator=g, dtype=torch.float64, device="cuda")
    e_vir = 0.1 + 2.9 * torch.rand(v, generator=g, dtype=torch.float64, device="cuda")
    B = _normal(g, X, n, n)
    B = B + B.transpose(1, 2)
    B *= (0.1 / math.sqrt(2.0)) * torch.exp(-torch.arange(X, dtype=torch.float64, device="cuda") / 15.0)[:, None, None]
    Bov = B[:, :o, o:].reshape(X, o * v)
    tau = (Bov.T @ Bov).view(o, v, o, v)
    tau /= (e_occ[:, None, None, None] + e_occ[None, None, :, None] - e_vir[None, :, None, None]
            - e_vir[None, None, None, :])
    tau = tau.permute(0, 2, 1, 3).contiguous()
    t1 = 0.1 * _normal(g, o, v)
    tau += t1[:, None, :, None] * t1[None, :, None, :]
    factors = {m: _normal(g, v if m in "ab" else o, R) for m in MODES}
    taus = [tau]
    for k in range(1, extra_taus + 1):
        Z = _normal(g, o, o, v, v)
        taus.append(taus[-1] + (0.3 ** k) * tau.square().mean().sqrt() / math.sqrt(2.0) * (Z + Z.permute(1, 0, 3, 2)))
    return B, taus, t1, factors


def _shapes(case):
    """Uneven instances: o in [4, 24], v in [40, 240], X = 3v, R in [2v, 4v]."""
    r = random.Random(case["shapes"])
    out = []
    for _ in range(case["count"]):
        o, v = r.randint(4, 24), r.randint(40, 240)
        out.append((o, v, 3 * v, r.randint(2 * v, 4 * v)))
    return out


def _host(factors):
    return {m: f.cpu() for m, f in factors.items()}


def _sizes(case):
    return case["o"], case["v"], case["X"], case["R"]


# ---- what a program has in hand, and one pass -----------------------------------


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        probs = []
        for k, (o, v, X, R) in enumerate(_shapes(case)):
            B, taus, _, fac = _inputs(o, v, X, R, 1000 * seed + k)
            probs.append(binding.CpAls(B, taus[0], _host(fac), precision=case["prec"]))
        return {"case": case, "probs": probs, "batch": binding.Batch(probs, nstreams=8)}
    o, v, X, R = _sizes(case)
    B, taus, t1, fac = _inputs(o, v, X, R, seed, 2 if kind == "cc" else 0)
    cp = binding.CpAls(B, taus[0], _host(fac), precision=case["prec"], r_chunk=case.get("r_chunk", 0), want_eta=kind == "cc",
                       dressed=bool(case.get("dressed")))
    if case.get("dressed"):
        cp.set_t1(t1)
    if case.get("fit"):
        cp.exact_contract()
    if kind in ("cpd", "cc"):
        cp.set_guess_policy("random")    # every solve starts from the guess given at the start
    return {"case": case, "cp": cp, "taus": taus}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        state["batch"].sweep(1, want_fits=False)
        return [p.fac for p in state["probs"]]
    cp = state["cp"]
    if kind == "sweep":
        fits = cp.sweep(1)
        out = dict(cp.factors())
        if case.get("fit"):
            out["fit"] = fits[0]
        return out
    if kind == "cpd":
        cp.solve(case["sweeps"], "fixed")
        return dict(cp.factors())
    if kind == "cc":
        out = {}
        for k in (1, 2):
            cp.set_tau(state["taus"][k])
            n, _, etas = cp.solve(case["sweeps"], "eta", 1e-9)
            out["n%d" % k], out["eta%d" % k] = n, etas[-1]
        out.update(cp.factors())
        return out
    if kind == "mttkrp":
        return cp.mttkrp(case["mode"])
    if kind == "energy":
        return cp.energy()
    if kind in ("exact", "exact64"):
        n2, E, R = cp.exact_contract(want_R=True, mixed=kind == "exact")
        return {"n2": n2, "E": E, "R": R}
    if kind == "reconstruct":
        return cp.reconstruct(symmetrise=True)
    raise ValueError(kind)


# ---- the work of a pass -----------------------------------------------------------


def _sweep_work(o, v, X, R):
    flops = 4.0 * o * o * v * v * R + 16.0 * X * v * v * R
    for dim in (v, v, o, o):
        flops += R ** 3 / 3.0 + 4.0 * dim * R * R
    n = o + v
    return 8.0 * (X * n * n + o * o * v * v + 2 * (2 * v + 2 * o + 1) * R), flops


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [_sweep_work(*s) for s in _shapes(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    o, v, X, R = _sizes(case)
    n = o + v
    b, f = _sweep_work(o, v, X, R)
    fac = 8.0 * (2 * v + 2 * o + 1) * R
    if kind == "sweep":
        return {"bytes": b, "flops": f}
    if kind == "cpd":
        return {"bytes": b, "flops": f * case["sweeps"]}
    if kind == "cc":
        return {"bytes": b + 8.0 * o * o * v * v, "flops": 2 * case["sweeps"] * f}
    if kind == "mttkrp":
        dim = v if case["mode"] in "ab" else o
        return {"bytes": 8.0 * (X * v * v + o * o * v * v + dim * R) + fac,
                "flops": 2.0 * o * o * v * v * R + 6.0 * X * v * v * R}
    if kind == "energy":
        return {"bytes": 8.0 * X * o * v + fac, "flops": 4.0 * X * o * v * R + 8.0 * X * o * R}
    if kind in ("exact", "exact64"):
        g = 1.0 * X * (o * v) * (o * v + 1)      # g[iajb] is symmetric
        return {"bytes": 8.0 * (X * n * n + 2 * o * o * v * v),
                "flops": g + 2.0 * X * v ** 4 + 2.0 * o * o * v ** 4}
    return {"bytes": fac + 8.0 * o * o * v * v, "flops": 2.0 * o * o * v * v * R}


# ---- the same results in 64 bits, plain torch --------------------------------------


def _chunks(R, per):
    step = max(1, min(R, int(2.0e8 // per)))
    return [(r, min(R, r + step)) for r in range(0, R, step)]


def _mttkrp64(Bv, Db, tau, U, mode):
    """M of one mode; R[a,b,i,j] = sum B[Q,a,c] Db[Q,b,d] tau[i,j,c,d]."""
    X, v, _ = Bv.shape
    o = tau.shape[0]
    R = U["a"].shape[1]
    tm = tau.reshape(o * o, v * v)
    out = torch.empty(v if mode in "ab" else o, R, dtype=torch.float64, device=Bv.device)
    for r0, r1 in _chunks(R, 2.0 * X * v):
        c = {m: U[m][:, r0:r1] for m in MODES}
        w = r1 - r0
        if mode in "ab":
            kr = (c["i"][:, None, :] * c["j"][None, :, :]).reshape(o * o, w)
            T = (tm.T @ kr).view(v, v, w).permute(2, 0, 1)                       # [r][c][d]
            if mode == "a":
                W = torch.matmul(Db.transpose(1, 2).reshape(X * v, v), c["b"]).view(X, v, w).permute(2, 1, 0)   # [r][d][Q]
                Y = torch.bmm(T, W)                                              # [r][c][Q]
                out[:, r0:r1] = Bv.permute(1, 2, 0).reshape(v, v * X) @ Y.reshape(w, v * X).T
            else:
                W = torch.matmul(Bv.transpose(1, 2).reshape(X * v, v), c["a"]).view(X, v, w).permute(2, 1, 0)   # [r][c][Q]
                Y = torch.bmm(T.transpose(1, 2), W)                              # [r][d][Q]
                out[:, r0:r1] = Db.permute(1, 2, 0).reshape(v, v * X) @ Y.reshape(w, v * X).T
        else:
            Wa = torch.matmul(Bv.transpose(1, 2).reshape(X * v, v), c["a"]).view(X, v, w).permute(2, 1, 0)      # [r][c][Q]
            Wb = torch.matmul(Db.transpose(1, 2).reshape(X * v, v), c["b"]).view(X, v, w).permute(2, 0, 1)      # [r][Q][d]
            P = (tm @ torch.bmm(Wa, Wb).reshape(w, v * v).T).view(o, o, w)       # [i][j][r]
            out[:, r0:r1] = (P * c["j"][None]).sum(1) if mode == "i" else (P * c["i"][:, None]).sum(0)
    return out


def _sweep64(Bv, Db, tau, U):
    """One ALS sweep in place; returns lam and the last MTTKRP."""
    for m in MODES:
        M = _mttkrp64(Bv, Db, tau, U, m)
        V = 1.0
        for q in MODES:
            if q != m:
                V = V * (U[q].T @ U[q])
        Ut = torch.cholesky_solve(M.T, torch.linalg.cholesky(V)).T
        lam = Ut.norm(dim=0)
        U[m] = Ut / lam
    return lam, M


def _norm2(U, lam):
    V = lam[:, None] * lam[None, :]
    for m in MODES:
        V = V * (U[m].T @ U[m])
    return V.sum()


def _dress(B, t1, o):
    return B[:, o:, o:] - 2.0 * torch.matmul(B[:, o:, :o], t1)


def _tensor64(Bv, tau):
    X, v, _ = Bv.shape
    o = tau.shape[0]
    R = torch.empty(v, v, o, o, dtype=torch.float64, device=Bv.device)
    tm = tau.reshape(o * o, v * v).T.contiguous()
    flat = Bv.reshape(X, v * v)
    for a in range(v):
        G = (Bv[:, a, :].T @ flat).view(v, v, v).transpose(0, 1)      # [b][c][d]
        R[a] = (G.reshape(v, v * v) @ tm).view(v, o, o)
    return R


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for k, (o, v, X, R) in enumerate(_shapes(case)):
            B, taus, _, U = _inputs(o, v, X, R, 1000 * seed + k)
            Bv = B[:, o:, o:].contiguous()
            lam, _ = _sweep64(Bv, Bv, taus[0], U)
            out.append(torch.cat([U[m].reshape(-1) for m in MODES] + [lam]))
        return out
    o, v, X, R = _sizes(case)
    B, taus, t1, U = _inputs(o, v, X, R, seed, 2 if kind == "cc" else 0)
    Bv = B[:, o:, o:].contiguous()
    Db = _dress(B, t1, o) if case.get("dressed") else Bv
    tau = taus[0]
    if kind == "mttkrp":
        return _mttkrp64(Bv, Db, tau, U, case["mode"])
    if kind in ("sweep", "cpd"):
        for _ in range(case.get("sweeps", 1)):
            lam, M = _sweep64(Bv, Db, tau, U)
        out = dict(U, lam=lam)
        if case.get("fit"):
            n2 = _tensor64(Bv, tau).square().sum()
            res = n2 - 2.0 * (M * U["j"] * lam).sum() + _norm2(U, lam)
            out["fit"] = float(1.0 - (res / n2).sqrt())
        return out
    if kind == "cc":
        out = {}
        for k in (1, 2):
            W = dict(U)
            lam = torch.ones(R, dtype=torch.float64, device="cuda")
            for _ in range(case["sweeps"]):
                old, lam0 = dict(W), lam
                lam, _ = _sweep64(Bv, Db, taus[k], W)
            cross = lam[:, None] * lam0[None, :]
            for m in MODES:
                cross = cross * (W[m].T @ old[m])
            n_old = _norm2(old, lam0)
            out["n%d" % k] = case["sweeps"]
            out["eta%d" % k] = float(((_norm2(W, lam) - 2.0 * cross.sum() + n_old) / n_old).sqrt())
        out.update(W, lam=lam)
        return out
    Bov = B[:, :o, o:]
    if kind == "energy":
        A = {}
        for x in "ij":
            for y in "ab":
                A[x + y] = ((Bov @ U[y]) * U[x][None]).sum(1)                     # [Q][r]
        return float((2.0 * A["ia"] * A["jb"] - A["ib"] * A["ja"]).sum())
    if kind in ("exact", "exact64"):
        Rt = _tensor64(Bv, tau)
        g = (Bov.reshape(X, o * v).T @ Bov.reshape(X, o * v)).view(o, v, o, v)    # [i][a][j][b]
        E = 2.0 * (Rt * g.permute(1, 3, 0, 2)).sum() - (Rt * g.permute(3, 1, 0, 2)).sum()
        return {"n2": float(Rt.square().sum()), "E": float(E), "R": Rt}
    ab = (U["a"][:, None, :] * U["b"][None, :, :]).reshape(v * v, R)
    ij = (U["i"][:, None, :] * U["j"][None, :, :]).reshape(o * o, R)
    Rt = (ab @ ij.T).view(v, v, o, o)
    return 0.5 * (Rt + Rt.permute(1, 0, 3, 2))
