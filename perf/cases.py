"""The work a user of this library has it do, as cases that can be timed.

A case is one system (or one batch of systems) of the grid-network model of
``paper_2510_05885_gb300.synth`` and one pass over it through the public
entry points:

  step      factor + refined solve in one call (``ncl_kkt_batch_factor_solve``,
            the call the benchmark times): one Newton step of the NCL loop
  separate  ``KKT.factor`` then ``KKT.solve``, as the README uses the library
  solve     ``KKT.solve`` on factors that are there already (a second right-hand
            side, the extrapolation step)
  adjoint   ``step`` and then ``KKT.adjoint``: forward and backward of a layer
            that differentiates through the solve
  slack     the condensed form with slacks: ``factor_k1s``, ``k1s_rhs``,
            ``solve``, ``slack_step``
  newton    ``newton_rhs``, ``solve``, ``newton_recover`` after ``factor``: the
            whole Newton step around the factorisation

Patterns are analysed once per process and shared (the symbolic analysis is
made once per pattern and reused across Newton steps); every state has a
handle of its own on that analysis, and values made from the seed.  The
settings are the benchmark's: the committed table of tuned cut-overs, and a
backward-error target at which the solution itself, not only its residual,
is settled to about ten digits (``ir_tol``).
"""
import math
import os

import numpy as np
import torch

import paper_2510_05885_gb300 as _pkg
from paper_2510_05885_gb300 import ncl_kkt as nk
from paper_2510_05885_gb300 import synth

TUNED = os.path.join(os.path.dirname(os.path.abspath(_pkg.__file__)), "tuned_gb300.txt")
F64 = torch.float64


def _case(call, form, rows, cols, rho, name=None, count=1, spread=0, nrhs=1, prec="fp32_ir"):
    # the solution's error is the condition number (which the penalty enters)
    # times the backward error
    tol = (1e-12 if rho < 1e6 else 1e-13) if form == "stabilized" else max(1e-15, 1e-11 / rho)
    c = {"call": call, "form": form, "rows": rows, "cols": cols, "rho": float(rho), "count": count,
         "spread": spread, "nrhs": nrhs, "prec": prec, "ir_tol": tol}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a small network in an outer loop that factors thousands of times: latency and launches count
        _case("step", "stabilized", 20, 25, 1e4, name="step-20x25"),
        # a mid-sized network, the condensed form
        _case("step", "condensed", 100, 100, 1e4, name="step-condensed-100"),
        # a mid-sized network, the stabilized form
        _case("step", "stabilized", 150, 150, 1e4, name="step-stabilized-150"),
        # the benchmark's default workload
        _case("step", "condensed", 300, 300, 1e5, name="step-condensed-300"),
        # the benchmark's largest single system
        _case("step", "stabilized", 700, 700, 1e6, name="step-stabilized-700"),
        # the scenarios of one network (one to three lines out in each), four right-hand sides
        _case("step", "stabilized", 100, 100, 1e4, name="scenarios-64x100", count=64, nrhs=4),
        # a mixed batch of networks of side 10 to 70, differentiated through
        _case("adjoint", "stabilized", 10, 70, 1e4, name="adjoint-mixed-64", count=64, spread=1),
        # several right-hand sides on the factors of the benchmark's default system
        _case("solve", "condensed", 300, 300, 1e5, name="solve-8rhs-300", nrhs=8),
        # one more right-hand side on the factors of an odd-sized network
        _case("solve", "stabilized", 93, 107, 1e4, name="solve-93x107"),
        # the plain FP64 path, factor and solve apart
        _case("separate", "condensed", 100, 100, 1e4, name="fp64-condensed-100", prec="fp64"),
        # inequality rows with slacks
        _case("slack", "condensed", 200, 200, 1e3, name="slack-200"),
        # right-hand side, factorisation, solve and the whole direction of one Newton step
        _case("newton", "stabilized", 61, 83, 1e4, name="newton-61x83"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        case = _any(rng)
        if _contained(case):
            return case


def _contained(case):
    """Whether reads of whole 32 x 32 blocks along the diagonals of the pivot
    blocks stay within the pages of the factor's storage.  The kernel that
    inverts these blocks read the rows of a last, narrower block up to the
    32nd, which only the block of a root can put past the end of the storage;
    a system where that could leave the last mapped page is not drawn."""
    pats = [_pattern(k) for k in _instances(case)]
    arrays = [(p.n, p.m, p.H_rowptr, p.H_colind, p.J_rowptr, p.J_colind) for p in pats]
    K = nk.KKT.batch(nk.STABILIZED if case["form"] == "stabilized" else nk.CONDENSED, arrays, host_only=1)
    col0, _, nrow = (a.astype(np.int64) for a in K.supernodes())
    ncol = np.diff(col0)
    width = (ncol + 3) // 4 * 4
    size = (nrow * width + 31) // 32 * 32
    last = ncol - 1 - (ncol - 1) % 32
    reach = int((np.cumsum(size) - size + (last + 31) * width + last + 31)[ncol > 32].max(initial=0))
    return all(reach * b <= -(-int(size.sum()) * b // (2 << 20)) * (2 << 20) for b in (4, 8))


def _any(rng):
    call = rng.choice(["step", "step", "step", "separate", "solve", "solve", "adjoint", "slack", "newton"])
    form = "condensed" if call == "slack" else rng.choice(["stabilized", "condensed"])
    prec = "fp64" if rng.random() < 0.15 else "fp32_ir"
    if call in ("step", "adjoint", "separate") and rng.random() < 0.35:
        if rng.random() < 0.5:
            # scenarios of one network
            count = _log_uniform(rng, 2, 64)
            side = _log_uniform(rng, 8, 100 if prec == "fp32_ir" else 50)
            return _case(call, "stabilized", side, max(2, side + rng.randint(-5, 5)), 1e4, count=count,
                         nrhs=rng.choice([1, 2, 4, 5]) if call != "adjoint" else rng.choice([1, 2]), prec=prec)
        lo = _log_uniform(rng, 5, 20)
        return _case(call, "stabilized", lo, lo + _log_uniform(rng, 5, 50), 1e4,
                     count=_log_uniform(rng, 4, 128 if prec == "fp32_ir" else 32), spread=1, prec=prec)
    hi = 110 if prec == "fp64" else 420
    rows = _log_uniform(rng, 6, hi)
    cols = max(2, min(hi, int(round(rows * rng.uniform(0.5, 1.6)))))
    rho = rng.choice([1e2, 1e3, 1e4, 1e5])
    nrhs = rng.choice([1, 1, 2, 3, 8]) if call in ("step", "separate", "solve") else 1
    return _case(call, form, rows, cols, rho, nrhs=nrhs, prec=prec)


# ---------------------------------------------------------------------------
# patterns and their analyses
# ---------------------------------------------------------------------------
_grids, _plans = {}, {}


def _instances(case):
    """(rows, cols, deleted edges) of every system of the case."""
    if case["spread"]:
        lo, hi, n = case["rows"], case["cols"], case["count"]
        sides = [lo + int(round((hi - lo) * i / max(n - 1, 1))) for i in range(n)]
        np.random.Generator(np.random.PCG64(n)).shuffle(sides)
        return [(s, s, ()) for s in sides]
    if case["count"] == 1:
        return [(case["rows"], case["cols"], ())]
    rng = np.random.Generator(np.random.PCG64(case["count"]))
    E = len(synth.grid_edges(case["rows"], case["cols"]))
    return [(case["rows"], case["cols"], tuple(sorted(int(e) for e in rng.choice(E, size=int(rng.integers(1, 4)), replace=False))))
            for _ in range(case["count"])]


def _pattern(key):
    if key not in _grids:
        _grids[key] = synth.make_pattern(key[0], key[1], np.asarray(key[2], dtype=np.int64) if key[2] else None)
    return _grids[key]


class _Plan:
    """The analysed pattern of a case and what its values are made from."""

    def __init__(self, case):
        self.stab = case["form"] == "stabilized"
        pats = [_pattern(k) for k in _instances(case)]
        self.pats = pats
        form = nk.STABILIZED if self.stab else nk.CONDENSED
        arrays = [(p.n, p.m, p.H_rowptr, p.H_colind, p.J_rowptr, p.J_colind) for p in pats]
        if len(arrays) == 1:
            self.base = nk.KKT(form, *arrays[0], host_only=1)
        else:
            self.base = nk.KKT.batch(form, arrays, host_only=1)
        n, m = np.array([p.n for p in pats]), np.array([p.m for p in pats])
        dims = n + (m if self.stab else 0)
        off = lambda v: np.concatenate([[0], np.cumsum(v)]).astype(np.int64)  # noqa: E731
        self.n, self.m = n, m
        self.noff, self.moff, self.doff = off(n), off(m), off(dims)
        self.dim = int(self.doff[-1])
        hoff = off([p.nnz_H for p in pats])
        # edge blocks in four groups, so that within a group no two blocks meet
        # (the sums of a bus's own entries then have one order)
        pos, grp, ends = [], [], []
        for i, p in enumerate(pats):
            b1, b2 = p.edges[:, 0], p.edges[:, 1]
            down = (b2 - b1) == p.C
            g = np.where(down, 2 + (b1 // p.C) % 2, (b1 % p.C) % 2)
            pos.append(p.edge_pos + hoff[i])
            grp.append(g)
            ends.append(np.stack([b1, b2], 1) + self.noff[i] // 4)
        pos, grp, ends = np.concatenate(pos), np.concatenate(grp), np.concatenate(ends)
        order = np.argsort(grp, kind="stable")
        self.cuts = [int(v) for v in np.searchsorted(grp[order], np.arange(5))]
        self.pos = torch.from_numpy(pos[order]).cuda()
        self.ends = torch.from_numpy(ends[order]).cuda()
        self.nnzH, self.nnzJ = int(hoff[-1]), int(sum(p.nnz_J for p in pats))
        self.nvar, self.ncon = int(self.noff[-1]), int(self.moff[-1])
        info = self.base.analysis
        self.nnz_L, self.nnz_A, self.flops = int(info.nnz_L), int(info.nnz_A), float(info.flops)


def _plan(case):
    key = (case["form"], case["rows"], case["cols"], case["count"], case["spread"])
    if key not in _plans:
        while len(_plans) >= 12:
            del _plans[next(iter(_plans))]
        _plans[key] = _Plan(case)
    return _plans[key]


def _values(case, seed):
    """H, J, Sigma, delta, rho and the right-hand sides, as ``synth`` draws
    them: an indefinite block of prescribed spectrum per edge, normal J,
    Sigma over four decades, delta the power of ten that certifies
    H + Sigma + delta I positive definite."""
    P = _plan(case)
    g = torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))
    rnd = lambda *s: torch.rand(*s, dtype=F64, device="cuda", generator=g)       # noqa: E731
    nrm = lambda *s: torch.randn(*s, dtype=F64, device="cuda", generator=g)      # noqa: E731
    E = len(P.pos)
    lam = 2.0 * rnd(E, 8) - 1.0
    B = torch.diag_embed(lam)
    for _ in range(8):    # random reflections on both sides keep the spectrum
        v = nrm(E, 8, 1)
        v = v / v.norm(dim=1, keepdim=True)
        B = B - 2.0 * v * (v * B).sum(1, keepdim=True)
        B = B - 2.0 * (v.transpose(1, 2) * B).sum(2, keepdim=True) * v.transpose(1, 2)
    la, lb = np.tril_indices(8)
    low = B[:, torch.from_numpy(la).cuda(), torch.from_numpy(lb).cuda()]
    neg = (-lam.min(dim=1).values).clamp(min=0.0)
    H = torch.zeros(P.nnzH, dtype=F64, device="cuda")
    cert = torch.zeros(P.nvar // 4, dtype=F64, device="cuda")
    for a, b in zip(P.cuts[:-1], P.cuts[1:]):
        if b > a:
            idx = P.pos[a:b].reshape(-1)
            H[idx] = H[idx] + low[a:b].reshape(-1)
            for k in range(2):
                cert[P.ends[a:b, k]] = cert[P.ends[a:b, k]] + neg[a:b]
    J = nrm(P.nnzJ)
    S = 10.0 ** (4.0 * rnd(P.nvar) - 2.0)
    slack = (S.reshape(-1, 4) - cert[:, None]).min(dim=1).values.cpu().numpy()
    delta = []
    for i in range(len(P.pats)):
        s = float(slack[P.noff[i] // 4:P.noff[i + 1] // 4].min())
        delta.append(0.0 if s > 0 else 10.0 ** math.floor(math.log10(-s) + 1.0))
    rhs = nrm(case["nrhs"], P.dim)
    v = {"H": H, "J": J, "S": S, "delta": delta, "rho": [case["rho"]] * len(P.pats), "B": rhs}
    if case["call"] == "slack":
        ss = 10.0 ** (6.0 * rnd(P.ncon) - 2.0)
        v["Ss"] = torch.where(rnd(P.ncon) < 0.4, torch.full_like(ss, math.inf), ss)   # 40 % equality rows
        v["RS"] = nrm(P.ncon)
    if case["call"] == "newton":
        x = nrm(P.nvar)
        lo, up = x - 0.1 - rnd(P.nvar), x + 0.1 + rnd(P.nvar)
        has_lo, has_up = rnd(P.nvar) < 0.7, rnd(P.nvar) < 0.5
        inf = torch.full_like(x, math.inf)
        v["pt"] = {"grad_phi": nrm(P.nvar), "x": x, "lower": torch.where(has_lo, lo, -inf),
                   "upper": torch.where(has_up, up, inf), "z_lower": torch.where(has_lo, rnd(P.nvar), 0 * x),
                   "z_upper": torch.where(has_up, rnd(P.nvar), 0 * x), "c": nrm(P.ncon), "y": nrm(P.ncon),
                   "y_k": nrm(P.ncon), "r": nrm(P.ncon)}
        v["mu"] = 1e-2
    return v


def prepare(case, seed):
    P = _plan(case)
    s = {"call": case["call"], "nrhs": case["nrhs"], "v": _values(case, seed)}
    s["K"] = nk.KKT.like(P.base, prec=case["prec"], ir_tol=case["ir_tol"], ir_max_iter=20, autotune_path=TUNED)
    if case["call"] in ("step", "adjoint"):
        s["X"] = torch.empty_like(s["v"]["B"])
    else:
        s["b"] = s["v"]["B"][0].clone() if case["nrhs"] == 1 else s["v"]["B"].t().contiguous()
    if case["call"] == "solve":
        _factor(s)
    return s


def _factor(s):
    v, K = s["v"], s["K"]
    one = K.count == 1
    return K.factor(v["H"], v["J"], v["S"], v["delta"][0] if one else v["delta"], v["rho"][0] if one else v["rho"])


def _inertia(infos):
    infos = infos if isinstance(infos, list) else [infos]
    return np.array([[f.n_pos, f.n_neg, f.n_zero, f.n_perturbed] for f in infos], dtype=np.int64)


def run(s):
    call, K, v = s["call"], s["K"], s["v"]
    if call in ("step", "adjoint"):
        X = s["X"]
        infos, _ = nk.ncl_kkt_batch_factor_solve(K._h, v["H"], v["J"], v["S"], v["delta"], v["rho"], s["nrhs"], v["B"],
                                                 K.dim, X, K.dim)
        out = {"X": X, "inertia": _inertia(infos)}
        if call == "adjoint":
            g = K.adjoint(X.t(), X.t())    # of 0.5 |x|^2
            out.update({k: g[k] for k in ("b", "H", "J", "Sigma", "scal")})
        return out
    if call == "separate":
        infos = _factor(s)
        X, _ = K.solve(s["b"])
        return {"X": X, "inertia": _inertia(infos)}
    if call == "solve":
        X, _ = K.solve(s["b"])
        return {"X": X}
    if call == "slack":
        info = K.factor_k1s(v["H"], v["J"], v["S"], v["Ss"], v["delta"][0], v["rho"][0])
        X, _ = K.solve(K.k1s_rhs(s["b"], v["RS"]))
        return {"X": X, "ds": K.slack_step(X, v["RS"]), "inertia": _inertia(info)}
    info = _factor(s)
    B = K.newton_rhs(v["pt"], v["mu"])
    X, _ = K.solve(B)
    out = K.newton_recover(v["pt"], v["mu"], X)
    out.update({"B": B, "inertia": _inertia(info)})
    return out


def work(case):
    """Each value of H, J, Sigma and the right-hand sides read once, the factor
    written once and read twice by one pair of triangular sweeps, the
    solution written; the factorisation's own operations."""
    P = _plan(case)
    esz = 4 if case["prec"] == "fp32_ir" else 8
    nr = case["nrhs"]
    vec = 8.0 * P.dim * nr
    vals = 8.0 * (P.nnzH + P.nnzJ + P.nvar)
    by, fl = 2.0 * vec + 2.0 * esz * P.nnz_L, 4.0 * P.nnz_L * nr
    if case["call"] != "solve":
        by += vals + esz * P.nnz_L
        fl += P.flops
    if case["call"] == "adjoint":
        by += 2.0 * vec + vals + 2.0 * esz * P.nnz_L
        fl += 4.0 * P.nnz_L * nr
    if case["call"] == "slack":
        by += 8.0 * 3 * P.ncon
    if case["call"] == "newton":
        by += 8.0 * (9 * P.nvar + 6 * P.ncon)
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# the same in 64 bits: conjugate gradients on the condensed form, refined on
# the system itself
# ---------------------------------------------------------------------------
def _csr(rows, cols, vals, shape):
    order = torch.argsort(rows * shape[1] + cols)
    rows, cols, vals = rows[order], cols[order], vals[order]
    ptr = torch.zeros(shape[0] + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=shape[0]), 0)
    return torch.sparse_csr_tensor(ptr, cols, vals, shape)


def _system(case, v):
    P = _plan(case)
    hr, hc, jr, jc, dual, prim = [], [], [], [], [], []
    for i, p in enumerate(P.pats):
        hr.append(np.repeat(np.arange(p.n), np.diff(p.H_rowptr)) + P.noff[i])
        hc.append(p.H_colind.astype(np.int64) + P.noff[i])
        jr.append(np.repeat(np.arange(p.m), np.diff(p.J_rowptr)) + P.moff[i])
        jc.append(p.J_colind.astype(np.int64) + P.noff[i])
        prim.append(P.doff[i] + np.arange(p.n))
        if P.stab:
            dual.append(P.doff[i] + p.n + np.arange(p.m))
    T = lambda a: torch.from_numpy(np.concatenate(a)).cuda()  # noqa: E731
    hr, hc, jr, jc = T(hr), T(hc), T(jr), T(jc)
    off = hr != hc
    Hs = _csr(torch.cat([hr, hc[off]]), torch.cat([hc, hr[off]]), torch.cat([v["H"], v["H"][off]]), (P.nvar, P.nvar))
    J = _csr(jr, jc, v["J"], (P.ncon, P.nvar))
    JT = _csr(jc, jr, v["J"], (P.nvar, P.ncon))
    per = lambda x, cnt: torch.from_numpy(np.repeat(np.asarray(x, dtype=np.float64), cnt)).cuda()  # noqa: E731
    diag = v["S"] + per(v["delta"], P.n)
    w = per(v["rho"], P.m)
    if "Ss" in v:
        fin = torch.isfinite(v["Ss"])
        w = torch.where(fin, w * torch.where(fin, v["Ss"], 1.0) / (w + torch.where(fin, v["Ss"], 1.0)), w)
    hd = torch.zeros(P.nvar, dtype=F64, device="cuda")
    hd[hr[~off]] = v["H"][~off]
    jd = torch.zeros(P.nvar, dtype=F64, device="cuda").index_add_(0, jc, v["J"] * v["J"] * w[jr])
    return {"H": Hs, "J": J, "JT": JT, "diag": diag, "w": w, "pre": 1.0 / (hd + diag + jd), "hr": hr, "hc": hc, "jr": jr,
            "jc": jc, "prim": T(prim), "dual": T(dual) if P.stab else None}


def _cg(S, b, tol=1e-13, most=40000):
    """K u = b for K = H + diag + J^T W J, diagonally preconditioned."""
    mul = lambda p: S["H"] @ p + S["diag"] * p + S["JT"] @ (S["w"] * (S["J"] @ p))  # noqa: E731
    x = torch.zeros_like(b)
    r = b.clone()
    z = S["pre"] * r
    p, rz = z.clone(), torch.dot(r, z)
    stop = float(rz) * tol * tol
    for it in range(most):
        q = mul(p)
        a = rz / torch.dot(p, q)
        x += a * p
        r -= a * q
        z = S["pre"] * r
        new = torch.dot(r, z)
        p = z + (new / rz) * p
        rz = new
        if it % 50 == 49 and not float(rz) > stop:
            break
    return x


def _apply(S, x):
    u = x[S["prim"]]
    y = torch.empty_like(x)
    if S["dual"] is None:
        y[S["prim"]] = S["H"] @ u + S["diag"] * u + S["JT"] @ (S["w"] * (S["J"] @ u))
    else:
        d = x[S["dual"]]
        y[S["prim"]] = S["H"] @ u + S["diag"] * u + S["JT"] @ d
        y[S["dual"]] = S["J"] @ u - d / S["w"]
    return y


def _solve64(S, b, steps=4):
    x = torch.zeros_like(b)
    r = b
    for _ in range(steps):
        f = r[S["prim"]]
        if S["dual"] is None:
            d = torch.empty_like(b)
            d[S["prim"]] = _cg(S, f, 1e-9)
        else:
            g = r[S["dual"]]
            u = _cg(S, f + S["JT"] @ (S["w"] * g), 1e-9)
            d = torch.empty_like(b)
            d[S["prim"]] = u
            d[S["dual"]] = S["w"] * (S["J"] @ u - g)
        x = x + d
        r = b - _apply(S, x)
    return x


def exact(case, seed):
    P = _plan(case)
    if P.dim * case["nrhs"] > 1_600_000:
        return None    # the iterations take too long
    v = _values(case, seed)
    S = _system(case, v)
    call = case["call"]
    if call in ("step", "adjoint"):
        X = torch.stack([_solve64(S, b) for b in v["B"]])
        out = {"X": X, "inertia": None}
        if call == "adjoint":
            G = torch.stack([_solve64(S, b) for b in X])
            prim, dual = S["prim"], S["dual"]
            out["b"] = G.t()
            hr, hc = prim[S["hr"]], prim[S["hc"]]
            both = (S["hr"] != S["hc"]).to(F64)
            out["H"] = -(G[:, hr] * X[:, hc] + both * G[:, hc] * X[:, hr]).sum(0)
            out["Sigma"] = -(G[:, prim] * X[:, prim]).sum(0)
            jr, jc = S["jr"], S["jc"]
            dsum = lambda t, o: [float(t[:, a:b].sum()) for a, b in zip(o[:-1], o[1:])]  # noqa: E731
            gd = dsum(-(G[:, prim] * X[:, prim]), P.noff)
            if dual is not None:
                out["J"] = -(G[:, dual[jr]] * X[:, prim[jc]] + G[:, prim[jc]] * X[:, dual[jr]]).sum(0)
                gr = dsum(-(G[:, dual] * X[:, dual]) / S["w"] ** 2, P.moff)
            else:
                jx, jg = (torch.stack([S["J"] @ t for t in T]) for T in (X, G))
                out["J"] = -(S["w"][jr] * (jg[:, jr] * X[:, jc] + jx[:, jr] * G[:, jc])).sum(0)
                gr = dsum(-jg * jx, P.moff)
            out["scal"] = torch.tensor([t for ab in zip(gd, gr) for t in ab], dtype=F64, device="cuda")
        return out
    if call in ("separate", "solve"):
        X = torch.stack([_solve64(S, b) for b in v["B"]])
        X = X[0] if case["nrhs"] == 1 else X.t()
        return {"X": X, "inertia": None} if call == "separate" else {"X": X}
    if call == "slack":
        rho, ss, rs = v["rho"][0], v["Ss"], v["RS"]
        fin = torch.isfinite(ss)
        inv = torch.where(fin, 1.0 / (torch.where(fin, ss, 1.0) + rho), 0.0 * rs)
        X = _solve64(S, v["B"][0] + S["JT"] @ (rho * inv * rs))
        return {"X": X, "ds": inv * (rho * (S["J"] @ X) + rs), "inertia": None}
    pt, rho, mu = v["pt"], v["rho"][0], v["mu"]
    below, above = 1.0 / (pt["x"] - pt["lower"]), 1.0 / (pt["upper"] - pt["x"])
    grad = pt["grad_phi"] - mu * below + mu * above
    B = torch.empty(P.dim, dtype=F64, device="cuda")
    if P.stab:
        B[S["prim"]] = -(grad - S["JT"] @ pt["y"])
        B[S["dual"]] = -(pt["c"] - (pt["y_k"] - pt["y"]) / rho)
    else:
        B[S["prim"]] = S["JT"] @ (pt["y_k"] - rho * pt["c"]) - grad
    X = _solve64(S, B)
    dx = X[S["prim"]]
    dy = -X[S["dual"]] if P.stab else -rho * (S["J"] @ dx + pt["c"]) + pt["y_k"] - pt["y"]
    return {"B": B, "dx": dx, "dy": dy, "dr": (dy - pt["y_k"] + pt["y"]) / rho - pt["r"],
            "dz_lower": -(pt["z_lower"] * dx - mu) * below - pt["z_lower"],
            "dz_upper": (pt["z_upper"] * dx + mu) * above - pt["z_upper"], "inertia": None}
