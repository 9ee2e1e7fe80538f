"""What the performance of this package is measured on: calls of its public entry points
(``paper_1705_10087_gb300.capi``) over the sizes it is used at.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges, ``prepare`` makes
what a program has in hand before the call (inputs, lambda, a handle or a server), ``run``
makes one pass, ``work`` says what the path cannot do without and ``exact`` gives the result
in float64 by plain torch (for solves: the minimiser of Eq. sparse_code).

Inputs follow the law of ``paper_1705_10087_gb300.synth`` (unit-norm Gaussian atoms,
Bernoulli-Gaussian activations, white noise; lambda = 0.1 lambda_max), drawn on the GPU.
Sizes and tolerances are those of its workloads, of the tests, or odd neighbours of them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1705_10087_gb300 import capi

DEV = "cuda"
# the four resident dictionaries (K, L, P) of the request stream
STREAM_DICTS = ((25, 64, 1), (25, 128, 7), (64, 64, 7), (64, 128, 1))


def listed():
    return [
        # the short single-channel signal cut into 10 segments: launches and latency
        {"name": "short", "kind": "solve", "K": 5, "P": 1, "L": 16, "T": 2000, "M": 10, "u": 0,
         "rho": 0.01, "sigma": 0.01, "tol": 1e-6, "host": False},
        # the long multichannel signal in the configuration the benchmark times
        {"name": "long", "kind": "solve", "K": 25, "P": 7, "L": 64, "T": 200_000, "M": 1024,
         "u": 24, "rho": 0.005, "sigma": 0.1, "tol": 1e-6, "host": False},
        # a very long single-channel recording, default segments of 2L-2 columns
        {"name": "verylong", "kind": "solve", "K": 25, "P": 1, "L": 200, "T": 5_000_000, "M": 0,
         "u": 24, "rho": 0.002, "sigma": 0.1, "tol": 1e-6, "host": False},
        # sizes of no special form, arrays in host memory, all defaults
        {"name": "odd_host", "kind": "solve", "K": 18, "P": 5, "L": 51, "T": 60_013, "M": 0,
         "u": 0, "rho": 0.005, "sigma": 0.1, "tol": 1e-6, "host": True},
        # a regularisation path: three lambdas, each solve continuing from the last Z
        {"name": "path", "kind": "path", "K": 25, "P": 7, "L": 64, "T": 100_003, "rho": 0.005,
         "sigma": 0.1, "tol": 1e-6},
        # signals of uneven length against one dictionary in one solve
        {"name": "batch", "kind": "batch", "K": 25, "P": 7, "L": 64, "n": 24, "T_min": 10_000,
         "T_max": 500_000, "lengths": 1, "u": 24, "rho": 0.005, "sigma": 0.1, "tol": 1e-6},
        # requests for four resident dictionaries through the serving engine
        {"name": "stream", "kind": "stream", "n": 16, "T_min": 5_000, "T_max": 100_000,
         "lengths": 1, "rho": 0.005, "sigma": 0.1, "tol": 1e-3},
        # a gray image with 8 x 8 atoms, automatic tiles
        {"name": "image", "kind": "image", "K": 8, "P": 1, "h": 8, "w": 8, "H": 512, "W": 512,
         "rho": 0.005, "sigma": 0.1, "tol": 1e-6},
        # a small colour image: launches and latency of the 2-D path
        {"name": "image_rgb", "kind": "image", "K": 6, "P": 3, "h": 6, "w": 6, "H": 96, "W": 80,
         "rho": 0.01, "sigma": 0.1, "tol": 1e-6},
        # only the start of a solve: beta0 = D~ * X and lambda_max, 64 atoms, a ragged length
        {"name": "beta0", "kind": "beta0", "K": 64, "P": 7, "L": 64, "T": 300_007, "rho": 0.005,
         "sigma": 0.1},
        # the checks of a given Z: objective and optimality report
        {"name": "report", "kind": "report", "K": 25, "P": 7, "L": 64, "T": 200_000,
         "rho": 0.005, "sigma": 0.1},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["path", "batch", "stream", "image", "image", "beta0",
                                       "report"])
    sig = {"rho": 0.005, "sigma": 0.1}
    if kind == "stream":
        return {"kind": kind, "n": rng.randint(4, 16), "T_min": 5_000,
                "T_max": _log_int(rng, 20_000, 100_000), "lengths": rng.randrange(1 << 20), **sig,
                "tol": 1e-3}
    if kind == "batch":
        return {"kind": kind, "K": 25, "P": 7, "L": 64, "n": rng.randint(2, 24),
                "T_min": rng.randint(500, 10_000), "T_max": _log_int(rng, 20_000, 500_000),
                "lengths": rng.randrange(1 << 20), "u": rng.choice([0, 24]), **sig, "tol": 1e-6}
    if kind == "image":
        K, P, h, w = rng.choice([(8, 1, 8, 8), (6, 3, 6, 6), (3, 2, 5, 4),
                                 (rng.randint(2, 12), 2, rng.randint(3, 9), rng.randint(3, 9))])
        return {"kind": kind, "K": K, "P": P, "h": h, "w": w, "H": _log_int(rng, 40, 512),
                "W": _log_int(rng, 40, 512), "rho": 0.005, "sigma": 0.1, "tol": 1e-6}
    # a dictionary of the workloads and tests, or one of no special form
    K, P, L = rng.choice([(5, 1, 16), (25, 7, 64), (18, 5, 51), (64, 7, 64), (25, 1, 200), None,
                          None]) or (rng.randint(4, 40), rng.randint(4, 7), rng.randint(8, 128))
    sig["rho"] = 0.002 if L > 128 else 0.01 if L == 16 else 0.005
    top = {"solve": 2_000_000, "path": 150_000, "beta0": 1_000_000, "report": 500_000}[kind]
    T = _log_int(rng, max(1000, 8 * L), min(top, 60_000_000 // K))
    case = {"kind": kind, "K": K, "P": P, "L": L, "T": T, **sig}
    if kind == "solve":
        most = max(1, T // (2 * L))
        case["M"] = rng.choice([0, 0, _log_int(rng, max(1, most // 4), most)])
        case["u"] = rng.choice([0, 24, 24])
        case["host"] = rng.random() < 0.25
    if kind in ("solve", "path"):
        case["tol"] = 1e-6
    return case


# ---------------------------------------------------------------- inputs

def _sizes(c):
    """Atom extents and signal extents of a case: ([L], [T]) or ([h, w], [H, W])."""
    return ([c["h"], c["w"]], [c["H"], c["W"]]) if c["kind"] == "image" else ([c["L"]], [c["T"]])


def _dictionary(g, K, P, ext):
    D = torch.randn((K, P, *ext), generator=g, device=DEV, dtype=torch.float64)
    return (D / D.flatten(1).norm(dim=1).view(K, *[1] * (D.ndim - 1))).float()


def _signal(g, D, ext, rho, sigma):
    """X [P, *ext] = sum_k Z_k * D_k + noise, and the Z [K, *valid] it was made from.
    The sum runs lag by lag as K x P products (the same bits on every run)."""
    K, P = D.shape[:2]
    lags = D.shape[2:]
    valid = [t - l + 1 for t, l in zip(ext, lags)]
    Z = torch.randn((K, *valid), generator=g, device=DEV)
    Z.mul_(torch.rand((K, *valid), generator=g, device=DEV) < rho)
    X = torch.randn((P, *ext), generator=g, device=DEV).mul_(sigma)
    Zf = Z.view(K, -1)
    for lag in np.ndindex(*lags):
        at = (slice(None), *(slice(o, o + v) for o, v in zip(lag, valid)))
        X[at] += (D[(slice(None), slice(None), *lag)].t().contiguous() @ Zf).view(P, *valid)
    return X, Z


def _smooth(n):
    """The least 2^a 3^b 5^c >= n (a transform length)."""
    best = 1 << max(0, (n - 1).bit_length())
    p5 = 1
    while p5 < best:
        p35 = p5
        while p35 < best:
            q = -(-n // p35)
            best = min(best, p35 << max(0, (q - 1).bit_length()))
            p35 *= 3
        p5 *= 5
    return best


class _Ops:
    """Convolution and correlation with D in float64, by transforms."""

    def __init__(self, D, ext):
        self.ext = ext
        self.lags = list(D.shape[2:])
        self.valid = [t - l + 1 for t, l in zip(ext, self.lags)]
        self.n = [_smooth(t) for t in ext]
        self.dims = tuple(range(-len(ext), 0))
        self.Df = torch.fft.rfftn(D.double(), s=self.n, dim=self.dims)

    def conv(self, Z):
        """sum_k Z_k * D_k  [P, *ext]"""
        Zf = torch.fft.rfftn(Z, s=self.n, dim=self.dims)
        out = torch.stack([(Zf * self.Df[:, p]).sum(0) for p in range(self.Df.shape[1])])
        out = torch.fft.irfftn(out, s=self.n, dim=self.dims)
        return out[(slice(None), *(slice(0, t) for t in self.ext))]

    def corr(self, R):
        """D~ * R  [K, *valid]"""
        Rf = torch.fft.rfftn(R, s=self.n, dim=self.dims)
        out = torch.stack([(self.Df[k].conj() * Rf).sum(0) for k in range(self.Df.shape[0])])
        out = torch.fft.irfftn(out, s=self.n, dim=self.dims)
        return out[(slice(None), *(slice(0, v) for v in self.valid))].contiguous()

    def lipschitz(self):
        """An upper bound of the largest eigenvalue of D~ * D (row sums of its symbol)."""
        K, P = self.Df.shape[:2]
        rows = []
        for p in range(P):
            rows.append(sum(((self.Df[:, p] * self.Df[:, q].conj()).sum(0)).abs()
                            for q in range(P)))
        return float(torch.stack(rows).max())


def _lambda_max(D, X):
    """max |D~ * X|, one atom at a time (long recordings)."""
    top = 0.0
    for k in range(D.shape[0]):
        top = max(top, float(_Ops(D[k:k + 1], list(X.shape[1:])).corr(X.double()).abs().max()))
    return top


def _make(c, seed):
    """D, X, the generating Z and lambda of a case with one signal or image."""
    lags, ext = _sizes(c)
    g = torch.Generator(DEV).manual_seed(int(seed))
    D = _dictionary(g, c["K"], c["P"], lags)
    X, Z = _signal(g, D, ext, c["rho"], c["sigma"])
    return D, X, Z, float(np.float32(0.1 * _lambda_max(D, X)))


class _Handle:
    """A solver handle that goes with the state that holds it."""

    def __init__(self, D, opts):
        self.opts = opts
        self.h = capi.csc_setup(D, opts)

    def __del__(self):
        capi.csc_destroy(self.h)


class _Server:
    def __init__(self, budget):
        self.s = capi.csc_server_create(hbm_budget_bytes=budget)

    def __del__(self):
        capi.csc_server_destroy(self.s)


def _lengths(c):
    """Signal lengths of a batch (uniform) or of a stream's requests (log-uniform), by the case."""
    r = np.random.RandomState(c["lengths"])
    if c["kind"] == "batch":
        return r.randint(c["T_min"], c["T_max"] + 1, c["n"]).astype(np.int64)
    return np.exp(r.uniform(np.log(c["T_min"]), np.log(c["T_max"]), c["n"])).astype(np.int64)


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "stream":
        g = torch.Generator(DEV).manual_seed(int(seed))
        srv = _Server(8 << 30)
        Ds = [_dictionary(g, K, P, [L]) for K, L, P in STREAM_DICTS]
        ids = [capi.csc_server_add_dictionary(srv.s, D) for D in Ds]
        req = []
        for i, T in enumerate(_lengths(c)):
            j = i % len(Ds)  # the dictionaries in turn
            X, Z = _signal(g, Ds[j], [int(T)], c["rho"], c["sigma"])
            req.append((ids[j], X.cpu().numpy(), torch.empty_like(Z)))
        return {"case": c, "server": srv, "requests": req}
    if kind == "batch":
        g = torch.Generator(DEV).manual_seed(int(seed))
        T = _lengths(c)
        D = _dictionary(g, c["K"], c["P"], [c["L"]])
        Xs = [_signal(g, D, [int(t)], c["rho"], c["sigma"])[0] for t in T]
        lam = [float(np.float32(0.1 * _lambda_max(D, X))) for X in Xs]
        Z = torch.empty((c["K"], int(T.sum()) - c["L"] + 1), device=DEV)
        return {"case": c, "D": D, "X": torch.cat(Xs, 1), "T": T, "lam": lam, "Z": Z,
                "handle": _Handle(D, capi.make_opts(updates_per_visit=c["u"]))}
    D, X, Z, lam = _make(c, seed)
    s = {"case": c, "D": D, "X": X, "lam": lam}
    if kind == "image":
        s["Z"] = torch.empty_like(Z)
    elif kind == "solve":
        s["Z"] = torch.empty_like(Z)
        if c["host"]:
            for k in ("D", "X", "Z"):
                s[k] = s[k].cpu().pin_memory()
        s["handle"] = _Handle(s["D"], capi.make_opts(segments=c["M"], updates_per_visit=c["u"]))
    elif kind == "path":
        s["lams"] = [float(np.float32(f * lam)) for f in (5.0, 2.0, 1.0)]
        s["Zs"] = [torch.empty_like(Z) for _ in s["lams"]]
        s["handle"] = _Handle(D, capi.make_opts())
    elif kind == "beta0":
        s["beta"] = torch.empty_like(Z)
        s["handle"] = _Handle(D, capi.make_opts())
    else:  # report: a handle with the signal on it, and the Z to check
        s["Z"] = Z
        s["handle"] = _Handle(D, capi.make_opts())
        capi.csc_init(s["handle"].h, X, lam)
    return s


# ---------------------------------------------------------------- one pass

def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "image":
        _, E, _ = capi.csc2d_solve(s["D"], s["X"], s["lam"], c["tol"], Z_out=s["Z"])
        return {"Z": s["Z"], "E": E}
    if kind == "stream":
        srv = s["server"].s
        at = {}
        for i, (d, X, _) in enumerate(s["requests"]):
            at[capi.csc_server_submit(srv, d, X, -0.1, c["tol"])] = i
        E = [0.0] * len(at)
        while at:
            _, _, ndone = capi.csc_server_step(srv)
            if not ndone:
                continue
            for rid in capi.csc_server_completed(srv):
                i = at.pop(rid)
                E[i] = capi.csc_server_fetch(srv, rid, s["requests"][i][2])["objective"]
        return {"Z": [q[2] for q in s["requests"]], "E": E}
    h = s["handle"].h
    if kind == "report":
        return {"E": capi.csc_objective(h, s["Z"]), **capi.csc_kkt(h, s["Z"])}
    capi.csc_setup(s["D"], s["handle"].opts, handle=h)
    if kind == "beta0":
        capi.csc_init(h, s["X"], s["lam"])
        capi.csc_get_beta(h, s["beta"])
        return {"beta": s["beta"], "lambda_max": capi.csc_lambda_max(h)}
    if kind == "batch":
        capi.csc_init_batch(h, s["X"], s["T"], s["lam"])
        capi.csc_solve(h, c["tol"], 1 << 40, s["Z"])
        return {"Z": s["Z"], "E": capi.csc_get_objectives(h, len(s["T"]))}
    if kind == "path":
        E = []
        for i, (lam, Z) in enumerate(zip(s["lams"], s["Zs"])):
            if i == 0:
                capi.csc_init(h, s["X"], lam)
            else:
                capi.csc_set_lambda(h, [lam])
            E.append(capi.csc_solve(h, c["tol"], 1 << 40, Z)[1])
        return {"Z": s["Zs"], "E": E}
    capi.csc_init(h, s["X"], s["lam"])
    _, E, _ = capi.csc_solve(h, c["tol"], 1 << 40, s["Z"])
    return {"Z": s["Z"], "E": E}


# ---------------------------------------------------------------- floors

def work(case):
    """Bytes: D, X in, Z (or beta) out.  Flops: beta0 (2 K P L per column) and, for a solve, one
    window update per activation the signal was made from (2 K (2L-1), 2-D alike)."""
    c, kind = case, case["kind"]
    if kind == "stream":
        parts = [(*(STREAM_DICTS[i % len(STREAM_DICTS)]), int(T))
                 for i, T in enumerate(_lengths(c))]
        parts = [(K, P, [L], [T]) for K, L, P, T in parts]
    elif kind == "batch":
        parts = [(c["K"], c["P"], [c["L"]], [int(T)]) for T in _lengths(c)]
    else:
        parts = [(c["K"], c["P"], *_sizes(c))]
    nbytes = flops = 0.0
    for K, P, lags, ext in parts:
        out = K * math.prod(t - l + 1 for t, l in zip(ext, lags))
        window = math.prod(2 * l - 1 for l in lags)
        nbytes += 4.0 * (K * P * math.prod(lags) + P * math.prod(ext) + out)
        beta0 = 2.0 * out * P * math.prod(lags)
        updates = 2.0 * c["rho"] * out * K * window
        solves = 3 if kind == "path" else 0 if kind in ("beta0", "report") else 1
        flops += ((updates if kind == "report" else beta0) + solves * updates)
        nbytes += 4.0 * (2 * out if kind == "path" else 0)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- float64 results

def _soft(U, lam):
    return U.sign() * (U.abs() - lam).clamp_min(0)


def _minimiser(ops, X, lam, Z, rounds=40):
    """The minimiser of Eq. sparse_code in float64, started at Z: accelerated proximal
    gradient steps (Beck & Teboulle 2009, with restarts), then conjugate gradients on the
    support it found, until signs and |D~ * residual| <= lambda hold.  None if they do not."""
    lip = ops.lipschitz()
    B = ops.corr(X)
    steps = 400
    for _ in range(rounds):
        Y, t = Z, 1.0
        for _ in range(steps):
            Zn = _soft(Y + (B - ops.corr(ops.conv(Y))) / lip, lam / lip)
            if float(((Y - Zn) * (Zn - Z)).sum()) > 0:
                t = 1.0  # restart (O'Donoghue & Candes 2015)
            tn = 0.5 * (1 + math.sqrt(1 + 4 * t * t))
            Y, Z, t = Zn + (t - 1) / tn * (Zn - Z), Zn, tn
        steps = 100
        S, sign = Z != 0, Z.sign()
        if not bool(S.any()):
            return Z if float(B.abs().max()) <= lam * (1 + 1e-12) else None
        # (D~ * D) z = B - lambda sign on the support
        r = torch.where(S, B - lam * sign - ops.corr(ops.conv(Z)), 0.0)
        p, rr, first = r, float((r * r).sum()), float((B * B * S).sum())
        for _ in range(400):
            if rr <= 1e-28 * first:
                break
            q = torch.where(S, ops.corr(ops.conv(p)), 0.0)
            a = rr / float((p * q).sum())
            Z, r = Z + a * p, r - a * q
            rn = float((r * r).sum())
            p, rr = r + (rn / rr) * p, rn
        keep = torch.where(Z.sign() == sign, Z, 0.0)
        G = B - ops.corr(ops.conv(keep))
        if bool((keep == Z).all()) and float((G.abs() * ~S).max()) <= lam * (1 + 1e-9):
            return Z
        Z = keep
    return None


def _objective(ops, X, Z, lam):
    return float(0.5 * (X - ops.conv(Z)).square().sum() + lam * Z.abs().sum())


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("batch", "stream"):
        return None
    if kind in ("solve", "path", "image"):
        # (about 20 seconds of transforms at most)
        if c["K"] * math.prod(_sizes(c)[1]) > (3 if kind == "path" else 6) * 1_000_000:
            return None
    D, X, Z, lam = _make(c, seed)
    ops = _Ops(D, list(X.shape[1:]))
    X = X.double()
    if kind == "beta0":
        beta = torch.cat([_Ops(D[k:k + 1], list(X.shape[1:])).corr(X) for k in range(c["K"])])
        return {"beta": beta, "lambda_max": float(beta.abs().max())}
    Z = Z.double()
    if kind == "report":
        norms = D.double().flatten(1).square().sum(1).view(-1, 1)
        r = ops.corr(X - ops.conv(Z))
        gap = (Z - _soft(r + norms * Z, lam) / norms).abs()
        return {"E": _objective(ops, X, Z, lam),
                "zero_excess": max(0.0, float((r.abs() * (Z == 0)).max()) - lam),
                "nonzero_gap": float((gap * (Z != 0)).max()), "max_delta_z": float(gap.max())}
    if kind == "path":
        Zs, E = [], []
        for lam_i in (float(np.float32(f * lam)) for f in (5.0, 2.0, 1.0)):
            Z = _minimiser(ops, X, lam_i, Z)
            if Z is None:
                return None
            Zs.append(Z)
            E.append(_objective(ops, X, Z, lam_i))
        return {"Z": Zs, "E": E}
    Z = _minimiser(ops, X, lam, Z)
    return None if Z is None else {"Z": Z, "E": _objective(ops, X, Z, lam)}
