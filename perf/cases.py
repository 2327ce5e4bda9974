"""Performance cases of the KPM library, measured through its public binding.

Every case is one call (or the short sequence of calls) that a program using the
library makes in its hot loop: a solve with its density of states, a batch of
disorder realisations, a burst of requests to the server, the spectral bounds, local
moments, and the error bars and thermodynamics worked out from per-vector moments.
Inputs are synthetic and come from the case's seed alone; the model arrays are drawn
and laid out on the GPU with torch and handed over as the library wants them (host
arrays for the operators).

A case is a dict of plain values with a "family":

  solve   kpm_moments and kpm_dos into device arrays, one handle kept.  lattice
          extents Lx, Ly, Lz (0: dimension absent); op "stencil" or "csr"; complex:
          spin-derived hoppings of the double-exchange model; W: on-site disorder
          width; dilution: share of bonds removed; nnn: next-nearest neighbours too
          (csr only); open_edge: the last dimension is not periodic.
  batch   kpm_batch_run of `count` 2D disorder realisations of uneven size.
  serve   a burst of `requests` DOS requests through a running server, results polled.
  dense   kpm_moments on a dense Hermitian (Wigner) matrix.
  bounds  kpm_bounds (Gershgorin and Lanczos) of a lattice operator.
  ldos    kpm_ldos_moments of a set of sites.
  stats   kpm_stats and kpm_thermo on a set of per-vector moments.

Solves use the padded Gershgorin enclosure for the rescaling, as the server's users do.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1105_5481_gb300 import kpm as K

DEV = "cuda"
PAD = 0.01
GOLDEN = 0x9E3779B97F4A7C15
L2_BYTES = 129e6   # vector blocks below this stay on the chip from product to product


# ---------------------------------------------------------------------------- the cases
def listed():
    return [
        # the small FP64 lattice of a parameter scan: latency and launches count
        dict(name="square_L32_fp64", family="solve", op="stencil", Lx=32, Ly=32, Lz=0, complex=False,
             W=1.0, dilution=0.0, nnn=False, open_edge=False, precision="fp64", M=256, R=8, S=1,
             K=1024),
        # the paper's evaluation: the 10x10x10 cube, 14 vectors x 128 realisations, FP64
        dict(name="cube10_S128_fp64", family="solve", op="stencil", Lx=10, Ly=10, Lz=10,
             complex=False, W=0.0, dilution=0.0, nnn=False, open_edge=False, precision="fp64", M=256,
             R=14, S=128, K=1024),
        # the mid-size spin lattice with FP32 vectors (half the moments of a full run)
        dict(name="cubic_spin_L64_fp32", family="solve", op="stencil", Lx=64, Ly=64, Lz=64,
             complex=True, W=0.0, dilution=0.0, nnn=False, open_edge=False, precision="fp32", M=512,
             R=64, S=1, K=1024),
        # the same lattice when FP64 vectors are asked for (a short run)
        dict(name="cubic_spin_L64_fp64", family="solve", op="stencil", Lx=64, Ly=64, Lz=64,
             complex=True, W=0.0, dilution=0.0, nnn=False, open_edge=False, precision="fp64", M=128,
             R=64, S=1, K=1024),
        # the largest operator: 4.1 million sites, diluted, as CSR (a short run of the
        # headline benchmark's recursion; its products do not change with M)
        dict(name="csr_spin_dilute_L160_fp32", family="solve", op="csr", Lx=160, Ly=160, Lz=160,
             complex=True, W=0.0, dilution=0.1, nnn=False, open_edge=False, precision="fp32", M=256,
             R=32, S=1, K=4096),
        # an irregular CSR with rows of up to 19 entries (next-nearest neighbours), odd extents
        dict(name="csr_nnn_61x50x73_fp32", family="solve", op="csr", Lx=61, Ly=50, Lz=73,
             complex=False, W=2.0, dilution=0.1, nnn=True, open_edge=False, precision="fp32", M=512,
             R=16, S=1, K=1024),
        # disorder average: 256 uneven 2D realisations in one batch
        dict(name="batch_2d_256", family="batch", count=256, L_lo=16, L_hi=128, M_lo=128, M_hi=2048,
             R=16, sizes=3),
        # a burst of mixed requests to the server
        dict(name="serve_burst_24", family="serve", requests=24, N_lo=1000, N_hi=300000, M_lo=256,
             M_hi=2048, sizes=5),
        # the paper's dense formulation at its largest matrix and vector count
        dict(name="dense_D4096_fp64", family="dense", D=4096, complex=False, R=1792, M=32),
        # spectral bounds of a million-site CSR before its first solve
        dict(name="bounds_csr_L100", family="bounds", op="csr", Lx=100, Ly=100, Lz=100, complex=True,
             W=0.0, dilution=0.1, nnn=False, open_edge=False, steps=30),
        # local density of states of 16 sites on a ragged lattice with one open edge
        dict(name="ldos_500x301_fp32", family="ldos", op="stencil", Lx=500, Ly=301, Lz=0,
             complex=False, W=4.0, dilution=0.0, nnn=False, open_edge=True, precision="fp32", M=512,
             sites=16),
        # error bars and thermodynamics from the per-vector moments of a solve
        dict(name="stats_64x2048_K4096", family="stats", nvec=64, M=2048, K=4096, temperatures=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["solve", "solve", "solve", "batch", "serve", "dense", "bounds", "ldos", "stats"])
    if family == "batch":
        lo = rng.randint(8, 40)
        mlo = 2 * rng.randint(32, 128)
        return dict(family="batch", count=_log_int(rng, 8, 256), L_lo=lo, L_hi=rng.randint(lo + 8, 128),
                    M_lo=mlo, M_hi=mlo + 2 * rng.randint(32, 800), R=rng.choice([4, 8, 13, 16, 24, 32]),
                    sizes=rng.randint(1, 10**6))
    if family == "serve":
        return dict(family="serve", requests=rng.randint(4, 16), N_lo=1000, N_hi=_log_int(rng, 10000, 150000),
                    M_lo=256, M_hi=_log_int(rng, 512, 1600), sizes=rng.randint(1, 10**6))
    if family == "dense":
        cplx = rng.random() < 0.25
        D = _log_int(rng, 100, 1000) if cplx else _log_int(rng, 100, 4096)
        return dict(family="dense", D=D, complex=cplx, R=rng.randint(1, 300 if cplx else 1792),
                    M=2 * rng.randint(2, 16))
    if family == "stats":
        return dict(family="stats", nvec=_log_int(rng, 2, 128), M=2 * _log_int(rng, 32, 2048),
                    K=_log_int(rng, 64, 8192), temperatures=rng.randint(1, 32))
    # the lattice families
    dims = rng.choice([2, 3])
    N = _log_int(rng, 200, 1000000 if family != "ldos" else 300000)
    side = max(4.0, N ** (1.0 / dims))
    ext = [max(3, int(round(side * rng.uniform(0.7, 1.4)))) for _ in range(dims)] + [0] * (3 - dims)
    op = rng.choice(["stencil", "csr"])
    c = dict(family=family, op=op, Lx=ext[0], Ly=ext[1], Lz=ext[2], complex=rng.random() < 0.5,
             W=rng.choice([0.0, 1.0, 4.0]), dilution=rng.choice([0.0, 0.1]) if op == "csr" else 0.0,
             nnn=op == "csr" and rng.random() < 0.4, open_edge=rng.random() < 0.3)
    if family == "bounds":
        return dict(c, steps=rng.choice([0, 10, 30, 30, 50]))
    if family == "ldos":
        return dict(c, precision=rng.choice(["fp32", "fp64"]), M=2 * _log_int(rng, 32, 256),
                    sites=rng.randint(1, 16))
    prec = rng.choice(["fp32", "fp64"])
    S = rng.choice([1, 1, 2, 16]) if N < 20000 else 1
    R = rng.choice([1, 4, 8, 14, 16, 32, 64])
    # row updates bounded so that no draw costs more than the largest listed cases
    n_sites = max(1, ext[0] * ext[1] * max(1, ext[2]))
    most = 3e9 if prec == "fp32" else 5e8
    M = min(2 * _log_int(rng, 32, 512), 2 * int(most / (n_sites * R * S)))
    return dict(c, precision=prec, M=max(8, M), R=R, S=S, K=_log_int(rng, 64, 4096))


# ------------------------------------------------------------------------ model arrays
def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _extents(case):
    return [e for e in (case["Lx"], case["Ly"], case["Lz"]) if e > 0]


class _Lattice:
    """A lattice Hamiltonian on the device: the neighbour table (idx, val: [N, W]), the
    diagonal, and what the stencil description needs (forward hoppings, mask)."""

    def __init__(self, case, seed):
        g = _generator(seed)
        self.L = L = _extents(case)
        d = len(L)
        self.periodic = [True] * d
        if case["open_edge"]:
            self.periodic[-1] = False
        n = int(np.prod(L))
        self.n = n
        self.complex = case["complex"]
        site = torch.arange(n, device=DEV)
        xs, rem = [], site
        for e in L:
            xs.append(rem % e)
            rem = rem // e
        stride = [int(np.prod(L[:k])) for k in range(d)]
        shifts = [tuple(int(k == j) for k in range(d)) for j in range(d)]
        if case["nnn"]:  # half of the diagonal neighbours; the other half are their reverses
            for i in range(d):
                for j in range(i + 1, d):
                    for s in (1, -1):
                        e = [0] * d
                        e[i], e[j] = 1, s
                        shifts.append(tuple(e))
        self.diag = (torch.rand(n, generator=g, device=DEV, dtype=torch.float64) - 0.5) * case["W"]
        self.has_diag = case["W"] != 0.0
        dt = torch.complex128 if self.complex else torch.float64
        if self.complex:
            th = torch.arccos(1 - 2 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64))
            ph = 2 * math.pi * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
            ci, si = torch.cos(th / 2), torch.sin(th / 2)
        cols, vals, keeps, self.hop = [], [], [], None
        fwd = []
        for e in shifts:
            to, back, there = torch.zeros_like(site), torch.zeros_like(site), None
            for k in range(d):
                to += ((xs[k] + e[k]) % L[k]) * stride[k]
                back += ((xs[k] - e[k]) % L[k]) * stride[k]
                if e[k] and not self.periodic[k]:
                    y = xs[k] + e[k]
                    ok = (y >= 0) & (y < L[k])
                    there = ok if there is None else there & ok
            scale = 1.0 if sum(abs(v) for v in e) == 1 else 0.3
            if self.complex:
                t = ci * ci[to] + si * si[to] * torch.polar(torch.ones_like(ph), ph[to] - ph)
                t = scale * t
            else:
                t = torch.full((n,), scale, device=DEV, dtype=dt)
            keep = torch.rand(n, generator=g, device=DEV) >= case["dilution"]
            if there is not None:
                keep &= there
            if len(fwd) < d:
                fwd.append(t)
            h = torch.where(keep, -t, torch.zeros((), device=DEV, dtype=dt))
            cols += [to, back]
            vals += [h, h[back].conj().resolve_conj()]
            keeps += [keep, keep[back]]
        self.idx, self.val, self.keep = torch.stack(cols, 1), torch.stack(vals, 1), torch.stack(keeps, 1)
        if self.complex:
            self.hop = torch.stack(fwd, 1)
        rad = self.val.abs().sum(1)
        emin, emax = float((self.diag - rad).min()), float((self.diag + rad).max())
        self.enclosure = emin, emax
        self.a, self.b = (emax - emin) / (2 - PAD), (emax + emin) / 2

    def handle(self, op):
        if op == "stencil":
            return K.kpm_create_stencil(
                len(self.L), self.L, periodic=self.periodic,
                onsite=self.diag.cpu().numpy() if self.has_diag else None,
                hop=self.hop.cpu().numpy() if self.hop is not None else None, t=1.0, complex_=self.complex)
        idx, val, keep = self.idx, self.val, self.keep
        if self.has_diag:
            me = torch.arange(self.n, device=DEV)[:, None]
            idx = torch.cat([idx, me], 1)
            val = torch.cat([val, self.diag.to(val.dtype)[:, None]], 1)
            keep = torch.cat([keep, torch.ones_like(me, dtype=torch.bool)], 1)
        order = torch.argsort(idx, dim=1, stable=True)
        idx, val, keep = (torch.gather(t, 1, order) for t in (idx, val, keep))
        rowptr = torch.zeros(self.n + 1, device=DEV, dtype=torch.int64)
        rowptr[1:] = keep.sum(1).cumsum(0)
        return K.kpm_create_csr(self.n, rowptr.cpu().numpy(), idx[keep].to(torch.int32).cpu().numpy(),
                                val[keep].cpu().numpy(), complex_=self.complex)

    def apply(self, x):
        """H x in 64 bits."""
        y = self.diag[:, None] * x
        for k in range(self.idx.shape[1]):
            y += self.val[:, k, None] * x[self.idx[:, k]]
        return y


def _batch_shapes(case):
    """Sizes of a batch: they belong to the case; the seed draws the disorder and the vectors."""
    r = np.random.default_rng(case["sizes"])
    n = case["count"]
    L = r.integers(case["L_lo"], case["L_hi"] + 1, n)
    M = case["M_lo"] + 2 * r.integers(0, (case["M_hi"] - case["M_lo"]) // 2 + 1, n)
    return L, M, 4.0 * r.random(n)


def _batch_instances(case, seed):
    L, M, W = _batch_shapes(case)
    vs = 7919 * int(seed) + np.arange(case["count"])
    out = []
    for k in range(case["count"]):
        c = dict(Lx=int(L[k]), Ly=int(L[k]), Lz=0, complex=False, W=float(W[k]), dilution=0.0, nnn=False,
                 open_edge=False)
        out.append((_Lattice(c, 1000003 * int(seed) + k), int(M[k]), int(vs[k])))
    return out


def _requests(case, seed):
    r = np.random.default_rng(case["sizes"])
    out = []
    for k in range(case["requests"]):
        dims = 2 if r.random() < 0.5 else 3
        n = math.exp(r.uniform(math.log(case["N_lo"]), math.log(case["N_hi"])))
        side = max(4, int(round(n ** (1.0 / dims))))
        c = dict(Lx=side, Ly=side, Lz=side if dims == 3 else 0, complex=bool(r.random() < 0.5), W=0.0,
                 dilution=0.0, nnn=False, open_edge=False)
        M = int(math.exp(r.uniform(math.log(case["M_lo"]), math.log(case["M_hi"])))) // 2 * 2
        out.append((c, 5003 * int(seed) + k, M, int(r.choice([8, 16, 32, 64])), 7000 * int(seed) + k))
    return out


SERVE_K = 1024


def _wigner(case, seed):
    D, g = case["D"], _generator(seed)
    h = (2 * torch.rand(D, D, generator=g, device=DEV, dtype=torch.float64) - 1) / math.sqrt(D)
    if case["complex"]:
        im = (2 * torch.rand(D, D, generator=g, device=DEV, dtype=torch.float64) - 1) / math.sqrt(D)
        h = torch.complex(h, im)
    u = torch.triu(h, 1)
    return u + u.mH + torch.diag(torch.diagonal(h).real).to(h.dtype)


def _wigner_scale(case):
    # the semicircle's edge is 2 sigma sqrt(D), sigma^2 = 1/(3D) (2/(3D) when complex), padded
    # by what the edge of a small matrix fluctuates
    edge = 2 * math.sqrt((2 if case["complex"] else 1) / 3.0)
    return edge * (1.1 + 3.0 / case["D"] ** (2.0 / 3.0))


def _pv(case, seed):
    """Per-vector moments like a solve's: a smooth decaying mean and a spread of 1/sqrt(N)."""
    g = _generator(seed)
    n = torch.arange(case["M"], device=DEV, dtype=torch.float64)
    mean = torch.cos(0.9 * n) * torch.exp(-n / 40.0)
    pv = mean + 1e-3 * torch.randn(case["nvec"], case["M"], generator=g, device=DEV, dtype=torch.float64)
    pv[:, 0] = 1.0
    return pv, 4.2, 0.1


def _betas(case):
    return np.geomspace(0.5, 200.0, case["temperatures"])


# ------------------------------------------------------------------------------- prepare
def prepare(case, seed):
    f = case["family"]
    s = dict(case=case, seed=int(seed))
    if f in ("solve", "ldos", "bounds"):
        lat = _Lattice(case, seed)
        s.update(h=lat.handle(case["op"]), a=lat.a, b=lat.b)
        if f == "solve":
            s.update(mu=torch.empty(case["M"], device=DEV, dtype=torch.float64),
                     E=torch.empty(case["K"], device=DEV, dtype=torch.float64),
                     rho=torch.empty(case["K"], device=DEV, dtype=torch.float64))
        if f == "ldos":
            s.update(sites=np.random.default_rng(seed).integers(0, lat.n, case["sites"]),
                     mu=torch.empty(case["sites"], case["M"], device=DEV, dtype=torch.float64))
    elif f == "batch":
        inst = _batch_instances(case, seed)
        hs = [lat.handle("stencil") for lat, _, _ in inst]
        Ms = [M for _, M, _ in inst]
        bt = K.kpm_batch_create(hs, Ms, case["R"], [lat.a for lat, _, _ in inst],
                                [lat.b for lat, _, _ in inst], [v for _, _, v in inst])
        s.update(batch=bt, mu=torch.empty(sum(Ms), device=DEV, dtype=torch.float64))
    elif f == "serve":
        reqs = []
        for c, ls, M, R, vs in _requests(case, seed):
            lat = _Lattice(c, ls)
            reqs.append((lat.handle("stencil"), M, R, lat.a, lat.b, vs))
        s.update(server=K.kpm_server_create(8 << 30), reqs=reqs)
    elif f == "dense":
        s.update(h=K.kpm_create_dense(_wigner(case, seed).cpu().numpy()), a=_wigner_scale(case),
                 mu=torch.empty(case["M"], device=DEV, dtype=torch.float64))
    else:
        s["pv"], s["a"], s["b"] = _pv(case, seed)
    return s


# ----------------------------------------------------------------------------------- run
def run(s):
    c = s["case"]
    f = c["family"]
    if f == "solve":
        K.kpm_moments(s["h"], c["M"], c["R"], s["a"], s["b"], seed=s["seed"], S=c["S"],
                      precision=c["precision"], out=s["mu"])
        K.kpm_dos(s["mu"], s["a"], s["b"], c["K"], E=s["E"], rho=s["rho"])
        return dict(mu=s["mu"], E=s["E"], rho=s["rho"])
    if f == "ldos":
        return K.kpm_ldos_moments(s["h"], s["sites"], c["M"], s["a"], s["b"], precision=c["precision"],
                                  out=s["mu"])
    if f == "bounds":
        return list(K.kpm_bounds(s["h"], c["steps"], PAD, seed=s["seed"]))
    if f == "batch":
        return K.kpm_batch_run(s["batch"], out=s["mu"])
    if f == "serve":
        ids = [K.kpm_server_submit(s["server"], h, M, R, a, b, seed=v, precision="fp32", K=SERVE_K)
               for h, M, R, a, b, v in s["reqs"]]
        out = []
        for i in ids:
            K.kpm_server_wait(s["server"], i)
            mu, _, rho, _ = K.kpm_server_poll(s["server"], i)
            out.append([mu, rho])
        return out
    if f == "dense":
        return K.kpm_moments(s["h"], c["M"], c["R"], s["a"], 0.0, seed=s["seed"], precision="fp64",
                             out=s["mu"])
    mean, err, E, rho, rho_err = K.kpm_stats(s["pv"], s["a"], s["b"], c["K"])
    return [mean, err, E, rho, rho_err, K.kpm_thermo(mean, s["a"], s["b"], c["K"], _betas(c), mu_c=0.3)]


# ---------------------------------------------------------------------------------- work
def _lattice_entries(case):
    d = len(_extents(case))
    w = 2 * d + (2 * d * (d - 1) if case["nnn"] else 0)
    return (1.0 - case["dilution"]) * w + (1 if case["W"] else 0)


def _solve_work(n, entries, cplx, prec, R, M, op_bytes, out_bytes):
    """One read of the operator and one write of the results; vector blocks that do not fit on
    the chip are also read twice and written once by every product, with the operator's
    values beside them.  Flops: the row's products, the recursion and the two dots."""
    sv = (8 if prec == "fp64" else 4) * (2 if cplx else 1)
    block = n * R * sv
    byts = op_bytes + out_bytes
    if 2 * block > L2_BYTES:
        byts += (M // 2) * (3 * block + op_bytes)
    per = (8 * entries + 12) if cplx else (2 * entries + 6)
    return dict(bytes=float(byts), flops=float(n * R * (M // 2) * per))


def _op_bytes(case, n, prec):
    v = (8 if prec == "fp64" else 4) * (2 if case["complex"] else 1)
    if case["op"] == "csr":
        return n * _lattice_entries(case) * (v + 4) + 8 * (n + 1)
    return n * ((len(_extents(case)) * v if case["complex"] else 0) + (v if case["W"] else 0))


def work(case):
    f = case["family"]
    if f in ("solve", "ldos", "bounds"):
        n = int(np.prod(_extents(case)))
        e = _lattice_entries(case)
        if f == "bounds":
            k = case["steps"]
            per = (8 * e if case["complex"] else 2 * e) + 10
            fl = n * (k * per + 2 * k * k * (4 if case["complex"] else 1)) + n * 2 * e
            vec = n * 8 * (2 if case["complex"] else 1)
            return dict(bytes=float(_op_bytes(case, n, "fp64") + (k * vec if k * vec > L2_BYTES else 0)),
                        flops=float(fl))
        prec = case["precision"]
        R, out = (case["R"] * case["S"], 8 * (case["M"] + 2 * case["K"])) if f == "solve" else (
            case["sites"], 8 * case["M"] * case["sites"])
        return _solve_work(n, e, case["complex"], prec, R, case["M"],
                           _op_bytes(case, n, prec), out)
    if f == "batch":
        L, M, _ = _batch_shapes(case)
        return dict(bytes=float((4 * L ** 2 + 8 * M).sum()),
                    flops=float((L ** 2 * (M // 2)).sum() * case["R"] * 16))
    if f == "serve":
        byts = flops = 0.0
        for c, _, M, R, _ in _requests(case, 0):
            n = int(np.prod(_extents(c)))
            d = len(_extents(c))
            w = _solve_work(n, 2 * d, c["complex"], "fp32", R, M, n * d * 8 if c["complex"] else 0,
                            8 * (M + SERVE_K))
            byts, flops = byts + w["bytes"], flops + w["flops"]
        return dict(bytes=byts, flops=flops)
    if f == "dense":
        m = 4 if case["complex"] else 1
        return dict(bytes=float(8 * m * case["D"] ** 2 / (2 if case["complex"] else 1) + 8 * case["M"]),
                    flops=float(2.0 * m * case["D"] ** 2 * case["R"] * (case["M"] // 2)))
    # a fast cosine transform per vector; the mean's DOS once more for the integrals
    k2 = max(case["K"], 2)
    return dict(bytes=float(8 * (case["nvec"] * case["M"] + 2 * case["M"] + 3 * case["K"])),
                flops=float(2.5 * (case["nvec"] + 1) * k2 * math.log2(k2) + 4 * case["nvec"] * case["M"]))


# --------------------------------------------------------------------------------- exact
def _splitmix(z):
    """SplitMix64 on int64 tensors (wrapping arithmetic)."""
    def sr(v, k):
        return (v >> k) & ((1 << (64 - k)) - 1)

    def sgn(u):
        return u - (1 << 64) if u >= 1 << 63 else u

    z = z + sgn(GOLDEN)
    z = (z ^ sr(z, 30)) * sgn(0xBF58476D1CE4E5B9)
    z = (z ^ sr(z, 27)) * sgn(0x94D049BB133111EB)
    return z ^ sr(z, 31)


def _u64(seed, stream, counter):
    key = (seed & ((1 << 64) - 1)) ^ ((GOLDEN * (1 + stream)) & ((1 << 64) - 1))
    return _splitmix(counter + (key - (1 << 64) if key >= 1 << 63 else key))


def _random_block(seed, n, R, S, cplx):
    """[n, S R] start vectors: counter (s R + r) n + i of stream 0."""
    c = torch.arange(S * R, device=DEV)[None, :] * n + torch.arange(n, device=DEV)[:, None]
    z = _u64(seed, 0, c)
    if cplx:
        ph = 2 * math.pi * (((z >> 11) & ((1 << 53) - 1)).double() * 2.0 ** -53)
        return torch.polar(torch.ones_like(ph), ph)
    return torch.where(z < 0, -1.0, 1.0).double()


def _moments(apply, v0, a, b, M):
    """Per-column moments [R, M] by the doubling form in 64 bits (columns scaled to norm^2 = n)."""
    n = v0.shape[0]
    mu = torch.empty(v0.shape[1], M, device=DEV, dtype=torch.float64)

    def dot(x, y):
        return (torch.view_as_real(x) * torch.view_as_real(y)).sum((0, 2)) if x.is_complex() else (x * y).sum(0)

    w, v = None, v0
    for k in range(M // 2):
        y = (apply(v) - b * v) / a
        y = y if w is None else y.mul_(2).sub_(w)
        A, B = dot(v, v) / n, dot(y, v) / n
        mu[:, 2 * k] = A if k == 0 else 2 * A - mu[:, 0]
        mu[:, 2 * k + 1] = B if k == 0 else 2 * B - mu[:, 1]
        w, v = v, y
    return mu


def _dos(mu, a, b, Kn):
    """Jackson-damped series on the Chebyshev nodes: (E, rho), rho [.., K]."""
    M = mu.shape[-1]
    n = torch.arange(M, device=DEV, dtype=torch.float64)
    t = math.pi / (M + 1)
    g = ((M - n + 1) * torch.cos(t * n) + torch.sin(t * n) / math.tan(t)) / (M + 1)
    c = mu * g
    c = torch.cat([c[..., :1], 2 * c[..., 1:]], -1)
    k = torch.arange(Kn, device=DEV)
    out = torch.zeros(*mu.shape[:-1], Kn, device=DEV, dtype=torch.float64)
    step = 2048
    for m0 in range(0, M, step):  # angles reduced in whole numbers first
        m = torch.arange(m0, min(M, m0 + step), device=DEV)
        ang = ((2 * k[None, :] + 1) * m[:, None]) % (4 * Kn)
        out += c[..., m0:m0 + step] @ torch.cos(ang.double() * (math.pi / (2 * Kn)))
    th = (k.double() + 0.5) * math.pi / Kn
    return a * torch.cos(th) + b, out / (math.pi * a * torch.sin(th))


def _exact_bounds(case, seed):
    lat = _Lattice(case, seed)
    n, k = lat.n, case["steps"]
    emin, emax = lat.enclosure
    if k:
        q = torch.where(_u64(seed, 6, torch.arange(n, device=DEV)) < 0, -1.0, 1.0).double()
        q = (q / math.sqrt(n)).to(lat.val.dtype)
        Q, al, be = [q], [], []
        for j in range(min(k, n)):
            y = lat.apply(Q[j][:, None])[:, 0]
            al.append(float(torch.vdot(Q[j], y).real))
            V = torch.stack(Q, 1)
            for _ in range(2):
                y = y - V @ (V.mH @ y)
            be.append(float(torch.linalg.vector_norm(y)))
            if be[-1] <= 1e-12 * max(1.0, abs(al[-1])):
                break
            Q.append(y / be[-1])
        m = len(al)
        t, u = np.linalg.eigh(np.diag(al) + np.diag(be[:m - 1], 1) + np.diag(be[:m - 1], -1))
        emax = min(emax, t[-1] + be[-1] * abs(u[-1, -1]))
        emin = max(emin, t[0] - be[-1] * abs(u[-1, 0]))
    return [float(emin), float(emax), float((emax - emin) / (2 - PAD)), float((emax + emin) / 2)]


def _exact_batch(case, seed):
    """All instances as one block-diagonal operator; the dots summed per instance."""
    inst = _batch_instances(case, seed)
    R, count = case["R"], case["count"]
    start = np.concatenate([[0], np.cumsum([lat.n for lat, _, _ in inst])])
    idx = torch.cat([lat.idx + int(start[k]) for k, (lat, _, _) in enumerate(inst)])
    val = torch.cat([lat.val / lat.a for lat, _, _ in inst])
    diag = torch.cat([(lat.diag - lat.b) / lat.a for lat, _, _ in inst])
    own = torch.repeat_interleave(torch.arange(count, device=DEV),
                                  torch.tensor([lat.n for lat, _, _ in inst], device=DEV))
    size = torch.tensor([lat.n * R for lat, _, _ in inst], device=DEV, dtype=torch.float64)
    v = torch.cat([_random_block(s, lat.n, R, 1, False) for lat, _, s in inst])
    Ms = [M for _, M, _ in inst]
    mu = torch.empty(count, max(Ms), device=DEV, dtype=torch.float64)
    w = None

    def dot(x, y):
        return torch.zeros(count, device=DEV, dtype=torch.float64).index_add_(0, own, (x * y).sum(1)) / size

    for k in range(max(Ms) // 2):
        y = diag[:, None] * v
        for j in range(idx.shape[1]):
            y.addcmul_(val[:, j, None], v[idx[:, j]])
        y = y if w is None else y.mul_(2).sub_(w)
        A, B = dot(v, v), dot(y, v)
        mu[:, 2 * k] = A if k == 0 else 2 * A - mu[:, 0]
        mu[:, 2 * k + 1] = B if k == 0 else 2 * B - mu[:, 1]
        w, v = v, y
    return torch.cat([mu[i, :Ms[i]] for i in range(count)])


def _exact_thermo(mu, a, b, case, mu_c):
    E, rho = _dos(mu, a, b, case["K"])
    th = (torch.arange(case["K"], device=DEV).double() + 0.5) * math.pi / case["K"]
    w = rho * a * math.pi * torch.sin(th) / case["K"]
    out = []
    for beta in _betas(case):
        x = float(beta) * (E - mu_c)
        f = torch.sigmoid(-x)
        ent = torch.sigmoid(-x.abs()) * x.abs() + torch.log1p(torch.exp(-x.abs()))
        out.append(torch.stack([(w * f).sum(), (w * E * f).sum(), (w * ent).sum(),
                                (w * x * x * f * torch.sigmoid(x)).sum()]))
    return torch.stack(out)


def exact(case, seed):
    f = case["family"]
    if f == "bounds":
        return _exact_bounds(case, seed)
    if f == "batch":
        return _exact_batch(case, seed)
    if f == "solve":
        lat = _Lattice(case, seed)
        v0 = _random_block(seed, lat.n, case["R"], case["S"], lat.complex)
        mu = _moments(lat.apply, v0, lat.a, lat.b, case["M"]).mean(0)
        E, rho = _dos(mu, lat.a, lat.b, case["K"])
        return dict(mu=mu, E=E, rho=rho)
    if f == "ldos":
        lat = _Lattice(case, seed)
        sites = np.random.default_rng(seed).integers(0, lat.n, case["sites"])
        v0 = torch.zeros(lat.n, case["sites"], device=DEV, dtype=lat.val.dtype)
        v0[torch.from_numpy(sites).to(DEV), torch.arange(case["sites"], device=DEV)] = math.sqrt(lat.n)
        return _moments(lat.apply, v0, lat.a, lat.b, case["M"])
    if f == "serve":
        out = []
        for c, ls, M, R, vs in _requests(case, seed):
            lat = _Lattice(c, ls)
            mu = _moments(lat.apply, _random_block(vs, lat.n, R, 1, lat.complex), lat.a, lat.b, M).mean(0)
            out.append([mu, _dos(mu, lat.a, lat.b, SERVE_K)[1]])
        return out
    if f == "dense":
        h = _wigner(case, seed)
        v0 = _random_block(seed, case["D"], case["R"], 1, case["complex"])
        return _moments(lambda x: h @ x, v0, _wigner_scale(case), 0.0, case["M"]).mean(0)
    pv, a, b = _pv(case, seed)
    nv = case["nvec"]
    mean = pv.mean(0)
    E, rho = _dos(pv, a, b, case["K"])
    rm = rho.mean(0)

    def err(x, m):
        return torch.sqrt(((x - m) ** 2).sum(0) / (max(nv - 1, 1) * nv))

    return [mean, err(pv, mean), E, rm, err(rho, rm), _exact_thermo(mean, a, b, case, 0.3)]
