"""The work that a program using this library has it do, as cases that can be timed and checked.

Every case goes through the Python binding's public calls.  ``listed()`` gives the fixed
cases, ``draw(rng)`` one more of the same ranges, ``prepare`` the inputs and the plan that a
program holds before the call, ``run`` one pass, ``work`` the bytes and operations the pass
cannot do without, and ``exact`` the same results in plain FP64 torch (no library code).

Kinds of case:
  apply     exx_apply, the ACE case (Psi_in = Psi_occ, occupied orbitals leading)
  separate  exx_apply on input functions other than the occupied orbitals (a block of trial
            vectors or a k-space block of an eigensolver)
  batched   exx_apply_batched: many small independent systems in one call
  build     ace_build: M, its Cholesky factor, xi
  ace       ace_apply: the compressed operator on a block of vectors
  step      exx_ace_step_host: one whole ACE outer step from and to host memory
  bloch     exx_apply_complex: one k - q term of a k-point calculation
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2501_16572_gb300 as exx

HSE_OMEGA = 0.106
FD_ORDER = 12
PREC = {"fp64": exx.EXX_PREC_FP64, "bf16x7": exx.EXX_PREC_BF16X7}
BATCH_SYSTEMS = 12


# ---- the cases --------------------------------------------------------------------------
def _grid(name, kind, n, h, bc, n_occ, n_in, prec="bf16x7"):
    c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "h": h, "bc": bc, "n_occ": n_occ, "n_in": n_in,
         "prec": prec}
    return {"name": name, **c} if name else c


def listed():
    return [
        # an isolated molecule on a 24^3 grid, every orbital occupied: the smallest call, two
        # batches of launches (the repository's smallest configuration)
        _grid("molecule24", "apply", (24, 24, 24), 0.3, "ddd", 16, 16),
        # a periodic crystal cell, screened exchange, 128 orbitals: the ordinary call
        _grid("crystal48", "apply", (48, 48, 48), 0.25, "ppp", 128, 128),
        # the mixed-boundary slab of the benchmark with a tenth of its orbitals, 78% occupied
        _grid("slab72", "apply", (72, 72, 144), 0.2, "ppd", 75, 96),
        # the paper's large slab grid: odd slices too wide for resident matrices
        _grid("slab117", "apply", (117, 117, 119), 0.2, "ppd", 31, 40),
        # trial vectors of an eigensolver on an odd-sized wire grid: no symmetry to use, no
        # 16-byte aligned rows
        _grid("wire_trial", "separate", (45, 39, 53), 0.3, "ddp", 40, 30),
        # a set of small molecules and cells of different sizes in one call
        {"name": "molecules12", "kind": "batched", "specs": 4, "prec": "bf16x7"},
        # the double-precision reference path, a plan's default precision
        _grid("double28", "apply", (28, 30, 33), 0.3, "dpd", 24, 32, "fp64"),
        # construction of the compressed operator on the benchmark's slab, half its orbitals
        _grid("build_slab", "build", (72, 72, 144), 0.2, "ppd", 512, 512),
        # the compressed operator on all bands of the slab, as a polynomial-filtered
        # eigensolver applies it many times in each outer step
        _grid("ace_slab", "ace", (72, 72, 144), 0.2, "ppd", 512, 512),
        # the compressed operator on a block of 16 vectors of the crystal cell
        _grid("ace_block16", "ace", (48, 48, 48), 0.25, "ppp", 128, 16),
        # a whole outer step from pinned host memory: apply, energy, build, copies
        _grid("step_host48", "step", (48, 48, 48), 0.25, "ppp", 100, 128),
        # one k - q term on a small cell with Bloch phases (FP64 only)
        _grid("bloch24", "bloch", (24, 20, 22), 0.3, "ppd", 12, 12),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "separate", "build", "ace", "ace", "step", "batched", "bloch"])
    if kind == "batched":
        return {"kind": "batched", "specs": rng.randrange(5, 1 << 20), "prec": "bf16x7"}
    while True:
        prec = "bf16x7"
        if kind == "bloch":
            n = tuple(rng.randint(12, 32) for _ in range(3))
            n_occ, n_in = rng.randint(2, 24), rng.randint(2, 24)
            prec = "fp64"
        elif kind in ("build", "ace"):
            n = tuple(rng.randint(20, 80) for _ in range(3))
            n_occ = _log(rng, 8, 512)
            n_in = n_occ if kind == "build" else _log(rng, 1, 512)
        else:
            n = (_log(rng, 16, 120), _log(rng, 16, 120), _log(rng, 16, 150))
            n_occ = _log(rng, 4, 160)
            n_in = _log(rng, 2, 160) if kind == "separate" else n_occ + rng.choice([0, int(0.28 * n_occ)])
            if kind == "apply" and rng.random() < 0.2:
                prec = "fp64"
        bc = "".join(rng.choice("dp") for _ in range(3))
        h = rng.choice([0.2, 0.25, 0.3])
        c = _grid(None, kind, n, h, bc, n_occ, n_in, prec)
        # more orbitals than a quarter of the grid's smooth functions cannot be independent
        if max(n_occ, n_in) * 40 > n[0] * n[1] * n[2]:
            continue
        w = work(c)
        if kind in ("build", "ace"):
            if w["flops"] > work(listed()[7])["flops"]:
                continue
        elif w["flops"] * (100 if prec == "fp64" else 1) > work(listed()[2])["flops"]:
            continue
        return c


def _specs(seed):
    """The systems of a batched case: axes U{20..64}, a boundary per axis, 8 to 160 orbitals."""
    rng = random.Random(int(seed))
    out = []
    for i in range(BATCH_SYSTEMS):
        n = tuple(rng.randint(20, 64) for _ in range(3))
        bc = "ddd" if i == 0 else "ppp" if i == 1 else "".join(rng.choice("dp") for _ in range(3))
        n_orb = rng.randint(8, 160)
        n_orb = min(n_orb, max(8, n[0] * n[1] * n[2] // 200))
        out.append(_grid(None, "apply", n, 0.3, bc, n_orb, n_orb))
    return out


# ---- inputs -----------------------------------------------------------------------------
def _N(c):
    return c["nx"] * c["ny"] * c["nz"]


def _kernel(c):
    # the unscreened kernel needs one axis that is not periodic
    slab = c["bc"] in ("ppp", "ppd")
    return (exx.EXX_KERNEL_ERFC, HSE_OMEGA) if slab else (exx.EXX_KERNEL_COULOMB, 0.0)


def _bcs(c):
    return [exx.EXX_BC_PERIODIC if b == "p" else exx.EXX_BC_DIRICHLET for b in c["bc"]]


def _orbitals(c, n_orb, seed):
    """Smooth localized functions, (n_orb, N): 6 Gaussians each and, with a periodic axis, 4
    plane waves under an envelope along the Dirichlet axes; slabs leave the top 30% empty."""
    rng = np.random.Generator(np.random.PCG64(seed))
    n, h = (c["nx"], c["ny"], c["nz"]), c["h"]
    per = [b == "p" for b in c["bc"]]
    L = [v * h for v in n]
    top = [0.7 if c["bc"] == "ppd" and d == 2 else 1.0 for d in range(3)]
    dev = torch.device("cuda")
    x = [torch.arange(v, dtype=torch.float64, device=dev) * h for v in n]
    fac = [[], [], []]
    amp = torch.from_numpy(rng.normal(0.0, 1.0, (n_orb, 6))).to(dev)
    sig = torch.from_numpy(rng.uniform(0.6, 1.5, (n_orb, 6, 1))).to(dev)
    for d in range(3):
        cen = torch.from_numpy(rng.uniform(0.2, 0.8, (n_orb, 6, 1)) * L[d] * top[d]).to(dev)
        g = sum(torch.exp(-(x[d] - cen + s * L[d]) ** 2 / (2 * sig ** 2)) for s in ((-1, 0, 1) if per[d] else (0,)))
        fac[d].append(g * amp[:, :, None] if d == 2 else g)
    if any(per):
        b = torch.from_numpy(rng.normal(0.0, 0.3, (n_orb, 4, 1))).to(dev)
        th = torch.from_numpy(rng.uniform(0.0, 2 * np.pi, (n_orb, 4, 1))).to(dev)
        ph, env = [], []
        for d in range(3):
            k = torch.from_numpy(rng.integers(0, 4, (n_orb, 4, 1)).astype(np.float64)).to(dev)
            ph.append(2 * np.pi / L[d] * k * x[d] if per[d] else 0 * k * x[d])
            env.append(torch.exp(-(x[d] - 0.5 * top[d] * L[d]) ** 2 / (2 * (0.15 * L[d]) ** 2)) if not per[d] else 1.0 + 0 * x[d])
        ph[2] = ph[2] + th
        # cos(a + b + c) as four products of one-dimensional factors
        for fx, fy, fz, s in ((torch.cos, torch.cos, torch.cos, 1), (torch.sin, torch.sin, torch.cos, -1),
                              (torch.sin, torch.cos, torch.sin, -1), (torch.cos, torch.sin, torch.sin, -1)):
            fac[0].append(fx(ph[0]) * env[0])
            fac[1].append(fy(ph[1]) * env[1])
            fac[2].append(fz(ph[2]) * env[2] * b * s)
    fx, fy, fz = (torch.cat(f, 1) for f in fac)
    out = torch.empty((n_orb, n[2], n[1] * n[0]), dtype=torch.float64, device=dev)
    for a in range(0, n_orb, 32):
        e = min(n_orb, a + 32)
        yx = (fy[a:e, :, :, None] * fx[a:e, :, None, :]).reshape(e - a, -1, n[1] * n[0])
        torch.bmm(fz[a:e].transpose(1, 2), yx, out=out[a:e])
    return out.reshape(n_orb, -1)


def _orthonormal(raw, dV):
    """Rows made orthonormal in the dV metric (Householder QR, or Cholesky QR for large blocks)."""
    if raw.shape[0] * raw.shape[1] <= 1 << 26:
        q, r = torch.linalg.qr(raw.mH.contiguous())
        s = torch.sign(torch.diagonal(r).real)
        return ((q * s) / math.sqrt(dV)).mH.resolve_conj().contiguous()
    g = raw @ raw.mH * dV
    # a small shift keeps the factor real when functions nearly depend on each other
    g.diagonal().add_(1e-10 * g.diagonal().mean())
    low = torch.linalg.cholesky(g)
    return torch.linalg.solve_triangular(low, raw, upper=False).contiguous()


def _occ(n_occ, n_in):
    """Fermi-Dirac occupations in [0, 2], the level at 97% of the occupied orbitals."""
    j = torch.arange(n_occ, dtype=torch.float64, device="cuda")
    f = 2.0 / (1.0 + torch.exp(0.002 * (j - int(0.97 * n_occ)) / 0.01))
    return torch.full_like(f, 2.0) if n_occ == n_in else f


def _inputs(c, seed):
    """The tensors of a case, the same for prepare and exact."""
    N, dV = _N(c), c["h"] ** 3
    kind, no, ni = c["kind"], c["n_occ"], c["n_in"]
    if kind == "bloch":
        z = [torch.complex(_orbitals(c, k, seed + s), _orbitals(c, k, seed + s + 1)) for k, s in ((no, 1000), (ni, 2000))]
        th = np.random.Generator(np.random.PCG64(seed + 3000)).uniform(-2.5, 2.5, 3)
        return {"psi": _orthonormal(z[0], dV), "phi": _orthonormal(z[1], dV), "f": _occ(no, ni), "theta": [float(t) for t in th]}
    if kind in ("apply", "step"):
        return {"psi": _orthonormal(_orbitals(c, ni, seed), dV), "f": _occ(no, ni)}
    if kind == "separate":
        return {"psi": _orthonormal(_orbitals(c, no, seed), dV), "phi": _orbitals(c, ni, seed + 1000), "f": _occ(no, no + 1)}
    psi = _orthonormal(_orbitals(c, no, seed), dV)
    # W = -v(r) psi with a positive smooth v: -Psi^T W is symmetric positive definite, as the
    # exchange matrix is
    v = 0.2 + _orbitals(c, 1, seed + 500)[0] ** 2
    if kind == "build":
        return {"psi": psi, "W": -v * psi}
    return {"xi": torch.sqrt(v) * psi, "phi": _orbitals(c, ni, seed + 1000)}


def _plan(c, theta=None):
    n, (k, om) = (c["nx"], c["ny"], c["nz"]), _kernel(c)
    if theta is not None:
        return exx.Plan.bloch(n, c["h"], _bcs(c), theta, FD_ORDER, k, om)
    p = exx.Plan(n, c["h"], _bcs(c), FD_ORDER, k, om)
    p.set_precision(PREC[c["prec"]])
    return p


def prepare(case, seed):
    if case["kind"] == "batched":
        subs = _specs(case["specs"])
        ins = [_inputs(s, seed * 64 + i) for i, s in enumerate(subs)]
        return {"kind": "batched", "plans": [_plan(s) for s in subs],
                "args": [(t["psi"], t["f"], t["psi"], torch.empty_like(t["psi"])) for t in ins],
                "stream": torch.cuda.Stream()}
    s = _inputs(case, seed)
    s["kind"], s["n_occ"] = case["kind"], case["n_occ"]
    s["plan"] = _plan(case, s.get("theta"))
    if case["kind"] == "step":
        s["psi"] = s["psi"].cpu().pin_memory()
        s["f"] = s["f"].cpu().pin_memory()
        s["xi"] = torch.empty_like(s["psi"]).pin_memory()
    elif case["kind"] == "build":
        s["xi"] = torch.empty_like(s["psi"])
        s["M"] = torch.empty((case["n_occ"], case["n_occ"]), dtype=torch.float64, device="cuda")
    else:
        s["out"] = torch.empty_like(s["phi"] if "phi" in s else s["psi"])
    return s


def run(state):
    kind = state["kind"]
    if kind == "batched":
        # the graph path wants a stream of its own
        st = state["stream"]
        st.wait_stream(torch.cuda.current_stream())
        out = exx.exx_apply_batched(state["plans"], state["args"], st)
        torch.cuda.current_stream().wait_stream(st)
        return out
    p = state["plan"]
    if kind == "apply":
        return p.apply(state["psi"][:state["n_occ"]], state["f"], state["psi"], state["out"])
    if kind == "separate":
        return p.apply(state["psi"], state["f"], state["phi"], state["out"])
    if kind == "build":
        return {"xi": p.ace_build(state["psi"], state["W"], state["xi"], state["M"]), "M": state["M"]}
    if kind == "ace":
        return p.ace_apply(state["xi"], state["phi"], state["out"])
    if kind == "step":
        e = p.ace_step_host(state["psi"], state["n_occ"], state["f"], state["xi"])
        return {"xi": state["xi"], "E": e}
    return p.apply_complex(state["psi"], state["f"], state["phi"], state["out"])


def _pairs(c):
    """Poisson problems that have to be solved: phi_mn = phi_nm among the occupied orbitals."""
    no, ni = c["n_occ"], c["n_in"]
    return no * (no + 1) // 2 + no * (ni - no) if c["kind"] in ("apply", "step") else no * ni


def work(case):
    if case["kind"] == "batched":
        ws = [work(s) for s in _specs(case["specs"])]
        return {"bytes": sum(w["bytes"] for w in ws), "flops": sum(w["flops"] for w in ws)}
    N, no, ni, kind = _N(case), case["n_occ"], case["n_in"], case["kind"]
    if kind == "build":   # M, its Cholesky factor and inverse, xi
        return {"bytes": 8.0 * (3 * N * no + no * no), "flops": 2.0 * N * no * no * 1.5 + no ** 3 * 2 / 3}
    if kind == "ace":
        return {"bytes": 8.0 * N * (no + 2 * ni), "flops": 4.0 * N * no * ni}
    el, mul = (16.0, 4.0) if kind == "bloch" else (8.0, 1.0)
    nin = no + ni if kind in ("bloch", "separate") else ni
    # six mode products a pair (2 n flops a point each), the pair density and the sums
    flops = mul * _pairs(case) * N * (4.0 * (case["nx"] + case["ny"] + case["nz"]) + 6)
    if kind == "step":
        flops += 2.0 * N * ni * ni * 1.5
    return {"bytes": el * N * (nin + ni), "flops": flops}


# ---- the same results in plain FP64 torch -------------------------------------------------
def _weights():
    """Centred second-derivative weights of order 12 (w[0] .. w[6])."""
    p = FD_ORDER // 2
    w = [0.0] * (p + 1)
    for k in range(1, p + 1):
        w[k] = 2.0 * (-1.0) ** (k + 1) / k ** 2 * math.factorial(p) ** 2 / (math.factorial(p - k) * math.factorial(p + k))
    w[0] = -2.0 * sum(w[1:])
    return w


def _axis(n, h, periodic, theta=None):
    w = _weights()
    D = np.zeros((n, n), dtype=complex)
    for i in range(n):
        for k in range(-len(w) + 1, len(w)):
            j = i + k
            ph = 1.0
            if periodic:
                ph = np.exp(1j * (theta or 0.0) * (j // n))
                j %= n
            if 0 <= j < n:
                D[i, j] += w[abs(k)] * ph
    D /= h * h
    lam, V = np.linalg.eigh(D if theta is not None and periodic else D.real)
    return lam, V


def _solver(c, theta=None):
    """rho (..., nz, ny, nx) -> f(L) rho."""
    k, om = _kernel(c)
    n = (c["nx"], c["ny"], c["nz"])
    ax = [_axis(n[d], c["h"], c["bc"][d] == "p", None if theta is None else theta[d]) for d in range(3)]
    lam = ax[0][0][None, None, :] + ax[1][0][None, :, None] + ax[2][0][:, None, None]
    if k == exx.EXX_KERNEL_COULOMB:
        F = -4 * np.pi / lam
    else:
        a = -lam
        tiny = np.abs(a) < 1e-13
        safe = np.where(tiny, 1.0, a)
        F = np.where(tiny, np.pi / om ** 2, -4 * np.pi * np.expm1(-safe / (4 * om ** 2)) / safe)
    dt = torch.float64 if theta is None else torch.complex128
    F = torch.from_numpy(F).to("cuda")
    X, Y, Z = (torch.from_numpy(np.ascontiguousarray(a[1])).to("cuda", dt) for a in ax)

    def axis_z(M, t):
        return torch.matmul(M, t.reshape(t.shape[0], n[2], -1)).reshape(t.shape)

    def solve(rho):
        t = torch.matmul(rho, X.conj())
        t = torch.matmul(Y.mH, t)
        t = axis_z(Z.mH, t) * F
        t = axis_z(Z, t)
        t = torch.matmul(Y, t)
        return torch.matmul(t, X.mT)

    return solve


def _exchange(c, psi, f, phi, aliased, theta=None):
    """-sum_m f_m psi_m f(L)(conj(psi_m) phi_n); aliased: phi[:n_occ] = psi, each pair once."""
    solve = _solver(c, theta)
    shape = (-1, c["nz"], c["ny"], c["nx"])
    no, ni, N = f.numel(), phi.shape[0], _N(c)
    out = torch.zeros_like(phi)
    step = max(1, (1 << 26) // N)
    for m in range(no):
        for a in range(m if aliased else 0, ni, step):
            e = min(ni, a + step)
            V = solve((psi[m].conj() * phi[a:e]).reshape(shape)).reshape(e - a, N)
            out[a:e] -= f[m] * psi[m] * V
            if aliased:
                lo, hi = max(a, m + 1), min(e, no)
                if hi > lo:
                    out[m] -= torch.einsum("n,nr,nr->r", f[lo:hi], psi[lo:hi], V[lo - a:hi - a])
    return out


def _xi(psi, W, dV):
    M = psi @ W.mT * dV
    low = torch.linalg.cholesky(-0.5 * (M + M.mT))
    return M, torch.linalg.solve_triangular(low, W, upper=False)


def exact(case, seed):
    if case["kind"] == "batched":
        outs = []
        for i, s in enumerate(_specs(case["specs"])):
            t = _inputs(s, seed * 64 + i)
            outs.append(_exchange(s, t["psi"], t["f"], t["psi"], True))
        return outs
    if work(case)["flops"] > 1.5e13:
        return None
    t, dV = _inputs(case, seed), case["h"] ** 3
    kind, no = case["kind"], case["n_occ"]
    if kind == "apply":
        return _exchange(case, t["psi"][:no], t["f"], t["psi"], True)
    if kind == "separate":
        return _exchange(case, t["psi"], t["f"], t["phi"], False)
    if kind == "build":
        M, xi = _xi(t["psi"], t["W"], dV)
        return {"xi": xi, "M": M.mT.contiguous()}   # the library's M is column-major
    if kind == "ace":
        return -dV * ((t["phi"] @ t["xi"].mT) @ t["xi"])
    if kind == "step":
        W = _exchange(case, t["psi"][:no], t["f"], t["psi"], True)
        E = 0.25 * dV * torch.einsum("n,nr,nr->", t["f"], t["psi"][:no], W[:no])
        return {"xi": _xi(t["psi"], W, dV)[1], "E": float(E)}
    return _exchange(case, t["psi"], t["f"], t["phi"], False, t["theta"])
