"""Performance cases of the eigensolver: what its users have it compute, through hq.Solver and hq.Batch.

Each case is a dict of plain values.  ``prepare`` makes what a user's program
holds before the call (a context with its potential set, device blocks),
``run`` makes one pass through the public calls, ``work`` states what a pass
cannot do without and ``exact`` gives the outputs in plain FP64 torch.

Inputs.  The potentials are the repository's family, the harmonic oscillator
with eight Gaussian wells, drawn from the seed; the adjoint and the refinement
need converged or nearly converged eigenvectors, which an off-centre
anisotropic oscillator gives in closed form (sums of 1-D eigenvalues).  Blocks
are iterates as they stand early in a run: oscillator eigenfunctions, slightly
mixed, scaled off orthonormality, with 2% of white noise; the warm start of a
step is the oscillator's inverse of that block.

Iteration counts of the inner solver are not among the outputs: they depend on
a stopping test met at a threshold.  Scalars and blocks of a mixed-precision
context are returned in its working precision (FP32).
"""
import math

import numpy as np
import torch

from paper_2605_25149_gb300 import hq

LO, HI = -6.0, 6.0


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # The smallest real problem, the 16^3 oscillator: launches and latency, four steps per call.
        dict(name="step_small", kind="step", m=16, N=8, prec="fp64", mg_fp32=1, nu=2, rtol=1e-10, tau=0.5, steps=4),
        # The headline step: FP64 PCG with the FP32 preconditioner and three sweeps per level.
        dict(name="step_fp64", kind="step", m=64, N=64, prec="fp64", mg_fp32=1, nu=3, rtol=1e-10, tau=0.4, steps=2),
        # The largest problem of the repository: one mixed-precision step at 128^3, N = 256.
        dict(name="step_mixed_large", kind="step", m=128, N=256, prec="mixed", mg_fp32=0, nu=2, rtol=1e-6, tau=0.4, steps=1),
        # Several uneven problems advanced by one graph launch (members of the batched workload's sides and widths).
        dict(name="batch_mixed", kind="batch", members="32x16,48x32,64x64,32x128,64x16,48x64,32x64,64x32", prec="mixed", mg_fp32=0, nu=2, rtol=1e-6, tau=0.4, steps=1),
        # The inner solve by itself with the library's default options (FP64 V-cycle), at the differentiation workload's size.
        dict(name="pcg_fp64", kind="pcg", m=64, N=32, prec="fp64", mg_fp32=0, nu=2, rtol=1e-10),
        # The same in mixed precision on the largest side of the batched workload.
        dict(name="pcg_mixed", kind="pcg", m=96, N=64, prec="mixed", mg_fp32=0, nu=2, rtol=1e-6),
        # The preconditioner alone on an odd grid with an odd number of columns (no vector loads).
        dict(name="vcycle_fp64_ragged", kind="vcycle", m=47, N=33, prec="fp64", mg_fp32=0, nu=2),
        # The FP64 operator y = (H + sigma) x alone.
        dict(name="operator_fp64", kind="operator", m=64, N=64, prec="fp64", mg_fp32=0, nu=2),
        # The update U C1 + W C2 of a mixed step, the dense contraction.
        dict(name="update_mixed", kind="gemm", m=64, N=128, prec="mixed", mg_fp32=0, nu=2),
        # Reading the result: eigenvalues, Ritz vectors and residuals of an iterate.
        dict(name="eigenpairs", kind="eigenpairs", m=64, N=64, prec="fp64", mg_fp32=1, nu=2, rtol=1e-10),
        # The density gradient by adjoint solves, from converged eigenvectors.
        dict(name="adjoint", kind="adjoint", m=48, N=32, prec="fp64", mg_fp32=1, nu=2, rtol=1e-10, solve_rtol=1e-11),
        # The final FP64 refinement of a nearly converged iterate: inexact Newton rounds.
        dict(name="refine", kind="refine", m=64, N=64, prec="fp64", mg_fp32=1, nu=3, rtol=1e-10, rounds=3, solve_rtol=1e-2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sizes(rng, m_lo, m_hi, n_lo, n_hi, most):
    """A grid side and a width, odd ones among them, of at most `most` point-columns."""
    while True:
        m, N = _log_int(rng, m_lo, m_hi), _log_int(rng, n_lo, n_hi)
        if m ** 3 * N <= most:
            return m, N


def draw(rng):
    kind = rng.choice(["step", "step", "batch", "pcg", "vcycle", "operator", "gemm", "eigenpairs", "adjoint", "refine"])
    prec, mg_fp32 = rng.choice([("fp64", 0), ("fp64", 1), ("mixed", 0)])
    mixed = prec == "mixed"
    most = 4e8 if mixed else (4e7 if mg_fp32 else 2e7)
    c = dict(kind=kind, prec=prec, mg_fp32=mg_fp32, nu=rng.choice([2, 2, 3]))
    rtol = 1e-6 if mixed else 1e-10
    if kind == "step":
        m, N = _sizes(rng, 12, 128, 4, 256, most)
        c.update(m=m, N=N, rtol=rtol, tau=0.4, steps=rng.choice([1, 2]))
    elif kind == "batch":
        members = []
        for _ in range(rng.randint(2, 8)):
            members.append("%dx%d" % _sizes(rng, 12, 72, 4, 128, most / 40))
        c.update(members=",".join(members), rtol=rtol, tau=0.4, steps=1)
    elif kind == "pcg":
        m, N = _sizes(rng, 12, 128, 4, 256, most)
        c.update(m=m, N=N, rtol=rtol)
    elif kind in ("vcycle", "operator"):
        m, N = _sizes(rng, 12, 128, 1, 256, 4e8 if mixed else 1e8)
        c.update(m=m, N=N)
    elif kind == "gemm":
        m, N = _sizes(rng, 24, 128, 4, 256, 2e8 if mixed else 2e7)
        c.update(m=m, N=N)
    elif kind == "eigenpairs":
        m, N = _sizes(rng, 16, 72, 4, 72, 1e8)
        c.update(m=m, N=N, rtol=rtol)
    else:
        m, N = _sizes(rng, 20, 56, 4, 40, 5e6)
        c.update(m=m, N=N, prec="fp64", mg_fp32=1, rtol=1e-10)
        c.update(solve_rtol=1e-11) if kind == "adjoint" else c.update(rounds=3, solve_rtol=1e-2)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _nodes(m):
    h = (HI - LO) / (m + 1)
    return h, LO + h * np.arange(1, m + 1)


class Oscillator:
    """-Delta_h/2 + (1/2) sum_d w_d^2 (x_d - c_d)^2 on the grid: 1-D eigenvectors per axis, and the
    N lowest sums of 1-D eigenvalues with their (i, j, k) mode numbers."""

    def __init__(self, m, N, omega=(1.0, 1.0, 1.0), centre=(0.0, 0.0, 0.0)):
        h, t = _nodes(m)
        self.m, self.h = m, h
        self.one, self.vec = [], []
        for w, c in zip(omega, centre):
            T = np.diag(1.0 / h ** 2 + 0.5 * w * w * (t - c) ** 2)
            T += np.diag(np.full(m - 1, -0.5 / h ** 2), 1) + np.diag(np.full(m - 1, -0.5 / h ** 2), -1)
            e, v = np.linalg.eigh(T)
            self.one.append(e)
            self.vec.append(v)
        low = [e[:24] for e in self.one]   # enough modes per axis for the lowest few hundred sums
        sums = low[2][:, None, None] + low[1][None, :, None] + low[0][None, None, :]
        order = np.argsort(sums, axis=None, kind="stable")[: N + 1]
        self.kji = np.unravel_index(order[:N], sums.shape)
        self.lam = sums.reshape(-1)[order]   # N + 1 values

    def cuda(self):
        self.vec = [torch.from_numpy(v).cuda() for v in self.vec]
        x, y, z = (torch.from_numpy(e).cuda() for e in self.one)
        self.lam3 = z[:, None, None] + y[None, :, None] + x[None, None, :]
        return self

    def lowest(self):
        """The N lowest eigenvectors (n x N), <.,.>-orthonormal."""
        k, j, i = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in self.kji)
        X, Y, Z = self.vec[0][:, i], self.vec[1][:, j], self.vec[2][:, k]
        f = (Z * self.h ** -1.5)[:, None, None, :] * (Y[:, None, :] * X[None, :, :])[None]
        return f.reshape(self.m ** 3, -1)

    def to_modes(self, b, back=False):
        m, N = self.m, b.shape[1]
        b = b.reshape(m, m, m, N)
        x, y, z = (v if back else v.T for v in self.vec)
        b = torch.matmul(x, b)                                                          # x axis
        b = torch.matmul(y, b.reshape(m, m, m * N)).reshape(m, m, m, N)                 # y axis
        return torch.matmul(z, b.reshape(m, m * m * N)).reshape(m ** 3, N)              # z axis

    def inverse(self, b, shift):
        """(oscillator + shift)^-1 b; shift: a number or one per column."""
        d = self.lam3.reshape(-1, 1) + shift
        return self.to_modes(self.to_modes(b) / d, back=True)


def _wells(m, rng):
    """The oscillator with eight Gaussian wells, n values, x fastest."""
    _, t = _nodes(m)
    t = torch.from_numpy(t).cuda()
    z, y, x = torch.meshgrid(t, t, t, indexing="ij")
    V = 0.5 * (x * x + y * y + z * z)
    depth, width = rng.uniform(1.0, 5.0, 8), rng.uniform(0.5, 1.5, 8)
    centre = rng.uniform(LO, HI, (8, 3))
    for d, w, c in zip(depth, width, centre):
        V = V - d * torch.exp(-((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2) / (2.0 * w * w))
    return V.reshape(-1).contiguous()


def _gapped(m, N, rng):
    """An off-centre anisotropic oscillator whose N-th and next eigenvalues are apart."""
    while True:
        omega, centre = rng.uniform(0.85, 1.35, 3), rng.uniform(-0.3, 0.3, 3)
        o = Oscillator(m, N, omega, centre)
        if o.lam[N] - o.lam[N - 1] > 0.08 and np.diff(o.lam[:N]).min(initial=1.0) > 5e-4:
            break
    o.cuda()
    _, t = _nodes(m)
    q = [torch.from_numpy(0.5 * w * w * (t - c) ** 2).cuda() for w, c in zip(omega, centre)]
    V = q[2][:, None, None] + q[1][None, :, None] + q[0][None, None, :]
    return o, V.reshape(-1).contiguous()


def _noise(shape, gen):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)


def _iterate(o, shift, rng, gen):
    """(U, Z): an early iterate and the oscillator's inverse of its smooth part."""
    N = len(o.lam) - 1
    scale = torch.from_numpy(1.15 * (1.0 + 0.05 * rng.standard_normal(N))).cuda()
    lam = torch.from_numpy(o.lam[:N]).cuda()
    f = o.lowest()
    U = f * scale
    U += 0.1 * torch.roll(f, 1, 1)
    Z = f * (scale / (lam + shift))
    Z += 0.1 * torch.roll(f, 1, 1) / (torch.roll(lam, 1) + shift)
    n = f.shape[0]
    del f
    for a in range(0, n, 1 << 18):   # 2% of white noise
        part = U[a:a + (1 << 18)]
        part += (0.02 / (HI - LO) ** 1.5) * _noise(part.shape, gen)
    return U, Z


def _shift_of(V, m):
    """The automatic shift of the operator (documented at hq_config)."""
    h = (HI - LO) / (m + 1)
    lb = 3.0 * (2.0 / (h * h)) * math.sin(math.pi / (2.0 * (m + 1))) ** 2 + float(V.min())
    return 0.0 if lb > 0.0 else 1.0 - lb


def _inputs(case, m, N, seed):
    """The seeded inputs of one problem, as FP64 tensors, rounded to the context's precision."""
    rng, gen = np.random.default_rng(seed), torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    d = {}
    if kind in ("adjoint", "refine"):
        d["osc"], d["V"] = _gapped(m, N, rng)
        d["U"] = d["osc"].lowest()
        if kind == "adjoint":
            # the density to match: that of the eigenvectors with a smooth relative change
            k = torch.arange(m ** 3, device="cuda", dtype=torch.float64) / m ** 3
            a, b = rng.uniform(0.05, 0.2, 2)
            d["rho"] = (d["U"] ** 2).sum(1) * (1.0 + a * torch.sin(6.0 * k) + b * torch.cos(17.0 * k))
        else:
            # 1e-3 of smooth error: the oscillator's inverse of white noise
            e = d["osc"].inverse(_noise((m ** 3, N), gen), 1.0)
            d["U"] = d["U"] + 1e-3 * e / (e.square().sum(0) * d["osc"].h ** 3).sqrt()
    else:
        d["osc"] = Oscillator(m, N).cuda()
        d["V"] = _wells(m, rng)
        U, Z = _iterate(d["osc"], _shift_of(d["V"], m), rng, gen)
        if case["prec"] == "mixed":
            for a in (U, Z):
                a.copy_(a.float())
        d["U"], d["Z"] = U, Z
        if kind == "gemm":
            d["C1"] = torch.eye(N, device="cuda", dtype=torch.float64) + 0.1 * _noise((N, N), gen) / math.sqrt(N)
            d["C2"] = 0.4 * _noise((N, N), gen) / math.sqrt(N)
    return d


def _members(case):
    if case["kind"] != "batch":
        return [(case["m"], case["N"])]
    return [tuple(int(v) for v in s.split("x")) for s in case["members"].split(",")]


def _solver(case, m, N):
    kw = dict(precision=case["prec"], mg_fp32=case["mg_fp32"], mg_nu1=case["nu"], mg_nu2=case["nu"])
    if "rtol" in case:
        kw.update(cg_rtol=case["rtol"])
    if "tau" in case:
        kw.update(tau=case["tau"])
    return hq.Solver(m, N, **kw)


def prepare(case, seed):
    problems = []
    for q, (m, N) in enumerate(_members(case)):
        d = _inputs(case, m, N, seed + 1000 * q)
        s = _solver(case, m, N)
        s.set_potential(d["V"])
        keep = {"s": s}
        kind = case["kind"]
        if kind in ("step", "batch", "eigenpairs"):
            keep.update(U=d["U"], Z=d["Z"])
        elif kind in ("adjoint", "refine"):
            keep.update(U=d["U"])
            if kind == "adjoint":
                s.set_state_device(d["U"], 0)
                keep.update(rho=d["rho"].cpu().numpy())
        else:
            keep.update(U=d["U"].to(s.dtype))
            if kind in ("gemm", "pcg"):
                keep.update(Z=d["Z"].to(s.dtype))
            if kind == "gemm":
                keep.update(C1=d["C1"], C2=d["C2"])
        problems.append(keep)
        del d
    state = {"case": case, "problems": problems}
    if case["kind"] == "batch":
        state["batch"] = hq.Batch([p["s"] for p in problems])
    return state


def run(state):
    case, problems = state["case"], state["problems"]
    kind, p = case["kind"], problems[0]
    s = p["s"]
    if kind == "step":
        s.set_state_device(p["U"], 0, p["Z"])
        g = s.step(case["steps"])
        return {"U": s.state_device()[0].to(s.dtype), "g": g}
    if kind == "batch":
        for q in problems:
            q["s"].set_state_device(q["U"], 0, q["Z"])
        g, _ = state["batch"].step(case["steps"])
        return {"U": [q["s"].state_device()[0].to(q["s"].dtype) for q in problems], "g": g.astype(np.float32)}
    if kind == "pcg":
        return s.block_pcg(p["U"], X0=p["Z"], rtol=case["rtol"])[0]
    if kind == "vcycle":
        return s.mg_vcycle(p["U"])
    if kind == "operator":
        return s.apply_operator(p["U"])
    if kind == "gemm":
        return s.block_gemm(p["U"], p["C1"], p["Z"], p["C2"])
    if kind == "eigenpairs":
        s.set_state_device(p["U"], 0, p["Z"])
        e = s.eigenpairs(vectors=True, vectors_on_device=True)
        paper = e["lam_paper"] if case["prec"] == "fp64" else e["lam_paper"].astype(np.float32)
        return {"lam_rr": e["lam_rr"], "vectors": e["vectors"], "residuals": e["residuals"], "lam_paper": paper}
    if kind == "adjoint":
        dV, loss, _ = s.grad_density(rho_target=p["rho"], rtol=case["solve_rtol"])
        return {"dV": dV, "loss": loss}
    s.set_state_device(p["U"], 0)
    s.refine(rounds=case["rounds"], rtol=case["solve_rtol"])
    return s.state_device()[0]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
# Block-PCG iterations of one inner solve from a warm start at these tolerances (nominal), and of one
# adjoint / refinement solve.
_ITERS = {"fp64": 7, "mixed": 4}
_ADJOINT_ITERS, _REFINE_ITERS = 60, 20


def _solve_flops(pc, nu, iters):
    """PCG: operator 8, updates and dots 12, V-cycle (10 per sweep, 9 residual, 24 transfers) on all levels 8/7."""
    return pc * iters * (20 + (10 * (2 * nu - 1) + 33) * 8.0 / 7.0)


def work(case):
    w = 4 if case["prec"] == "mixed" else 8
    nbytes = flops = 0.0
    kind, nu = case["kind"], case["nu"]
    for m, N in _members(case):
        n, pc = float(m) ** 3, float(m) ** 3 * N
        if kind in ("step", "batch"):
            dense = 2 * pc * (0.5 * 4 * N + N + 2 * N + N + N)
            flops += case["steps"] * (2 * _solve_flops(pc, nu, _ITERS[case["prec"]]) + dense)
            nbytes += 3 * 8 * pc + 8 * n
        elif kind == "pcg":
            flops += _solve_flops(pc, nu, _ITERS[case["prec"]])
            nbytes += 3 * w * pc + 8 * n
        elif kind == "vcycle":
            flops += _solve_flops(pc, nu, 1) - 20 * pc
            nbytes += 2 * w * pc + 8 * n
        elif kind == "operator":
            flops += 8 * pc
            nbytes += 2 * w * pc + 8 * n
        elif kind == "gemm":
            flops += 4 * pc * N
            nbytes += 3 * w * pc + 16.0 * N * N
        elif kind == "eigenpairs":
            flops += _solve_flops(pc, nu, _ITERS[case["prec"]]) + 8 * pc + 2 * pc * (2 * N + N + 0.5 * N + N + 2 * N)
            nbytes += 3 * 8 * pc + 8 * n
        else:
            its = _ADJOINT_ITERS if kind == "adjoint" else case["rounds"] * _REFINE_ITERS
            flops += _solve_flops(pc, nu, its) + 2 * its * 4 * pc * N
            nbytes += 2 * 8 * pc + 8 * n
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the outputs in FP64, without the library
# ---------------------------------------------------------------------------
def _operator(x, V, sigma, m):
    h = (HI - LO) / (m + 1)
    c = 0.5 / (h * h)
    x4 = x.reshape(m, m, m, -1)
    y = (6.0 * c + sigma + V).reshape(m, m, m, 1) * x4
    for d in range(3):
        y.narrow(d, 1, m - 1).sub_(x4.narrow(d, 0, m - 1), alpha=c)
        y.narrow(d, 0, m - 1).sub_(x4.narrow(d, 1, m - 1), alpha=c)
    return y.reshape(x.shape)


def _solve(osc, V, sigma, b, x):
    """(H + sigma)^-1 b by conjugate gradients preconditioned with the oscillator's inverse."""
    m = osc.m
    shift = max(sigma, 0.0)
    bn = b.square().sum(0).sqrt()
    for _ in range(2):   # restarted once from the true residual
        r = b - _operator(x, V, sigma, m)
        z = osc.inverse(r, shift)
        p, rz = z.clone(), (r * z).sum(0)
        for _ in range(200):
            if bool((r.square().sum(0).sqrt() <= 1e-14 * bn).all()):
                break
            q = _operator(p, V, sigma, m)
            a = rz / (p * q).sum(0).clamp_min(1e-300)
            x = x + a * p
            r = r - a * q
            z = osc.inverse(r, shift)
            new = (r * z).sum(0)
            p = z + (new / rz.clamp_min(1e-300)) * p
            rz = new
    return x


def _transfer(mf, mc):
    """1-D interpolation (mf x mc) from mc to mf nodes of the same interval, zero at its ends."""
    f = np.arange(1, mf + 1)[:, None] * (mc + 1.0) / (mf + 1.0)
    return torch.from_numpy(np.maximum(0.0, 1.0 - np.abs(f - np.arange(1, mc + 1)[None, :]))).cuda()


def _along_axes(T, b, m_in):
    """T applied along x, y and z of an m_in^3 block."""
    m, N = T.shape[0], b.shape[1]
    b = torch.matmul(T, b.reshape(m_in, m_in, m_in, N))
    b = torch.matmul(T, b.reshape(m_in, m_in, m * N))
    return torch.matmul(T, b.reshape(m_in, m * m * N)).reshape(m ** 3, N)


def _vcycle(r, V, sigma, m, nu, omega=0.8):
    h = (HI - LO) / (m + 1)
    if m <= 4:
        A = _operator(torch.eye(m ** 3, device="cuda", dtype=torch.float64), V, sigma, m)
        return torch.linalg.solve(A, r)
    w = (omega / (3.0 / (h * h) + V + sigma))[:, None]
    z = w * r
    for _ in range(nu - 1):
        z = z + w * (r - _operator(z, V, sigma, m))
    mc = m // 2
    P = _transfer(m, mc)
    rc = ((mc + 1.0) / (m + 1.0)) ** 3 * _along_axes(P.T.contiguous(), r - _operator(z, V, sigma, m), m)
    z = z + _along_axes(P, _vcycle(rc, _coarse_potential(V, m, mc), sigma, mc, nu, omega), mc)
    for _ in range(nu):
        z = z + w * (r - _operator(z, V, sigma, m))
    return z


def _coarse_potential(V, m, mc):
    """V interpolated trilinearly at the mc^3 coarse nodes."""
    s = np.arange(1, mc + 1)[:, None] * (m + 1.0) / (mc + 1.0)
    T = torch.from_numpy(np.maximum(0.0, 1.0 - np.abs(s - np.arange(1, m + 1)[None, :]))).cuda()
    return _along_axes(T, V[:, None], m)[:, 0].contiguous()


def _step(osc, V, sigma, U, Z, tau):
    N, h3 = U.shape[1], osc.h ** 3
    W = _solve(osc, V, sigma, U, Z)
    S, Pwu, Q = h3 * U.T @ U, h3 * W.T @ U, h3 * W.T @ W
    g = (W - U @ Pwu).square().sum().mul(h3).sqrt()
    eye = torch.eye(N, device="cuda", dtype=torch.float64)
    M = torch.cat([torch.cat([eye - 0.5 * tau * Pwu.T, 0.5 * tau * S], 1), torch.cat([-0.5 * tau * Q, eye + 0.5 * tau * Pwu], 1)])
    XY = torch.linalg.solve(M, torch.cat([S, Pwu]))
    C1, C2 = eye - tau * XY[N:], tau * XY[:N]
    Uh = U @ C1 + W @ C2
    Zh = _solve(osc, V, sigma, Uh, W @ (C1 + torch.linalg.solve(S, Pwu.T) @ C2))
    return Uh - tau * Zh @ (h3 * Uh.T @ Uh - eye), Zh, g


def _signs(X):
    return X * torch.sign(X.gather(0, X.abs().argmax(0)[None]))


def _exact_ritz(osc, V, sigma, U, Z):
    h3 = osc.h ** 3
    AU = _operator(U, V, 0.0, osc.m)
    L = torch.linalg.cholesky(h3 * U.T @ U)
    K = h3 * U.T @ AU
    C = torch.linalg.solve_triangular(L, torch.linalg.solve_triangular(L, 0.5 * (K + K.T), upper=False).T, upper=False)
    lam, Y = torch.linalg.eigh(0.5 * (C + C.T))
    Cv = torch.linalg.solve_triangular(L.T, Y, upper=True)
    W = _solve(osc, V, sigma, U, Z)
    P = h3 * W.T @ U
    return {"lam_rr": lam, "vectors": _signs(U @ Cv), "residuals": (AU @ Cv - (U @ Cv) * lam).square().sum(0).mul(h3).sqrt(),
            "lam_paper": 1.0 / torch.linalg.eigvalsh(0.5 * (P + P.T)).flip(0) - sigma}


def exact(case, seed):
    sizes = _members(case)
    if sum(m ** 3 * N for m, N in sizes) * (case.get("steps", 1)) > 1e8 and case["kind"] in ("step", "batch", "pcg"):
        return None   # over about 20 seconds
    outs = []
    kind = case["kind"]
    for q, (m, N) in enumerate(sizes):
        d = _inputs(case, m, N, seed + 1000 * q)
        osc, V, U = d["osc"], d["V"], d["U"]
        sigma = _shift_of(V, m)
        if kind in ("step", "batch"):
            Z = d["Z"]
            for _ in range(case["steps"]):
                U, Z, g = _step(osc, V, sigma, U, Z, case["tau"])
            outs.append((U, g))
        elif kind == "pcg":
            return _solve(osc, V, sigma, U, d["Z"])
        elif kind == "vcycle":
            return _vcycle(U, V, sigma, m, case["nu"])
        elif kind == "operator":
            return _operator(U, V, sigma, m)
        elif kind == "gemm":
            return U @ d["C1"] + d["Z"] @ d["C2"]
        elif kind == "eigenpairs":
            return _exact_ritz(osc, V, sigma, U, d["Z"])
        elif kind == "adjoint":
            # the complement's resolvent is diagonal in the oscillator's modes
            rho = (U ** 2).sum(1)
            G = osc.h ** 3 * (rho - d["rho"])
            lam = torch.from_numpy(osc.lam[:N]).cuda()
            b = osc.to_modes(G[:, None] * U)
            rows = np.ravel_multi_index(osc.kji, (m, m, m))
            b[torch.from_numpy(rows).cuda()] = 0.0
            den = osc.lam3.reshape(-1, 1) - lam
            den[torch.from_numpy(rows).cuda()] = 1.0
            xi = osc.to_modes(b / den, back=True)
            return {"dV": -2.0 * (U * xi).sum(1), "loss": 0.5 * osc.h ** 3 * (rho - d["rho"]).square().sum()}
        else:
            return _signs(osc.lowest())   # the eigenvectors that the refinement converges to
    if kind == "step":
        return {"U": outs[0][0], "g": outs[0][1]}
    return {"U": [u for u, _ in outs], "g": torch.stack([g for _, g in outs])}
