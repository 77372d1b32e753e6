"""The work that users of this framework have it do, as measured cases.

Every case goes through the Python entry points (``binding.Context``, ``binding.batch_transmission``,
``autograd.transmission``) on the seeded synthetic junctions of ``problems``.  Kinds:

* ``apply``    y_k = A(E_k) x_k for n vectors: the bare operator, for a user's own Krylov method.
* ``columns``  Green's-function columns G(E) e_j.
* ``T``        transmission T(E) over energies and right-lead columns.
* ``window``   T(E) over an energy window from one Krylov space per column (shifted solves).
* ``grad``     T(E) and its gradient with respect to the local potential (forward and adjoint solves).
* ``batch``    T(E) of several uneven junctions in one call.
* ``block``    columns by block solves, several right-hand sides sharing one Krylov space.

Precisions: ``fp64`` (complex FP64 recurrence, the library's default tolerances) and ``mixed`` (complex FP32
recurrence under FP64 refinement, taken to a true residual of 1e-12, so that what comes back is an FP64-grade
result; where T is wanted its goal-oriented finish is taken to 1e-10 for the same reason).  The window's stopping
rule is a recurrence estimate with no goal-oriented finish: its tolerance is 1e-15, so that the small T of nearly
closed channels settle too.  Iteration counts and residual estimates are diagnostics and are not among the outputs.
"""
import math

import numpy as np
import torch

from paper_1401_0782_gb300 import autograd as AG
from paper_1401_0782_gb300 import binding as B
from paper_1401_0782_gb300 import problems as P

DEV = "cuda:0"


def listed():
    bench = dict(nx=24, ny=24, nz=120, h=0.35, R=4, wells=20, lmax=1, n_cap=8, wells_seed=1)  # the benchmark's junction
    small = dict(nx=16, ny=16, nz=64, h=0.35, R=4, wells=8, lmax=1, n_cap=6, wells_seed=2)    # a test-sized junction
    guide = dict(nx=8, ny=8, nz=48, h=0.5, R=1, wells=0, lmax=0, n_cap=16, wells_seed=0)      # the hard-wall waveguide
    large = dict(nx=48, ny=48, nz=192, h=0.3, R=6, wells=60, lmax=2, n_cap=6, wells_seed=4)   # the adjoint junction, s/p/d projectors
    return [
        # one vector on the smallest grid: what a user's own eigensolver or Krylov loop calls; launches and copies count
        dict(name="apply_guide_fp64_1", kind="apply", precision="fp64", n=1, **guide),
        # many vectors on the benchmark junction in complex64: the matvec at bandwidth
        dict(name="apply_bench_fp32_256", kind="apply", precision="mixed", n=256, **bench),
        # odd, ragged planes, no even row and no multiple of a tile: any grid that a DFT code hands over
        dict(name="apply_odd_fp32_16", kind="apply", precision="mixed", n=16, nx=23, ny=19, nz=101, h=0.35, R=3,
             wells=12, lmax=1, n_cap=7, wells_seed=3),
        # the largest grid, widest stencil and nine projectors an atom, in FP64
        dict(name="apply_large_fp64_8", kind="apply", precision="fp64", n=8, **large),
        # a handful of columns of a small junction: latency of the iteration
        dict(name="columns_small_mixed_8", kind="columns", precision="mixed", n_e=1, n_cols=8, e_lo=0.2, e_hi=0.2, **small),
        # a lead plane's worth of columns at one energy: the solver at bandwidth
        dict(name="columns_bench_mixed_144", kind="columns", precision="mixed", n_e=1, n_cols=144, e_lo=0.2, e_hi=0.2, **bench),
        # an energy scan of the waveguide: very many very small systems
        dict(name="T_guide_fp64_32x32", kind="T", precision="fp64", n_e=32, n_cols=32, e_lo=0.05, e_hi=2.0, **guide),
        # T at one energy of the benchmark junction in plain FP64
        dict(name="T_bench_fp64_16", kind="T", precision="fp64", n_e=1, n_cols=16, e_lo=0.2, e_hi=0.2, **bench),
        # an energy window above the first transverse level of the leads, where the junction conducts, from one Krylov
        # space a column
        dict(name="window_bench_16x16", kind="window", precision="fp64", n_e=16, n_cols=16, e_lo=0.40, e_hi=0.48, **bench),
        # T and dT/dV (forward and adjoint) at two energies, the step of an inverse design
        dict(name="grad_small_fp64_8x2", kind="grad", precision="fp64", n_e=2, n_cols=8, e_lo=0.18, e_hi=0.22, **small),
        # a screening run: uneven junctions, a few columns each, one pool
        dict(name="batch_mixed_8", kind="batch", precision="mixed", junctions=8, sizes=11, xy_lo=12, xy_hi=28, z_lo=48,
             z_hi=128, n_e=1, n_cols=4, e_lo=0.2, e_hi=0.2, R=4),
        # the columns of one energy by block solves
        dict(name="block_small_16x32", kind="block", precision="mixed", block=16, n_e=1, n_cols=32, e_lo=0.2, e_hi=0.2, **small),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_grid(rng, n_hi, nz_hi):
    """A junction with independent sides, odd ones as likely as even ones, at a spacing and order in use."""
    R = rng.choice([1, 2, 3, 4, 4, 4, 5, 6])
    nx, ny, nz = rng.randint(10, n_hi), rng.randint(10, n_hi), rng.randint(36, nz_hi)
    return dict(nx=nx, ny=ny, nz=nz, h=rng.choice([0.3, 0.35, 0.4]), R=R, wells=rng.randint(3, 20), lmax=rng.choice([0, 1, 1, 2]),
                n_cap=rng.randint(4, 9), wells_seed=rng.randint(1, 10**6))


def draw(rng):
    kind = rng.choice(["apply", "apply", "columns", "columns", "T", "window", "grad", "batch", "block"])
    prec = rng.choice(["fp64", "mixed"])
    e = round(rng.uniform(0.17, 0.23), 4)
    if kind == "apply":
        g = _draw_grid(rng, 40, 160)
        n = _log_int(rng, 1, max(1, min(256, 256 * 69120 // (g["nx"] * g["ny"] * g["nz"]))))
        return dict(kind=kind, precision=prec, n=n, **g)
    if kind == "batch":
        return dict(kind=kind, precision=prec, junctions=rng.randint(2, 6), sizes=rng.randint(1, 10**6), xy_lo=12, xy_hi=22, z_lo=40,
                    z_hi=80, n_e=rng.randint(1, 2), n_cols=rng.randint(1, 4), e_lo=e, e_hi=round(e + 0.02, 4), R=rng.choice([2, 4]))
    if kind == "T" and rng.random() < 0.4:
        nx, ny = rng.randint(5, 12), rng.randint(5, 12)
        return dict(kind=kind, precision="fp64", n_e=rng.randint(1, 32), n_cols=rng.randint(1, 32), e_lo=0.1, e_hi=1.8, nx=nx, ny=ny,
                    nz=rng.randint(40, 64), h=0.5, R=rng.choice([1, 2]), wells=0, lmax=0, n_cap=16, wells_seed=0)
    g = _draw_grid(rng, 20, 72)
    if kind == "window":
        e = round(rng.uniform(0.3, 0.5), 4)
        return dict(kind=kind, precision="fp64", n_e=rng.randint(4, 16), n_cols=_log_int(rng, 1, 16), e_lo=e, e_hi=round(e + 0.05, 4), **g)
    n_cols = _log_int(rng, 1, 32)
    if kind == "block":
        return dict(kind=kind, precision="mixed", block=rng.choice([4, 8, 16]), n_e=1, n_cols=max(4, n_cols), e_lo=e, e_hi=e, **g)
    n_e = rng.randint(1, 2)
    if kind == "grad":
        return dict(kind=kind, precision="fp64", n_e=n_e, n_cols=min(12, n_cols), e_lo=e, e_hi=round(e + 0.02, 4), **g)
    if kind == "T":
        prec = "fp64"
    return dict(kind=kind, precision=prec, n_e=n_e, n_cols=n_cols, e_lo=e, e_hi=round(e + 0.02, 4), **g)


# ---- inputs ------------------------------------------------------------------

def _perturbed(j, seed):
    """The junction with its potential moved a little, as each step of a self-consistent or design loop moves it."""
    return j.with_potential(j.v_loc + 0.01 * np.random.default_rng(seed).standard_normal(j.N))


def _junction(case, seed):
    if case["wells"] == 0:
        j = P.waveguide(case["nx"], case["ny"], case["nz"], case["h"], n_cap=case["n_cap"], fd_half_order=case["R"])
    else:
        j = P.molecular_junction(seed=case["wells_seed"], nx=case["nx"], ny=case["ny"], nz=case["nz"], h=case["h"], fd_half_order=case["R"],
                                 n_wells=case["wells"], lmax=case["lmax"], n_cap=case["n_cap"])
    return _perturbed(j, seed)


def _batch(case, seed):
    """Uneven junctions: the sizes and wells belong to the case, the perturbation of the potentials to the seed."""
    r, out = np.random.default_rng(case["sizes"]), []
    for k in range(case["junctions"]):
        nxy, nz = int(r.integers(case["xy_lo"], case["xy_hi"] + 1)), int(r.integers(case["z_lo"], case["z_hi"] + 1))
        n_cap, wells = int(r.integers(6, 11)), int(r.integers(5, 21))
        j = P.molecular_junction(seed=case["sizes"] * 64 + k, nx=nxy, ny=nxy, nz=nz, fd_half_order=case["R"], n_wells=wells, n_cap=n_cap)
        out.append(_perturbed(j, seed * 64 + k))
    return out


def _energies(case):
    return np.linspace(case["e_lo"], case["e_hi"], case["n_e"])


def _options(case):
    if case["kind"] == "window":
        return B.default_opts(B.RSN_FP64, tol=1e-15)
    if case["precision"] == "fp64":
        return B.default_opts(B.RSN_FP64)
    # columns: the residual criterion alone; T: the goal-oriented finish as well
    return B.default_opts(B.RSN_MIXED, tol=1e-12, tol_T=1e-10 if case["kind"] == "batch" else 0.0)


def _vectors(case, seed, N):
    g = torch.Generator(device=DEV).manual_seed(seed)
    x = torch.randn(case["n"], N, 2, generator=g, device=DEV, dtype=torch.float64)
    x = torch.view_as_complex(x)
    return x if case["precision"] == "fp64" else x.to(torch.complex64)


def _inputs(case, seed):
    """Everything a pass starts from, on the host but for the vectors of ``apply``."""
    s = dict(case=case)
    if case["kind"] == "batch":
        s["junctions"] = _batch(case, seed)
        s["cols"] = [P.column_subset(j, case["n_cols"], seed + k) for k, j in enumerate(s["junctions"])]
    else:
        s["junction"] = j = _junction(case, seed)
    if case["kind"] == "apply":
        s["E"] = np.random.default_rng(seed).uniform(0.16, 0.24, case["n"])
        s["x"] = _vectors(case, seed, j.N)
    else:
        s["E"] = _energies(case)
    if case["kind"] not in ("apply", "batch"):
        s["cols"] = P.column_subset(j, case["n_cols"], seed)
    if case["kind"] == "grad":
        s["w"] = np.random.default_rng(seed).uniform(0.5, 1.5, case["n_e"])
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    if case["kind"] == "batch":
        s["ctx"] = [B.Context(0).set_junction(j) for j in s["junctions"]]
    else:
        s["ctx"] = B.Context(0).set_junction(s["junction"])
    if case["kind"] == "grad":
        s["v"] = torch.tensor(s["junction"].v_loc, dtype=torch.float64, device=DEV, requires_grad=True)
        s["w"] = torch.tensor(s["w"], dtype=torch.float64, device=DEV)
    if case["kind"] != "apply":
        s["opts"] = _options(case)
    return s


def run(s):
    case, kind, ctx = s["case"], s["case"]["kind"], s["ctx"]
    if kind == "apply":
        return ctx.apply(s["E"], s["x"], B.RSN_FP64 if case["precision"] == "fp64" else B.RSN_MIXED)
    if kind == "columns":
        return ctx.solve_columns(s["E"], s["cols"], s["opts"])[0]
    if kind == "T":
        return ctx.transmission(s["E"], s["cols"], s["opts"])
    if kind == "window":
        return ctx.transmission_shifted(s["E"], s["cols"], s["opts"])
    if kind == "block":
        return ctx.solve_columns_block(s["E"], s["cols"], case["block"], opts=s["opts"])[0]
    if kind == "batch":
        # one spectrum of the set: T of a long, closed junction is 1e-20 of an open one's
        return np.concatenate(B.batch_transmission(ctx, [s["E"]] * len(ctx), s["cols"], s["opts"]))
    T = AG.transmission(ctx, s["v"], s["E"], s["cols"], s["opts"])
    return {"T": T.detach(), "dV": torch.autograd.grad(T, s["v"], s["w"])[0]}


def work(case):
    """Inputs once and outputs once; for the solves the flops of about ten Krylov iterations a grid plane (what the
    24x24x120 junction takes in FP64), each a stencil, the local and projector terms, and the COCG recurrence."""
    if case["kind"] == "batch":
        r, n_pts, planes = np.random.default_rng(case["sizes"]), [], []
        for _ in range(case["junctions"]):
            nxy, nz = int(r.integers(case["xy_lo"], case["xy_hi"] + 1)), int(r.integers(case["z_lo"], case["z_hi"] + 1))
            r.integers(6, 11), r.integers(5, 21)
            n_pts.append(nxy * nxy * nz)
            planes.append(nz)
    else:
        n_pts, planes = [case["nx"] * case["ny"] * case["nz"]], [case["nz"]]
    op = 2 * (7 * case["R"] + 4) + 16  # flops a point of one operator application, projectors about 16
    el = 16 if case["precision"] == "fp64" else 8
    if case["kind"] == "apply":
        return {"bytes": n_pts[0] * (2 * el * case["n"] + 16), "flops": n_pts[0] * case["n"] * op}
    systems = case["n_cols"] * (1 if case["kind"] == "window" else case["n_e"]) * (2 if case["kind"] == "grad" else 1)
    flops = sum(systems * n * 10 * z * (op + 40) for n, z in zip(n_pts, planes))
    out = case["n_e"] * case["n_cols"] * n_pts[0] * 16 if case["kind"] in ("columns", "block") else 8 * case["n_e"] * len(n_pts)
    return {"bytes": sum(24 * n for n in n_pts) + out, "flops": flops}


# ---- the same in 64 bits, plain torch ----------------------------------------

class _Operator:
    """A(E) = E - H + i Gamma on [systems, nz, ny, nx] complex128 tensors."""

    def __init__(self, j):
        R, f = j.fd_half_order, math.factorial
        c = [0.0] + [2.0 * (-1) ** (k + 1) * f(R) ** 2 / (k * k * f(R - k) * f(R + k)) for k in range(1, R + 1)]
        c[0] = -2.0 * sum(c)
        self.w = [v / (2.0 * j.h * j.h) for v in c]
        self.shape, self.N = (j.nz, j.ny, j.nx), j.N
        t = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device=DEV)  # noqa: E731
        self.gl, self.gr = t(j.gamma_l), t(j.gamma_r)
        self.diag = torch.complex(3.0 * self.w[0] - t(j.v_loc), self.gl + self.gr)
        self.atoms = []
        off, last = np.asarray(j.proj_offsets), None
        for p in range(j.proj_ekb.size):
            idx, val = j.proj_idx[off[p]:off[p + 1]], j.proj_val[off[p]:off[p + 1]]
            if last is not None and np.array_equal(last, idx):
                self.atoms[-1][1].append(val)
                self.atoms[-1][2].append(j.proj_ekb[p])
            else:
                self.atoms.append([idx, [val], [j.proj_ekb[p]]])
            last = idx
        self.atoms = [(torch.tensor(np.asarray(i), dtype=torch.int64, device=DEV), t(np.stack(v)).to(torch.complex128), t(e))
                      for i, v, e in self.atoms]

    def __call__(self, E, x):
        """E: [S] float64, x: [S, N] complex128."""
        y = (self.diag + E[:, None]) * x
        ur, yr = (torch.view_as_real(v).view(-1, *self.shape, 2) for v in (x, y))
        for m in range(1, len(self.w)):
            for d in (1, 2, 3):
                n = ur.shape[d] - m
                if n > 0:
                    yr.narrow(d, m, n).add_(ur.narrow(d, 0, n), alpha=self.w[m])
                    yr.narrow(d, 0, n).add_(ur.narrow(d, m, n), alpha=self.w[m])
        for idx, val, e in self.atoms:
            y.index_add_(1, idx, ((x[:, idx] @ val.T) * -e) @ val)
        return y


def _solve(A, E, b):
    """COCG in complex128, far past the residual's rounding floor: the small entries of a column go on converging there."""
    x, r, p = torch.zeros_like(b), b.clone(), b.clone()
    rho = (r * r).sum(1)
    b2 = torch.view_as_real(b).square().sum((1, 2))
    one, zero = torch.ones_like(rho), torch.zeros_like(rho)
    live = b2 > 0
    for k in range(1, 15001):
        q = A(E, p)
        alpha = torch.where(live, rho / torch.where(live, (p * q).sum(1), one), zero)
        x.addcmul_(alpha[:, None], p)
        r.addcmul_(alpha[:, None], q, value=-1)
        new = (r * r).sum(1)
        p.mul_(torch.where(live, new / torch.where(live, rho, one), zero)[:, None]).add_(r)
        rho = new
        live &= torch.view_as_real(r).square().sum((1, 2)) > 1e-38 * b2  # a finished system stays as it is
        if k % 50 == 0 and not bool(live.any()):
            break
    return x


def _columns(A, E, cols):
    """[n_e * n_cols, N] columns and the energy of each."""
    Es = torch.tensor(np.repeat(E, len(cols)), dtype=torch.float64, device=DEV)
    b = torch.zeros(Es.numel(), A.N, dtype=torch.complex128, device=DEV)
    b[torch.arange(Es.numel(), device=DEV), torch.tensor(np.tile(cols, len(E)).astype(np.int64), device=DEV)] = 1.0
    return _solve(A, Es, b), Es


def _transmission(A, x, n_e, cols):
    t = (A.gl * torch.view_as_real(x).square().sum(-1)).sum(1).view(n_e, -1)
    return 4.0 * t @ A.gr[torch.tensor(cols.astype(np.int64), device=DEV)]


def exact(case, seed):
    kind = case["kind"]
    s = _inputs(case, seed)
    if kind == "batch":
        out = []
        for j, cols in zip(s["junctions"], s["cols"]):
            A = _Operator(j)
            out.append(_transmission(A, _columns(A, s["E"], cols)[0], len(s["E"]), cols).cpu().numpy())
        return np.concatenate(out)
    A = _Operator(s["junction"])
    if kind == "apply":
        return A(torch.tensor(s["E"], dtype=torch.float64, device=DEV), s["x"].to(torch.complex128))
    x, Es = _columns(A, s["E"], s["cols"])
    if kind in ("columns", "block"):
        return x.view(len(s["E"]), len(s["cols"]), -1)
    T = _transmission(A, x, len(s["E"]), s["cols"])
    if kind != "grad":
        return T.cpu().numpy()
    lam = _solve(A, Es, A.gl * x.conj())
    wt = torch.tensor(np.repeat(s["w"], len(s["cols"])), device=DEV) * 8.0 * A.gr[torch.tensor(np.tile(s["cols"], len(s["E"])).astype(np.int64), device=DEV)]
    return {"T": T, "dV": (wt[:, None] * (lam * x).real).sum(0)}
