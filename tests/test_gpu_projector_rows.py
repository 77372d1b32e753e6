"""Projector term of the operator application and of the COCG update: rows of a
block of points, coefficients in whole quads per atom.  Sizes at which the row
tables can go wrong (planes that are no multiple of a block, odd point counts,
1 to 16 projectors an atom, more entries a point than one layer, repeated points
in an atom's index list, more atoms than the shared-memory staging holds), each
against the dense operator of the CPU oracle.

Tolerances: an application sums at most (6 R + 1 + projectors at a point) products;
in FP64 1e-13 of the largest entry, in FP32 2e-6 of it (the parity bounds of the
operator); a solved column meets its residual target 1e-12 times the condition
number (below 1e3 for these CAPs), 1e-9."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_1401_0782_gb300 import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_0782_gb300 import binding
    return binding


def _with_projectors(j, n_atoms, np_atom, support, repeat, seed):
    """`n_atoms` groups of `np_atom` projectors on `support` random points each
    (sorted; `repeat`: the first point once more at the end of the list)."""
    r = np.random.default_rng(seed)
    off, idx, val, ekb = [0], [], [], []
    for _ in range(n_atoms):
        pts = np.sort(r.choice(j.N, size=support, replace=False))
        if repeat:
            pts = np.concatenate([pts, pts[:1]])
        for _ in range(np_atom):
            v = r.standard_normal(pts.size)
            idx.append(pts)
            val.append(v / np.linalg.norm(v))
            off.append(off[-1] + pts.size)
            ekb.append(r.uniform(-0.5, 0.5))
    return dataclasses.replace(j, proj_offsets=np.array(off, np.int64), proj_idx=np.concatenate(idx).astype(np.int32),
                               proj_val=np.concatenate(val), proj_ekb=np.array(ekb))


CASES = [
    # nx, ny, nz, atoms, projectors an atom, support, repeated point
    (8, 8, 24, 3, 4, 200, False),     # whole blocks
    (7, 5, 23, 4, 1, 150, False),     # odd points, one projector (a quad of one value)
    (9, 7, 20, 6, 5, 600, True),      # two quads, a repeated point, several layers
    (10, 6, 17, 12, 9, 700, False),   # three quads, up to twelve atoms a point
    (6, 6, 22, 3, 16, 300, True),     # four quads
]


def _apply_ref(j, E, x):
    A = [O.system_matrix(j, float(e)) for e in E]
    return np.stack([a @ v for a, v in zip(A, x)])


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[:3])) + f"_np{c[4]}")
@pytest.mark.parametrize("n", [1, 3, 130])
def test_apply_with_projector_rows(B, case, n):
    nx, ny, nz, atoms, npa, support, repeat = case
    j = P.tiny_junction(seed=3, nx=nx, ny=ny, nz=nz, fd_half_order=2)
    j = _with_projectors(j, atoms, npa, support, repeat, 5)
    ctx = B.Context(0).set_junction(j)
    r = np.random.default_rng(n)
    x = r.standard_normal((n, j.N)) + 1j * r.standard_normal((n, j.N))
    E = r.uniform(0.1, 0.3, n)
    ref = _apply_ref(j, E, x)
    top = np.abs(ref).max()
    y = ctx.apply(E, torch.tensor(x, device="cuda"), B.RSN_FP64).cpu().numpy()
    assert np.abs(y - ref).max() <= 1e-13 * top
    y = ctx.apply(E, torch.tensor(x.astype(np.complex64), device="cuda"), B.RSN_MIXED).cpu().numpy()
    assert np.abs(y - ref).max() <= 2e-6 * top
    ctx.close()


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[:3])) + f"_np{c[4]}")
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_solve_with_projector_rows(B, case, prec):
    nx, ny, nz, atoms, npa, support, repeat = case
    j = P.tiny_junction(seed=3, nx=nx, ny=ny, nz=nz, fd_half_order=2)
    j = _with_projectors(j, atoms, npa, support, repeat, 5)
    ctx = B.Context(0).set_junction(j)
    cols = j.right_columns()[::11][:7]  # an odd number of slots: odd vectors start off a 16-byte boundary
    p = B.RSN_FP64 if prec == "fp64" else B.RSN_MIXED
    x, _, rel = ctx.solve_columns([0.21], cols, B.default_opts(p, tol=1e-12, tol_T=0.0))
    assert rel.max() <= 1e-12
    A = O.system_matrix(j, 0.21)
    b = np.zeros((j.N, cols.size), complex)
    b[cols, np.arange(cols.size)] = 1.0
    ref = np.linalg.solve(A.toarray() if hasattr(A, "toarray") else np.asarray(A), b).T
    got = x[0].cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-9 * np.linalg.norm(ref)
    ctx.close()


def test_more_atoms_than_the_staging_holds(B):
    # 2,000 single-projector atoms: 128 KB of quads in FP64, 64 KB in FP32
    j = P.tiny_junction(seed=3, nx=8, ny=8, nz=20, fd_half_order=2)
    j = _with_projectors(j, 2000, 1, 12, False, 7)
    ctx = B.Context(0).set_junction(j)
    r = np.random.default_rng(0)
    x = r.standard_normal((2, j.N)) + 1j * r.standard_normal((2, j.N))
    ref = _apply_ref(j, [0.2, 0.25], x)
    for prec, dt, tol in ((B.RSN_FP64, torch.complex128, 1e-13), (B.RSN_MIXED, torch.complex64, 4e-6)):
        y = ctx.apply([0.2, 0.25], torch.tensor(x, device="cuda").to(dt), prec).cpu().numpy()
        assert np.abs(y - ref).max() <= tol * np.abs(ref).max()
    cols = j.right_columns()[:3]
    x64, _, rel = ctx.solve_columns([0.2], cols, B.default_opts(B.RSN_FP64))
    assert rel.max() <= 1e-13
    ctx.close()


@pytest.mark.parametrize("n", [3000, 6000, 14200, 28700])
def test_as_many_projectors_as_the_shared_memory_holds(B, n):
    # coefficients beside the sums of four blocks of points: above 48 KB from 2,544
    # projectors in FP64 (the update 1,520) and 5,616 in FP32; 14,200 fill an SM's shared
    # memory in FP64 beside one block's sums (the update reads them where they lie),
    # 28,700 in FP32.  Bounds as above; a point holds up to 3 n / 640 entries of about
    # 0.01, which adds little to the roundings of an entry of the result.
    j = P.tiny_junction(seed=3, nx=4, ny=4, nz=40, fd_half_order=1)
    j = _with_projectors(j, n, 1, 3, False, 7)
    j = dataclasses.replace(j, proj_ekb=0.04 * j.proj_ekb)
    ctx = B.Context(0).set_junction(j)
    r = np.random.default_rng(0)
    x = r.standard_normal((5, j.N)) + 1j * r.standard_normal((5, j.N))
    E = [0.2, 0.21, 0.22, 0.23, 0.24]
    A = O.system_matrix(j, 0.0)
    ref = np.stack([A @ v + e * v for e, v in zip(E, x)])
    for prec, dt, tol in ((B.RSN_FP64, torch.complex128, 1e-13), (B.RSN_MIXED, torch.complex64, 4e-6)):
        if n > 14200 and prec == B.RSN_FP64:
            continue
        y = ctx.apply(E, torch.tensor(x, device="cuda").to(dt), prec).cpu().numpy()
        assert np.abs(y - ref).max() <= tol * np.abs(ref).max()
    if n <= 14200:
        cols = j.right_columns()[:3]
        A2 = O.system_matrix(j, 0.2)
        b = np.zeros((j.N, 3), complex)
        b[cols, np.arange(3)] = 1.0
        g_ref = np.linalg.solve(A2.toarray(), b).T
        for prec in (B.RSN_FP64, B.RSN_MIXED):
            g, _, rel = ctx.solve_columns([0.2], cols, B.default_opts(prec, tol=1e-12, tol_T=0.0))
            assert rel.max() <= 1e-12
            assert np.linalg.norm(g[0].cpu().numpy() - g_ref) <= 1e-9 * np.linalg.norm(g_ref)
    ctx.close()


def test_infinities_of_an_application(B):
    # an infinite entry at a support point: the projection is infinite, not NaN, and so
    # is the result on the rest of the support, in both precisions
    j = P.tiny_junction(seed=3, nx=8, ny=8, nz=24, fd_half_order=2)
    j = _with_projectors(j, 1, 1, 700, False, 5)
    pts = np.asarray(j.proj_idx)
    x = np.ones((1, j.N), complex)
    x[0, pts[3]] = np.inf
    z, yx = np.divmod(np.arange(j.N), 64)
    far = np.abs(z - z[pts[3]]) > 2
    sup = np.zeros(j.N, bool)
    sup[pts] = True
    v = np.zeros(j.N)
    v[pts] = np.asarray(j.proj_val)
    sign = -np.sign(v * v[pts[3]] * j.proj_ekb[0])
    ctx = B.Context(0).set_junction(j)
    for prec, dt in ((B.RSN_FP64, torch.complex128), (B.RSN_MIXED, torch.complex64)):
        y = ctx.apply([0.2], torch.tensor(x, device="cuda").to(dt), prec).cpu().numpy()[0]
        assert np.all(np.isfinite(y[far & ~sup]))
        assert np.array_equal(y.real[far & sup], np.where(sign > 0, np.inf, -np.inf)[far & sup]), prec
        assert np.all(np.isfinite(y.imag[far]))
    ctx.close()


def test_results_do_not_depend_on_the_number_of_systems(B):
    # FP64 columns solved alone, with a few others and in a pool whose z chunks differ
    j = P.molecular_junction(seed=9, nx=10, ny=9, nz=34, n_wells=3, n_cap=4)
    ctx = B.Context(0).set_junction(j)
    cols = j.right_columns()
    o = B.default_opts(B.RSN_FP64)
    alone = ctx.solve_columns([0.2], cols[:1], o)[0][0, 0]
    few = ctx.solve_columns([0.2], cols[:5], o)[0][0, 0]
    many = ctx.solve_columns([0.2], cols, o)[0][0, 0]
    assert torch.equal(alone, few) and torch.equal(alone, many)
    ctx.close()
