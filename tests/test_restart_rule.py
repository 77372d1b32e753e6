"""The restart rule of the FP64 recurrence (the header's own function, compiled for
the host): its bounds, its count across the checks of a goal phase, that it stays out
of ordinary COCG histories, and that it brings a recurrence back that lost its
conjugacy."""
import ctypes as ct
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle as O
from paper_1401_0782_gb300 import problems as P

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include "rsn_internal.h"
extern "C" int step(double* rmin2, int* rmin_it, double nrm, int total) {
  return rsn::watch_step(*rmin2, *rmin_it, nrm, total);
}
"""


class Watch:
    def __init__(self, lib, nrm=1.0, total=0):
        self.lib, self.rmin2, self.rmin_it = lib, ct.c_double(nrm), ct.c_int(total)

    def step(self, nrm, total):
        return bool(self.lib.step(ct.byref(self.rmin2), ct.byref(self.rmin_it), ct.c_double(nrm), total))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cuda = os.path.join(os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("watch")
    (d / "watch.cpp").write_text(SRC)
    p = subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", cuda, "-I",
                        os.path.join(ROOT, "paper_1401_0782_gb300", "csrc"), str(d / "watch.cpp"), "-o", str(d / "watch.so")],
                       capture_output=True, text=True)
    assert p.returncode == 0, p.stderr
    return ct.CDLL(str(d / "watch.so"))


def test_bounds(lib):
    w = Watch(lib)
    assert not w.step(1e10, 1) and w.step(1.0001e10, 2)  # 1e5 times the start
    w = Watch(lib)
    assert not any(w.step(2.0, k) for k in range(1, 3000))  # a plateau above 1e-4 ||b|| is slow convergence
    w = Watch(lib)
    assert not w.step(1e-8, 10) and w.rmin_it.value == 10
    first = next(k for k in range(11, 3000) if w.step(2e-8, k))
    assert first == 411  # more than 400 past the minimum
    w = Watch(lib, 1e-9, 2000)
    first = next(k for k in range(2001, 9000) if w.step(2e-9, k))
    assert first == 4001  # a long-running system: more than half of its iterations (2001 of 4001)


def test_goal_phase_checks_do_not_reset_the_count(lib):
    # the count is in the system's own iterations: a check that only begins a new cycle
    # at iteration 700 passes no argument that could change it (501 > 1001 / 2)
    w = Watch(lib, 1e-12, 500)
    fired = [k for k in range(501, 1200) if w.step(1.5e-12, k)]
    assert fired[0] == 1001


def _cocg(A, b, lib, spoil=None, max_iter=4000, tol=1e-13):
    """COCG with the rule; once the residual is below `spoil` the direction is replaced
    by a random one (conjugacy lost).  Returns the iterations, the restarts and the true residual."""
    x, r, p, w, restarts = np.zeros_like(b), b.copy(), b.copy(), Watch(lib), 0
    rho, nrm = r @ r, 1.0
    for k in range(1, max_iter + 1):
        if spoil and nrm <= spoil ** 2:
            spoil = None
            g = np.random.default_rng(0)
            p = (g.standard_normal(b.size) + 1j * g.standard_normal(b.size)) * np.linalg.norm(p)
        q = A @ p
        a = rho / (p @ q)
        x += a * p
        r -= a * q
        nrm = np.linalg.norm(r) ** 2
        if nrm <= tol ** 2:
            break
        if w.step(nrm, k):
            restarts += 1
            r = b - A @ x
            p, rho, w = r.copy(), r @ r, Watch(lib, np.linalg.norm(r) ** 2, k)
            continue
        new = r @ r
        p = r + (new / rho) * p
        rho = new
    return k, restarts, np.linalg.norm(b - A @ x)


JUNCTIONS = {
    "junction": lambda: (P.molecular_junction(seed=3, nx=10, ny=10, nz=36, n_wells=4, n_cap=5), (0.15, 0.2, 0.25)),
    "waveguide": lambda: (P.waveguide(8, 8, 48), (0.3, 0.8, 1.5)),
}


@pytest.mark.parametrize("name", sorted(JUNCTIONS))
def test_ordinary_systems_and_a_lost_recurrence(lib, name):
    j, energies = JUNCTIONS[name]()
    for E in energies:
        A = O.system_matrix(j, E).tocsr()
        b = np.zeros(j.N, complex)
        b[j.right_columns()[3]] = 1.0
        its, restarts, res = _cocg(A, b, lib)
        assert restarts == 0 and res <= 1e-11, (E, its, restarts, res)
        _, restarts, res = _cocg(A, b, lib, spoil=1e-6)
        assert 1 <= restarts <= 3 and res <= 1e-10, (E, restarts, res)
