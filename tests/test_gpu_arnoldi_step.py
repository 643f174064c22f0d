"""The Arnoldi step as one kernel (systems of at most 160 dot-product chunks)
and as separate kernels (larger ones): solves to a given residual, checked
with the operator itself (am_apply_operator, which the parity tests compare
with the oracle).  One chunk and few, both sides of the limit, restart lengths
1, around a warp and the largest, several systems of which some stop at
once."""
import numpy as np
import pytest

from paper_2107_10800_gb300 import build, binding, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.lib()


def chains(seed, n_chains, bodies=8):
    return W.chains_free_space(seed, n_chains=n_chains, bodies_per_chain=bodies,
                               box=10.0 * max(1.0, n_chains / 4.0) ** (1.0 / 3.0))


def residual(s, U, phi, lam, F):
    """|b - A y| / |b| with b = (0, -F, 0) (no slip, passive links)."""
    y = np.concatenate([lam.ravel(), U.ravel(), phi.ravel()])
    b = np.concatenate([np.zeros(lam.size), -F.ravel(), np.zeros(phi.size)])
    return np.linalg.norm(s.apply_operator(y) - b) / np.linalg.norm(b)


# 12 blobs a body: 34 (13 and 23 links more) to about 16,000 unknowns
@pytest.mark.parametrize("n_chains, bodies", [(1, 1), (1, 2), (4, 8), (26, 8), (28, 8), (45, 8)])
@pytest.mark.parametrize("precision, tol", [("fp64", 1e-11), ("mixed", 1e-9)])
def test_solve_reaches_its_residual(n_chains, bodies, precision, tol):
    w = chains(3, n_chains, bodies)
    s = binding.Solver.from_workload(w, precision=precision, tol=tol, max_iter=2000)
    U, phi, lam, st = s.solve()
    assert st["status"] == 0 and st["rel_residual"] <= tol
    check = binding.Solver.from_workload(w)  # the FP64 operator
    # the solver's residual is computed with the same operator up to rounding
    assert residual(check, U, phi, lam, w["F"]) <= 1.01 * tol + 1e-13


@pytest.mark.parametrize("restart", [1, 2, 31, 32, 33, 65, 200])
def test_restart_lengths(restart):
    w = chains(5, 2)
    s = binding.Solver.from_workload(w, tol=1e-11, restart=restart, max_iter=5000)
    U, phi, lam, st = s.solve()
    assert st["status"] == 0
    assert residual(s, U, phi, lam, w["F"]) <= 1.01e-11 + 1e-13
    if restart == 200:
        full = st["iterations"]
        s50 = binding.Solver.from_workload(w, tol=1e-11, restart=full, max_iter=5000)
        assert s50.solve()[3]["iterations"] == full


def test_systems_stop_by_themselves():
    ws = [chains(7, 1), chains(8, 6), chains(9, 3), chains(10, 1, 2)]
    ws[2] = dict(ws[2], F=np.zeros_like(ws[2]["F"]))  # nothing to solve
    s = binding.Solver.from_workloads(ws, tol=1e-11)
    U, phi, lam, st = s.solve()
    assert st["status"] == 0
    for k, (w, (u, p, l)) in enumerate(zip(ws, s.split(U, phi, lam))):
        one = binding.Solver.from_workload(w, tol=1e-11)
        if k == 2:
            assert not np.any(u) and not np.any(l)
            continue
        assert residual(one, u, p, l, w["F"]) <= 1.01e-11 + 1e-13
        u1 = one.solve()[0]
        assert np.abs(u - u1).max() <= 1e-9 * np.abs(u1).max()
