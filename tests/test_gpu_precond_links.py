"""The factorisation of the link block of the preconditioner (pivoted Cholesky
without exchanges): chains of linked bodies whose link rows fill part of a
panel, whole panels, and the panel's place in shared memory and one row more
(FP64 240 rows, FP32 455), with every link once or twice (half of the rows
dependent).  The solution of the preconditioner's system has to satisfy the
force and link rows of the full operator, which hold no mobility: FP64 rounding
times the condition of a chain of n links (n^2 <= 1e5) and of a body's block
(below 1e3) stays below 1e-7, FP32 factors (6e-8 n^2 for the link block) below
1e-2 up to 160 links."""
import numpy as np
import pytest

from paper_2107_10800_gb300 import build, binding

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.lib()


def chain(links, twice, precision):
    M, n = links + 1, 4
    t = np.arange(n) - 0.5 * (n - 1)
    rho = np.stack([0.3 * np.cos(2 * t), 0.3 * np.sin(2 * t), 0.21 * t], axis=1)
    s = binding.Solver(eta=1.0, a=0.1, wall=0, precision=precision)
    s.set_bodies(3.0 * np.arange(M)[:, None] * np.array([[1.0, 0.0, 0.0]]), np.tile([1.0, 0, 0, 0], (M, 1)),
                 n * np.arange(M + 1), np.tile(rho, (M, 1)), np.zeros((M, 6)), np.zeros(M, int))
    b = np.repeat(np.arange(links), 2 if twice else 1)
    k = 0.01 * (b % 7)[:, None]
    s.set_constraints(b, b + 1, np.concatenate([1.5 + 0 * k, 0.1 + k, -0.2 + 0 * k], axis=1),
                      np.concatenate([-1.5 + 0 * k, 0.1 + k, 0.3 - k], axis=1))
    return s, 3 * n * M, 6 * M, 3 * len(b)


@pytest.mark.parametrize("precision, tol", [("fp64", 1e-7), ("mixed", 1e-2)])
@pytest.mark.parametrize("links, twice", [(1, 0), (1, 1), (10, 0), (11, 0), (22, 1), (62, 0), (80, 0), (81, 0),
                                          (40, 1), (41, 1), (151, 0), (152, 0)])
def test_force_and_link_rows_hold(links, twice, precision, tol):
    s, nl, nu, nc = chain(links, twice, precision)
    rng = np.random.default_rng(links)
    # a consistent right-hand side: link velocities of some body velocities
    y0 = np.concatenate([np.zeros(nl), rng.standard_normal(nu), np.zeros(nc)])
    r = rng.standard_normal(nl + nu + nc)
    r[nl + nu:] = s.apply_operator(y0)[nl + nu:]
    z = s.apply_precond(r)
    back = s.apply_operator(z)
    scale = max(np.abs(r).max(), np.abs(z[nl + nu:]).max())
    assert np.abs((back - r)[nl:]).max() <= tol * scale
