"""The body preconditioner built by clusters of 1, 2, 4 and 8 blocks: the
number of large bodies decides which.  A handle of M bodies without links
against handles of single bodies (always clusters of 8): the same
block-diagonal problems, FP64 factorisations of 75 and 111 rows (1e-11) and
FP32 ones (their rounding times the condition of a body's block, below 1e3:
1e-4)."""
import numpy as np
import pytest

from paper_2107_10800_gb300 import build, binding

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.lib()


def body(n):
    """n blobs of radius 0.1 on a helix, neighbours 0.21 apart along the axis."""
    t = np.arange(n) - 0.5 * (n - 1)
    return np.stack([0.3 * np.cos(t), 0.3 * np.sin(t), 0.21 * t], axis=1)


def handle(q, sizes, precision):
    M = len(q)
    s = binding.Solver(eta=1.0, a=0.1, wall=0, precision=precision)
    s.set_bodies(q, np.tile([1.0, 0, 0, 0], (M, 1)), np.concatenate([[0], np.cumsum(sizes)]),
                 np.concatenate([body(n) for n in sizes]), np.zeros((M, 6)), np.arange(M))
    return s


@pytest.mark.parametrize("precision, tol", [("fp64", 1e-11), ("mixed", 1e-4)])
@pytest.mark.parametrize("M", [1, 30, 90, 160, 216, 310])
def test_every_cluster_size_builds_the_same(M, precision, tol):
    sizes = [25 if k % 3 else 37 for k in range(M)] + [4, 5]  # and two small ones
    q = 20.0 * np.arange(M + 2)[:, None] * np.array([[1.0, 0.0, 0.0]])
    s = handle(q, sizes, precision)
    rng = np.random.default_rng(M)
    nb = sum(sizes)
    r = rng.standard_normal(3 * nb + 6 * (M + 2))
    z = s.apply_precond(r)
    off = np.concatenate([[0], np.cumsum(sizes)])
    for k in sorted({0, M // 2, M - 1, M, M + 1}):
        one = handle(q[k:k + 1], sizes[k:k + 1], precision)
        lam, vel = slice(3 * off[k], 3 * off[k + 1]), slice(3 * nb + 6 * k, 3 * nb + 6 * k + 6)
        ref = one.apply_precond(np.concatenate([r[lam], r[vel]]))
        got = np.concatenate([z[lam], z[vel]])
        assert np.abs(got - ref).max() <= tol * np.abs(ref).max()
