"""Preconditioner blocks of bodies of one shape (one built, the others rotated
from it) against handles of single bodies at the same pose.  More bodies than
SMs of 3 to 12 blobs, more clusters than SMs of 25 and 37 blobs, several shapes
mixed, a blob moved by one bit (a shape of its own), and every body scaled by
its own factor (no shape shared: every block built, by clusters of 4, 2 and 1).
FP64: blocks of condition below 1e3, 1e-11 of the largest entry; FP32 factors:
1e-4.  Above a wall the blocks depend on the pose: the same comparison there."""
import numpy as np
import pytest

from paper_2107_10800_gb300 import build, binding

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.lib()


def body(n):
    t = np.arange(n) - 0.5 * (n - 1)
    return np.stack([0.3 * np.cos(t), 0.3 * np.sin(t), 0.21 * t], axis=1)


def handle(q, theta, rhos, wall, precision):
    M = len(q)
    s = binding.Solver(eta=1.0, a=0.1, wall=wall, precision=precision)
    s.set_bodies(q, theta, np.concatenate([[0], np.cumsum([len(r) for r in rhos])]), np.concatenate(rhos),
                 np.zeros((M, 6)), np.arange(M))
    return s


def check(rhos, wall, precision, tol, seed):
    M = len(rhos)
    rng = np.random.default_rng(seed)
    q = 20.0 * np.arange(M)[:, None] * np.array([[1.0, 0.0, 0.0]]) + np.array([0.0, 0.0, 9.0])
    theta = rng.standard_normal((M, 4))
    theta /= np.linalg.norm(theta, axis=1)[:, None]
    s = handle(q, theta, rhos, wall, precision)
    off = np.concatenate([[0], np.cumsum([len(r) for r in rhos])])
    nb = off[-1]
    r = rng.standard_normal(3 * nb + 6 * M)
    z = s.apply_precond(r)
    for k in sorted({0, 1, 2, M // 3, M // 2, M - 2, M - 1}):
        one = handle(q[k:k + 1], theta[k:k + 1], rhos[k:k + 1], wall, precision)
        lam, vel = slice(3 * off[k], 3 * off[k + 1]), slice(3 * nb + 6 * k, 3 * nb + 6 * k + 6)
        ref = one.apply_precond(np.concatenate([r[lam], r[vel]]))
        got = np.concatenate([z[lam], z[vel]])
        assert np.abs(got - ref).max() <= tol * np.abs(ref).max()


def moved():
    r = body(12)
    r[5, 1] = np.nextafter(r[5, 1], 1.0)
    return r


CASES = {
    "three blobs": [body(3)] * 200,
    "twelve blobs": [body(12)] * 200,
    "large": [body(25)] * 24 + [body(37)] * 6,
    "shapes": [body(12), body(25), body(11), moved()] * 50,
    "one bit": [body(12)] * 160 + [moved()] * 2 + [body(12)],
    "none shared": [(1.0 + 1e-3 * k) * body(25) for k in range(160)],
    "few clusters": [(1.0 + 1e-3 * k) * body(25) for k in range(45)],
}


@pytest.mark.parametrize("precision, tol", [("fp64", 1e-11), ("mixed", 1e-4)])
@pytest.mark.parametrize("name", CASES)
def test_shared_shapes(name, precision, tol):
    check(CASES[name], 0, precision, tol, len(name))


@pytest.mark.parametrize("precision, tol", [("fp64", 1e-11), ("mixed", 1e-4)])
def test_above_a_wall_every_body_is_built(precision, tol):
    check([body(12)] * 200, 1, precision, tol, 5)
