"""The mixed product of many systems of at most 32 blobs (a warp per system) and
the step to larger ones: sizes around a block of 16 sources and the limit,
systems of one size and of several, free space and wall, far from the origin,
against the FP64 product with the bar of the mixed tests; and solves, in which
systems stop one after the other.  FP64 handles on few tiles of 128, whose steps
are split, beside tiles of 32."""
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


def handle(sizes, wall, precision, tile, offset=0.0):
    """A system per list of body sizes."""
    s = binding.Solver(eta=1.0, a=0.1, wall=wall, precision=precision, n_systems=len(sizes), tol=1e-8)
    for k, g in enumerate(sizes):
        M = len(g)
        q = np.stack([offset + 1.5 * np.arange(M), 0.1 * k + 0 * np.arange(M), 18.0 + 0 * np.arange(M)], axis=1)
        rng = np.random.default_rng(k)
        th = rng.standard_normal((M, 4))
        s.set_bodies(q, th / np.linalg.norm(th, axis=1)[:, None], np.concatenate([[0], np.cumsum(g)]),
                     np.concatenate([body(n) for n in g]), rng.standard_normal((M, 6)), np.arange(M), system=k)
    s.set_mobility_layout(3, tile)
    return s


SIZES = {
    "smallest": [[3]],
    "blocks of sources": [[15], [16], [17], [31], [32]],
    "two bodies": [[5, 11], [16, 16], [3, 4, 5]] * 30,
    "one larger": [[12]] * 9 + [[33]],
}


@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("name", SIZES)
def test_product(name, wall):
    for offset in (0.0, 200.0):
        s = handle(SIZES[name], wall, "mixed", 32, offset)
        lam = np.random.default_rng(1).standard_normal((s.Nb, 3))
        ref = s.apply_mobility_ex(lam, "fp64")
        for _ in range(2):
            u = s.apply_mobility_ex(lam, "mixed")
            assert np.abs(u - ref).max() <= 1e-5 * np.abs(ref).max()
        assert np.array_equal(s.apply_mobility_ex(lam, "mixed"), u)


@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("name", SIZES)
def test_solve(name, wall):
    U, phi, lam, st = handle(SIZES[name], wall, "mixed", 32).solve()
    assert st["status"] == 0
    ref = handle(SIZES[name], wall, "fp64", 32).solve()[0]
    # both within 1e-8 of their right side; a body's blob mobility is conditioned below 1e3
    assert np.abs(U - ref).max() <= 1e-5 * np.abs(ref).max()


@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("sizes", [[[40, 40, 40]], [[130]], [[12]] * 5, [[100, 157], [3]]])
def test_fp64_tiles_of_128(sizes, wall):
    a, b = (handle(sizes, wall, "fp64", t) for t in (32, 128))
    lam = np.random.default_rng(2).standard_normal((a.Nb, 3))
    ref = a.apply_mobility(lam)
    for arithmetic, tol in (("fp64", 1e-12), ("mixed", 1e-5), ("df64", 1e-11)):
        assert np.abs(b.apply_mobility_ex(lam, arithmetic) - ref).max() <= tol * np.abs(ref).max()
