"""The preconditioner's one-launch apply (every body and every articulated
body's links in 64 rows) against the three-kernel apply, which a handle takes
as soon as one body is larger: the same articulated bodies with a lone body of
23 blobs (69 rows) far away.  Body rows below, at and above one warp and at the
limit, link rows likewise, one articulated body and many, with and without
links.  Both apply the same factors, so they differ by the order of sums: FP64
1e-11; FP32 factors (64-term FP32 sums times a body's condition below 1e3) 1e-4
of the largest entry."""
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


def handle(groups, precision, lone):
    """groups: one list of body sizes per articulated body, its bodies linked in
    a chain (and in a ring where the list is marked by a leading 0)."""
    sizes, assembly, bp, bq = [], [], [], []
    for g in groups:
        ring, g = g[0] == 0, [n for n in g if n]
        first = len(sizes)
        for k, n in enumerate(g):
            if k:
                bp.append(first + k - 1), bq.append(first + k)
            assembly.append(first)
            sizes.append(n)
        if ring:
            bp.append(first + len(g) - 1), bq.append(first)
    if lone:
        assembly.append(len(sizes))
        sizes.append(23)
    assembly = np.unique(assembly, return_inverse=True)[1]
    M = len(sizes)
    q = 6.0 * np.arange(M)[:, None] * np.array([[1.0, 0.0, 0.0]])
    s = binding.Solver(eta=1.0, a=0.1, wall=0, precision=precision)
    s.set_bodies(q, np.tile([1.0, 0, 0, 0], (M, 1)), np.concatenate([[0], np.cumsum(sizes)]),
                 np.concatenate([body(n) for n in sizes]), np.zeros((M, 6)), assembly)
    if bp:
        x = np.arange(len(bp))[:, None]
        s.set_constraints(bp, bq, np.concatenate([3.0 + 0 * x, 0.1 + 0.01 * x, -0.2 + 0 * x], axis=1),
                          np.concatenate([-3.0 + 0 * x, 0.2 + 0 * x, 0.3 - 0.01 * x], axis=1))
    return s, sum(sizes), M, len(bp)


GROUPS = {
    "smallest body": [[3]],
    "no links": [[k] for k in (3, 5, 10, 11, 20, 21)],
    "warp edges": [[10, 11, 21], [11, 10], [21, 3, 20, 10]],
    "one chain": [[12] * 8],
    "longest chain": [[5] * 22],
    "ring": [[0, 11, 12, 13, 21]],
    "many": [[12] * 8, [7, 3]] * 60,
}


@pytest.mark.parametrize("precision, tol", [("fp64", 1e-11), ("mixed", 1e-4)])
@pytest.mark.parametrize("name", GROUPS)
def test_small_apply_matches_large(name, precision, tol):
    small, nb, M, P = handle(GROUPS[name], precision, False)
    large, nb2, M2, _ = handle(GROUPS[name], precision, True)
    assert (nb2, M2) == (nb + 23, M + 1)
    r = np.random.default_rng(nb).standard_normal(3 * nb + 6 * M + 3 * P)
    lam, vel, phi = r[:3 * nb], r[3 * nb:3 * nb + 6 * M], r[3 * nb + 6 * M:]
    z = small.apply_precond(r)
    y = large.apply_precond(np.concatenate([lam, np.ones(69), vel, np.ones(6), phi]))
    parts = [y[:3 * nb], y[3 * nb2:3 * nb2 + 6 * M], y[3 * nb2 + 6 * M2:]]
    for got, ref in zip(np.split(z, [3 * nb, 3 * nb + 6 * M]), parts):
        if ref.size:
            assert np.abs(got - ref).max() <= tol * np.abs(ref).max()
