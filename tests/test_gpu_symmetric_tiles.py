"""The symmetric FP64 product on warp tiles at the sizes where its items
change: edges of the 32-blob tiles, of the groups of 64 and 128 blobs and of
the step splits of small systems, one system and several, against the
one-direction FP64 product of the same handle (both sum at most 1,300 terms in
FP64: 1e-12 as the other FP64 product tests)."""
import numpy as np
import pytest

from paper_2107_10800_gb300 import build, binding, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.lib()


def handle(rs, wall):
    s = binding.Solver(eta=1.0, a=0.1, wall=wall, n_systems=len(rs))
    for k, r in enumerate(rs):
        n = len(r)
        s.set_bodies(r, np.tile([1.0, 0, 0, 0], (n, 1)), np.arange(n + 1), np.zeros((n, 3)), np.zeros((n, 6)),
                     np.arange(n), system=k)
    return s


@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("sizes", [(1,), (2,), (31,), (32,), (33,), (65,), (129,), (300,), (577,), (833,), (1281,),
                                   (1, 40, 333), (64, 65, 3, 128)])
@pytest.mark.parametrize("tile", [32, 64, 128])
def test_symmetric_tiles_match_one_direction(sizes, wall, tile):
    rs, lams = zip(*[W.random_blobs(7 + n, n, a=0.1, wall=wall) for n in sizes])
    lam = np.concatenate(lams)
    s = handle(rs, wall)
    s.set_mobility_layout(1, 0)
    ref = s.apply_mobility(lam)
    s.set_mobility_layout(3, tile)
    for _ in range(2):  # the second call finds the first one's partial sums
        u = s.apply_mobility(lam)
        assert np.abs(u - ref).max() <= 1e-12 * np.abs(ref).max()
    for arithmetic, tol in (("mixed", 1e-5), ("df64", 1e-11)):  # on the same layout
        u = s.apply_mobility_ex(lam, arithmetic)
        assert np.abs(u - ref).max() <= tol * np.abs(ref).max()
