"""Row ranges of the stateless mobility products whose sources are split into
parts with slots of their own: few rows of many blobs, many rows, shares that
are not whole tiles, a scratch of the least size.  The same rows in one call
and one by one of 97 rows (clusters, one launch) have to agree: FP64 by the
order of sums, 1e-13 of the largest entry; mixed, where the FP32 blocks of 16
sources are the same in every split and their sums have 48 bits, 1e-12."""
import numpy as np
import pytest

from paper_2107_10800_gb300 import build, binding, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    build.build()
    binding.lib()
    return t


def rows_of(torch, dr, dl, n, row0, rows, wall, prec):
    work = binding.rpy_matvec_rows_workspace(n, rows, prec)
    # the scratch starts as NaN: nothing of it may be read before it is written
    w = torch.full(((work + 7) // 8 + 64,), float("nan"), dtype=torch.float64, device="cuda")
    p = (w.data_ptr() + 255) // 256 * 256
    end = (p - w.data_ptr()) // 8 + (work + 7) // 8
    w[end:] = 7.0  # behind the scratch: stays
    u = torch.full((rows, 3), float("nan"), dtype=torch.float64, device="cuda")
    binding.rpy_matvec_rows_ptr(dr.data_ptr(), dl.data_ptr(), u.data_ptr(), n, row0, rows, 1.0, 0.1, wall, prec, p,
                                work, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert bool((w[end:] == 7.0).all())
    return u.cpu().numpy()


@pytest.mark.parametrize("prec, tol", [("fp64", 1e-13), ("mixed", 1e-12)])
@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("n, row0, rows", [(513, 0, 511), (2251, 1000, 562), (3001, 1, 2999), (5063, 3, 632),
                                           (5063, 3798, 1265), (7594, 17, 949), (17086, 8000, 2135),
                                           (30011, 29000, 1011)])
def test_rows_in_one_call_and_in_pieces(torch, n, row0, rows, wall, prec, tol):
    r, lam = W.random_blobs(n + rows, n, a=0.1, wall=wall)
    r = r + np.array([20.0, -15.0, 0.0])
    dr, dl = torch.tensor(r, device="cuda"), torch.tensor(lam, device="cuda")
    u = rows_of(torch, dr, dl, n, row0, rows, wall, prec)
    assert np.array_equal(rows_of(torch, dr, dl, n, row0, rows, wall, prec), u)  # nothing depends on scheduling
    for at in sorted({0, rows // 3, rows - 97}):
        piece = rows_of(torch, dr, dl, n, row0 + at, 97, wall, prec)
        assert np.abs(u[at:at + 97] - piece).max() <= tol * np.abs(u).max()
