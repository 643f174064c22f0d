"""The stateless mobility products (am_rpy_matvec, its rows and its
allocation-free form) at the sizes where their kernels change: one blob, the
edges of the clusters' groups and shares, the step from the cluster product to
the symmetric one, edges of its tiles and groups, and scratch too small for
it.  References: the product of a handle in FP64 (its own tests compare it
with the oracle) with the bars of those tests, 1e-12 FP64 and 1e-5 mixed."""
import numpy as np
import pytest

from paper_2107_10800_gb300 import build, binding, workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "mixed": 1e-5}


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    build.build()
    binding.lib()
    return t


def reference(r, lam, wall):
    n = len(r)
    s = binding.Solver(eta=1.0, a=0.1, wall=wall)
    s.set_bodies(r, np.tile([1.0, 0, 0, 0], (n, 1)), np.arange(n + 1), np.zeros((n, 3)), np.zeros((n, 6)),
                 np.arange(n))
    s.set_mobility_layout(1, 0)
    return s.apply_mobility(lam)


def run(torch, r, lam, wall, prec, work=None, row0=0, rows=0):
    n = len(r)
    dr, dl = torch.tensor(r, device="cuda"), torch.tensor(lam, device="cuda")
    u = torch.full((rows or n, 3), float("nan"), dtype=torch.float64, device="cuda")
    if work is None:
        work = binding.rpy_matvec_rows_workspace(n, rows, prec) if rows else binding.rpy_matvec_workspace(n, prec)
    # the scratch starts as NaN: nothing of it may be read before it is written
    w = torch.full(((work + 7) // 8 + 32,), float("nan"), dtype=torch.float64, device="cuda")
    p = (w.data_ptr() + 255) // 256 * 256
    st = torch.cuda.current_stream().cuda_stream
    if rows:
        binding.rpy_matvec_rows_ptr(dr.data_ptr(), dl.data_ptr(), u.data_ptr(), n, row0, rows, 1.0, 0.1, wall, prec,
                                    p, work, st)
    else:
        binding.rpy_matvec_ptr(dr.data_ptr(), dl.data_ptr(), u.data_ptr(), n, 1.0, 0.1, wall, prec, p, work, st)
    torch.cuda.synchronize()
    return u.cpu().numpy()


def err(u, ref):
    return np.abs(u - ref).max() / np.abs(ref).max()


@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 7, 31, 33, 129, 255, 256, 257, 1024, 1217, 3072, 3073, 2368, 2433, 4097])
def test_whole_product(torch, n, wall):
    r, lam = W.random_blobs(100 + n, n, a=0.1, wall=wall)
    r = r + np.array([20.0, -15.0, 0.0])
    ref = reference(r, lam, wall)
    for prec in ("fp64", "mixed"):
        u = run(torch, r, lam, wall, prec)
        assert err(u, ref) <= TOL[prec]
        assert np.array_equal(run(torch, r, lam, wall, prec), u)  # nothing depends on scheduling
        # the least scratch a caller may pass: the product without partial sums
        least = binding.rpy_matvec_rows_workspace(n, n, prec)
        assert err(run(torch, r, lam, wall, prec, work=least), ref) <= TOL[prec]


@pytest.mark.parametrize("n", [20479, 20481, 21000])  # 160 and 161 tiles of 128: groups of one, of two
def test_large_products(torch, n):
    r, lam = W.random_blobs(n, n, a=0.1, wall=1)
    ref = run(torch, r, lam, 1, "fp64", row0=n - 2000, rows=2000)
    assert err(run(torch, r, lam, 1, "mixed")[n - 2000:], ref) <= TOL["mixed"]
    assert err(run(torch, r, lam, 1, "fp64")[n - 2000:], ref) <= TOL["fp64"]
    # the paired-lane and double-float products of a handle on the same tiles
    s = binding.Solver(eta=1.0, a=0.1, wall=1, precision="mixed")
    s.set_bodies(r, np.tile([1.0, 0, 0, 0], (n, 1)), np.arange(n + 1), np.zeros((n, 3)), np.zeros((n, 6)),
                 np.arange(n))
    s.set_mobility_layout(3, 128)
    for _ in range(2):  # the second call finds the first one's partial sums
        assert err(s.apply_mobility_ex(lam, "mixed")[n - 2000:], ref) <= TOL["mixed"]
    assert err(s.apply_mobility_ex(lam, "df64")[n - 2000:], ref) <= 1e-11


@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("n, row0, rows", [(1, 0, 1), (40, 39, 1), (500, 3, 129), (2600, 100, 2500), (3000, 2999, 1)])
def test_rows(torch, n, row0, rows, wall):
    r, lam = W.random_blobs(n, n, a=0.1, wall=wall)
    ref = reference(r, lam, wall)[row0:row0 + rows]
    scale = np.abs(reference(r, lam, wall)).max()
    for prec in ("fp64", "mixed"):
        u = run(torch, r, lam, wall, prec, row0=row0, rows=rows)
        assert np.abs(u - ref).max() <= TOL[prec] * scale


def test_scratch_limits(torch):
    n = 5000
    for prec in ("fp64", "mixed"):
        least = binding.rpy_matvec_rows_workspace(n, n, prec)
        assert least <= binding.rpy_matvec_workspace(n, prec)
        with pytest.raises(binding.AmError) as e:
            binding.rpy_matvec_ptr(256, 256, 256, n, 1.0, 0.1, 0, prec, 256, least - 1, None)
        assert e.value.code == binding.AM_ERR_ARG


@pytest.mark.parametrize("n", [300, 5000])
def test_under_capture(torch, n):
    r, lam = W.random_blobs(n, n, a=0.1, wall=1)
    for prec in ("fp64", "mixed"):
        ref = run(torch, r, lam, 1, prec)
        dr, dl = torch.tensor(r, device="cuda"), torch.tensor(lam, device="cuda")
        u = torch.zeros_like(dr)
        work = binding.rpy_matvec_workspace(n, prec)
        w = torch.empty(work + 256, dtype=torch.uint8, device="cuda")
        p = (w.data_ptr() + 255) // 256 * 256
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            binding.rpy_matvec_ptr(dr.data_ptr(), dl.data_ptr(), u.data_ptr(), n, 1.0, 0.1, 1, prec, p, work,
                                   torch.cuda.current_stream().cuda_stream)
        for _ in range(2):
            u.zero_()
            g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(u.cpu().numpy(), ref)
