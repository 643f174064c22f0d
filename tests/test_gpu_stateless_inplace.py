"""Stateless mobility products whose output shares memory with an input: u in
place of lambda, in place of r, one blob further on, and a range of rows in
its own place in lambda or r.  Every entry point has to give, bit for bit, what
it gives with an output of its own: one launch of clusters (FP64 below 256
blobs, fewer rows, little scratch, mixed with one and with two targets per
thread), several parts, and the symmetric product."""
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


def product(torch, pr, pl, pu, n, wall, prec, form, row0, rows):
    st = torch.cuda.current_stream().cuda_stream
    if form == "noalloc":
        binding.rpy_matvec_noalloc_ptr(pr, pl, pu, n, 1.0, 0.1, wall, prec, st)
        return
    # "least": the smallest scratch the entry point takes
    nbytes = binding.rpy_matvec_workspace(n, prec) if form == "full" else \
        binding.rpy_matvec_rows_workspace(n, rows, prec)
    w = torch.full(((nbytes + 7) // 8 + 32,), float("nan"), dtype=torch.float64, device="cuda")
    p = (w.data_ptr() + 255) // 256 * 256
    if form == "rows":
        binding.rpy_matvec_rows_ptr(pr, pl, pu, n, row0, rows, 1.0, 0.1, wall, prec, p, nbytes, st)
    else:
        binding.rpy_matvec_ptr(pr, pl, pu, n, 1.0, 0.1, wall, prec, p, nbytes, st)


@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n, form, row0, rows", [
    (40, "full", 0, 0), (200, "full", 0, 0), (255, "noalloc", 0, 0), (1000, "least", 0, 0), (1000, "full", 0, 0),
    (5000, "full", 0, 0), (5000, "least", 0, 0), (5000, "noalloc", 0, 0), (9000, "least", 0, 0),
    (200, "rows", 50, 97), (1000, "rows", 903, 97), (7000, "rows", 4000, 2333), (9000, "rows", 0, 3000)])
def test_output_shares_an_input(torch, n, form, row0, rows, prec, wall):
    r, lam = W.random_blobs(n + rows, n, a=0.1, wall=wall)
    rows = rows or n
    # one blob of room behind each input
    both = {"r": r, "lam": lam}
    buf = {k: torch.zeros((n + 1, 3), dtype=torch.float64, device="cuda") for k in both}

    def fill():
        for k, v in both.items():
            buf[k][:n] = torch.tensor(v, device="cuda")

    def at(k, i):
        return buf[k].data_ptr() + 24 * i

    fill()
    u = torch.full((rows, 3), float("nan"), dtype=torch.float64, device="cuda")
    product(torch, at("r", 0), at("lam", 0), u.data_ptr(), n, wall, prec, form, row0, rows)
    torch.cuda.synchronize()
    assert bool(torch.isfinite(u).all())
    for k in both:
        for i in {row0, row0 + 1}:
            for _ in range(3):
                fill()
                product(torch, at("r", 0), at("lam", 0), at(k, i), n, wall, prec, form, row0, rows)
                torch.cuda.synchronize()
                assert bool((buf[k][i:i + rows] == u).all()), (k, i)
                other = "lam" if k == "r" else "r"
                assert np.array_equal(buf[other][:n].cpu().numpy(), both[other])
