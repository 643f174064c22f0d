"""Which way the preconditioner is built and applied.  Blocks: every body's
built, or, of many bodies of one shape in free space, one built and the others
rotated from it in another launch.  Apply: in one launch, or in two (bodies
without links) where bodies are larger or too many articulated bodies have few
bodies each; the lines and the times on both sides stand beside the rules in
api.cu and precond.cu.  Told by the launches of one am_apply_precond; the results against
handles of one articulated body, FP64 1e-11, FP32 factors 1e-4 of the largest
entry."""
import numpy as np
import pytest

from paper_2107_10800_gb300 import build, binding

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "mixed": 1e-4}


@pytest.fixture(scope="module")
def sms():
    torch = pytest.importorskip("torch")
    build.build()
    binding.lib()
    return torch.cuda.get_device_properties(0).multi_processor_count


def body(n):
    t = np.arange(n) - 0.5 * (n - 1)
    return np.stack([0.3 * np.cos(t), 0.3 * np.sin(t), 0.21 * t], axis=1)


def handle(q, blobs, assembly, precision, wall):
    M = len(q)
    s = binding.Solver(eta=1.0, a=0.1, wall=wall, precision=precision)
    s.set_bodies(q, np.tile([1.0, 0, 0, 0], (M, 1)), blobs * np.arange(M + 1), np.tile(body(blobs), (M, 1)),
                 np.zeros((M, 6)), assembly)
    return s


def check(M, blobs, per, precision, wall, launches):
    k = np.arange(M)
    q = 8.0 * np.stack([k % 16, k // 16 % 16, 1 + k // 256], axis=1)
    s = handle(q, blobs, k // per, precision, wall)
    r = np.random.default_rng(M + blobs).standard_normal(s.n)
    s.apply_precond(r)
    l0 = binding.kernel_launches()
    z = s.apply_precond(r)
    assert binding.kernel_launches() - l0 == launches
    nb = 3 * blobs
    for a in {0, M // (2 * per), M // per - 1}:
        i, j = a * per, min(M, (a + 1) * per)
        one = handle(q[i:j], blobs, np.zeros(j - i, int), precision, wall)
        lam, vel = slice(nb * i, nb * j), slice(nb * M + 6 * i, nb * M + 6 * j)
        ref = one.apply_precond(np.concatenate([r[lam], r[vel]]))
        got = np.concatenate([z[lam], z[vel]])
        assert np.abs(got - ref).max() <= TOL[precision] * np.abs(ref).max()


# pose, bodies' blocks and N~: three launches besides the apply (above a wall every body is built)
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("sm, rest, blobs, per, apply", [
    (0, 5, 12, 1, 1), (0, 5, 13, 1, 2), (0, 5, 21, 1, 2), (4, 0, 4, 1, 1), (4, 1, 4, 1, 2), (8, 2, 4, 2, 2),
    (20, 4, 4, 4, 1)])
def test_apply_in_one_launch_or_two(sms, sm, rest, blobs, per, apply, precision):
    check(sm * sms + rest, blobs, per, precision, 1, 3 + apply)


@pytest.mark.parametrize("precision, sm, rest, blobs, rotated", [
    ("fp64", 1, 0, 4, 0), ("fp64", 1, 1, 4, 1), ("mixed", 1, 1, 4, 0), ("mixed", 3, 0, 12, 0), ("mixed", 3, 1, 4, 1),
    ("mixed", 3, 1, 12, 1), ("mixed", 0, 19, 25, 0), ("mixed", 0, 20, 25, 1)])
def test_blocks_built_or_rotated(sms, precision, sm, rest, blobs, rotated):
    if sm == 0 and sms // 8 != 19:
        pytest.skip("the line of large bodies lies elsewhere")
    # 25 blobs: 75 rows, applied in two launches
    check(sm * sms + rest, blobs, 1, precision, 0, 3 + rotated + (1 if blobs <= 12 else 2))
