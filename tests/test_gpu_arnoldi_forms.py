"""The Arnoldi step's way back from one kernel to the separate kernels: a
cooperative launch that the runtime refuses ends neither in a loop on the host
nor in another answer than the separate kernels give.  From the graph and from
steps launched by the host (which kernel timing does), with one system and
several, FP64 and mixed, in solves and in time steps."""
import numpy as np
import pytest

from paper_2107_10800_gb300 import build, binding, workloads as W

pytestmark = pytest.mark.gpu

FUSED, SEPARATE, REFUSED = 0, 1, 2


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.lib()


def solver(n_systems, precision, form, timing):
    ws = [W.chains_free_space(20 + k, n_chains=k + 2, bodies_per_chain=8, box=12.0) for k in range(n_systems)]
    s = binding.Solver.from_workloads(ws, precision=precision, tol=1e-9, restart=20)
    s.set_mobility_layout(3, 32)  # no autotuning: the same sums in every handle
    s.set_arnoldi_step(form)
    if timing:
        s.mobility_timing(True)
    return s


@pytest.mark.parametrize("timing", [False, True])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n_systems", [1, 3])
@pytest.mark.parametrize("form", [REFUSED])
def test_way_back(n_systems, precision, form, timing):
    ref, s = (solver(n_systems, precision, f, timing) for f in (SEPARATE, form))
    for _ in range(2):  # the second solve has the separate kernels from its start
        a, b = ref.solve(), s.solve()
        assert a[3]["status"] == b[3]["status"] == 0
        assert a[3]["iterations"] == b[3]["iterations"] and a[3]["restarts"] == b[3]["restarts"]
        for x, y in zip(a[:3], b[:3]):
            assert np.array_equal(x, y)
    s.set_arnoldi_step(form)
    for k in range(2):
        a, b = ref.step(0.1 * k, 1e-3), s.step(0.1 * k, 1e-3)
        assert a[-1]["status"] == b[-1]["status"] == 0
    s.set_arnoldi_step(form)
    ref.step_rk2(0.2, 1e-3), s.step_rk2(0.2, 1e-3)
    for sysi in range(n_systems):
        for x, y in zip(ref.bodies(sysi), s.bodies(sysi)):
            assert np.array_equal(x, y)
    # and the one kernel again
    s.set_arnoldi_step(FUSED)
    assert s.solve()[3]["status"] == 0
