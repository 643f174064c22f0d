"""The Arnoldi step's way back from one kernel to the separate kernels: a
cooperative launch that the runtime refuses, or a wait of its blocks that runs
out, ends neither in a loop on the host nor in a failed solve nor in another
answer than the separate kernels give.  From the graph and from steps launched
by the host (which kernel timing does), with one system and several, FP64 and
mixed, in solves and in time steps; and handles that solve at once, on threads
and streams of their own."""
import threading

import numpy as np
import pytest

from paper_2107_10800_gb300 import build, binding, workloads as W

pytestmark = pytest.mark.gpu

FUSED, SEPARATE, REFUSED, LATE = 0, 1, 2, 3


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
@pytest.mark.parametrize("form", [REFUSED, LATE])
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


def test_unknown_form():
    with pytest.raises(binding.AmError) as e:
        binding.Solver().set_arnoldi_step(4)
    assert e.value.code == binding.AM_ERR_ARG


def test_solves_at_once():
    # two handles of eight systems, each with about 590 step blocks of the 608 that a GPU of 152
    # SMs holds at four a SM: on two streams they cannot all be resident at once
    hs = [binding.Solver.from_workloads([W.chains_free_space(40 + 8 * k + i, n_chains=12, bodies_per_chain=8, box=24.0)
                                         for i in range(8)], tol=1e-9) for k in range(2)]
    for s in hs:
        s.set_mobility_layout(3, 64)
    ref = [s.solve() for s in hs]
    out, errors = [None, None], []

    def work(k):
        try:
            out[k] = [hs[k].solve() for _ in range(20)]
        except Exception as e:  # shown by the assertion below
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for k in range(2):
        for U, phi, lam, st in out[k]:
            assert st["status"] == 0
            # both are within 1e-9 of their right side; a solve that went over to the separate kernels
            # rounds otherwise.  A thousandfold of it covers the conditioning of a few bodies in contact
            assert np.abs(U - ref[k][0]).max() <= 1e-6 * np.abs(ref[k][0]).max()
