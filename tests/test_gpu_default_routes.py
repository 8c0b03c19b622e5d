"""The default routes of the solves beyond their kernels: statistics, memory, streams, the rules.

Tolerances.  Two routes to the same iterations differ in the order and the rounding of float32
sums: a solve after a fixed number of iterations agrees to 2e-5 (about 1e-7 a step, a 2x2 block's
condition below 10, a few steps).  Counts and statistics are exact."""
import ctypes as C

import numpy as np
import pytest

import test_gpu_moments as tmo
from paper_2412_10072_gb300 import qc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = 2e-5


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-30))


@pytest.fixture
def dirty():
    """Leaves freed device memory of small allocations that is not zero."""
    lib = qc.load()
    ptrs = []
    for size in (256, 1024, 4096, 1 << 14, 1 << 16) * 32:
        p = C.c_void_p()
        assert lib.cudaMalloc(C.byref(p), C.c_size_t(size)) == 0
        assert lib.cudaMemset(p, 0x11, C.c_size_t(size)) == 0
        ptrs.append(p)
    assert lib.cudaDeviceSynchronize() == 0
    for p in ptrs[5:]:                # the first ones stay, and with them the driver's blocks
        assert lib.cudaFree(p) == 0
    yield
    for p in ptrs[:5]:
        assert lib.cudaFree(p) == 0


def _terms(obs, iters, **kw):
    return [qc.Term.from_spec(s, obs.n_ant, max_iter=k, tol=0.0, **kw) for s, k in zip(obs.terms, iters)]


@pytest.mark.parametrize("iters,epochs", [((4, 40), 2), ((40, 4), 2), ((3, 3), 9), ((3, 5), 9)])
def test_iteration_statistics(dirty, iters, epochs):
    """Two terms of unlike max_iter on a new solver, and more term solves than are collected at
    once: with tol = 0 every solve takes all of its iterations."""
    obs = tmo._chain_obs(5, ("diag", "diag"), n_ant=9, n_time=24, n_chan=33, t_int=(12, 24), f_int=(33, 11))
    gains = []
    for kernel in (0, 3):
        S = qc.Solver.from_obs(obs)
        T = _terms(obs, iters)
        st = S.solve(T, n_epochs=epochs, kernel=kernel)
        S.close()
        assert st.n_iter_max == max(iters)
        assert st.acc_launches == epochs * sum(iters)
        assert all((t.iters == k).all() for t, k in zip(T, iters))
        gains.append(T)
    # beyond the first epochs the rounding differences of the two routes stay at their fixed point
    for a, b in zip(*gains):
        assert _rel(a.gains, b.gains) < TOL
