"""The default routes of the solves beyond their kernels: statistics, memory, streams, the rules.

Tolerances.  Two routes to the same iterations differ in the order and the rounding of float32
sums: a solve after a fixed number of iterations agrees to 2e-5 (about 1e-7 a step, a 2x2 block's
condition below 10, a few steps).  Counts and statistics are exact."""
import ctypes as C

import numpy as np
import pytest

import oracle as O
import test_gpu_moments as tmo
from paper_2412_10072_gb300 import qc, synth

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


# (kind, n_ant, n_time, n_chan, t_int, f_int): slots of one addition and of several, one slot over the
# whole scan (flushes of several row blocks and chunks), intervals across chunk edges, a channel each
DEPTHS = [("diag", 7, 60, 16, 4, 4), ("diag", 7, 120, 200, 8, 40), ("full", 7, 60, 256, 8, 40), ("diag", 7, 120, 512, 120, 512),
          ("full", 7, 120, 512, 120, 512), ("phase", 9, 48, 130, 12, 33), ("full", 8, 40, 290, 1, 290),
          ("diag", 9, 160, 40, 160, 1)]


@pytest.mark.parametrize("m16", [False, True])
@pytest.mark.parametrize("shape", DEPTHS, ids=lambda s: "%s-%d-%dx%d-%dx%d" % s)
def test_sums_hold_their_precision(shape, m16):
    """The error of the default solve against the oracle does not grow with the interval.  Rounding
    the result to float32 alone is 2.4e-8 (rms, relative); sums of 16 to 32 float32 terms, added in 64
    bits, leave another 2e-8 after averaging over the terms, on few antennas a little more: 6e-8."""
    kind, n_ant, n_time, n_chan, ti, fi = shape
    obs = tmo._chain_obs(60 + n_ant, (kind,), n_ant=n_ant, n_time=n_time, n_chan=n_chan, t_int=(ti,), f_int=(fi,))
    rng = np.random.default_rng(1)
    start = tmo._start(obs.terms[0], rng)
    S = qc.Solver.from_obs(obs, model_fp16=m16)
    T = qc.Term.from_spec(obs.terms[0], n_ant, gains=start, max_iter=6, tol=0.0)
    st = S.solve([T])
    s3 = S.solve([qc.Term.from_spec(obs.terms[0], n_ant, gains=start, max_iter=6, tol=0.0)], kernel=3)
    S.close()
    assert st.acc_bytes < s3.acc_bytes             # the sums, not the samples an iteration
    if m16:                                        # the model as the solver holds it: float16 and a scale a baseline
        m = obs.model.view(np.float32).reshape(*obs.model.shape, 2)
        key = obs.ant1.astype(np.int64) * n_ant + obs.ant2
        scale = np.zeros(n_ant * n_ant, np.float32)
        np.maximum.at(scale, key, np.abs(m).max(axis=(1, 2, 3)))
        s = scale[key][:, None, None, None]
        h = (m * (np.float32(1) / s)).astype(np.float16).astype(np.float32) * s
        obs.model = np.ascontiguousarray(h).view(np.complex64)[..., 0]
    P = O.OracleProblem.from_obs(obs)
    o = O.OracleTerm.from_spec(obs.terms[0], n_ant, params=start.astype(np.float64 if kind == "phase" else np.complex128),
                               max_iter=6, tol=0.0)
    O.solve(P, [o], damping_mode=1)
    err = np.linalg.norm(np.asarray(T.gains, dtype=o.params.dtype) - o.params) / np.linalg.norm(o.params)
    assert err < 6e-8, err


def _delay_case(seed, n_ant, n_time, n_chan, t_int, twice=False, oracle=True):
    """A delay term over intervals of t_int times, with truth as start: data, terms of both sides."""
    rng = np.random.default_rng(seed)
    p, q = synth.baselines(n_ant)
    ant1, ant2 = np.tile(p, n_time), np.tile(q, n_time)
    tidx = np.repeat(np.arange(n_time, dtype=np.int32), p.size)
    if twice:                                       # a second row of every pair and time, the other way round
        ant1, ant2, tidx = np.concatenate([ant1, ant2]), np.concatenate([ant2, ant1]), np.tile(tidx, 2)
    nu = np.linspace(0.9, 1.7, n_chan)
    tm = synth.interval_map(n_time, t_int)
    nt = int(tm[-1]) + 1
    par = np.zeros((nt, 1, n_ant, 4), np.float32)
    par[..., 0::2] = rng.uniform(-1, 1, (nt, 1, n_ant, 2))
    par[..., 1::2] = rng.uniform(-0.1, 0.1, (nt, 1, n_ant, 2))
    ph = par[tm, 0][:, None, :, 0::2] + 2 * np.pi * nu[None, :, None, None] * par[tm, 0][:, None, :, 1::2]
    g = np.exp(1j * ph)                             # [time][chan][ant][2]
    shp = (ant1.size, n_chan, 4)
    model = np.ones(shp) * rng.uniform(0.5, 1.5, shp)
    gp, gq = g[tidx, :, ant1], g[tidx, :, ant2].conj()
    data = model * (gp[..., [0, 0, 1, 1]] * gq[..., [0, 1, 0, 1]])
    start = (par + rng.normal(0, 1, par.shape) * [0.1, 0.01, 0.1, 0.01]).astype(np.float32)
    args = (data.astype(np.complex64), model.astype(np.complex64), rng.uniform(0.5, 1.5, shp).astype(np.float32),
            np.zeros(shp[:2], np.uint8), ant1.astype(np.int32), ant2.astype(np.int32), tidx, n_ant, n_time)
    fm = np.zeros(n_chan, np.int32)
    G = lambda: qc.Term("delay", tm, fm, nt, 1, n_ant, gains=start, max_iter=8, tol=0.0, chan_freq=nu)  # noqa: E731
    o = O.OracleTerm("delay", tm, fm, nt, 1, n_ant, params=start.astype(np.float64), chan_freq=nu, max_iter=8, tol=0.0)
    if oracle:
        O.solve_term(O.OracleProblem(*args), [o], 0, damping_mode=1)

    def phases(u):                                  # at every channel, against antenna 0
        v = np.asarray(u, np.float64)[:, 0][:, None, :, 0::2] + \
            2 * np.pi * nu[None, :, None, None] * np.asarray(u, np.float64)[:, 0][:, None, :, 1::2]
        return v - v[:, :, :1]
    return args, G, phases(o.params), phases


@pytest.mark.parametrize("n_ant,n_time,n_chan,t_int,twice", [(3, 20000, 4, 20000, False), (5, 300, 33, 100, True),
                                                             (9, 64, 40, 2, False), (9, 16, 40, 1, True),
                                                             (6, 50, 64, 3, False), (5, 70, 40, 33, False),
                                                             (220, 4, 3, 2, False), (221, 4, 3, 2, False)])
def test_delay_products_hold_their_precision(n_ant, n_time, n_chan, t_int, twice):
    """Products of many samples and of few, rows of both orientations, antennas at the limit of a
    CTA's shared memory and beyond it.  A phase at a channel carries the rounding of its two float32
    parameters, 2^-25 of 1 and of 10.7 x 0.1, and that of antenna 0: 7e-8 (rms); 1e-7."""
    args, G, want, phases = _delay_case(11, n_ant, n_time, n_chan, t_int, twice)
    S = qc.Solver(*args)
    T = G()
    S.solve([T])
    S.close()
    err = np.sqrt(np.mean((phases(T.gains) - want) ** 2))
    assert err < 1e-7, err


@pytest.mark.parametrize("n_ant,tol", [(7, 1e-2), (7, 1e-4), (7, 1e-6), (130, 1e-3), (130, 1e-5)])
def test_delay_convergence(n_ant, tol):
    """The iterations of every interval, and with them the convergence test on the change of the
    gains (more antennas than the block of the update takes at once, large and small changes), are
    those of the chain rule per sample."""
    args, G, _, phases = _delay_case(12, n_ant, 24, 50, 1 if n_ant < 100 else 6, oracle=False)
    out = []
    for kernel in (0, 3):
        S = qc.Solver(*args)
        T = G()
        T.max_iter, T.tol = 12, tol
        S.solve([T], kernel=kernel)
        S.close()
        out.append(T)
    assert np.array_equal(out[0].iters, out[1].iters)
    assert 1 < out[0].iters.min() and out[0].iters.max() < 12
    assert np.sqrt(np.mean((phases(out[0].gains) - phases(out[1].gains)) ** 2)) < 2e-7


@pytest.mark.parametrize("n_chan", [1, 33, 70])
def test_chi2_beyond_float(n_chan):
    """chi^2 is a 64-bit sum of float32 terms: finite where a row's terms together exceed the largest
    float32, with every term itself representable; NaN and infinite terms stay what they are."""
    rng = np.random.default_rng(n_chan)
    n_ant, n_time = 4, 3
    p, q = synth.baselines(n_ant)
    ant1, ant2 = np.tile(p, n_time).astype(np.int32), np.tile(q, n_time).astype(np.int32)
    tidx = np.repeat(np.arange(n_time, dtype=np.int32), p.size)
    shp = (ant1.size, n_chan, 4)
    data = ((1 + rng.random(shp)) * 1e16 * np.exp(1j * rng.uniform(0, 6, shp))).astype(np.complex64)
    weight = rng.uniform(2e5, 8e5, shp).astype(np.float32)           # terms of 2e37 to 3.2e38

    def chi2(d, w):
        S = qc.Solver(d, np.zeros(shp, np.complex64), w, np.zeros(shp[:2], np.uint8), ant1, ant2, tidx, n_ant, n_time)
        T = qc.Term("diag", np.zeros(n_time, np.int32), np.zeros(n_chan, np.int32), 1, 1, n_ant, solve=False)
        v = S.residual([T])
        S.close()
        return v

    term = weight * (data.real.astype(np.float32) ** 2 + data.imag.astype(np.float32) ** 2)
    assert np.isfinite(term).all() and (n_chan == 1 or term.sum(dtype=np.float64) > 4e39)
    want = float((weight.astype(np.float64) * np.abs(data.astype(np.complex128)) ** 2).sum())
    assert abs(chi2(data, weight) - want) <= 2e-7 * want             # four float32 roundings a term, averaged
    bad = data.copy()
    bad[5, n_chan // 2, 1] = np.nan
    assert np.isnan(chi2(bad, weight))
    bad[5, n_chan // 2, 1] = np.inf
    assert np.isinf(chi2(bad, weight)) or np.isnan(chi2(bad, weight))


def test_failed_call_keeps_no_stream():
    """A call that fails half-way on a caller's stream leaves nothing of that stream behind: the
    stream is destroyed before the next call and before the solver is closed."""
    lib = qc.load()
    obs = tmo._chain_obs(7, ("diag",), n_ant=6, n_time=8, n_chan=20, t_int=(4,), f_int=(20,))
    want = _terms(obs, (5,))
    S = qc.Solver.from_obs(obs)
    S.solve(want)

    def failing(buffer, n, stream, user):
        return 1

    for fails in ("allocation", "allreduce"):
        for _ in range(2):
            st = C.c_void_p()
            assert lib.cudaStreamCreate(C.byref(st)) == 0
            F = qc.Solver.from_obs(obs)
            with pytest.raises(qc.QCError):
                if fails == "allocation":
                    lib.qc_test_fail_alloc(3)
                    F.solve(_terms(obs, (5,)), stream=st.value, kernel=3)
                else:
                    F.solve(_terms(obs, (5,), reduce=True), stream=st.value, allreduce=failing)
            lib.qc_test_fail_alloc(0)
            assert lib.cudaStreamDestroy(st) == 0
            got = _terms(obs, (5,))
            F.solve(got)
            F.close()
            assert _rel(got[0].gains, want[0].gains) < 1e-6
    S.close()


def test_staging_limit():
    """Host gains beyond the pinned block's limit (16 MB) go directly; the first call, which has no
    block yet, and the next ones agree, also when a call needs a larger block than the one before."""
    n_ant, n_time, n_chan = 4, 700, 256
    obs = tmo._chain_obs(8, ("diag",), n_ant=n_ant, n_time=n_time, n_chan=n_chan, t_int=(1,), f_int=(1,), flag_frac=0.0)
    small = [synth.TermSpec("diag", synth.interval_map(n_time, 350), synth.interval_map(n_chan, 128), 2, 2)]
    assert obs.terms[0].truth.size * 8 > 16 << 20
    S = qc.Solver.from_obs(obs)
    seen = {}
    for kind in ("small", "large", "small", "large", "small"):
        T = qc.Term.from_spec((small if kind == "small" else obs.terms)[0], n_ant, max_iter=4, tol=0.0)
        S.solve([T])
        assert (T.iters == 4).all()
        g = seen.setdefault(kind, T.gains)
        assert _rel(T.gains, g) < 1e-6 and _rel(g, np.ones(1)) > 1e-3
    S.close()
    # residuals and flags alone: direct copies first, the block from the eighth call on
    R = qc.Solver.from_obs(obs)
    fixed = _terms(obs, (1,), solve=False)
    chi2 = [R.residual(fixed) for _ in range(10)]
    flags = [R.mad_flag(fixed)[1] for _ in range(3)]
    R.close()
    assert max(chi2) - min(chi2) <= 1e-12 * chi2[0] and len(set(flags)) == 1


@pytest.mark.parametrize("kinds,n_ant,t_int", [(("diag",), 100, 8), (("diag",), 160, 8), (("diag",), 160, 1), (("full",), 70, 8),
                                               (("full",), 110, 8), (("phase",), 160, 8), (("full", "diag"), 130, 8),
                                               (("diag",), 257, 8)])
def test_many_antennas(kinds, n_ant, t_int):
    """Few intervals of many antennas: a launch for all iterations or one each (and beyond 256
    antennas the samples), against the samples; statistics of either count the same iterations, and
    asking for the sums is no other result."""
    n_time, n_chan = 8, 16
    obs = tmo._chain_obs(90, kinds, n_ant=n_ant, n_time=n_time, n_chan=n_chan, t_int=(t_int, n_time), f_int=(n_chan, n_chan))
    rng = np.random.default_rng(2)
    start = [tmo._start(s, rng) for s in obs.terms]
    S = qc.Solver.from_obs(obs)
    out = []
    for kw in (dict(), dict(moments=True), dict(kernel=3)):
        T = [qc.Term.from_spec(s, n_ant, gains=g, max_iter=4, tol=0.0) for s, g in zip(obs.terms, start)]
        st = S.solve(T, **kw)
        assert st.n_iter_max == 4 and st.acc_launches == 4 * len(kinds)
        out.append((T, st))
    S.close()
    assert (out[0][1].acc_bytes < out[2][1].acc_bytes) == (n_ant <= 256)
    for T, _ in out[:2]:
        for a, b in zip(T, out[2][0]):
            assert _rel(a.gains, b.gains) < TOL
            assert np.array_equal(a.gain_flags, b.gain_flags) and np.array_equal(a.iters, b.iters)


@pytest.mark.parametrize("t_int,n_chan", [(1, 60), (3, 64)])
def test_delay_bytes_tell_the_route(t_int, n_chan):
    """qc_stats.acc_bytes of a delay term from products: the samples once (80 B unflagged, a byte of
    flags each), then 32 B per pair and channel of the intervals iterated on; on the samples all of them
    an iteration.  Intervals of one time on a full grid are stored, the others added."""
    args, G, _, _ = _delay_case(13, 8, 12, n_chan, t_int, oracle=False)
    st = []
    for kernel in (0, 3):
        S = qc.Solver(*args)
        T = G()
        st.append(S.solve([T], kernel=kernel))
        S.close()
    n_pair, n_int, its = 28, 12 // t_int, 8
    samples = 12 * n_pair * n_chan * 81
    assert st[0].acc_bytes == samples + its * 32 * n_pair * n_chan * n_int
    assert st[1].acc_bytes == its * samples
    assert st[0].vis_iters == st[1].vis_iters == its * 12 * n_pair * n_chan


@pytest.mark.parametrize("n_ant,n_time,n_chan,products", [(8, 1, 64, True), (128, 1, 64, False), (128, 8, 512, True)])
def test_delay_route_of_few_intervals(n_ant, n_time, n_chan, products):
    """One CTA per time interval and 32 channels walks all pairs: few of them with many antennas
    iterate on the samples (qc_stats.acc_bytes tells), with the same result."""
    args, G, _, phases = _delay_case(14, n_ant, n_time, n_chan, 1, oracle=False)
    out = []
    for kernel in (0, 3):
        S = qc.Solver(*args)
        T = G()
        T.max_iter = 3
        out.append((T, S.solve([T], kernel=kernel).acc_bytes))
        S.close()
    assert (out[0][1] < out[1][1]) == products
    assert np.sqrt(np.mean((phases(out[0][0].gains) - phases(out[1][0].gains)) ** 2)) < 2e-7


def test_autotune_keeps_the_faster_route():
    """Tuning the persistent kernel does not take the default solves of the shape class from the sums
    where those are faster; asking for the shape's own launch does, and a second batch of the class
    behaves like the first."""
    import test_gpu_batch as tb
    b = tb.small_batch(n=40, seed_base=4200)
    S = tb.solver_of(b)
    g0, f0, i0, st0 = S.solve(max_iter=6, tol=0.0)
    assert st0.depth == 0                                # from sums
    best, _ = S.autotune()
    S2 = tb.solver_of(b)
    for solver in (S, S2):
        g1, f1, i1, st1 = solver.solve(max_iter=6, tol=0.0)
        g2, f2, i2, st2 = solver.solve(max_iter=6, tol=0.0, use_graph=False)
        assert st1.depth == 0 or st1.depth == best.depth and best.ms < st0.ms
        assert st2.depth == best.depth and st2.bytes > st0.bytes
        assert _rel(g1, g0) < TOL and _rel(g2, g0) < TOL
        assert np.array_equal(f1, f0) and np.array_equal(f2, f0) and np.array_equal(i1, i0)
    S.close()
    S2.close()


@pytest.mark.parametrize("kinds", [("diag",), ("full",), ("full", "diag")])
def test_unchanged_gains_converge_at_any_tolerance(kinds):
    """An interval without data does not change its gains: that is below a tolerance whose square
    underflows, so one iteration is all, as on the samples; a tolerance of zero takes them all."""
    obs = tmo._chain_obs(21, kinds, n_ant=6, n_time=8, n_chan=33, t_int=(4, 8), f_int=(33, 33))
    obs.flag = np.ones_like(obs.flag)
    for tol, its in ((1e-200, 1), (0.0, 5)):
        for kw in (dict(), dict(kernel=3)):
            S = qc.Solver.from_obs(obs)
            T = [qc.Term.from_spec(s, obs.n_ant, max_iter=5, tol=tol) for s in obs.terms]
            S.solve(T, **kw)
            S.close()
            assert all((t.iters == its).all() for t in T), (tol, kw)
    import test_gpu_batch as tb
    b = tb.small_batch(n=5, seed_base=77)
    b.flag = np.ones_like(np.array(b.flag))
    S = tb.solver_of(b)
    for kw in (dict(), dict(threads=256)):
        _, _, it, _ = S.solve(max_iter=5, tol=1e-200, **kw)
        assert (it == 1).all()
    S.close()


@pytest.fixture
def lib():
    lib = qc.load()
    yield lib
    lib.qc_test_fail_alloc(0)
    if hasattr(lib, "qc_test_free_bytes"):
        lib.qc_test_free_bytes(-1)


def test_routes_leave_room(lib):
    """A default route whose workspace would take more than half of the free memory is left for the
    iterations on the samples; asking for the sums is not refused."""
    import test_gpu_batch as tb
    obs = tmo._chain_obs(31, ("diag",), n_ant=8, n_time=40, n_chan=64, t_int=(8,), f_int=(64,))
    args, G, _, _ = _delay_case(15, 8, 12, 64, 1, oracle=False)
    b = tb.small_batch(n=6, seed_base=92)

    def routes():
        S = qc.Solver.from_obs(obs)
        r = [S.solve(_terms(obs, (4,))).acc_bytes]
        S.close()
        S = qc.Solver(*args)
        r.append(S.solve([G()]).acc_bytes)
        S.close()
        S = tb.solver_of(b)
        r.append(S.solve(max_iter=4, tol=0.0)[3].bytes)
        S.close()
        return r

    free = routes()
    lib.qc_test_free_bytes(1000)
    full = routes()
    assert all(a < c for a, c in zip(free, full))
    S = qc.Solver.from_obs(obs)
    assert S.solve(_terms(obs, (4,)), moments=True).acc_bytes == free[0]
    S.close()


@pytest.mark.parametrize("what", ["sums", "delay"])
def test_failed_workspace_falls_back(lib, what):
    """Each allocation of a default solve failing in turn: QC_ENOMEM where the samples need it too, else
    the samples, with the result and the statistics of kernel 3, and nothing is lost."""
    if what == "sums":
        obs = tmo._chain_obs(32, ("diag", "full"), n_ant=6, n_time=24, n_chan=40, t_int=(8, 24), f_int=(40, 40))
        make, terms = (lambda: qc.Solver.from_obs(obs)), (lambda: _terms(obs, (4, 3)))
    else:
        args, G, _, _ = _delay_case(16, 6, 12, 64, 1, oracle=False)
        make, terms = (lambda: qc.Solver(*args)), (lambda: [G()])
    base = lib.qc_test_live_allocs()
    S = make()
    want = terms()
    ref = S.solve(want, kernel=3)
    S.close()
    fell = 0
    for n in range(1, 60):
        S = make()
        T = terms()
        lib.qc_test_fail_alloc(n)
        try:
            st = S.solve(T)
        except qc.QCError as e:
            assert e.code == qc.QC_ENOMEM
            lib.qc_test_fail_alloc(0)
            st = S.solve(terms())                        # the context still works
            assert st.n_iter_max == ref.n_iter_max
            S.close()
            assert lib.qc_test_live_allocs() == base
            continue
        lib.qc_test_fail_alloc(0)
        S.close()
        assert lib.qc_test_live_allocs() == base
        assert st.n_iter_max == ref.n_iter_max
        for a, c in zip(T, want):
            assert _rel(a.gains, c.gains) < TOL and np.array_equal(a.iters, c.iters)
        fell += st.acc_bytes > 0.9 * ref.acc_bytes
        if n > 40:
            break
    assert fell >= 2, fell


@pytest.mark.parametrize("kinds,n_time", [(("diag",), 1100), (("full", "diag"), 600), (("diag", "full"), 1100)])
def test_long_time_maps(kinds, n_time):
    """Time maps longer than the pass keeps in shared memory (512 integrations behind a full term, 1024
    elsewhere)."""
    obs = tmo._chain_obs(41, kinds, n_ant=3, n_time=n_time, n_chan=20, t_int=(50, n_time), f_int=(20, 10))
    out = []
    for kernel in (0, 3):
        S = qc.Solver.from_obs(obs)
        T = _terms(obs, (4, 4))
        st = S.solve(T, kernel=kernel)
        S.close()
        out.append((T, st.acc_bytes))
    assert out[0][1] < out[1][1]
    for a, b in zip(out[0][0], out[1][0]):
        assert _rel(a.gains, b.gains) < TOL
