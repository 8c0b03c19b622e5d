"""Edge sizes of the kernels behind the default solves, and of the sample counts, the residual and
flagging passes and the warm-start network.

Tolerances.  A solve is compared after a fixed number of iterations from one start (no
convergence test in between).  The sums carry about 1e-7 of relative error whatever their length,
a step multiplies it by the condition of a 2x2 block (below 10 with the sample counts used here),
and four steps add up: 4e-6, and the fixed term enters rounded to float32.  2e-5 leaves a
factor of four.  Delay parameters: the gains at a channel carry the delay's error times 2 pi nu,
about 10, over a lever arm of the band of 0.25 in relative terms: 1e-4, as for the other delay
tests.  Flags, counts and unit-gain residual decisions are exact."""
import numpy as np
import pytest

import oracle as O
import test_gpu_batch as tb
import test_gpu_delay as td
import test_gpu_mad as tm
import test_gpu_moments as tmo
from oracle import mlp as OM
from oracle.mad_flag import mad_flag, mad_flag_per_baseline
from paper_2412_10072_gb300 import qc, synth

pytestmark = pytest.mark.gpu

TOL = 2e-5
ITERS = 4


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-30))


@pytest.mark.parametrize("n_ant,n_chan", [(2, 31), (33, 33), (65, 1)])
@pytest.mark.parametrize("kinds", [("diag",), ("phase",), ("full",), ("diag", "phase"), ("full", "diag"),
                                   ("diag", "full")])
def test_default_solve_from_sums(kinds, n_ant, n_chan):
    """Every form of the sums (plain diagonal, diagonal with a full term to the left, full; the
    other term to the right or left, per channel or per time) against the oracle, and with the
    FP16 model against the iterations on the samples.  One and several chunks, a ragged last
    chunk, one pair and more pairs than a warp has lanes."""
    n_time = 24
    obs = tmo._chain_obs(800 + n_ant, kinds, n_ant=n_ant, n_time=n_time, n_chan=n_chan,
                         t_int=(12 if n_chan > 1 else 24, 24), f_int=(max(1, n_chan // 2), 1))
    rng = np.random.default_rng(n_chan)
    start = [tmo._start(s, rng) for s in obs.terms]

    def gpu(kernel, **kw):
        S = qc.Solver.from_obs(obs, **kw)
        T = [qc.Term.from_spec(s, n_ant, gains=g, max_iter=ITERS, tol=0.0) for s, g in zip(obs.terms, start)]
        st = S.solve(T, kernel=kernel)
        S.close()
        return T, st

    P = O.OracleProblem.from_obs(obs)
    ot = [O.OracleTerm.from_spec(s, n_ant, params=g.astype(np.float64 if s.kind == "phase" else np.complex128),
                                 max_iter=ITERS, tol=0.0) for s, g in zip(obs.terms, start)]
    O.solve(P, ot, damping_mode=1)
    gt, st = gpu(0)
    assert st.acc_bytes < gpu(3)[1].acc_bytes        # one pass and the sums against a pass an iteration
    for g, o in zip(gt, ot):
        assert _rel(np.asarray(g.gains, dtype=o.params.dtype), o.params) < TOL
        assert np.array_equal(g.gain_flags, o.gain_flags)
    h, s16 = gpu(0, model_fp16=True)
    r, r16 = gpu(3, model_fp16=True)
    assert s16.acc_bytes <= r16.acc_bytes             # equal where the FP16 rows are too short for sums to pay
    for a, b in zip(h, r):
        assert _rel(a.gains, b.gains) < TOL
        assert np.array_equal(a.gain_flags, b.gain_flags)


@pytest.mark.parametrize("variant", ["right diag", "left diag", "right full", "two intervals", "missing rows", "fp16"])
def test_delay_term_from_products(variant):
    """The delay iterations on per-(interval, pair, channel) products, in every chain that they
    accept, on a grid of times and pairs with holes, and with the FP16 model."""
    other = {"right diag": "B", "left diag": "B", "right full": "G"}.get(variant)
    pb = td._problem(77, n_fint=2 if variant == "two intervals" else 1, other=other)
    if variant == "missing rows":
        keep = np.random.default_rng(3).random(pb["ant1"].size) < 0.8
        for k in ("data", "model", "weight", "flag", "ant1", "ant2", "tidx"):
            pb[k] = pb[k][keep]
    ot, n = td._oracle_terms(pb, max_iter=ITERS, tol=0.0)
    P = td._oracle_problem(pb)
    flip = variant in ("left diag", "right full")      # the other order of the chain than the problem's own
    if flip:
        ot, n = ot[::-1], 1 - n
    O.solve_term(P, ot, n, damping_mode=1)
    out = []
    for kernel in (0, 2):
        S = qc.Solver(pb["data"], pb["model"], pb["weight"], pb["flag"], pb["ant1"], pb["ant2"], pb["tidx"], td.N_ANT,
                      td.N_TIME, model_fp16=variant == "fp16")
        gt, _ = td._gpu_terms(pb, max_iter=ITERS, tol=0.0)
        if flip:
            gt = gt[::-1]
        S.solve(gt, kernel=kernel)
        S.close()
        out.append((td._referenced(gt[n].gains, pb), np.array(gt[n].gain_flags)))
    assert np.abs(out[0][0] - out[1][0]).max() <= td.GAIN_TOL
    assert np.array_equal(out[0][1], out[1][1])
    if variant != "fp16":
        assert np.abs(out[0][0] - td._referenced(ot[n].params, pb)).max() <= td.GAIN_TOL
        assert np.array_equal(out[0][1], ot[n].gain_flags)


@pytest.mark.parametrize("m16", [False, True])
def test_batch_from_sums(m16):
    """The batch's default solve against its iterations on the samples: 2 to 70 antennas, a pair of
    more samples than one segment, both orientations in one problem, an incomplete grid,
    autocorrelations, a fully flagged problem."""
    shapes = [(1, 2, 300, 40, 0.1), (2, 33, 3, 5, 0.2), (3, 65, 2, 7, 0.1), (4, 70, 3, 3, 0.0), (5, 8, 4, 33, 0.3),
              (6, 5, 4, 1, 0.0)]
    b = synth.make_batch(shapes)
    rng = np.random.default_rng(0)
    row_of = np.concatenate([np.repeat(np.arange(b.row_offset[i], b.row_offset[i + 1]), b.n_chan[i])
                             for i in range(b.n_prob)])
    swap = (rng.random(b.ant1.size) < 0.3)
    swap[b.row_offset[5]:] = False
    b.ant1, b.ant2 = np.where(swap, b.ant2, b.ant1), np.where(swap, b.ant1, b.ant2)
    s = swap[row_of]
    for name in ("data", "model"):
        x = np.array(getattr(b, name))
        x[s] = np.conj(x[s][:, [0, 2, 1, 3]])
        setattr(b, name, x)
    w = np.array(b.weight)
    w[s] = w[s][:, [0, 2, 1, 3]]
    b.weight = w
    r4 = int(b.row_offset[4])
    b.ant2[r4 + 3] = b.ant1[r4 + 3]                    # an autocorrelation; its pair misses a time
    b.flag = np.array(b.flag)
    b.flag[b.vis_offset[5]:] = 1
    S = tb.solver_of(b, model_fp16=m16)
    g0, f0, i0, st0 = S.solve(max_iter=ITERS, tol=0.0)
    g1, f1, i1, st1 = S.solve(max_iter=ITERS, tol=0.0, threads=256)
    S.close()
    assert st0.bytes < st1.bytes                       # one pass and the sums against a pass an iteration
    assert np.array_equal(f0, f1) and np.array_equal(i0, i1)
    assert _rel(g0, g1) < TOL


@pytest.mark.parametrize("n_chan", [1, 33, 65])
@pytest.mark.parametrize("n_terms", [1, 3])
def test_residual_and_flags(n_chan, n_terms):
    """With unit gains the residual is the float32 difference: the flags equal the oracle's bit for
    bit, the residual to an ulp of the data; rows of one, one and a bit, and two chunks and a bit."""
    pb = tm._problem(40 + n_chan, n_chan=n_chan)
    S = qc.Solver(pb["data"], pb["model"], pb["weight"], pb["flag"], pb["ant1"], pb["ant2"], pb["tidx"], pb["n_ant"],
                  pb["n_time"])
    T = [tm._unit_term(pb) for _ in range(n_terms)]
    got, n = S.mad_flag(T, threshold=4.0)
    got_b, n_b = S.mad_flag(T, threshold=4.0, per_baseline=True)
    _, r = S.residual(T, want_resid=True)
    S.close()
    d = pb["data"] - pb["model"]
    want, (_, _, n_want) = mad_flag(d, pb["weight"], pb["flag"], pb["ant1"], pb["ant2"], threshold=4.0)
    want_b, nb_want = mad_flag_per_baseline(d, pb["weight"], pb["flag"], pb["ant1"], pb["ant2"], threshold=4.0)
    np.testing.assert_array_equal(got, want)
    np.testing.assert_array_equal(got_b, want_b)
    assert n == n_want and n_b == nb_want
    ot = [O.OracleTerm("diag", np.zeros(pb["n_time"], np.int32), np.zeros(n_chan, np.int32), 1, 1, pb["n_ant"])]
    P = O.OracleProblem(pb["data"], pb["model"], pb["weight"], pb["flag"], pb["ant1"], pb["ant2"], pb["tidx"],
                        pb["n_ant"], pb["n_time"])
    _, r_o = O.residual(P, ot, want_resid=True)
    assert np.abs(r - r_o).max() <= 2.0 ** -23 * np.abs(pb["data"]).max()


@pytest.mark.parametrize("n_ant,n_time,n_chan,f_int", [(3, 2, 1, 1), (40, 60, 70, 7), (65, 40, 33, 1), (65, 40, 64, 64)])
def test_sample_counts(n_ant, n_time, n_chan, f_int):
    """The throughput and byte accounting counts every sample of an interval once: units of one row
    and of many, with time intervals that end inside a unit, channels of one and of several
    intervals in a chunk, autocorrelations left out."""
    rng = np.random.default_rng(n_ant)
    p, q = np.triu_indices(n_ant)
    ant1, ant2 = np.tile(p, n_time).astype(np.int32), np.tile(q, n_time).astype(np.int32)
    tidx = np.repeat(np.arange(n_time, dtype=np.int32), p.size)
    shp = (ant1.size, n_chan, 4)
    one = np.ones(shp, np.complex64)
    flag = (rng.random(shp[:2]) < 0.3).astype(np.uint8)
    S = qc.Solver(one, one, np.ones(shp, np.float32), flag, ant1, ant2, tidx, n_ant, n_time)
    tm_, fm = synth.interval_map(n_time, 7), synth.interval_map(n_chan, f_int)
    T = qc.Term("diag", tm_, fm, int(tm_[-1]) + 1, int(fm[-1]) + 1, n_ant, max_iter=2, tol=0.0)
    st = S.solve([T], kernel=3)
    S.close()
    cross = ant1 != ant2
    assert st.vis_iters == 2 * int(cross.sum()) * n_chan
    assert st.acc_bytes == 2 * int(cross.sum()) * n_chan + 2 * 80 * int((flag[cross] == 0).sum())


@pytest.mark.parametrize("n", [1, 31, 33, 4097])
def test_network_tiles(n):
    """Forward and backward of the warm-start network at the edges of its 32-row tiles, with the
    tolerances of its other tests."""
    torch = pytest.importorskip("torch")
    from paper_2412_10072_gb300 import warmstart as ws
    rng = np.random.default_rng(n)
    flat = (OM.init(4) * 0.7).astype(np.float32)
    x = rng.standard_normal((n, 10)).astype(np.float32)
    t = rng.standard_normal((n, 4)).astype(np.float32)
    net = ws.MLP(torch.from_numpy(flat))
    xd, t_d = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    z = torch.empty((n, 384), dtype=torch.float32, device="cuda")
    y = net.forward(xd, z)
    grad = torch.zeros(OM.NPARAM, dtype=torch.float32, device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    assert ws._lib().qc_mlp_backward(net.params.data_ptr(), xd.data_ptr(), z.data_ptr(), y.data_ptr(), t_d.data_ptr(),
                                     n, grad.data_ptr(), loss.data_ptr(), None) == 0
    torch.cuda.synchronize()
    f64 = flat.astype(np.float64)
    y_want, _ = OM.forward(f64, x.astype(np.float64))
    assert _rel(y.cpu().numpy(), y_want) < 1e-5
    assert _rel(grad.cpu().numpy(), OM.backward(f64, x.astype(np.float64), t.astype(np.float64))) < 1e-4
