"""What is timed of this framework: calibration solves, residuals, flagging and warm-start training.

Each case is one call (or the two or three calls in a row) that a user's program makes through the
public entry points of ``paper_2412_10072_gb300``: ``qc.Solver`` (``solve``, ``residual``,
``mad_flag``), ``qc.BatchSolver.solve`` and ``warmstart.MLP.train_step``.  ``prepare`` makes an
observation on the GPU (point sources seen by an east-west array, true gains, noise, flags) and the
staged ``Solver`` or ``BatchSolver`` that such a program keeps; ``run`` builds the terms from their
initial estimates and solves.

Outputs are the gains, the gain flags, chi^2, residuals and flags.  Iteration counts are left out: an
interval stops when its relative change falls below 1e-6, which is within the rounding of the
complex64 data, so the count of an interval on the edge differs from run to run.

``exact`` is the same method in 64 bits with plain torch: for a solved term, the sums of products of
data and model over each (interval, antenna pair), then the iterations on them.
"""
import math

import numpy as np
import torch

from paper_2412_10072_gb300 import qc, warmstart

DEV = "cuda"
C_LIGHT = 299792458.0
MAX_ITER, TOL = 20, 1e-6
EXACT_SAMPLES = 9e7          # larger observations take exact() over 20 seconds


def listed():
    return [
        # the smallest call: one short scan of a 7-antenna array, a diagonal term, then its chi^2;
        # latency and launches count
        {"name": "small_diag", "op": "solve", "n_ant": 7, "n_time": 60, "n_chan": 16, "chain": "diag:4x4",
         "epochs": 1, "fp16": False, "moments": False, "chi2": True},
        # an ordinary single-term solve with ragged sizes: intervals of 5 x 17 leave remainders in
        # time and frequency, 131 channels are no multiple of a warp
        {"name": "ragged_diag", "op": "solve", "n_ant": 27, "n_time": 61, "n_chan": 131, "chain": "diag:5x17",
         "epochs": 1, "fp16": False, "moments": False, "chi2": False},
        # the flagship: full-Jones G per integration, then the diagonal bandpass B over all times
        {"name": "large_GB", "op": "solve", "n_ant": 64, "n_time": 300, "n_chan": 512,
         "chain": "full:1x512 band:300x1", "epochs": 3, "fp16": False, "moments": False, "chi2": False},
        # the same chain with the model held as float16 pairs
        {"name": "fp16_GB", "op": "solve", "n_ant": 64, "n_time": 75, "n_chan": 512,
         "chain": "full:1x512 band:75x1", "epochs": 2, "fp16": True, "moments": False, "chi2": False},
        # the same chain with qc_opts.moments (solve from sums) asked for
        {"name": "sums_GB", "op": "solve", "n_ant": 64, "n_time": 85, "n_chan": 512,
         "chain": "full:1x512 band:85x1", "epochs": 3, "fp16": False, "moments": True, "chi2": False},
        # a residual delay and phase per integration, from the estimate of an earlier solve
        {"name": "delay_K", "op": "solve", "n_ant": 64, "n_time": 75, "n_chan": 512, "chain": "delay:1x512",
         "epochs": 1, "fp16": False, "moments": False, "chi2": False},
        # the KdE chain: K over both directions, then the direction-dependent dE
        {"name": "kde_two_dirs", "op": "solve", "n_ant": 64, "n_time": 64, "n_chan": 512,
         "chain": "delay:1x512 dddiag:16x128", "epochs": 2, "fp16": False, "moments": False, "chi2": False},
        # thousands of small uneven intervals in one call
        {"name": "batch_uneven", "op": "batch", "n_prob": 1024, "max_ant": 64, "max_time": 16, "max_chan": 64,
         "shape_seed": 1000, "moments": False},
        # the same kind of batch, solved from per-baseline sums
        {"name": "batch_sums", "op": "batch", "n_prob": 512, "max_ant": 64, "max_time": 16, "max_chan": 64,
         "shape_seed": 2000, "moments": True},
        # residual visibilities and chi^2 of a calibrated observation, odd channel count
        {"name": "residual_out", "op": "residual", "n_ant": 64, "n_time": 60, "n_chan": 509,
         "chain": "full:1x509 band:60x1"},
        # flagging outliers of the calibrated residual, over all baselines
        {"name": "mad_flag", "op": "mad", "n_ant": 64, "n_time": 75, "n_chan": 512, "chain": "full:1x512 band:75x1",
         "per_baseline": False},
        # one training step of the warm-start network on a mini-batch
        {"name": "mlp_train", "op": "mlp", "rows": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["single", "chain", "chain", "delay", "kde", "batch", "batch", "residual", "mad", "mlp"])
    if op == "mlp":
        return {"op": "mlp", "rows": _log_int(rng, 256, 65536)}
    if op == "batch":
        return {"op": "batch", "n_prob": _log_int(rng, 8, 1024), "max_ant": rng.randint(9, 64),
                "max_time": rng.randint(2, 16), "max_chan": rng.randint(4, 64),
                "shape_seed": rng.randrange(1, 1 << 20), "moments": rng.random() < 0.4}
    n_ant, n_chan = rng.randint(7, 64), _log_int(rng, 16, 512)
    cap = 3e7 if op in ("delay", "kde") else 6e7
    most = max(4, min(150, int(cap / (n_ant * (n_ant - 1) / 2 * n_chan))))
    n_time = _log_int(rng, 4, most)
    if op == "delay":
        n_chan = max(n_chan, 48)
        return {"op": "solve", "n_ant": n_ant, "n_time": n_time, "n_chan": n_chan,
                "chain": "delay:%dx%d" % (rng.choice([1, 1, 2]), n_chan), "epochs": 1, "fp16": False, "moments": False,
                "chi2": False}
    if op == "kde":
        n_chan = max(n_chan, 48)
        return {"op": "solve", "n_ant": n_ant, "n_time": n_time, "n_chan": n_chan,
                "chain": "delay:1x%d dddiag:%dx%d" % (n_chan, rng.randint(2, 16), rng.randint(16, 128)), "epochs": 2,
                "fp16": False, "moments": False, "chi2": False}
    if op == "single":
        # enough samples a baseline for the solve to be well conditioned
        kind = rng.choice(["diag", "diag", "phase", "full"])
        chain = "%s:%dx%d" % (kind, rng.randint(2, 8), rng.randint(4, 40))
        return {"op": "solve", "n_ant": n_ant, "n_time": n_time, "n_chan": n_chan, "chain": chain, "epochs": 1,
                "fp16": kind != "phase" and rng.random() < 0.2, "moments": rng.random() < 0.25,
                "chi2": rng.random() < 0.5}
    chain = "%s:1x%d band:%dx1" % (rng.choice(["full", "full", "diag"]), n_chan, n_time)
    if op == "residual":
        return {"op": "residual", "n_ant": n_ant, "n_time": n_time, "n_chan": n_chan, "chain": chain}
    if op == "mad":
        return {"op": "mad", "n_ant": n_ant, "n_time": n_time, "n_chan": n_chan, "chain": chain,
                "per_baseline": rng.random() < 0.4}
    fp16 = rng.random() < 0.25
    return {"op": "solve", "n_ant": n_ant, "n_time": max(8, n_time), "n_chan": max(32, n_chan),
            "chain": "%s:1x%d band:%dx1" % (rng.choice(["full", "full", "diag"]), max(32, n_chan), max(8, n_time)),
            "epochs": rng.randint(1, 3), "fp16": fp16, "moments": not fp16 and rng.random() < 0.3, "chi2": False}


# ---------------------------------------------------------------------------
# observations
# ---------------------------------------------------------------------------

def _terms(case):
    """The chain as dicts: kind, interval maps and counts."""
    out = []
    for word in case["chain"].split():
        kind, size = word.split(":")
        dt, df = (int(v) for v in size.split("x"))
        nt, nf = case["n_time"], case["n_chan"]
        out.append({"kind": kind, "t_map": (np.arange(nt) // dt).astype(np.int32),
                    "f_map": (np.arange(nf) // df).astype(np.int32), "n_tint": -(-nt // dt), "n_fint": -(-nf // df)})
    return out


def _freqs(n_chan):
    return 0.856e9 + (np.arange(n_chan) + 0.5) * (0.856e9 / n_chan)


def _truth(term, n_ant, rng):
    """True gains of a term [n_tint][n_fint][n_ant][4] (delay: parameters; dddiag: [..][n_ant][2][4])."""
    nt, nf, kind = term["n_tint"], term["n_fint"], term["kind"]
    if kind == "delay":
        k = np.zeros((nt, nf, n_ant, 4))
        k[..., 0::2] = rng.uniform(-np.pi, np.pi, (nt, nf, n_ant, 2))
        k[..., 1::2] = rng.normal(0, 1, (1, 1, n_ant, 2)) + 0.05 * np.cumsum(rng.normal(0, 1, (nt, nf, n_ant, 2)), 0)
        return k
    if kind == "dddiag":
        amp = 1 + np.array([0.02, 0.1])[:, None] * rng.standard_normal((nt, nf, n_ant, 2, 2))
        ph = np.array([0.05, 1.0])[:, None] * rng.uniform(-np.pi, np.pi, (nt, nf, n_ant, 2, 2))
        g = np.zeros((nt, nf, n_ant, 2, 4), complex)
        g[..., 0::3] = amp * np.exp(1j * ph)
        return g
    g = np.zeros((nt, nf, n_ant, 4), complex)
    if kind == "phase":
        return rng.uniform(-1, 1, (1, 1, n_ant, 2)) + 0.1 * rng.standard_normal((nt, nf, n_ant, 2))
    if kind == "band":       # smooth bandpass
        x = np.arange(nf)[:, None, None] / max(1, nf)
        ph = sum(rng.uniform(0, 0.5, (1, n_ant, 2)) * np.cos(2 * np.pi * (j + 1) * x + rng.uniform(0, 6.28, (1, n_ant, 2)))
                 for j in range(4))
        g[..., 0::3] = rng.normal(1, 0.1, (1, nf, n_ant, 2)) * np.exp(1j * ph[None])
        return g
    ph = rng.uniform(-np.pi, np.pi, (1, 1, n_ant, 2)) + 0.05 * np.cumsum(rng.standard_normal((nt, nf, n_ant, 2)), 0)
    g[..., 0::3] = (1 + 0.05 * rng.standard_normal((nt, nf, n_ant, 2))) * np.exp(1j * ph)
    if kind == "full":
        g[..., 1:3] = 0.05 * (rng.standard_normal((nt, nf, n_ant, 2)) + 1j * rng.standard_normal((nt, nf, n_ant, 2)))
    return g


def _per_channel(term, values, nu, ant, t):
    """2x2 Jones [n][n_chan][(dir)][4] (complex128 on the GPU) of antennas `ant` at times `t`."""
    ti = torch.as_tensor(term["t_map"], device=DEV, dtype=torch.long)[t]
    fm = torch.as_tensor(term["f_map"], device=DEV, dtype=torch.long)
    v = torch.as_tensor(values, device=DEV)
    g = v[ti[:, None], fm[None, :], ant[:, None]]
    if term["kind"] == "delay":
        ph = g[..., 0::2] + 2 * math.pi * g[..., 1::2] * nu[None, :, None]
        g = torch.polar(torch.ones_like(ph), ph)
    elif term["kind"] == "phase":
        g = torch.polar(torch.ones_like(g), g)
    if g.shape[-1] == 2:
        z = torch.zeros_like(g[..., 0])
        g = torch.stack([g[..., 0], z, z, g[..., 1]], -1)
    return g.to(torch.complex128)


def _mul(a, b):
    """2x2 products of [..., 4] arrays."""
    return torch.stack([a[..., 0] * b[..., 0] + a[..., 1] * b[..., 2], a[..., 0] * b[..., 1] + a[..., 1] * b[..., 3],
                        a[..., 2] * b[..., 0] + a[..., 3] * b[..., 2], a[..., 2] * b[..., 1] + a[..., 3] * b[..., 3]], -1)


def _herm(a):
    return torch.stack([a[..., 0], a[..., 2], a[..., 1], a[..., 3]], -1).conj()


def _sky(rng, n_src, flux=None):
    r, a = np.deg2rad(1.0) * np.sqrt(rng.uniform(0, 1, n_src)), rng.uniform(0, 2 * np.pi, n_src)
    s = rng.uniform(0.1, 1.0, n_src) if flux is None else np.full(n_src, flux)
    q, u = 0.05 * rng.standard_normal(n_src), 0.05 * rng.standard_normal(n_src)
    return {"l": r * np.cos(a), "m": r * np.sin(a), "coef": np.stack([s * (1 + q), s * u, s * (1 - q)], 1)}


def _predict(delay, nu, coef):
    """[n][n_chan][4] complex64 of sources with the given delays [n][src] (s), frequencies [n_chan] (Hz)."""
    turns = delay[:, None, :] * nu[None, :, None]
    ph = ((turns - torch.round(turns)) * (-2 * math.pi)).float()
    v = torch.polar(torch.ones_like(ph), ph) @ coef
    return torch.stack([v[..., 0], v[..., 1], v[..., 1], v[..., 2]], -1)


def _uvw(x, p, q, ha):
    b = x[q] - x[p]
    dec = math.radians(-30.0)
    return b * np.cos(ha), b * np.sin(ha) * math.sin(dec), -b * np.sin(ha) * math.cos(dec)


def _delays(uvw, sky):
    n = np.sqrt(1 - sky["l"] ** 2 - sky["m"] ** 2) - 1
    u, v, w = (torch.as_tensor(c, device=DEV, dtype=torch.float64)[:, None] for c in uvw)
    s = [torch.as_tensor(c, device=DEV, dtype=torch.float64)[None] for c in (sky["l"], sky["m"], n)]
    return (u * s[0] + v * s[1] + w * s[2]) / C_LIGHT


def _observation(case, seed):
    """data, model, weight, flag of a scan on the GPU, its row metadata, and the true gains."""
    rng = np.random.default_rng([seed, 71])
    gen = torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 13)
    n_ant, n_time, n_chan = case["n_ant"], case["n_time"], case["n_chan"]
    terms = _terms(case)
    n_dir = 2 if "dddiag" in case["chain"] else 1
    p, q = (v.astype(np.int32) for v in np.triu_indices(n_ant, 1))
    n_bl = p.size
    x = np.sort(rng.uniform(0, 125.0 * n_ant, n_ant))
    has = np.linspace(-0.5, 0.5, n_time)
    nu = torch.as_tensor(_freqs(n_chan), device=DEV)
    skies = [_sky(rng, 8)] + ([_sky(rng, 1, 5.0)] if n_dir == 2 else [])
    coefs = [torch.as_tensor(s["coef"], device=DEV).to(torch.complex64) for s in skies]
    truth = [_truth(t, n_ant, rng) for t in terms]
    n_row, sigma = n_time * n_bl, 0.05
    data = torch.empty((n_row, n_chan, 4), dtype=torch.complex64, device=DEV)
    model = torch.empty((n_row, n_chan) + ((2,) if n_dir == 2 else ()) + (4,), dtype=torch.complex64, device=DEV)
    weight = torch.empty((n_row, n_chan, 4), dtype=torch.float32, device=DEV).uniform_(0.5, 1.5, generator=gen)
    flag = (torch.rand((n_row, 1), device=DEV, generator=gen) < 0.1).expand(n_row, n_chan).to(torch.uint8).contiguous()
    pd, qd = (torch.as_tensor(v, device=DEV, dtype=torch.long) for v in (p, q))
    step = max(1, int(4e6 / (n_bl * n_chan)))
    for t0 in range(0, n_time, step):
        t1 = min(n_time, t0 + step)
        ts = np.arange(t0, t1)
        uvw = _uvw(x, np.tile(p, ts.size), np.tile(q, ts.size), np.repeat(has[ts], n_bl))
        tt = torch.arange(t0, t1, device=DEV).repeat_interleave(n_ant)
        aa = torch.arange(n_ant, device=DEV).repeat(ts.size)
        rows = slice(t0 * n_bl, t1 * n_bl)
        ip = (torch.arange(ts.size, device=DEV)[:, None] * n_ant + pd[None]).reshape(-1)
        iq = (torch.arange(ts.size, device=DEV)[:, None] * n_ant + qd[None]).reshape(-1)
        jones = [_per_channel(t, v, nu / 1e9, aa, tt).to(torch.complex64) for t, v in zip(terms, truth)]
        d = 0
        for k, (sky, coef) in enumerate(zip(skies, coefs)):
            m = _predict(_delays(uvw, sky), nu, coef)
            (model[rows, :, k] if n_dir == 2 else model[rows]).copy_(m)
            c = None
            for t, j in zip(terms, jones):
                j = j[:, :, k] if t["kind"] == "dddiag" else j
                c = j if c is None else _mul(c, j)
            d = d + _mul(_mul(c[ip], m), _herm(c[iq]))
        noise = torch.randn((t1 - t0) * n_bl, n_chan, 4, 2, device=DEV, generator=gen)
        data[rows] = d + torch.view_as_complex(noise) * sigma
    return {"data": data, "model": model, "weight": weight, "flag": flag, "ant1": np.tile(p, n_time),
            "ant2": np.tile(q, n_time), "time": np.repeat(np.arange(n_time, dtype=np.int32), n_bl), "terms": terms,
            "truth": truth, "start": _start(terms, truth, n_ant, rng, case["op"])}


def _start(terms, truth, n_ant, rng, op):
    """Initial estimates: unit gains; a delay term starts from an earlier solve's estimate; residuals
    and flagging take solved gains."""
    out = []
    for t, v in zip(terms, truth):
        if op != "solve":
            out.append(v.astype(np.complex64))
        elif t["kind"] == "delay":
            off = np.stack([rng.normal(0, 0.1, v[..., 0].shape), rng.normal(0, 0.02, v[..., 0].shape)] * 2, -1)
            out.append((v + off).astype(np.float32))
        else:
            out.append(None)
    return out


def _solver_terms(s):
    case, out = s["case"], []
    for t, g in zip(s["terms"], s["start"]):
        kind = {"band": "diag", "dddiag": "diag"}.get(t["kind"], t["kind"])
        dd = t["kind"] == "dddiag"
        out.append(qc.Term(kind, t["t_map"], t["f_map"], t["n_tint"], t["n_fint"], case["n_ant"], gains=g,
                           solve=case["op"] == "solve", max_iter=MAX_ITER, tol=TOL, dd=dd, n_dir=2 if dd else 1,
                           chan_freq=_freqs(case["n_chan"]) / 1e9 if kind == "delay" else None))
    return out


# ---------------------------------------------------------------------------
# batches
# ---------------------------------------------------------------------------

def _shapes(case):
    r = np.random.default_rng(case["shape_seed"])
    n = case["n_prob"]
    return (r.integers(7, case["max_ant"] + 1, n), r.integers(1, case["max_time"] + 1, n),
            r.integers(1, case["max_chan"] + 1, n), r.uniform(0, 0.5, n))


def _batch(case, seed):
    rng = np.random.default_rng([seed, 72])
    gen = torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 17)
    na, nt, nc, frac = _shapes(case)
    n_prob, n_src = case["n_prob"], 5
    a1, a2, uvw, n_rows, skies = [], [], [], [], []
    for i in range(n_prob):
        p, q = (v.astype(np.int32) for v in np.triu_indices(na[i], 1))
        x = np.sort(rng.uniform(0, 1000.0, na[i]))
        a1.append(np.tile(p, nt[i]))
        a2.append(np.tile(q, nt[i]))
        uvw.append(np.stack(_uvw(x, a1[-1], a2[-1], np.repeat(rng.uniform(-0.3, 0.3) + 0.002 * np.arange(nt[i]), p.size))))
        n_rows.append(a1[-1].size)
        skies.append(_sky(rng, n_src))
    n_rows = np.array(n_rows)
    row_off = np.concatenate([[0], np.cumsum(n_rows)]).astype(np.int64)
    vis_off = np.concatenate([[0], np.cumsum(n_rows * nc)]).astype(np.int64)
    gain_off = np.concatenate([[0], np.cumsum(na)]).astype(np.int64)
    ant1, ant2 = np.concatenate(a1), np.concatenate(a2)
    g = (1 + 0.05 * rng.standard_normal((gain_off[-1], 2))) * np.exp(1j * rng.uniform(-np.pi, np.pi, (gain_off[-1], 2)))
    gt = torch.as_tensor(g, device=DEV).to(torch.complex64)
    u = torch.as_tensor(np.concatenate(uvw, 1), device=DEV)
    lmn = torch.as_tensor(np.stack([np.stack([s["l"], s["m"], np.sqrt(1 - s["l"] ** 2 - s["m"] ** 2) - 1])
                                    for s in skies]), device=DEV)
    coef = torch.as_tensor(np.stack([s["coef"] for s in skies]), device=DEV).to(torch.complex64)
    prob_of_row = torch.as_tensor(np.repeat(np.arange(n_prob), n_rows), device=DEV)
    delay = torch.einsum("cr,rck->rk", u, lmn[prob_of_row]) / C_LIGHT
    ncd = torch.as_tensor(nc, device=DEV)
    rows_v0 = torch.as_tensor(np.repeat(vis_off[:-1] - row_off[:-1] * nc, n_rows), device=DEV)
    row_vis0 = rows_v0 + torch.arange(row_off[-1], device=DEV) * ncd[prob_of_row]
    gp = torch.as_tensor(ant1, device=DEV, dtype=torch.long) + torch.as_tensor(gain_off[:-1], device=DEV)[prob_of_row]
    gq = torch.as_tensor(ant2, device=DEV, dtype=torch.long) + torch.as_tensor(gain_off[:-1], device=DEV)[prob_of_row]
    nv = int(vis_off[-1])
    data = torch.empty((nv, 4), dtype=torch.complex64, device=DEV)
    model = torch.empty((nv, 4), dtype=torch.complex64, device=DEV)
    weight = torch.empty((nv, 4), dtype=torch.float32, device=DEV).uniform_(0.5, 1.5, generator=gen)
    flag = torch.empty(nv, dtype=torch.uint8, device=DEV)
    fr = torch.as_tensor(frac, device=DEV, dtype=torch.float32)
    n_row, at, step = int(row_off[-1]), 0, 1 << 17
    while at < n_row:
        end = min(n_row, at + step)
        reps = ncd[prob_of_row[at:end]]
        v0 = int(row_vis0[at])
        row = torch.repeat_interleave(torch.arange(at, end, device=DEV), reps)
        v1 = v0 + row.numel()
        ch = torch.arange(v0, v1, device=DEV) - row_vis0[row]
        turns = delay[row] * (1.4e9 + 1e6 * ch.double())[:, None]
        ph = ((turns - torch.round(turns)) * (-2 * math.pi)).float()
        m = torch.einsum("vk,vkc->vc", torch.polar(torch.ones_like(ph), ph), coef[prob_of_row[row]])
        m = torch.stack([m[:, 0], m[:, 1], m[:, 1], m[:, 2]], 1)
        G, H = gt[gp[row]], gt[gq[row]].conj()
        outer = torch.stack([G[:, 0] * H[:, 0], G[:, 0] * H[:, 1], G[:, 1] * H[:, 0], G[:, 1] * H[:, 1]], 1)
        noise = torch.randn(v1 - v0, 4, 2, device=DEV, generator=gen)
        model[v0:v1] = m
        data[v0:v1] = outer * m + 0.01 * torch.view_as_complex(noise)
        flag[v0:v1] = (torch.rand(v1 - v0, device=DEV, generator=gen) < fr[prob_of_row[row]]).to(torch.uint8)
        at = end
    return {"data": data, "model": model, "weight": weight, "flag": flag, "ant1": ant1, "ant2": ant2,
            "row_off": row_off, "vis_off": vis_off, "n_chan": nc.astype(np.int32), "n_ant": na.astype(np.int32),
            "prob_of_row": prob_of_row, "n_rows": n_rows}


# ---------------------------------------------------------------------------
# the interface
# ---------------------------------------------------------------------------

def prepare(case, seed):
    if case["op"] == "mlp":
        gen = torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 19)
        n = case["rows"]
        net = warmstart.MLP.load(warmstart.DEFAULT_CHECKPOINT)
        # mini-batch rows as the features pass gives them: relative normal-equation terms, amplitude
        # ratios near 1 and the previous interval's gains; the targets have drifted from those
        x = torch.randn(n, 10, device=DEV, generator=gen)
        x[:, :2].abs_().mul_(0.5)
        x[:, 4:6].mul_(0.05).add_(1.0)
        y = x[:, 6:10] + 0.08 * torch.randn(n, 4, device=DEV, generator=gen)
        # the optimiser in mid-training
        net.m.normal_(0, 1e-4, generator=gen)
        net.v.uniform_(1e-7, 1e-6, generator=gen)
        net.step = 1000
        return {"case": case, "net": net, "x": x, "y": y.contiguous()}
    if case["op"] == "batch":
        b = _batch(case, seed)
        torch.cuda.synchronize()
        s = qc.BatchSolver(b["data"], b["model"], b["weight"], b["flag"], b["ant1"], b["ant2"], b["row_off"],
                           b["vis_off"], b["n_chan"], b["n_ant"])
        return {"case": case, "solver": s}
    o = _observation(case, seed)
    torch.cuda.synchronize()
    s = qc.Solver(o["data"], o["model"], o["weight"], o["flag"], o["ant1"], o["ant2"], o["time"], case["n_ant"],
                  case["n_time"], model_fp16=case.get("fp16", False))
    st = {"case": case, "solver": s, "terms": o["terms"], "start": o["start"]}
    if case["op"] == "residual":
        st["out"] = torch.empty((s.n_row, s.n_chan, 4), dtype=torch.complex64, device=DEV)
    if case["op"] == "mad":
        st["out"] = torch.empty((s.n_row, s.n_chan), dtype=torch.uint8, device=DEV)
    return st


def run(state):
    case = state["case"]
    if case["op"] == "mlp":
        net = state["net"]
        loss = net.train_step(state["x"], state["y"], lr=1e-4)
        return {"params": net.params, "grad": net.grad, "m": net.m, "v": net.v, "loss": loss.float()}
    if case["op"] == "batch":
        g, flags, _, _ = state["solver"].solve(max_iter=MAX_ITER, tol=TOL, moments=case["moments"])
        return {"gains": g, "flags": flags}
    s, terms = state["solver"], _solver_terms(state)
    if case["op"] == "residual":
        chi2, res = s.residual(terms, resid_out=state["out"])
        return {"chi2": chi2, "residual": res}
    if case["op"] == "mad":
        flags, n = s.mad_flag(terms, threshold=5.0, out=state["out"], per_baseline=case["per_baseline"])
        return {"flags": flags, "n": n}
    s.solve(terms, n_epochs=case["epochs"], moments=case["moments"])
    out = {}
    for i, t in enumerate(terms):
        out["gains%d" % i], out["flags%d" % i] = t.gains, t.gain_flags
    if case["chi2"]:
        out["chi2"] = s.residual(terms)
    return out


def _samples(case):
    if case["op"] == "batch":
        na, nt, nc, _ = _shapes(case)
        return int((na * (na - 1) // 2 * nt * nc).sum()), int(na.sum()) * 17
    n_vis = case["n_ant"] * (case["n_ant"] - 1) // 2 * case["n_time"] * case["n_chan"]
    gains = sum(t["n_tint"] * t["n_fint"] * case["n_ant"] *
                {"delay": 17, "phase": 9, "dddiag": 66}.get(t["kind"], 33) for t in _terms(case))
    return n_vis, gains


def work(case):
    """Every input once and every output once; a solve forms the normal equations of each solved term
    from the samples at least once an epoch (about 300 operations a sample for a full-Jones term, 120
    for a diagonal one, both antennas)."""
    if case["op"] == "mlp":
        n, p = case["rows"], 34948
        return {"bytes": 4 * (n * 14 + 8 * p), "flops": 6 * n * p}
    n, gains = _samples(case)
    if case["op"] == "batch":
        return {"bytes": 81 * n + gains, "flops": 120 * n}
    if case["op"] == "residual":
        return {"bytes": (81 + 32) * n + gains, "flops": 100 * n}
    if case["op"] == "mad":
        return {"bytes": 82 * n + gains, "flops": 110 * n}
    per = sum(300 if t["kind"] == "full" else 120 for t in _terms(case)) * case["epochs"]
    b = 81 + (32 if "dddiag" in case["chain"] else 0) - (16 if case["fp16"] else 0)
    return {"bytes": b * n + gains + (b * n if case["chi2"] else 0), "flops": per * n}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _iterate(kind, H_b, g0, nu=None):
    """Algorithm 1 on sums: H_b(g) -> per-antenna blocks JHJ [b][a][n][n] and b = J^H W d [b][a][n] at
    the gains; g: [b][a][n] (phase and delay: real parameters)."""
    g = g0.clone()
    flags = torch.zeros(g.shape[:2], dtype=torch.int8, device=DEV)
    active = torch.ones(g.shape[0], dtype=torch.bool, device=DEV)
    for k in range(1, MAX_ITER + 1):
        old = H_b.gains(g)
        H, r = H_b(g, old)
        tr = torch.diagonal(H, dim1=-2, dim2=-1).real.sum(-1)
        eye = torch.eye(H.shape[-1], dtype=H.dtype, device=DEV)
        ok = tr > 0
        inv = torch.linalg.inv_ex(torch.where(ok[..., None, None], H, eye))[0]
        cond = H.abs().sum(-2).amax(-1) * inv.abs().sum(-2).amax(-1)
        ok = ok & (cond <= 1e12)
        step = torch.where(ok[..., None], (inv @ r[..., None])[..., 0], torch.zeros_like(r))
        new = g + (1.0 if k % 2 else 0.5) * step
        g = torch.where(active[:, None, None], new, g)
        flags = torch.where(active[:, None], (~ok).to(torch.int8), flags)
        now = H_b.gains(g)
        num, den = H_b.norms(now - old), H_b.norms(now)
        delta = torch.where(den > 0, torch.sqrt(num / den), torch.zeros_like(den))
        active = active & ~(delta < TOL)
        if not bool(active.any()):
            break
    return g, flags


class _Full:
    """Sums of a full-Jones term: S[b][p][q][k][j][l][m][n][o] over dense antenna pairs."""

    def __init__(self, S, T):
        self.S, self.T = S, T

    def gains(self, g):
        return g

    def norms(self, x):
        return (x.abs() ** 2).sum((1, 2))

    def __call__(self, g, _):
        G = g.reshape(*g.shape[:2], 2, 2)
        W = torch.einsum("bqjm,bqjo->bqjmo", G, G.conj())
        blk = torch.einsum("bpqkjlmno,bqjmo->bpkln", self.S, W)
        r = torch.einsum("bpqkjlm,bqjm->bpkl", self.T, G) - torch.einsum("bpkln,bpkn->bpkl", blk, G)
        H = torch.zeros((*g.shape[:2], 4, 4), dtype=g.dtype, device=DEV)
        H[..., :2, :2], H[..., 2:, 2:] = blk[:, :, 0], blk[:, :, 1]
        return H, r.reshape(*g.shape[:2], 4)


class _Diag:
    """Sums of a diagonal (or phase-only) term: S[b][p][q][a][c][a'][c'] and T[b][p][q][a][c]."""

    def __init__(self, S, T, phase=False):
        self.S, self.T, self.phase = S, T, phase

    def gains(self, g):
        return torch.polar(torch.ones_like(g), g) if self.phase else g

    def norms(self, x):
        return (x.abs() ** 2).sum((1, 2))

    def __call__(self, _, g):
        W = torch.einsum("bqc,bqd->bqcd", g, g.conj())
        H = torch.einsum("bpqacxd,bqcd->bpax", self.S, W)
        r = torch.einsum("bpqac,bqc->bpa", self.T, g) - torch.einsum("bpax,bpx->bpa", H, g)
        if self.phase:
            H = 2 * (g.conj()[..., :, None] * g[..., None, :] * H).real
            r = 2 * (g.conj() * r).imag
        return H, r


class _Delay:
    """A delay term from per-channel sums S[t][ch][p][q][k][j] (real), T (complex); parameters [t][a][4]."""

    def __init__(self, S, T, nu, f_map, n_fint):
        self.S, self.T, self.om = S, T, 2 * math.pi * nu
        self.f_map, self.n_fint = f_map, n_fint

    def gains(self, g):                     # [t*f][a][4] -> [t][ch][a][2]
        v = g.reshape(-1, self.n_fint, *g.shape[1:])[:, self.f_map]
        ph = v[..., 0::2] + v[..., 1::2] * self.om[:, None, None]
        return torch.polar(torch.ones_like(ph), ph)

    def _bins(self, x):                     # sum channels into intervals: [t][ch][...] -> [t*f][...]
        z = torch.zeros((x.shape[0], self.n_fint) + x.shape[2:], dtype=x.dtype, device=DEV)
        return z.index_add_(1, self.f_map, x).flatten(0, 1)

    def norms(self, x):
        return self._bins((x.abs() ** 2).sum((2, 3)))

    def __call__(self, _, g):
        h = self.S.sum((3, 5))              # |g_q| = 1
        r = torch.einsum("tcpqkj,tcqj->tcpk", self.T, g) - h * g
        ri = 2 * (g.conj() * r).imag
        om = self.om[None, :, None, None]
        s0, s1, s2 = (self._bins(2 * h * om ** i) for i in range(3))
        r0, r1 = self._bins(ri), self._bins(ri * om)
        H = torch.zeros((*s0.shape[:2], 4, 4), dtype=torch.float64, device=DEV)
        b = torch.zeros((*s0.shape[:2], 4), dtype=torch.float64, device=DEV)
        for c in range(2):
            i = 2 * c
            H[..., i, i], H[..., i, i + 1], H[..., i + 1, i], H[..., i + 1, i + 1] = s0[..., c], s1[..., c], s1[..., c], s2[..., c]
            b[..., i], b[..., i + 1] = r0[..., c], r1[..., c]
        return H, b


class _DirDiag:
    """A direction-dependent diagonal term: S[b][p][q][d][e][k][j], T[b][p][q][d][k][j]; gains [b][a*dir][2]."""

    def __init__(self, S, T):
        self.S, self.T = S, T

    def gains(self, g):
        return g

    def norms(self, x):
        return (x.abs() ** 2).sum((1, 2))

    def __call__(self, g, _):
        nd = self.S.shape[3]
        G = g.reshape(g.shape[0], -1, nd, 2)
        H = torch.einsum("bpqdkj,bqdj->bpdk", torch.diagonal(self.S, dim1=3, dim2=4).permute(0, 1, 2, 5, 3, 4),
                         (G.abs() ** 2).to(G.dtype))
        W = torch.einsum("bqdj,bqej->bqdej", G, G.conj())
        V = torch.einsum("bpqdekj,bqdej->bpdek", self.S, W)
        r = torch.einsum("bpqdkj,bqdj->bpdk", self.T, G) - torch.einsum("bpdek,bpek->bpdk", V, G)
        return torch.diag_embed(H).flatten(1, 2), r.flatten(1, 2)


def _dense(x, y, p, q, n_ant):
    """[b][bl][...] of baselines (p, q) and of their conjugates -> [b][n_ant][n_ant][...]."""
    z = torch.zeros((x.shape[0], n_ant, n_ant) + x.shape[2:], dtype=x.dtype, device=DEV)
    z[:, p, q], z[:, q, p] = x, y
    return z


def _exact_chain(case, o):
    """Gains (in the layout of qc.Term) and flags of every term after all epochs, in 64 bits."""
    n_ant, n_time, n_chan = case["n_ant"], case["n_time"], case["n_chan"]
    p, q = (torch.as_tensor(v, device=DEV) for v in np.triu_indices(n_ant, 1))
    n_bl, nu = p.numel(), torch.as_tensor(_freqs(n_chan) / 1e9, device=DEV)
    n_dir = 2 if "dddiag" in case["chain"] else 1
    data = o["data"].view(n_time, n_bl, n_chan, 4)
    model = o["model"].view(n_time, n_bl, n_chan, n_dir, 4)
    weight = o["weight"].view(n_time, n_bl, n_chan, 4)
    flag = o["flag"].view(n_time, n_bl, n_chan)
    scale = None
    if case.get("fp16"):
        scale = torch.view_as_real(model).abs().amax((0, 2, 3, 4, 5))
        scale = torch.where(scale > 0, scale, torch.ones_like(scale))[None, :, None, None, None, None]
    terms = o["terms"]
    cur, flags = [], []
    for t, g in zip(terms, o["start"]):
        nd = 2 if t["kind"] == "dddiag" else 1
        if t["kind"] in ("delay", "phase"):
            w = 4 if t["kind"] == "delay" else 2
            cur.append(torch.zeros(t["n_tint"], t["n_fint"], n_ant, w, dtype=torch.float64, device=DEV) if g is None
                       else torch.as_tensor(g.astype(np.float64), device=DEV))
        elif g is not None:
            cur.append(torch.as_tensor(g.astype(np.complex128), device=DEV))
        else:
            u = torch.zeros((t["n_tint"], t["n_fint"], n_ant) + ((nd,) if nd > 1 else ()) + (4,), dtype=torch.complex128,
                            device=DEV)
            u[..., 0] = u[..., 3] = 1
            cur.append(u)
        flags.append(torch.zeros(cur[-1].shape[:3] + ((nd,) if nd > 1 else ()), dtype=torch.int8, device=DEV))
    ants = torch.arange(n_ant, device=DEV)

    def jones(i, t):                        # [ant][ch][(dir)][4] of term i at time t
        return _per_channel(terms[i], cur[i], nu, ants, torch.full((n_ant,), t, device=DEV))

    def sample(t):
        m = model[t]
        if scale is not None:
            inv = (1.0 / scale[0])
            m = torch.view_as_complex((torch.view_as_real(m) * inv).half().float() * scale[0])
        w = torch.where(flag[t][..., None] == 0, weight[t].double(), torch.zeros((), dtype=torch.float64, device=DEV))
        return data[t].to(torch.complex128), m.to(torch.complex128), w

    def chain_of(idx, t, d):
        c = None
        for i in idx:
            j = jones(i, t)
            j = j[:, :, d] if terms[i]["kind"] == "dddiag" else j
            c = j if c is None else _mul(c, j)
        return c

    def solve(n):
        term = terms[n]
        kind, nf = term["kind"], term["n_fint"]
        fm = torch.as_tensor(term["f_map"], device=DEV, dtype=torch.long)
        for ti in range(term["n_tint"]):
            S = T = None
            for t in np.nonzero(term["t_map"] == ti)[0]:
                t = int(t)
                D, M, w = sample(t)
                Xs, left = [], []
                for d in range(n_dir):
                    R, L = chain_of(range(n + 1, len(terms)), t, d), chain_of(range(n), t, d)
                    X = M[:, :, d]
                    Xs.append(X if R is None else _mul(_mul(R[p], X), _herm(R[q])))
                    left.append(L)
                if kind == "full":
                    X = Xs[0].reshape(n_bl, n_chan, 2, 2)
                    wk, Dk = w.reshape(n_bl, n_chan, 2, 2), D.reshape(n_bl, n_chan, 2, 2)
                    edges = [int(e) for e in np.searchsorted(term["f_map"], np.arange(nf + 1))]
                    s, tt = [], []
                    for f in range(nf):
                        c = slice(edges[f], edges[f + 1])
                        A = X[:, c].flatten(2)
                        wA = (wk[:, c].flatten(2)[:, :, :, None] * A[:, :, None, :].conj())       # [bl][c][kj][u]
                        s.append((wA.flatten(2).transpose(1, 2) @ A).reshape(n_bl, 2, 2, 2, 2, 2, 2))
                        tt.append((wA * Dk[:, c].flatten(2)[..., None]).sum(1).reshape(n_bl, 2, 2, 2, 2))
                    s, tt = torch.stack(s), torch.stack(tt)
                elif kind == "delay":
                    X = sum(Xs)
                    s = (w * X.abs() ** 2).transpose(0, 1).reshape(n_chan, n_bl, 2, 2)
                    tt = (w * X.conj() * D).transpose(0, 1).reshape(n_chan, n_bl, 2, 2)
                elif kind == "dddiag":
                    E = torch.stack([X if L is None else _mul(_mul(L[p], X), _herm(L[q])) for X, L in zip(Xs, left)], 2)
                    z = lambda *v: torch.zeros((n_bl, nf) + v, dtype=torch.complex128, device=DEV)  # noqa: E731
                    ss = w[:, :, None, None, :] * E.conj()[:, :, :, None] * E[:, :, None]
                    s = z(n_dir, n_dir, 4).index_add_(1, fm, ss).transpose(0, 1).reshape(nf, n_bl, n_dir, n_dir, 2, 2)
                    tt = z(n_dir, 4).index_add_(1, fm, (w * D)[:, :, None] * E.conj()).transpose(0, 1)
                    tt = tt.reshape(nf, n_bl, n_dir, 2, 2)
                else:                       # diagonal or phase-only, with or without a term to its left
                    X = Xs[0].reshape(n_bl, n_chan, 2, 2)
                    z = lambda *v: torch.zeros((n_bl, nf) + v, dtype=torch.complex128, device=DEV)  # noqa: E731
                    if left[0] is None:     # E_kj,ab = M_kj for (a, b) = (k, j): diagonal sums
                        s4 = z(4).index_add_(1, fm, (w * X.flatten(2).abs() ** 2).to(torch.complex128))
                        s = torch.diag_embed(s4).transpose(0, 1).reshape(nf, n_bl, 2, 2, 2, 2)
                        tt = z(4).index_add_(1, fm, w * X.flatten(2).conj() * D).transpose(0, 1).reshape(nf, n_bl, 2, 2)
                    else:
                        Lp, Lq = left[0][p].reshape(n_bl, n_chan, 2, 2), left[0][q].reshape(n_bl, n_chan, 2, 2)
                        E = (Lp[:, :, :, None, :, None] * X[:, :, None, None] * Lq.conj()[:, :, None, :, None, :]).flatten(4)
                        E = E.flatten(2, 3)                                                    # [bl][c][kj][ab]
                        wE = w[..., None] * E.conj()
                        s = z(4, 4).index_add_(1, fm, wE.transpose(2, 3) @ E)
                        s = s.transpose(0, 1).reshape(nf, n_bl, 2, 2, 2, 2)
                        tt = z(4).index_add_(1, fm, (wE * D[..., None]).sum(2)).transpose(0, 1).reshape(nf, n_bl, 2, 2)
                S, T = (s, tt) if S is None else (S + s, T + tt)
            if kind == "full":
                Sd = _dense(S, S.conj().permute(0, 1, 3, 2, 5, 4, 7, 6), p, q, n_ant)
                Td = _dense(T, T.conj().permute(0, 1, 3, 2, 5, 4), p, q, n_ant)
                H, g0 = _Full(Sd, Td), cur[n][ti]
            elif kind == "delay":
                Sd = _dense(S, S.transpose(-1, -2), p, q, n_ant)
                Td = _dense(T, T.conj().transpose(-1, -2), p, q, n_ant)
                H, g0 = _Delay(Sd[None], Td[None], nu, fm, nf), cur[n][ti]
            elif kind == "dddiag":
                Sd = _dense(S, S.conj().transpose(-1, -2), p, q, n_ant)
                Td = _dense(T, T.conj().transpose(-1, -2), p, q, n_ant)
                H, g0 = _DirDiag(Sd, Td), cur[n][ti][..., 0::3].flatten(1, 2)
            else:
                Sd = _dense(S, S.conj().permute(0, 1, 3, 2, 5, 4), p, q, n_ant)
                Td = _dense(T, T.conj().transpose(-1, -2), p, q, n_ant)
                H = _Diag(Sd, Td, kind == "phase")
                g0 = cur[n][ti] if kind == "phase" else cur[n][ti][..., 0::3]
            g, f = _iterate(kind, H, g0)
            flags[n][ti] = f.reshape(flags[n][ti].shape)
            if kind in ("full", "delay", "phase"):
                cur[n][ti] = g
            else:
                cur[n][ti][..., 0::3] = g.reshape(cur[n][ti][..., 0::3].shape)

    if case["op"] == "solve":
        for _ in range(case["epochs"]):
            for n in range(len(terms)):
                solve(n)
    return cur, flags, (sample, chain_of, n_dir, p, q)


def exact(case, seed):
    if case["op"] == "mlp":
        return _exact_mlp(case, seed)
    if case["op"] == "mad" or (case["op"] != "residual" and _samples(case)[0] > EXACT_SAMPLES):
        return None
    if case["op"] == "batch":
        return _exact_batch(case, seed)
    o = _observation(case, seed)
    cur, flags, (sample, chain_of, n_dir, p, q) = _exact_chain(case, o)
    out = {}
    if case["op"] == "solve":
        for i, (g, f) in enumerate(zip(cur, flags)):
            out["gains%d" % i], out["flags%d" % i] = g, None
    if case["op"] == "residual" or case["chi2"]:
        chi2, res = 0.0, []
        for t in range(case["n_time"]):
            D, M, w = sample(t)
            for d in range(n_dir):
                c = chain_of(range(len(cur)), t, d)
                D = D - _mul(_mul(c[p], M[:, :, d]), _herm(c[q]))
            chi2 += float((w * D.abs() ** 2).sum())
            if case["op"] == "residual":
                res.append(torch.where(o["flag"].view(case["n_time"], p.numel(), -1)[t][..., None] == 0, D,
                                       torch.zeros_like(D)))
        out["chi2"] = torch.tensor(chi2, dtype=torch.float64)
        if res:
            out["residual"] = torch.cat(res)
    return out


def _exact_batch(case, seed):
    b = _batch(case, seed)
    n_prob, A = case["n_prob"], int(b["n_ant"].max())
    row_p = torch.as_tensor(b["ant1"], device=DEV, dtype=torch.long)
    row_q = torch.as_tensor(b["ant2"], device=DEV, dtype=torch.long)
    slot = (b["prob_of_row"] * A + row_p) * A + row_q
    nc = torch.as_tensor(b["n_chan"], device=DEV, dtype=torch.long)[b["prob_of_row"]]
    S = torch.zeros(n_prob * A * A, 4, dtype=torch.float64, device=DEV)
    T = torch.zeros(n_prob * A * A, 4, dtype=torch.complex128, device=DEV)
    first, n_row = torch.cumsum(nc, 0) - nc, nc.numel()
    for at in range(0, n_row, 1 << 17):
        end = min(n_row, at + (1 << 17))
        v0, v1 = int(first[at]), int(first[end - 1] + nc[end - 1])
        w = torch.where(b["flag"][v0:v1, None] == 0, b["weight"][v0:v1].double(),
                        torch.zeros((), dtype=torch.float64, device=DEV))
        m, d = b["model"][v0:v1].to(torch.complex128), b["data"][v0:v1].to(torch.complex128)
        lo = first[at:end] - v0                            # a row's samples are contiguous
        for acc, x in ((S, w * m.abs() ** 2), (T, w * m.conj() * d)):
            c = torch.cat([torch.zeros_like(x[:1]), torch.cumsum(x, 0)])
            acc.index_add_(0, slot[at:end], c[lo + nc[at:end]] - c[lo])
    S, T = S.view(n_prob, A, A, 2, 2), T.view(n_prob, A, A, 2, 2)
    S = S + S.permute(0, 2, 1, 4, 3)                       # a baseline fills one of its two places
    T = T + T.conj().permute(0, 2, 1, 4, 3)
    real = torch.arange(A, device=DEV)[None] < torch.as_tensor(b["n_ant"], device=DEV)[:, None]

    class Sums:
        def gains(self, g):
            return g

        def norms(self, x):
            return ((x.abs() ** 2).sum(2) * real).sum(1)

        def __call__(self, g, _):
            h = torch.einsum("bpqkj,bqj->bpk", S, g.abs() ** 2)
            r = torch.einsum("bpqkj,bqj->bpk", T, g) - h * g
            return torch.diag_embed(h).to(g.dtype), r

    g, _ = _iterate("diag", Sums(), torch.ones(n_prob, A, 2, dtype=torch.complex128, device=DEV))
    return {"gains": g[real], "flags": None}


def _exact_mlp(case, seed):
    s = prepare(case, seed)
    net = s["net"]
    w = net.params.double().requires_grad_(True)
    x, y = s["x"].double(), s["y"].double()
    h, at = x, 0
    for out_d, in_d in ((128, 10), (128, 128), (128, 128), (4, 128)):
        W, b = w[at:at + out_d * in_d].view(out_d, in_d), w[at + out_d * in_d:at + out_d * in_d + out_d]
        at += out_d * in_d + out_d
        h = h @ W.T + b
        if out_d != 4:
            h = 0.5 * h * (1 + torch.erf(h / math.sqrt(2.0)))
    loss = ((h + x[:, 6:10] - y) ** 2).mean()
    g, = torch.autograd.grad(loss, w)
    m, v = 0.9 * net.m.double() + 0.1 * g, 0.999 * net.v.double() + 0.001 * g * g
    k = net.step + 1
    p = net.params.double() - 1e-4 * (m / (1 - 0.9 ** k)) / (torch.sqrt(v / (1 - 0.999 ** k)) + 1e-8)
    return {"params": p, "grad": g, "m": m, "v": v, "loss": loss.detach()}
