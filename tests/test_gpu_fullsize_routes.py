"""The full-size workload (64 antennas, 300 times x 512 channels, G full per time then B diagonal per
channel, 3 epochs) on the routes that the other full-size tests leave out: the streaming kernel per
sample with the complex64 model, which reduce, divergence flagging and longer chains iterate
on, and the default route with the FP16 model.  The checks and tolerances are those tests'."""
import numpy as np
import pytest

import test_gpu_fullsize as tf
import test_gpu_fullsize_fp16 as t16
from paper_2412_10072_gb300 import qc, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def full():
    torch = pytest.importorskip("torch")
    setup = synth.plain_large_setup(seed=1, n_ant=64, n_time=300, n_chan=512)
    obs = synth.make_observation_device(setup, noise=0.05, noise_seed=1000, device="cuda:0")

    def solve(kernel, fp16):
        S = qc.Solver(obs["data"], obs["model"], obs["weight"], obs["flag"], setup.ant1, setup.ant2, setup.time_idx,
                      setup.n_ant, setup.n_time, model_fp16=fp16)
        terms = [qc.Term.from_spec(s, setup.n_ant, max_iter=20, tol=1e-6) for s in setup.terms]
        st = S.solve(terms, n_epochs=3, kernel=kernel)
        torch.cuda.synchronize()
        S.close()
        return terms, st

    yield setup, obs, solve
    del obs
    torch.cuda.empty_cache()


def test_per_sample_kernel(full):
    setup, obs, solve = full
    terms, st = solve(3, False)
    assert st.acc_bytes > 40 * 25e9                    # the samples every iteration
    for check in (tf.test_sampled_g_intervals_are_stationary, tf.test_sampled_b_intervals_are_stationary,
                  tf.test_full_size_chi2_matches_oracle_on_sampled_rows):
        check((setup, obs, terms))


def test_fp16_default_route(full):
    setup, obs, solve = full
    terms, st = solve(0, True)
    ref, st3 = solve(3, True)
    assert st.acc_bytes < 0.2 * st3.acc_bytes          # six passes and the sums
    deq = t16._dequantized(obs["model"], setup.n_ant * (setup.n_ant - 1) // 2)
    assert t16._steps(setup, obs, deq, terms) < t16.GAIN_TOL
    for a, b in zip(terms, ref):                       # both stopped at a relative change of 1e-6
        assert np.linalg.norm(a.gains - b.gains) < 1e-5 * np.linalg.norm(b.gains)
        assert np.array_equal(a.gain_flags, b.gain_flags)
