"""Calls and puts of an FP32 pricing are kept as pairs of a sign and a strike, or as
signed strikes where pairs would cost a block an SM: prices of mixed option sets, strikes of
zero among them, match the FP64 oracle on the same streams (1e-5, the pricer's
FP32 tolerance; past 1800 steps by the square root of their number, as the
per-step errors of the SFU functions, times sqrt(h), add up) at sizes where a
block's tables take a quarter, a third or most of an SM's shared memory."""
import numpy as np
import pytest

import oracle as O
import paper_2407_20713_gb300 as sg

pytestmark = pytest.mark.gpu

P = [0.3, 0.6, -0.4, 0.7]


@pytest.mark.parametrize("options,steps,paths", [
    (1, 12, 3000), (37, 60, 3000), (16, 40, 512 * 152 * 4 + 1),
    # 49-60 KB a block (four, then three blocks an SM), 512 options
    (400, 1400, 700), (400, 1800, 700), (512, 1200, 700),
    # 164 KB
    (512, 8000, 300),
])
def test_mixed_option_sets_match_the_oracle(options, steps, paths):
    T = np.where(np.arange(options) % 3 == 0, 0.5, 1.0)
    K = np.linspace(0.0, 1.8, options) if options > 1 else np.array([1.0])
    ic = (np.arange(options) % 2).astype(np.int8)  # the strike of zero is a put; the next test has the call
    ref, rse = O.mc_price(O.HAGAN, P, 1.0, T, K, is_call=ic, n_paths=paths, steps_per_year=steps, seed=9, n_threads=8)
    got, gse = sg.mc_price(sg.HAGAN, P, 1.0, T, K, is_call=ic, n_paths=paths, steps_per_year=float(steps), seed=9)
    tol = 1e-5 * max(1.0, (steps / 1800) ** 0.5)
    assert np.max(np.abs(got.cpu().numpy() - ref)) <= tol
    assert np.max(np.abs(gse.cpu().numpy() - rse)) <= tol


@pytest.mark.parametrize("call", [0, 1])
def test_a_strike_of_zero(call):
    T, K, ic = np.array([0.5]), np.array([0.0]), np.array([call], dtype=np.int8)
    ref, _ = O.mc_price(O.HAGAN, P, 1.0, T, K, is_call=ic, n_paths=5000, steps_per_year=20, seed=9, n_threads=8)
    got, _ = sg.mc_price(sg.HAGAN, P, 1.0, T, K, is_call=ic, n_paths=5000, steps_per_year=20.0, seed=9)
    assert abs(got.item() - ref[0]) <= 1e-5
    if call == 0:
        assert got.item() == 0.0


def test_too_many_steps_and_options_stay_refused():
    with pytest.raises(Exception):
        sg.mc_price(sg.HAGAN, P, 1.0, np.ones(512), np.ones(512), n_paths=100, steps_per_year=8192.0,
                    prec=sg.FP64)
