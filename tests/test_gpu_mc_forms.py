"""The FP32 log-Euler pricer has two forms of its path loop (a thread runs four
paths of a block, or two threads two each), steps its time grid two steps at
a time with landings at either of them, and may leave the last round of a
grid with one live pair.  A range of few blocks (sabr_mc_shard_partials) runs
the second form over paths that the whole grid runs in the first, so the two
are compared bit for bit; the grids and rounds are compared with the FP64
oracle on the same streams (1e-5, the pricer's FP32 tolerance)."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2407_20713_gb300 as sg

pytestmark = pytest.mark.gpu

PARAMS = {sg.HAGAN: [0.3, 0.6, -0.4, 0.7], sg.DYN_I: [0.3, 0.7, -0.6, 0.9, 0.5, 1.2],
          sg.DYN_II: [0.3, 0.8, -0.5, 0.7, 1.1, 0.6, 0.1, 0.2, 0.25, -0.2]}

# maturities that end at the first and at the second step of a block of two,
# in the same block, at the first step of all, and after a single step
GRIDS = [([0.25], 4), ([0.1, 0.2, 0.3], 10), ([0.1, 0.25, 0.3, 0.35, 1.0], 20), ([1.0 / 12, 0.5, 0.51], 12)]


@pytest.mark.parametrize("model", list(PARAMS))
@pytest.mark.parametrize("grid", range(len(GRIDS)))
@pytest.mark.parametrize("strikes", [1, 16, 17])
def test_both_forms_of_the_path_loop_agree_bit_for_bit(model, grid, strikes):
    mats, spy = GRIDS[grid]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n_paths = 512 * (sms + 40) - 77  # more blocks than SMs, the last one ragged
    T = np.repeat(mats, strikes)
    K = np.tile(np.linspace(0.7, 1.3, strikes), len(mats))
    ic = (np.arange(T.size) % 2).astype(np.int8)
    kw = dict(is_call=ic, n_paths=n_paths, steps_per_year=float(spy), seed=11)
    blocks, _ = sg.mc_shard_layout(model, PARAMS[model], 1.0, T, K, **kw)
    assert blocks == sms + 40
    whole, se = sg.mc_price(model, PARAMS[model], 1.0, T, K, **kw)
    half = blocks // 2
    parts = [sg.mc_shard_partials(model, PARAMS[model], 1.0, T, K, blocks, b, n, **kw)
             for b, n in ((0, half), (half, blocks - half))]
    got, gse = sg.mc_shard_reduce(model, PARAMS[model], 1.0, T, K, blocks, torch.cat(parts), **kw)
    assert torch.equal(got, whole) and torch.equal(gse, se)


@pytest.mark.parametrize("grid", range(len(GRIDS)))
@pytest.mark.parametrize("n_paths", [2, 130, 512 * 152 + 1])
def test_landings_match_the_oracle(grid, n_paths):
    mats, spy = GRIDS[grid]
    T = np.repeat(mats, 3)
    K = np.tile([0.9, 1.0, 1.1], len(mats))
    ref, rse = O.mc_price(O.DYN_I, PARAMS[sg.DYN_I], 1.0, T, K, n_paths=n_paths, steps_per_year=spy, seed=3, n_threads=8)
    got, gse = sg.mc_price(sg.DYN_I, PARAMS[sg.DYN_I], 1.0, T, K, n_paths=n_paths, steps_per_year=spy, seed=3)
    assert np.max(np.abs(got.cpu().numpy() - ref)) <= 1e-5
    assert np.max(np.abs(gse.cpu().numpy() - rse)) <= 1e-5


@pytest.mark.parametrize("extra", [100, 512 * 152, 512 * 152 * 3 + 5])
def test_the_last_round_of_the_grid_matches_the_oracle(extra):
    n_paths = 512 * 4 * 152 + extra  # one whole round of the four-block grid and part of another
    T = np.array([0.25, 0.5])
    K = np.array([0.95, 1.05])
    ref, _ = O.mc_price(O.HAGAN, PARAMS[sg.HAGAN], 1.0, T, K, n_paths=n_paths, steps_per_year=4, seed=5, n_threads=8)
    got, _ = sg.mc_price(sg.HAGAN, PARAMS[sg.HAGAN], 1.0, T, K, n_paths=n_paths, steps_per_year=4, seed=5)
    assert np.max(np.abs(got.cpu().numpy() - ref)) <= 1e-5
