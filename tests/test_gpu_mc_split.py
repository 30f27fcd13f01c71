"""The FP32 log-Euler pricer runs one pair of paths a thread where a launch has at
most one block an SM and 128 steps or more.  Ranges of a grid
(sabr_mc_shard_partials) with a block an SM are compared bit for bit with the
whole grid, which has more, on both sides of the line, with landings at either
step of a block of two."""
import numpy as np
import pytest
import torch

import paper_2407_20713_gb300 as sg

pytestmark = pytest.mark.gpu

PARAMS = {sg.HAGAN: [0.3, 0.6, -0.4, 0.7], sg.DYN_I: [0.3, 0.7, -0.6, 0.9, 0.5, 1.2],
          sg.DYN_II: [0.3, 0.8, -0.5, 0.7, 1.1, 0.6, 0.1, 0.2, 0.25, -0.2]}
MATS = [0.1, 0.25, 0.3, 0.35, 1.0]


@pytest.mark.parametrize("model", list(PARAMS))
@pytest.mark.parametrize("steps_per_year", [120, 125, 126, 130, 200, 500])
@pytest.mark.parametrize("strikes", [1, 17])
def test_both_forms_of_the_path_loop_agree_bit_for_bit(model, steps_per_year, strikes):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    T = np.repeat(MATS, strikes)
    K = np.tile(np.linspace(0.7, 1.3, strikes) if strikes > 1 else [1.0], len(MATS))
    ic = (np.arange(T.size) % 2).astype(np.int8)
    kw = dict(is_call=ic, n_paths=512 * (sms + 40) - 77, steps_per_year=float(steps_per_year), seed=11)
    blocks, _ = sg.mc_shard_layout(model, PARAMS[model], 1.0, T, K, **kw)
    assert blocks == sms + 40
    whole, se = sg.mc_price(model, PARAMS[model], 1.0, T, K, **kw)
    half = blocks // 2
    parts = [sg.mc_shard_partials(model, PARAMS[model], 1.0, T, K, blocks, b, n, **kw)
             for b, n in ((0, half), (half, blocks - half))]
    got, gse = sg.mc_shard_reduce(model, PARAMS[model], 1.0, T, K, blocks, torch.cat(parts), **kw)
    assert torch.equal(got, whole) and torch.equal(gse, se)
