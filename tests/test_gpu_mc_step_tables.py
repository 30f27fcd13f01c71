"""A dynamic model's step table is built by the path blocks of a small launch and
by a launch of its own otherwise.  Ranges of a grid (sabr_mc_shard_partials) that
build theirs give the whole grid's prices, which read one, bit for bit; the
cliquet is compared with the FP64 oracle on both sides of the line (1e-5 in
FP32, 1e-10 in FP64: the tolerances of the full-size tests)."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2407_20713_gb300 as sg

pytestmark = pytest.mark.gpu

PARAMS = {sg.DYN_I: [0.3, 0.7, -0.6, 0.9, 0.5, 1.2], sg.DYN_II: [0.3, 0.8, -0.5, 0.7, 1.1, 0.6, 0.1, 0.2, 0.25, -0.2]}


@pytest.mark.parametrize("prec", [sg.FP32, sg.FP64])
@pytest.mark.parametrize("model", list(PARAMS))
@pytest.mark.parametrize("steps", [150, 151, 255, 256])
def test_built_and_read_tables_agree_bit_for_bit(model, prec, steps):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    T = np.repeat([0.5, 1.0], 3)
    K = np.tile([0.8, 1.0, 1.2], 2)
    per_block = 512 if prec == sg.FP32 else 384
    kw = dict(n_paths=per_block * (2 * sms) - 5, steps_per_year=float(steps), seed=11, prec=prec)
    blocks, _ = sg.mc_shard_layout(model, PARAMS[model], 1.0, T, K, **kw)
    assert blocks == 2 * sms  # two blocks an SM read a table from 151 steps on, one builds up to 256
    whole, se = sg.mc_price(model, PARAMS[model], 1.0, T, K, **kw)
    parts = [sg.mc_shard_partials(model, PARAMS[model], 1.0, T, K, blocks, b, sms, **kw) for b in (0, sms)]
    got, gse = sg.mc_shard_reduce(model, PARAMS[model], 1.0, T, K, blocks, torch.cat(parts), **kw)
    assert torch.equal(got, whole) and torch.equal(gse, se)


@pytest.mark.parametrize("prec,tol", [(sg.FP32, 1e-5), (sg.FP64, 1e-10)])
@pytest.mark.parametrize("model", list(PARAMS))
@pytest.mark.parametrize("steps,paths", [(12, 1000), (128, 500), (129, 500), (100, 64 * 4 * 152 * 3 + 7)])
def test_cliquet_with_built_and_read_tables_matches_the_oracle(model, prec, tol, steps, paths):
    if prec == sg.FP64:
        paths = min(paths, 2000)
    args = (1.0, 4, -0.02, 0.02, 0.0, 0.2)
    ref, rse = O.mc_cliquet(model, PARAMS[model], 1.0, *args, disc=0.9, n_paths=paths, steps_per_year=steps, seed=7,
                            n_threads=8)
    got, gse = sg.mc_cliquet(model, PARAMS[model], 1.0, *args, discount=0.9, n_paths=paths, steps_per_year=float(steps),
                             seed=7, prec=prec)
    assert abs(got.item() - ref) <= tol and abs(gse.item() - rse) <= tol
