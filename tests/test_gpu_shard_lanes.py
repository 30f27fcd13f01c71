"""Chain shards of FP32 dynamic fits run each chain on as many lanes as the
shard's own chains leave, its sums in the order of the whole problem's lanes.  A
plan, one shard with every chain, two unequal shards and many small shards (all
lanes a chain) give the same calibration bit for bit."""
import numpy as np
import pytest

import paper_2407_20713_gb300 as sg
from paper_2407_20713_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TRUTH = {sg.DYN_I: [0.25, 0.8, -0.5, 0.7, 0.6, 0.9], sg.DYN_II: [0.25, 0.8, -0.4, 0.6, 0.8, 0.9, 0.1, 0.15, 0.2, -0.1]}
BOX = {sg.DYN_I: (W.DYN1_LO, W.DYN1_HI), sg.DYN_II: (W.DYN2_LO, W.DYN2_HI)}


def problem(model, mats, strikes, chains):
    T = np.repeat(0.1 + 0.15 * np.arange(mats), strikes)[1:]
    K = np.tile(np.linspace(0.75, 1.25, strikes), mats)[1:]
    mkt = sg.implied_vol(model, TRUTH[model], 1.0, T, K, prec=sg.FP64).cpu().numpy()
    lo, hi = BOX[model]
    return sg.CalibrationProblem(model=model, T=T, K=K, market=mkt, lo=lo, hi=hi, prec=sg.FP32, n_chains=chains,
                                 n_levels=3, chain_len=9, seed=5)


def sharded(pb, cuts):
    shards = [sg.Shard(pb, a, b - a) for a, b in zip(cuts[:-1], cuts[1:])]
    for lv in range(pb.n_levels):
        f, _, x = min((s.level(lv) for s in shards), key=lambda p: (p[0], p[1]))
        for s in shards:
            s.restart(f, x)
    parts = [s.result() for s in shards]
    best, _ = min(parts, key=lambda p: (p[0].misfit, p[1]))
    return (tuple(best.params), best.misfit, best.misfit_fp64, sum(r.n_evals for r, _ in parts),
            sum(r.n_accepts for r, _ in parts), {r.status for r, _ in parts}, best.restart_misfit)


@pytest.mark.parametrize("model", [sg.DYN_I, sg.DYN_II])
@pytest.mark.parametrize("mats,strikes,chains", [(12, 21, 8192), (7, 9, 4001), (2, 11, 8001), (33, 5, 9001),
                                                 (64, 3, 2500)])
def test_shards_of_any_size_equal_the_plan(model, mats, strikes, chains):
    pb = problem(model, mats, strikes, chains)
    r = sg.calibrate(pb)
    whole = (tuple(r.params), r.misfit, r.misfit_fp64, r.n_evals, r.n_accepts, {r.status}, r.restart_misfit)
    assert sharded(pb, [0, chains]) == whole
    assert sharded(pb, [0, chains // 3, chains]) == whole
    assert sharded(pb, list(range(0, chains, 301)) + [chains]) == whole
