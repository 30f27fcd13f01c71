"""Static problems of few chains run in one launch that looks several steps
ahead, with one to four warps a chain (sa_small.cu).  A shard that holds all
chains of a problem runs the same calibration level by level with the one-step
or two-step loops of the level kernel; the two must agree bit for bit -- every
step's decision, counter and sum is the same -- over the shapes' edges: a
window longer than the level, windows that end inside a draw of 32 steps, more
lanes than quotes, several rounds of quotes a lane, ragged chain counts on both
sides of the shapes' limits, and boxes that most proposals leave."""
import numpy as np
import pytest

import paper_2407_20713_gb300 as sg
from paper_2407_20713_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def problem(model, prec, mats, strikes, chains, levels, length, seed=5, hi=None, **kw):
    T = np.repeat(0.25 * (1 + np.arange(mats)), strikes)
    K = np.tile(np.linspace(0.7, 1.3, strikes), mats)
    mkt = sg.implied_vol(sg.HAGAN, [0.25, 0.7, -0.4, 0.5], 1.0, T, K, prec=sg.FP64).cpu().numpy()
    mkt = mkt * (1 + 1e-3 * np.random.default_rng(seed).normal(size=T.size))
    return sg.CalibrationProblem(model=model, T=T, K=K, market=mkt, lo=W.STATIC_LO, hi=hi or W.STATIC_HI, prec=prec,
                                 n_chains=chains, n_levels=levels, chain_len=length, seed=seed, **kw)


def level_by_level(pb):
    s = sg.Shard(pb, 0, pb.n_chains)
    for lv in range(pb.n_levels):
        f, _, x = s.level(lv)
        s.restart(f, x)
    r, _ = s.result()
    return r


def same(a, b):
    assert np.array_equal(a.params, b.params) and np.array_equal(a.restart_params, b.restart_params)
    assert (a.misfit, a.misfit_fp64, a.restart_misfit) == (b.misfit, b.misfit_fp64, b.restart_misfit)
    assert (a.n_evals, a.n_accepts, a.status) == (b.n_evals, b.n_accepts, b.status)


CASES = [
    # model, mats, strikes, chains, levels, length
    (sg.HAGAN, 1, 15, 64, 35, 40), (sg.HAGAN, 1, 3, 7, 5, 33), (sg.HAGAN, 1, 4, 1, 3, 100), (sg.HAGAN, 2, 9, 152, 4, 31),
    (sg.HAGAN, 1, 15, 64, 3, 1), (sg.HAGAN, 1, 15, 64, 3, 5), (sg.HAGAN, 5, 41, 153, 3, 20), (sg.HAGAN, 9, 33, 305, 3, 17),
    (sg.HAGAN, 3, 21, 609, 3, 20), (sg.HAGAN, 12, 41, 1216, 2, 9), (sg.OBLOJ, 1, 15, 64, 6, 33), (sg.OBLOJ, 4, 17, 303, 3, 20),
    (sg.OBLOJ, 2, 41, 1000, 2, 12), (sg.HAGAN, 1, 12, 64, 4, 0),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
def test_fp32_equals_the_level_kernels(case):
    model, mats, strikes, chains, levels, length = case
    pb = problem(model, sg.FP32, mats, strikes, chains, levels, length)
    same(sg.calibrate(pb), level_by_level(pb))


@pytest.mark.parametrize("case", [(sg.HAGAN, 1, 15, 64, 4, 33), (sg.HAGAN, 2, 21, 153, 2, 9), (sg.HAGAN, 1, 5, 305, 2, 9),
                                  (sg.OBLOJ, 1, 9, 30, 3, 17), (sg.EXPANDED, 2, 20, 64, 4, 40)],
                         ids=lambda c: "-".join(map(str, c)))
def test_fp64_equals_the_level_kernels(case):
    model, mats, strikes, chains, levels, length = case
    pb = problem(model, sg.FP64, mats, strikes, chains, levels, length)
    same(sg.calibrate(pb), level_by_level(pb))


@pytest.mark.parametrize("prec", [sg.FP32, sg.FP64])
def test_proposals_that_leave_the_box(prec):
    # a box the size of a step around the start: most windows hold several
    # proposals outside, some nothing else; and a coordinate held fixed at 0
    pb = problem(sg.HAGAN, prec, 1, 15, 50, 4, 37, hi=[2.0, 0.0, 1 - 1e-6, 3.0], step0=2.0, x0=[0.3, 0.0, 0.0, 0.4])
    r = sg.calibrate(pb)
    assert 0 < r.n_evals < 0.5 * 50 * 4 * 37
    same(r, level_by_level(pb))

