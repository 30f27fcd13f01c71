"""A chain's misfit is summed in the order of its G lanes whichever lanes run
it: fewer lanes playing the G in plans and in the server (dynamic models, and
Hagan requests of the server), or all of them, level by level, in a shard.  The
calibrations must agree bit for bit over lane splits, maturity counts below, at
and above the lanes, ragged quote counts (chunks and remainders of the quote
loop) and chain counts that leave part of a warp without a chain."""
import numpy as np
import pytest

import paper_2407_20713_gb300 as sg
from paper_2407_20713_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TRUTH = {sg.HAGAN: [0.25, 0.7, -0.4, 0.5], sg.DYN_I: [0.25, 0.8, -0.5, 0.7, 0.6, 0.9],
         sg.DYN_II: [0.25, 0.8, -0.4, 0.6, 0.8, 0.9, 0.1, 0.15, 0.2, -0.1]}
BOX = {sg.HAGAN: (W.STATIC_LO, W.STATIC_HI), sg.DYN_I: (W.DYN1_LO, W.DYN1_HI), sg.DYN_II: (W.DYN2_LO, W.DYN2_HI)}


def problem(model, mats, strikes, chains, levels=3, length=9, seed=5, drop=0):
    T = np.repeat(0.1 + 0.15 * np.arange(mats), strikes)
    K = np.tile(np.linspace(0.75, 1.25, strikes), mats)
    T, K = T[drop:], K[drop:]
    mkt = sg.implied_vol(model, TRUTH[model], 1.0, T, K, prec=sg.FP64).cpu().numpy()
    lo, hi = BOX[model]
    return sg.CalibrationProblem(model=model, T=T, K=K, market=mkt, lo=lo, hi=hi, prec=sg.FP32, n_chains=chains,
                                 n_levels=levels, chain_len=length, seed=seed)


def level_by_level(pb):
    s = sg.Shard(pb, 0, pb.n_chains)
    for lv in range(pb.n_levels):
        f, _, x = s.level(lv)
        s.restart(f, x)
    return s.result()[0]


def same(a, b):
    assert np.array_equal(a.params, b.params) and np.array_equal(a.restart_params, b.restart_params)
    assert (a.misfit, a.misfit_fp64, a.restart_misfit) == (b.misfit, b.misfit_fp64, b.restart_misfit)
    assert (a.n_evals, a.n_accepts, a.status) == (b.n_evals, b.n_accepts, b.status)


# mats, strikes, chains: 4 of 8 lanes, 16 of 32, 8 of 32, 4 of 32, all of them;
# one maturity, one quote a maturity, 64 maturities
SHAPES = [(12, 21, 8192), (12, 21, 2050), (7, 9, 4001), (33, 5, 9001), (1, 11, 20001), (2, 1, 8192), (5, 21, 301),
          (64, 3, 5000), (3, 40, 10007)]


@pytest.mark.parametrize("model", [sg.DYN_I, sg.DYN_II])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(map(str, s)))
def test_dynamic_plans_equal_all_lanes(model, shape):
    mats, strikes, chains = shape
    pb = problem(model, mats, strikes, chains, drop=min(3, mats * strikes - 1))
    same(sg.calibrate(pb), level_by_level(pb))


@pytest.mark.parametrize("model", [sg.HAGAN, sg.DYN_I, sg.DYN_II])
def test_server_requests_equal_all_lanes(model):
    shapes = [(1, 5, 60), (1, 24, 257), (2, 25, 500), (4, 33, 1024), (12, 41, 1000), (64, 2, 90), (3, 17, 7)]
    pbs = [problem(model, m, s, c, levels=4, length=7, seed=i, drop=i % 3) for i, (m, s, c) in enumerate(shapes)]
    srv = sg.Server(device_bytes=1 << 28, max_active=16, max_quotes=512)
    tickets = [srv.submit(p) for p in pbs]
    for p, t in zip(pbs, tickets):
        same(srv.wait(t, timeout_ms=60000), level_by_level(p))
    srv.close()


def test_one_lane_batches_equal_level_by_level_launches(monkeypatch):
    # every chain one lane: the queue kernel that holds their loops alone
    shapes = [(1, 21), (1, 20), (3, 9), (1, 9), (2, 22)]
    pbs = [problem(sg.HAGAN, m, s, 9000 + i, levels=3, length=8, seed=i) for i, (m, s) in enumerate(shapes)]
    plan = sg.Plan(pbs)
    plan.run()
    queued = plan.results()
    launches = plan.stats()[0]
    plan.close()
    monkeypatch.setenv("SABR_PLAN_QUEUE", "0")
    plan = sg.Plan(pbs)
    plan.run()
    levelwise = plan.results()
    assert launches == 4 and plan.stats()[0] == 1 + 3 + 1
    plan.close()
    for a, b in zip(queued, levelwise):
        same(a, b)
