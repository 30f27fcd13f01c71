"""The few-chain kernel (sa_small.cu) decides windows of steps, and goes step by
step after levels in which its chains accepted less than half of what they
evaluated.  Both kinds of levels, and changes between them in one calibration,
are compared bit for bit with the level kernels (a shard that holds every
chain), over the kernel's shapes; the launch counts say that the few-chain
kernel ran, up to its limit of chains and not past it."""
import numpy as np
import pytest
import torch

import paper_2407_20713_gb300 as sg
from paper_2407_20713_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def problem(model, prec, mats, strikes, chains, levels, length, **kw):
    T = np.repeat(0.25 * (1 + np.arange(mats)), strikes)
    K = np.tile(np.linspace(0.7, 1.3, strikes), mats)
    mkt = sg.implied_vol(sg.HAGAN, [0.25, 0.7, -0.4, 0.5], 1.0, T, K, prec=sg.FP64).cpu().numpy()
    mkt = mkt * (1 + 1e-3 * np.random.default_rng(5).normal(size=T.size))
    return sg.CalibrationProblem(model=model, T=T, K=K, market=mkt, lo=W.STATIC_LO, hi=W.STATIC_HI, prec=prec,
                                 n_chains=chains, n_levels=levels, chain_len=length, seed=5, **kw)


def result(r):
    return (tuple(r.params), tuple(r.restart_params), r.misfit, r.misfit_fp64, r.restart_misfit, r.n_evals, r.n_accepts,
            r.status)


def level_by_level(pb):
    s = sg.Shard(pb, 0, pb.n_chains)
    for lv in range(pb.n_levels):
        f, _, x = s.level(lv)
        s.restart(f, x)
    return result(s.result()[0])


def planned(pb):
    plan = sg.Plan([pb])
    plan.run()
    r, launches = plan.results()[0], plan.stats()[0]
    plan.close()
    return r, launches


# shapes of the kernel: (chains as a function of the SM count, quotes)
FP32_SHAPES = [(lambda n: 64, 15), (lambda n: n, 64), (lambda n: n, 65), (lambda n: 2 * n + 1, 33),
               (lambda n: 4 * n, 5), (lambda n: 4 * n + 1, 24), (lambda n: 8 * n, 15), (lambda n: 1, 2)]
FP64_SHAPES = [(lambda n: 30, 15), (lambda n: n + 1, 7), (lambda n: 2 * n + 1, 9), (lambda n: 4 * n, 5)]
# start temperatures from "nearly everything is accepted" to "nearly nothing"
TEMPS = [(0.0, 0.95), (0.3, 0.5), (30.0, 0.05), (1e-7, 0.999)]


@pytest.mark.parametrize("T0,factor", TEMPS)
@pytest.mark.parametrize("model", [sg.HAGAN, sg.OBLOJ])
@pytest.mark.parametrize("shape", range(len(FP32_SHAPES)))
def test_fp32_at_any_acceptance(shape, model, T0, factor):
    chains, strikes = FP32_SHAPES[shape]
    pb = problem(model, sg.FP32, 1, strikes, chains(sms()), 6, 37, T0=T0, factor=factor)
    r, launches = planned(pb)
    # init, the few-chain kernel, finalize; FP32 Hagan with one pair of quotes has
    # one lane a chain and keeps the queue kernel (with its reset)
    assert launches == (4 if model == sg.HAGAN and strikes <= 2 else 3)
    assert result(r) == level_by_level(pb)


@pytest.mark.parametrize("T0,factor", TEMPS)
@pytest.mark.parametrize("model", [sg.HAGAN, sg.OBLOJ, sg.EXPANDED])
@pytest.mark.parametrize("shape", range(len(FP64_SHAPES)))
def test_fp64_at_any_acceptance(shape, model, T0, factor):
    chains, strikes = FP64_SHAPES[shape]
    pb = problem(model, sg.FP64, 1, strikes, chains(sms()), 5, 33, T0=T0, factor=factor)
    r, launches = planned(pb)
    assert launches == 3
    assert result(r) == level_by_level(pb)


@pytest.mark.parametrize("prec,most", [(sg.FP32, 8), (sg.FP64, 4)])
def test_the_limit_of_chains(prec, most):
    pb = problem(sg.HAGAN, prec, 1, 15, most * sms() + 1, 3, 10)
    r, launches = planned(pb)
    assert launches != 3
    assert result(r) == level_by_level(pb)


def test_acceptance_that_comes_back():
    # the coldest start accepts little; a cooling factor above one is refused,
    # so the way back is the box: a start at its corner, where most proposals
    # are outside or uphill, and whose levels move into the middle
    pb = problem(sg.HAGAN, sg.FP32, 1, 15, 64, 30, 40, T0=0.05, factor=0.6, x0=[0.999, 0.0, 0.9, 2.9], step0=0.3)
    r, launches = planned(pb)
    assert launches == 3
    assert result(r) == level_by_level(pb)
