"""FP32 and FP64 Hagan chains on several lanes outside the few-chain kernel: a
batch of small problems (none alone of its kind) and single problems just above
the few-chain limit run the speculative loop of the queue and level kernels.  It
is compared bit for bit with the one-step loop, and the two launch shapes with
each other, at chain lengths below and beside the speculation depth."""
import numpy as np
import pytest
import torch

import paper_2407_20713_gb300 as sg
from paper_2407_20713_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def smile(strikes, chains, levels, length, prec, seed):
    T, K = np.ones(strikes), np.linspace(0.7, 1.3, strikes)
    mkt = sg.implied_vol(sg.HAGAN, [0.25, 0.7, -0.4, 0.5], 1.0, T, K, prec=sg.FP64).cpu().numpy()
    mkt = mkt * (1 + 1e-3 * np.random.default_rng(seed).normal(size=strikes))
    return sg.CalibrationProblem(model=sg.HAGAN, T=T, K=K, market=mkt, lo=W.STATIC_LO, hi=W.STATIC_HI, prec=prec,
                                 n_chains=chains, n_levels=levels, chain_len=length, seed=seed)


def result(r):
    return (tuple(r.params), tuple(r.restart_params), r.misfit, r.misfit_fp64, r.restart_misfit, r.n_evals, r.n_accepts,
            r.status)


def run(problems):
    plan = sg.Plan(problems)
    plan.run()
    out, launches = [result(r) for r in plan.results()], plan.stats()[0]
    plan.close()
    return out, launches


@pytest.mark.parametrize("prec", [sg.FP32, sg.FP64])
@pytest.mark.parametrize("length", [1, 2, 3, 5, 7, 40])
def test_batches_of_small_problems(prec, length, monkeypatch):
    pbs = [smile(st, ch, 4, length, prec, 3 + i) for i, (st, ch) in enumerate([(8, 20), (15, 48), (4, 1), (31, 200)])]
    spec, _ = run(pbs)
    monkeypatch.setenv("SABR_SPECULATE", "0")
    plain, _ = run(pbs)
    assert spec == plain and all(r[-1] == 0 for r in spec)


@pytest.mark.parametrize("length", [1, 2, 31])
def test_single_problems_above_the_few_chain_limit(length, monkeypatch):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    pb = smile(15, 8 * sms + 1, 4, length, sg.FP32, 9)
    queued, launches = run([pb])
    assert launches == 4  # init, queue reset, the queue kernel, finalize
    monkeypatch.setenv("SABR_PLAN_QUEUE", "0")
    levels, launches = run([pb])
    assert launches == 1 + 4 + 1
    monkeypatch.setenv("SABR_SPECULATE", "0")
    plain, _ = run([pb])
    assert queued == levels == plain
