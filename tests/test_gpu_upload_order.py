"""A calibration's tables reach the device before its kernels read them, on
whatever stream it runs: warm calls on side streams (which do not wait for the
default stream) reuse the kept arena, where a late upload would leave the
problem of the call before."""
import threading

import numpy as np
import pytest
import torch

import paper_2407_20713_gb300 as sg
from paper_2407_20713_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def smile(i):
    # one size for all, another market and seed each
    T, K = np.ones(15), np.linspace(0.7, 1.3, 15)
    mkt = 0.15 + 0.01 * i + (0.02 + 0.003 * i) * (K - 1) ** 2
    return sg.CalibrationProblem(model=sg.HAGAN, T=T, K=K, market=mkt, lo=W.STATIC_LO, hi=W.STATIC_HI, n_chains=64,
                                 n_levels=2, chain_len=5, seed=i)


def result(r):
    return (tuple(r.params), r.misfit, r.misfit_fp64, r.n_evals, r.n_accepts, r.status)


def test_warm_calls_on_side_streams_run_their_own_problem():
    alone = [result(sg.calibrate(smile(i))) for i in range(12)]
    assert len(set(alone)) == 12
    bad = []

    def work(k):
        stream = torch.cuda.Stream()
        for i in range(60):
            j = (5 * i + k) % 12
            if result(sg.calibrate(smile(j), stream=stream)) != alone[j]:
                bad.append((k, i))

    work(0)
    threads = [threading.Thread(target=work, args=(k,)) for k in range(1, 5)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


@pytest.mark.parametrize("graph", [False, True])
def test_a_plan_runs_on_a_side_stream_right_after_its_creation(graph):
    alone = [result(sg.calibrate(smile(i))) for i in range(6)]
    for i in range(24):
        plan = sg.Plan([smile(i % 6)], use_graph=graph)
        stream = torch.cuda.Stream()
        plan.run(stream=stream)
        assert result(plan.results()[0]) == alone[i % 6]
