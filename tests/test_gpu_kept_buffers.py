"""Buffers kept between calls: the blocking calibrations' arena and results,
and the pricers' two scratches.  Calls of different sizes in any order, on
several streams and from several threads at once give what each gives alone."""
import threading

import numpy as np
import pytest
import torch

import paper_2407_20713_gb300 as sg
from paper_2407_20713_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def calibration(i):
    T, K = np.ones(9 + i), np.linspace(0.7, 1.3, 9 + i)
    mkt = np.full(T.size, 0.2) + 0.02 * (K - 1) ** 2
    return sg.CalibrationProblem(model=sg.HAGAN, T=T, K=K, market=mkt, lo=W.STATIC_LO, hi=W.STATIC_HI,
                                 n_chains=(20, 3000, 64, 9000)[i % 4], n_levels=3, chain_len=10, seed=i)


def result(r):
    return (tuple(r.params), r.misfit, r.misfit_fp64, r.n_evals, r.n_accepts, r.status)


def price(i, stream=None):
    n = 1 + 3 * (i % 5)
    T = np.repeat([0.25, 0.5], n)
    K = np.tile(np.linspace(0.8, 1.2, n), 2)
    if i % 3 == 2:
        return sg.mc_cliquet(sg.DYN_I, [0.3, 0.7, -0.6, 0.9, 0.5, 1.2], 1.0, 1.0, 4, -0.02, 0.02, 0.0, 0.2,
                             n_paths=3000 + 7 * i, steps_per_year=20.0, seed=i, stream=stream)
    return sg.mc_price(sg.HAGAN, [0.3, 0.6, -0.4, 0.7], 1.0, T, K, n_paths=2000 + 501 * i, steps_per_year=30.0, seed=i,
                       stream=stream, scheme=sg.MC_BESSEL if i % 3 else None)


def test_calls_of_many_sizes_and_threads():
    alone = [result(sg.calibrate(calibration(i))) for i in range(8)]
    batch = [result(r) for r in sg.calibrate_batch([calibration(i) for i in (0, 2)])]
    prices = [[t.cpu() for t in price(i)] for i in range(12)]
    assert alone[0] == batch[0] and alone[2] == batch[1]
    bad = []

    def work(k):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            for i in range(8):
                j = (3 * i + k) % 8
                if result(sg.calibrate(calibration(j), stream=stream)) != alone[j]:
                    bad.append(("calibrate", k, j))
            got = [(j, price(j, stream)) for j in ((5 * i + k) % 12 for i in range(24))]
            stream.synchronize()
            for j, v in got:
                if not all(torch.equal(a.cpu(), b) for a, b in zip(v, prices[j])):
                    bad.append(("price", k, j))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_prices_in_a_row_before_any_is_read():
    ref = [[t.cpu() for t in price(i)] for i in range(10)]
    got = [price(i) for i in range(10)]  # enqueued without waiting
    torch.cuda.synchronize()
    for a, b in zip(got, ref):
        assert all(torch.equal(x.cpu(), y) for x, y in zip(a, b))
