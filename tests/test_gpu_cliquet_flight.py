"""Cliquets in flight: a call returns without waiting for the calls before it,
on one stream or several, and every one prices what it prices alone."""
import pytest
import torch

import paper_2407_20713_gb300 as sg

pytestmark = pytest.mark.gpu


def price(i, stream=None):
    return sg.mc_cliquet(sg.DYN_I if i % 2 else sg.HAGAN, [0.3, 0.7, -0.6, 0.9, 0.5, 1.2], 1.0, 1.0, 4, -0.02, 0.02, 0.0,
                         0.2, n_paths=3000 + 7 * i, steps_per_year=20.0, seed=i, stream=stream)


@pytest.mark.parametrize("streams", [1, 3])
def test_calls_do_not_wait_for_calls_in_flight(streams):
    alone = [[t.cpu() for t in price(i)] for i in range(14)]
    side = [torch.cuda.Stream() for _ in range(streams)]
    blocker = torch.cuda.Event()
    with torch.cuda.stream(side[0]):
        torch.cuda._sleep(1_000_000_000)  # about half a second
        blocker.record()
    for s in side[1:]:
        s.wait_event(blocker)
    got = [price(i, side[i % streams]) for i in range(14)]
    assert not blocker.query()
    torch.cuda.synchronize()
    for a, b in zip(got, alone):
        assert all(torch.equal(x.cpu(), y) for x, y in zip(a, b))
    # the kept scratches are free again
    again = [[t.cpu() for t in price(i)] for i in range(14)]
    assert all(torch.equal(x, y) for a, b in zip(again, alone) for x, y in zip(a, b))
