"""The pricing's work count over the live reset dates only (CPU)."""
import pytest

import bench
from paper_2211_17005_gb300 import workload


@pytest.mark.parametrize("name,n,G", [("paper", 100, 10), ("batched", 120, 10), ("small", 50, 5), ("paper", 20, 10)])
def test_mean_count_adds_the_live_dates_one_by_one(name, n, G):
    wl = workload.make(name, M=256, n_steps=n)
    E, C, P = wl.model.E, wl.model.C, len(wl.portfolios)
    total = 0
    for j in range(1, n + 1):
        t = j * wl.grid.horizon / n
        live = [T for T in range(1, G + 1) if T >= t - 1e-9]   # coupon dates not yet past
        if live:
            total += E * (20 + 12 * len(live) + P * C * (2 * len(live) + 1)) + 3 * P * C + 6
    assert bench.price_instr_mean(wl) == pytest.approx(total / n, rel=1e-12)


def test_count_of_the_timed_workload():
    # half the reset dates and one more on average: 5.5 of 10
    assert bench.price_instr_mean(workload.make("paper", M=256)) == pytest.approx(1850.0)
