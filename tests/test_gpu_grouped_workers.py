"""The grouped schedule's counts where the period of the deal, twice the workers,
passes 2^31."""
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_more_workers_than_two_to_the_thirty(lib, reading):
    n = 3 << 29                                     # workers; the period is 3 * 2^30
    M, N, K, tile = 1 << 30, 1 << 20, 64, (64, 64, 64, 2, 1)
    theta = O.prior_theta(152, reading=reading)
    theta[3] = 0.0                                  # a tile's time does not depend on the working set
    launch = float(theta[0]) + (float(theta[13]) if reading else 0.0)
    tau = lib.pm_grouped_predict([64], 64, K, [64], [64], *tile[2:], 1, theta, 1) - launch
    # 2^39 tiles: 170 periods and 2^31 tiles more, so the busiest worker has 2 * 170 + 2
    tiles = 2 * (M // 64) * (N // 64)
    per, rem = divmod(tiles, 2 * n)
    assert (per, rem) == (170, 1 << 31)
    t = lib.pm_grouped_predict([M, M], N, K, [64, 64], [64, 64], *tile[2:], 1, theta, n)
    assert t == pytest.approx(launch + 342 * tau, rel=1e-4)
