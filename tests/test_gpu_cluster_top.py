"""Which coarse tail the settings of cluster_tail run: 1 the cluster, also where its
top level has 16^3 cells (the whole grid, or a level of its own), 0 and 2 one block.
The two add in different orders, so equal bits mean the same kernel."""

import numpy as np
import pytest

from gpu_helpers import rel_l2
from oracle import pfc_oracle as O
from test_gpu_cluster import AGREE_RTOL, TOL, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,settings", [
    (16, dict(nu1=0, nu2=1, inner_cycles=2, jacobi_factor=4, coarse_sweeps=2)),
    (16, dict(nu1=1, nu2=2, inner_cycles=2, jacobi_factor=3, coarse_sweeps=4, coarsest=8)),
    (64, dict(nu1=0, nu2=1, inner_cycles=2, jacobi_factor=4, coarse_sweeps=2)),
])
def test_mode_one_is_the_cluster_and_two_is_zero(n, settings):
    h, eps, dt = 1.0, 0.025, 0.0125
    rng = np.random.default_rng(n)
    phi0 = 0.07 + 0.05 * rng.uniform(-1, 1, (n, n, n))
    out = {c: run(n, h * n, eps, dt, phi0, 3, c, **settings) for c in (0, 1, 2)}
    assert out[2][0] == out[0][0]
    for x, y in zip(out[2][1], out[0][1]):
        assert np.array_equal(x, y)
    assert not np.array_equal(out[1][1][0], out[0][1][0])
    assert all(abs(a - b) <= 1 for a, b in zip(out[1][0], out[0][0]))
    for x, y in zip(out[1][1][:3], out[0][1][:3]):
        assert rel_l2(x, y) <= AGREE_RTOL
    # rows 1 and 3 of the cluster run's last step in the oracle's FP64
    a, mu, om, b = out[1][1]
    p = O.Params(eps=eps, tau=dt)
    r = O.residual(O.source_S(b, b, h, p), [a, mu, om], b, h, p)
    assert np.sqrt(np.mean(r[0] ** 2 + r[2] ** 2) / 3) <= TOL * 1.0001
