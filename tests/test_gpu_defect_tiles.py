"""The FP64 defect's two tiles: blocks of four rows, and of eight where columns of
four are more than the partial-sum slots."""

import numpy as np
import pytest

from gpu_helpers import host
from paper_1611_06288_gb300 import workloads as W
from paper_1611_06288_gb300.solver import PFCBatch

pytestmark = pytest.mark.gpu


def test_tiles_give_the_same_fields():
    """8^3: with one plane a block, 600 members are 9600 blocks of four rows, within
    the 9728 slots; 1000 are 16000 of four and 8000 of eight.  Rows are the same
    arithmetic whatever the tile."""
    n, dt = 8, 0.02
    rng = np.random.default_rng(3)
    for count, planes in ((600, (1, 2, 8)), (1000, (1, 8))):
        eps = list(rng.uniform(0.05, 0.2, count))
        phi0 = 0.1 + 0.05 * rng.uniform(-1, 1, (count, n, n, n))
        out = []
        for z in (0, *planes):
            b = PFCBatch(n, 0.8 * n, eps, dt, phi0, tol=1e-9, defect_planes=z,
                         **W.ENSEMBLE_SETTINGS)
            b.step(2)
            out.append((b.status()[0], host(b.phi())))
            b.close()
        for its, phi in out[1:]:
            assert list(its) == list(out[0][0])
            assert np.array_equal(phi, out[0][1])
