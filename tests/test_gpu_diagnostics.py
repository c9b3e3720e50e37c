"""The energy and mass sums of the stored states, formed by blocks that add their
components row by row: one cell a thread and fewer, several, ragged remainders
of four cells, and ensembles, against the CPU oracle on the same fields."""

import numpy as np
import pytest

from gpu_helpers import host
from oracle import pfc_oracle as O
from paper_1611_06288_gb300 import workloads as W
from paper_1611_06288_gb300.solver import PFCBatch, PFCSolver

pytestmark = pytest.mark.gpu

# F's terms cancel to no less than 1 / 20 of the largest at these fields; a sum
# of N <= 10^6 terms on each side is off by at most ~100 eps = 1.1e-14 of its
# terms' magnitudes in the trees used, and the stored Laplacian by 2e-15.
RTOL = 1e-12


def check(d, a, b, h, eps):
    assert d["energy"] == pytest.approx(O.energy(a, h, eps), rel=RTOL)
    assert d["modified_energy"] == pytest.approx(O.modified_energy(a, b, h, eps), rel=RTOL)
    assert d["mass"] == pytest.approx(O.mass(a, h), rel=RTOL)
    assert d["grad_sq"] == pytest.approx(O.grad_norm2_sq(a, h), rel=RTOL)


def start(n, seed):
    return 0.3 + 0.1 * np.random.default_rng(seed).uniform(-1, 1, (n, n, n))


@pytest.mark.parametrize("n", [4, 16, 40, 80])
def test_step_diagnostics_of_one_run(n):
    s = PFCSolver(n, 0.8 * n, 0.1, 0.01, start(n, n), tol=1e-9, precision="mixed",
                  step_diagnostics=True)
    s.step(1)
    b = host(s.phi())
    s.step(1)
    check(s.diagnostics(), host(s.phi()), b, 0.8, 0.1)
    s.close()


@pytest.mark.parametrize("n,count", [(16, 3), (8, 40), (8, 64)])
def test_step_diagnostics_of_an_ensemble(n, count):
    eps = list(np.linspace(0.05, 0.25, count))
    phi0 = np.stack([start(n, m) for m in range(count)])
    s = PFCBatch(n, 0.8 * n, eps, 0.01, phi0, tol=1e-9, step_diagnostics=True,
                 **W.ENSEMBLE_SETTINGS)
    s.step(1)
    b = host(s.phi())
    s.step(1)
    a = host(s.phi())
    for m, d in enumerate(s.diagnostics()):
        check(d, a[m], b[m], 0.8, eps[m])
    s.close()
