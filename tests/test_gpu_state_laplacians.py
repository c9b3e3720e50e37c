"""pfc_set_state forms both fields' Laplacians in one launch, and copies the field
where no previous one is given: the same state either way, on sizes that a block
does and does not divide; the first step's source reads them."""

import numpy as np
import pytest

from gpu_helpers import host, rel_l2
from oracle import pfc_oracle as O
from paper_1611_06288_gb300.solver import PFCSolver

pytestmark = pytest.mark.gpu

# Both sides converge the same nonlinear system to an RMS residual of 1e-11; the
# fields are O(0.1) and the inverse O(1).
RTOL = 1e-9


def start(n, seed):
    return 0.1 + 0.05 * np.random.default_rng(seed).uniform(-1, 1, (n, n, n))


@pytest.mark.parametrize("n,precision", [(4, "mixed"), (16, "mixed"), (24, "mixed"),
                                         (80, "mixed"), (8, "fp64"), (64, "fp64")])
def test_state_with_and_without_a_previous_field(n, precision):
    a, b = start(n, 1), start(n, 2)
    out = []
    for prev in (None, a, b):
        s = PFCSolver(n, 0.8 * n, 0.1, 0.05, start(n, 3), tol=1e-11, max_cycles=200,
                      precision=precision)
        s.set_state(a, prev)
        s.step(1)
        out.append(host(s.phi()))
        s.close()
    assert np.array_equal(out[0], out[1])        # phi^{-1} := phi^0 is the default
    if n <= 16:
        ref = O.run(b, 1, 0.8, O.Params(eps=0.1, tau=0.05), tol=1e-11, phi1=a)[0]
        assert rel_l2(out[2], ref) <= RTOL
    else:
        assert not np.array_equal(out[2], out[1])
