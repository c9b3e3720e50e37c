"""The FP32 smoothing passes that march in z (sizes that are multiples of 4):
block, row and plane-column remainders, against the CPU oracle."""

import numpy as np
import pytest
import torch

from gpu_helpers import assert_close_field, dev, empty, from_split, host, to_split
from oracle import pfc_oracle as O
from paper_1611_06288_gb300 import binding as B

pytestmark = pytest.mark.gpu

EPS, TAU = 0.1, 0.05
# One pass forms each value from about 40 FP32 operations on terms of the size
# of its result, so its relative error is below 40 * 2^-24 ~ 2.4e-6; two
# sweeps (the second contracts the first one's error) stay below 1e-5.
F32_RTOL = 1e-5


def fields(n):
    rng = np.random.default_rng(500 + n)
    d = [(0.1 * rng.standard_normal((n,) * 3)).astype(np.float32) for _ in range(3)]
    r = [rng.standard_normal((n,) * 3).astype(np.float32) for _ in range(3)]
    q = (0.5 + 0.1 * rng.random((n,) * 3)).astype(np.float32)
    return d, r, q


# rows of one thread (4), of 5, 17 and 19 (no divisor of a block), of 33 in two
# parts of 17 (132); one plane a thread at the small sizes, two at 76, four at 132
@pytest.mark.parametrize("n", [4, 8, 20, 68, 76, 132])
@pytest.mark.parametrize("kind", ["rb", "jacobi"])
@pytest.mark.parametrize("zero_init", [True, False])
def test_marching_passes_match_oracle(n, kind, zero_init):
    h = 0.8
    d, r, q = fields(n)
    if zero_init:
        d = [np.zeros_like(x) for x in d]
    g = [dev(to_split(x), torch.float32) for x in d]
    if zero_init:
        for x in g:
            x.fill_(float("nan"))
    rq = [dev(to_split(x), torch.float32) for x in (*r, q)]
    if kind == "rb":
        B.pfc_op_lin_smooth(n, h, EPS, TAU, 2, zero_init, *g, *rq)
    else:
        t = [empty(n, torch.float32) for _ in range(3)]
        B.pfc_op_lin_jacobi(n, h, EPS, TAU, 2, 0.7, zero_init, *g, *t, *rq)
    f64 = lambda v: [x.astype(np.float64) for x in v]
    ref = O.linear_smooth(f64(d), f64(r), q.astype(np.float64), h, O.Params(eps=EPS, tau=TAU), 2,
                          kind)
    for x, y, name in zip(g, ref, ("d_phi", "d_mu", "d_om")):
        assert_close_field(from_split(host(x)), y, F32_RTOL, name)
