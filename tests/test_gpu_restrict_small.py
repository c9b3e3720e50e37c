"""FP32 residual restriction on small levels (three threads a coarse cell) and just
past their bound, with rows, columns and planes that no block divides, against the
CPU oracle."""

import numpy as np
import pytest
import torch

from gpu_helpers import assert_close_field, dev, empty, from_split, host, to_split
from oracle import pfc_oracle as O
from paper_1611_06288_gb300 import binding as B

pytestmark = pytest.mark.gpu

EPS, TAU, H = 0.1, 0.05, 0.8
# A value is the mean of 8 rows of at most 10 FP32 terms, summed in 40 operations;
# its terms are up to 30 times the result's scale: 40 * 30 * 2^-24 ~ 7e-5.
F32_RTOL = 1e-4


# coarse sizes 2, 10, 22, 24 (below 2^14 cells) and 26 (past them)
@pytest.mark.parametrize("n", [4, 20, 44, 48, 52])
def test_restricted_residual_matches_oracle(n):
    rng = np.random.default_rng(n)
    f32 = lambda: rng.standard_normal((n,) * 3).astype(np.float32)
    d, r, q = [f32() for _ in range(3)], [f32() for _ in range(3)], f32()
    out = [empty(n // 2, torch.float32) for _ in range(3)]
    put = lambda x: dev(to_split(x), torch.float32)
    B.pfc_op_lin_residual_restrict(n, H, EPS, TAU, False, *map(put, d), *map(put, r), put(q), *out)
    f64 = lambda v: [x.astype(np.float64) for x in v]
    jd = O.jacobian_apply(f64(d), q.astype(np.float64), H, O.Params(eps=EPS, tau=TAU))
    for g, x, y, name in zip(out, f64(r), jd, ("r1", "r2", "r3")):
        assert_close_field(from_split(host(g)), O.restrict(x - y), F32_RTOL, name)
