"""The FP64 transfers of the FAS cycle over both sides of their size rule (coarse
levels from 32^3 take the block-sum restriction and the tiled prolongation) and
with buffers that rule the 16-byte loads out, against the CPU oracle."""

import numpy as np
import pytest
import torch

from gpu_helpers import assert_close_field, host
from oracle import pfc_oracle as O
from paper_1611_06288_gb300 import binding as B

pytestmark = pytest.mark.gpu

EPS, TAU, H = 0.1, 0.05, 0.8
# Every value is a sum of at most 60 FP64 terms no larger than 12 / H^2 times
# the largest field value (about 20): 60 * 20 * 2^-53 ~ 1.3e-13.
FP64_RTOL = 1e-12


def field(x, shift):
    """x on the device, its first element `shift` doubles into an allocation."""
    t = torch.empty(x.size + shift, dtype=torch.float64, device="cuda")[shift:].view(x.shape)
    return t.copy_(torch.from_numpy(np.ascontiguousarray(x)))


# 62: the largest level of the small kernels; 64: the first of the large ones;
# 68 and 76: coarse sizes 34 and 38, ragged in the tiles of 32 x 4 columns and in
# the planes of a block
@pytest.mark.parametrize("n", [2, 16, 62, 64, 68, 76])
@pytest.mark.parametrize("shift", [0, 1])
def test_restriction_and_prolongation(n, shift):
    rng = np.random.default_rng(40 + n)
    nc = n // 2
    b = 0.2 + 0.1 * rng.standard_normal((n, n, n))
    u = [b + 0.02 * rng.standard_normal(b.shape), rng.standard_normal(b.shape),
         rng.standard_normal(b.shape)]
    S = [b, rng.standard_normal(b.shape), rng.standard_normal(b.shape)]
    prm = O.Params(eps=EPS, tau=TAU)
    d = [field(x, shift) for x in (*u, *S, b)]
    out = [field(np.zeros((nc,) * 3), shift) for _ in range(6)]
    B.pfc_op_residual_restrict(n, H, EPS, TAU, *d, *out)
    for g, x, name in zip(out[:3], O.residual(S, u, b, H, prm), ("r1", "r2", "r3")):
        assert_close_field(host(g), O.restrict(x), FP64_RTOL, name)
    for g, x in zip(out[3:], u):
        assert_close_field(host(g), O.restrict(x), 1e-15, "u")
    v = [rng.standard_normal((nc,) * 3) for _ in range(3)]
    w = [rng.standard_normal((nc,) * 3) for _ in range(3)]
    dw = [field(x, shift) for x in w]
    B.pfc_op_prolong_correct(n, *[field(x, shift) for x in v], *dw, *d[:3])
    for g, x, vv, ww in zip(d[:3], u, v, w):
        assert_close_field(host(g), x + O.prolong(vv - ww), 1e-14, "u + P(v - w)")
    for g, ww in zip(dw, w):
        assert np.array_equal(host(g), ww)            # the inputs stay as they were
