"""Jacobi sweeps in pairs on levels larger than L2 holds: the bits of single sweeps,
for even and odd counts, from zero and from d, with row tiles that do not divide
the level; and small grids of an ensemble against runs made one at a time."""

import numpy as np
import pytest
import torch

from gpu_helpers import host, rel_l2
from paper_1611_06288_gb300 import binding as B
from paper_1611_06288_gb300.solver import PFCBatch, PFCSolver

pytestmark = pytest.mark.gpu

EPS, TAU, H, W = 0.1, 0.05, 0.8, 0.7


# 132: the first size past the bound, rows of 33 threads; 216: nine rows of 54;
# 256: the largest, rows of a whole warp; 260: past it, single sweeps
@pytest.mark.parametrize("n", [132, 216, 256, 260])
@pytest.mark.parametrize("sweeps", [2, 3, 4])
@pytest.mark.parametrize("zero_init", [False, True])
def test_pairs_equal_single_sweeps(n, sweeps, zero_init):
    g = torch.Generator(device="cuda").manual_seed(n)
    f32 = lambda: torch.randn(n ** 3, generator=g, device="cuda", dtype=torch.float32)
    d0 = [f32() for _ in range(3)]
    r, q = [f32() for _ in range(3)], 0.5 + 0.1 * f32()
    nan = float("nan")
    out = []
    for calls in ([sweeps], [1] * sweeps):
        d = [torch.full_like(x, nan) if zero_init else x.clone() for x in d0]
        t = [torch.full_like(x, nan) for x in d0]
        for i, s in enumerate(calls):
            B.pfc_op_lin_jacobi(n, H, EPS, TAU, s, W, zero_init and i == 0, *d, *t, *r, q)
        torch.cuda.synchronize()
        out.append(d)
    for a, b in zip(*out):
        assert torch.isfinite(a).all()
        assert torch.equal(a, b)


def test_pairs_with_fields_at_any_element():
    """A field off a 16-byte boundary takes single sweeps."""
    n = 132
    g = torch.Generator(device="cuda").manual_seed(1)
    f32 = lambda s: torch.randn(n ** 3 + s, generator=g, device="cuda", dtype=torch.float32)[s:]
    d0, r, q = [f32(0) for _ in range(3)], [f32(0) for _ in range(3)], f32(0)
    out = []
    for s in (0, 2):
        move = lambda x: torch.cat([x[:s], x])[s:].clone() if s == 0 else torch.cat([x[:s], x])[s:]
        d, t = [move(x) if s else x.clone() for x in d0], [torch.empty_like(x) for x in d0]
        B.pfc_op_lin_jacobi(n, H, EPS, TAU, 2, W, False, *d, *t, *r, q)
        torch.cuda.synchronize()
        out.append([host(x) for x in d])
    for a, b in zip(*out):
        assert np.array_equal(a, b)


# the three row widths that ensembles reach; past the bound, their single runs far
# below it
@pytest.mark.parametrize("n,count,factor", [(64, 13, 2), (48, 33, 3), (80, 5, 4)])
def test_ensemble_in_pairs_equals_single_runs(n, count, factor):
    kw = dict(tol=1e-11, max_cycles=80, nu1=1, nu2=1, inner_cycles=2, jacobi_factor0=factor,
              stiff_hi=1e9, stiff_lo=0.0)
    rng = np.random.default_rng(n)
    eps = list(rng.uniform(0.05, 0.2, count))
    phi0 = 0.1 + 0.05 * rng.uniform(-1, 1, (count, n, n, n))
    b = PFCBatch(n, 0.8 * n, eps, 0.05, phi0, **kw)
    b.step(2)
    got = host(b.phi())
    b.close()
    for m in (0, count // 2, count - 1):
        s = PFCSolver(n, 0.8 * n, eps[m], 0.05, phi0[m], precision="mixed", **kw)
        s.step(2)
        assert rel_l2(got[m], host(s.phi())) <= 1e-10, m
        s.close()
