"""u += d in the last smoothing pass of a correction, on red-black and Jacobi
finest levels, and beside it for double-float states: steps against the CPU
oracle.  A cell that the pass left out or added to twice would keep the residual
above the tolerance."""

import functools

import numpy as np
import pytest
import torch

from gpu_helpers import host, rel_l2
from oracle import pfc_oracle as O
from paper_1611_06288_gb300 import binding as B
from paper_1611_06288_gb300.solver import PFCBatch, PFCSolver

pytestmark = pytest.mark.gpu

# Both sides converge the same nonlinear system to an RMS residual of 1e-11 (the
# double-float one to 1e-10); the fields are O(0.1) and the inverse O(1).
RTOL = 1e-9
L_PER_CELL, DT = 0.8, 0.05
JACOBI = dict(tol=1e-11, max_cycles=400, nu1=1, nu2=1, stiff_hi=1e9, stiff_lo=0.0)


def start(n, seed):
    return 0.1 + 0.05 * np.random.default_rng(seed).uniform(-1, 1, (n, n, n))


@functools.lru_cache(maxsize=None)
def reference(n, seed, eps):
    return O.run(start(n, seed), 2, L_PER_CELL, O.Params(eps=eps, tau=DT), tol=1e-11)


# 40: rows of ten threads, no divisor of a block; 64 without pre-smoothing: the
# prolongation fuses with the only sweep unless that one adds to u
@pytest.mark.parametrize("n,kw", [(40, {}), (40, dict(inner_cycles=2, jacobi_factor0=3)),
                                  (40, dict(policy="rb")),
                                  (64, dict(nu1=0, jacobi_factor0=1))])
@pytest.mark.parametrize("precision", ["mixed", "mixed_df"])
def test_folded_steps_match_oracle(n, kw, precision):
    args = {**JACOBI, **kw}
    if precision == "mixed_df":
        args["tol"] = 1e-10
    s = PFCSolver(n, L_PER_CELL * n, 0.1, DT, start(n, n), precision=precision, **args)
    s.step(2)
    ref = reference(n, n, 0.1)
    assert rel_l2(host(s.phi()), ref[0]) <= RTOL
    s.close()


def test_folded_ensemble_matches_oracle():
    n, eps = 40, [0.05, 0.1, 0.2]
    b = PFCBatch(n, L_PER_CELL * n, eps, DT, np.stack([start(n, m) for m in range(3)]), **JACOBI)
    b.step(2)
    phi = host(b.phi())
    for m in range(3):
        assert rel_l2(phi[m], reference(n, m, eps[m])[0]) <= RTOL, m
    b.close()


@pytest.mark.parametrize("policy", ["hybrid", "rb"])
def test_adjoint_field_at_any_element(policy):
    """The adjoint's z is the caller's: one that rules 16-byte moves out takes the
    separate u += d and gives the same bits."""
    n = 40
    s = PFCSolver(n, L_PER_CELL * n, 0.1, DT, start(n, 1), precision="mixed",
                  **{**JACOBI, "policy": policy})
    s.step(1)
    phi_k = s.phi().clone()
    s.step(1)
    phi = s.phi().clone()
    g = torch.from_numpy(start(n, 2)).cuda()
    out = []
    for shift in (0, 1):
        z = torch.zeros(3 * n ** 3 + shift, dtype=torch.float64, device="cuda")[shift:]
        gk, gkm1 = torch.zeros_like(g), torch.zeros_like(g)
        torch.cuda.synchronize()
        eb, cycles = B.pfc_adjoint_step(s.ctx, phi, phi_k, g, gk, gkm1, z, 1e-8)
        out.append((eb, cycles, host(gk), host(gkm1), host(z)))
    assert out[0][1] >= 1 and out[0][:2] == out[1][:2]
    for x, y in zip(out[0][2:], out[1][2:]):
        assert np.array_equal(x, y)
    s.close()
