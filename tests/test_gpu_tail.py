"""One correction of the mixed solver on grids whose coarse levels run in the
one-block tail, against the oracle's smoothers and transfers in FP64: the update
itself, not the field that the outer loop converges to."""

import numpy as np
import pytest

from gpu_helpers import host
from oracle import pfc_oracle as O
from paper_1611_06288_gb300.solver import PFCBatch

pytestmark = pytest.mark.gpu

DT = 0.05


def level_cycle(l, last, d, r, q, h, prm, kind, p):
    """One V-cycle on J d = r (levels l .. last, every one smoothed by `kind`)."""
    if l == last:
        return O.linear_smooth([np.zeros_like(x) for x in r], r, q[l], h, prm,
                               p["coarse_sweeps"], kind)
    f = (p["jacobi_factor0"] if l == 0 else p["jacobi_factor"]) if kind == "jacobi" else 1
    d = O.linear_smooth(d, r, q[l], h, prm, p["nu1"] * f, kind)
    rho = [O.restrict(x - y) for x, y in zip(r, O.jacobian_apply(d, q[l], h, prm))]
    e = level_cycle(l + 1, last, [np.zeros_like(x) for x in rho], rho, q, 2 * h, prm, kind, p)
    d = [x + O.prolong(y) for x, y in zip(d, e)]
    return O.linear_smooth(d, r, q[l], h, prm, p["nu2"] * f, kind)


def correction(u, b, h, n, coarsest, prm, kind, p):
    """(residual of u, update of one correction)."""
    r = O.residual(O.source_S(b, b, h, prm), u, b, h, prm)
    q = [O.jacobian_coefficient(u[0], b, prm)]
    while n > coarsest:
        n //= 2
        q.append(O.restrict(q[-1]))
    d = [np.zeros_like(x) for x in r]
    for _ in range(p["inner_cycles"]):
        d = level_cycle(0, len(q) - 1, d, r, q, h, prm, kind, p)
    return r, d


# 4, 8, 12, 16: the whole cycle in the tail, its top from zero and (second cycle)
# from d; 20, 24, 28: a coarsest level of 10, 12 and 14 cells alone or under one
# more; 14^3 is the size whose threads hold two positions each
@pytest.mark.parametrize("n,coarsest", [(4, 2), (8, 2), (12, 6), (16, 2), (16, 8), (20, 10),
                                        (24, 6), (28, 14)])
@pytest.mark.parametrize("kind,nu1,nu2,factor,sweeps", [
    ("rb", 1, 2, 1, 3), ("rb", 0, 1, 1, 2), ("jacobi", 1, 1, 3, 3), ("jacobi", 0, 1, 2, 4),
    ("jacobi", 2, 1, 1, 1)])
@pytest.mark.parametrize("members,cycles", [(1, 1), (3, 2)])
def test_one_correction(n, coarsest, kind, nu1, nu2, factor, sweeps, members, cycles):
    """FP32 against FP64.  A cell's solve rounds sums of about 20 terms of the size
    of d (h = 1: the couplings are 1 to 6, det > 6) to 2^-24, 20 * 2^-24 / 6 < 2e-7
    of the largest |d| a sweep; at most 40 sweeps and transfers: 1e-5.  One wrong
    neighbour or weight is 1e-2."""
    L, eps = float(n), [0.05, 0.15, 0.25][:members]
    p = dict(nu1=nu1, nu2=nu2, jacobi_factor=factor, jacobi_factor0=factor, coarse_sweeps=sweeps,
             inner_cycles=cycles)
    rng = np.random.default_rng(100 * n + coarsest + 7 * sweeps)
    phi0 = 0.1 * np.arange(1, members + 1)[:, None, None, None] \
        + 0.05 * rng.uniform(-1, 1, (members, n, n, n))

    def batch(tol):
        return PFCBatch(n, L, eps, DT, phi0, tol=tol, coarsest=coarsest, coarse_stiffness=0.0,
                        policy="rb" if kind == "rb" else "hybrid", stiff_hi=1e9, stiff_lo=0.0, **p)

    b = batch(1e-9)
    mu, om = host(b.mu()), host(b.omega())
    b.close()
    ref = []
    for m in range(members):
        prm = O.Params(eps=eps[m], tau=DT, jacobi_weight=0.7)
        u = [phi0[m], mu[m], om[m]]
        r, d = correction(u, phi0[m], 1.0, n, coarsest, prm, kind, p)
        v = [x + y for x, y in zip(u, d)]
        ref.append((O.rms(r), O.rms(O.residual(O.source_S(phi0[m], phi0[m], 1.0, prm), v,
                                               phi0[m], 1.0, prm)), u, d))
    # a tolerance that every member meets after one correction, none before it
    first, then = min(x[0] for x in ref), max(x[1] for x in ref)
    assert then < 0.9 * first
    b = batch(float(np.sqrt(first * then)))
    b.step(1)
    assert list(b.status()[0]) == [1] * members
    got = [host(f()) for f in (b.phi, b.mu, b.omega)]
    b.close()
    for m, (_, _, u, d) in enumerate(ref):
        scale = max(float(np.abs(x).max()) for x in d)
        for f in range(3):
            err = float(np.abs(got[f][m] - u[f] - d[f]).max())
            assert err <= 1e-5 * scale, (m, f, err / scale)
