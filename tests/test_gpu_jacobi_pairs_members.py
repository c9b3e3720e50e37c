"""Jacobi sweeps in pairs over the members of an ensemble: member m is one run's
field moved by whole coarsest cells of the periodic box, so its result is that
run's, moved alike, bit for bit (every sum of the scheme and of the cycle keeps its
order under such a move)."""

import pytest
import torch

from paper_1611_06288_gb300.solver import PFCBatch

pytestmark = pytest.mark.gpu


# every finest level that an ensemble's grid can have in the three widths of the
# kernel, with the fewest members whose fields pass its bound of 86 MiB; one run
# alone stays below it and takes single sweeps
@pytest.mark.parametrize("n,coarsest,members", [
    (40, 10, 36), (48, 12, 21), (56, 14, 13), (64, 16, 9), (80, 10, 5), (96, 12, 3),
    (112, 14, 2), (128, 16, 2)])
@pytest.mark.parametrize("nu1,factor", [(0, 4), (1, 3)])
def test_members_equal_single_runs(n, coarsest, members, nu1, factor):
    assert 40 * n ** 3 * members > 86 << 20 >= 40 * n ** 3
    kw = dict(tol=1e-9, max_cycles=80, nu1=nu1, nu2=1, inner_cycles=2, jacobi_factor0=factor,
              jacobi_factor=factor, stiff_hi=1e9, stiff_lo=0.0, coarsest=coarsest)
    g = torch.Generator(device="cuda").manual_seed(n)
    one = 0.1 + 0.05 * (2 * torch.rand((n, n, n), generator=g, device="cuda",
                                       dtype=torch.float64) - 1)
    s, c = 2 * n // coarsest, coarsest // 2
    moves = [(s * (m % c), s * (m // c % c), s * ((3 * m + m // (c * c)) % c))
             for m in range(members)]
    assert len(set(moves)) == members
    run = PFCBatch(n, 0.8 * n, [0.1], 0.05, one[None], **kw)
    run.step(2)
    ref = [f()[0] for f in (run.phi, run.mu, run.omega)]
    cycles = int(run.status()[0][0])
    run.close()
    b = PFCBatch(n, 0.8 * n, [0.1] * members, 0.05,
                 torch.stack([one.roll(d, (0, 1, 2)) for d in moves]), **kw)
    b.step(2)
    assert [int(x) for x in b.status()[0]] == [cycles] * members
    for f, x in zip((b.phi, b.mu, b.omega), ref):
        y = f()
        for m, d in enumerate(moves):
            assert torch.equal(y[m], x.roll(d, (0, 1, 2))), m
    b.close()
