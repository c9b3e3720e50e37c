"""The quotient of the pointwise solve against an IEEE division.  One sweep from
phi = mu = omega = 0 with S1 = S3 = 0 leaves mu = st2 / det on the cells that see
only zeros, with st2 and det formed here in the kernel's own roundings (h and tau
powers of two, so the level's constants are exact)."""

from fractions import Fraction

import numpy as np
import pytest
import torch

from gpu_helpers import dev, host
from paper_1611_06288_gb300 import binding as B

pytestmark = pytest.mark.gpu

N = 16


def fma(a, b, c):
    """Exact a b + c, rounded once."""
    return np.array([float(Fraction(x) * Fraction(y) + Fraction(z))
                     for x, y, z in np.broadcast(a, b, c)])


def colour0():
    k, j, i = np.indices((N, N, N))
    return (i + j + k) % 2 == 0


def first_mu(lin, e, S2, b, eps=0.0):
    """mu of the colour-0 cells after one sweep at h = 2^-e, tau = 1."""
    z = lambda: dev(np.zeros((N, N, N)))
    phi, mu, om, S1, S3 = (z() for _ in range(5))
    B.pfc_op_smooth(N, 2.0 ** -e, eps, 1.0, lin, 1, phi, mu, om, S1, dev(S2), S3, dev(b))
    return host(mu)[colour0()]


# det from just above 1 past 2^123, where the division itself takes over, to 2^970
@pytest.mark.parametrize("lin", [B.PFC_NEWTON, B.PFC_PICARD])
@pytest.mark.parametrize("e", [-4, 0, 3, 10, 18, 19, 20, 21, 80, 160])
def test_quotient_is_the_rounded_one(lin, e):
    """The last operation rounds a quotient that is right to about 2^-89 (a
    reciprocal to 2^-44, squared by the remainder): at most one ulp from the IEEE
    quotient, and equal but for near ties, one value in 2^36."""
    rng = np.random.default_rng(e + 100)
    cQ = 0.5 + 18.0 * 2.0 ** (4 * e)
    kap = 6.0 * 2.0 ** (2 * e)
    u = 10.0 ** rng.uniform(-3, 1, (N, N, N))
    b = np.where(rng.random((N, N, N)) < 0.5, 0.0, np.sqrt(4.0 * u * cQ))
    top = int(0.5 * np.log2(kap * cQ))
    S2 = rng.choice([-1.0, 1.0], (N, N, N)) * np.ldexp(rng.uniform(1, 2, (N, N, N)),
                                                      top + rng.integers(-40, 41, (N, N, N)))
    at = colour0()
    q4 = b[at] * b[at]
    num = fma(0.25, q4 * b[at], S2[at])
    det = fma(kap, fma(0.25, q4, cQ), 1.0)
    ref = num / det
    assert np.isfinite(ref).all() and (ref != 0).all()
    got = first_mu(lin, e, S2, b)
    assert (np.abs(got - ref) <= np.spacing(np.abs(ref))).all()
    assert (got == ref).mean() > 0.999


@pytest.mark.parametrize("e", [-4, 0, 21])
def test_quotient_of_infinities_and_largest_values(e):
    """Numerators without a finite remainder give what a division gives."""
    S2 = np.ones((N, N, N))
    special = np.array([np.inf, -np.inf, np.nan, np.finfo(float).max, -np.finfo(float).max,
                        0.0, 2.0 ** 1022, 2.0 ** -1000])
    at = colour0()
    flat = np.flatnonzero(at)
    S2.ravel()[flat[:len(special)]] = special
    det = fma(6.0 * 2.0 ** (2 * e), 0.5 + 18.0 * 2.0 ** (4 * e), 1.0)
    ref = S2.ravel()[flat] / det
    got = first_mu(B.PFC_NEWTON, e, S2, np.zeros((N, N, N)))
    assert np.array_equal(got, ref, equal_nan=True), (got[:8], ref[:8])


@pytest.mark.parametrize("j", [3, 40, 125, 131, 300])
def test_quotient_by_negative_determinants(j):
    """eps = 1 + 2^j makes (1 - eps)/2 + 18/h^4 and with it det negative, which the
    operation accepts: what a division gives, to one ulp."""
    e = 0 if j > 10 else -4
    rng = np.random.default_rng(j)
    S2 = rng.uniform(-2, 2, (N, N, N))
    det = fma(6.0 * 2.0 ** (2 * e), -(2.0 ** (j - 1)) + 18.0 * 2.0 ** (4 * e), 1.0)
    assert det < 1
    ref = S2[colour0()] / det
    got = first_mu(B.PFC_NEWTON, e, S2, np.zeros((N, N, N)), 1.0 + 2.0 ** j)
    assert (np.abs(got - ref) <= np.spacing(np.abs(ref))).all()


# n = 6: one cell a thread; 16: two
@pytest.mark.parametrize("n", [6, 16])
@pytest.mark.parametrize("e", [-4, 0, 3, 10, 19])
def test_fp32_quotient_within_its_bound(n, e):
    """The FP32 solve's quotient: a reciprocal to one ulp, 2^-23 relative, and one
    rounded product, 2^-24.  One Jacobi sweep of weight 1 from zero with r1 = r3 = 0
    leaves d2 = r2 times it; det from just above 1 to 2^121."""
    rng = np.random.default_rng(n + e)
    f32 = lambda x: np.asarray(x).astype(np.float32)
    Q0, kap = 18.0 * 2.0 ** (4 * e), 6.0 * 2.0 ** (2 * e)
    q = f32(Q0 * 10.0 ** rng.uniform(-3, 0.5, n ** 3))
    r2 = f32(rng.choice([-1.0, 1.0], n ** 3) * np.ldexp(rng.uniform(1, 2, n ** 3),
                                                        rng.integers(0, 41, n ** 3)))
    # kap Q + 1 rounded once: kap Q is exact here, and a 1 below its last place still
    # ends a tie
    kq = kap * f32(q.astype(float) + Q0).astype(float)
    det = f32(np.where(kq + 1.0 == kq, np.nextafter(kq, np.inf), kq + 1.0)).astype(float)
    z = lambda: torch.zeros(n ** 3, device="cuda")
    d, t = [z() for _ in range(3)], [z() for _ in range(3)]
    up = lambda x: dev(x, torch.float32)
    B.pfc_op_lin_jacobi(n, 2.0 ** -e, 0.0, 1.0, 1, 1.0, True, *d, *t, z(), up(r2), z(), up(q))
    ref = r2.astype(float) / det
    bound = (2.0 ** -23 + 2.0 ** -24) * (1 + 2.0 ** -23)
    assert (np.abs(host(d[1]) - ref) <= bound * np.abs(ref)).all()
