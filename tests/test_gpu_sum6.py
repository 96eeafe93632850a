"""GPU: the FP64 neighbour sum, done on the integer pipes, at the edges of its range.

With lambda = m2 = 0, dt = dx = 1 and pi = 0 one FP64 step gives pi' = nb - 6 phi and
phi' = phi + pi', so the neighbour sum nb shows in the result.  The reference is the exact
rational sum.  Derivation of the tolerance, with u = 2^-53 and M the largest neighbour: the sum is
off by at most u |nb| + 6 units of 2^-59 M (bits below its fixed-point grid) or, outside the grid's
exponent range, by the five FP64 additions' 3 u sum|phi_i|; -6 phi is rounded once and its fma with
nb once, each at most u (6 |phi| + |nb|): in all below 6 u (sum|phi_i| + 6 |phi|) + 2^-56 M, plus
the smallest subnormal for each rounding.  (The range's high end, 2^1017, cannot be seen in a step:
phi^2 overflows above 2^512 and the step gives NaN whatever the sum.)"""
from fractions import Fraction
from functools import reduce

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
SHAPE = (6, 4, 5)  # nx, ny, nz


@pytest.fixture(scope="module")
def lf2():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1508_05610_gb300 import build, lf2 as binding
    build.build()
    binding.load()
    return binding


def values(kind, rng):
    n = SHAPE[::-1] + (1,)
    v = rng.standard_normal(n)
    if kind == "spread":  # exponents up to 140 apart: small operands drop below the grid
        return np.ldexp(v, rng.integers(-70, 70, n))
    if kind == "equal":  # all significands full, sums of up to six equal values
        return np.where(rng.random(n) < 0.5, 1.0, -1.0) * (2.0 - 2.0 ** -52)
    if kind == "cancel":  # sums that vanish or keep only the last bits
        return np.where(np.indices(n).sum(0) % 2 == 0, 1.0, -1.0) * (1.0 + 2.0 ** -52 * rng.integers(0, 3, n))
    if kind == "zeros":
        return np.where(rng.random(n) < 0.6, 0.0, v) * np.where(rng.random(n) < 0.5, 1.0, -1.0)
    assert kind == "low"  # around the low end of the grid's range (2^-959), and subnormal
    return np.ldexp(v, rng.integers(-1073, -950, n))


@pytest.mark.parametrize("kernel", ["site", "stream", "tblock"])
@pytest.mark.parametrize("kind", ["spread", "equal", "cancel", "zeros", "low"])
def test_neighbour_sum_against_exact_rationals(lf2, kind, kernel):
    phi = values(kind, np.random.default_rng(5))
    p = lf2.params(dx=1.0, dt=1.0, lam=0.0, eta=0.0, m2=0.0)
    steps = 2 if kernel == "tblock" else 1
    with lf2.System(SHAPE, 1, "f64") as s, lf2.System(SHAPE, 1, "f64") as t:
        for q in (s, t):
            q.upload(phi, np.zeros_like(phi))
        if kernel == "tblock":
            lf2.lf2_leapfrog_ex(s.phi, s.pi, p, steps, kernel=lf2.LF2_KERNEL_TBLOCK, depth=2, cx=1, tile_x=4, tile_y=4)
        else:
            lf2.lf2_leapfrog_ex(s.phi, s.pi, p, steps, kernel={"site": 1, "stream": 2}[kernel])
        lf2.lf2_leapfrog_ex(t.phi, t.pi, p, steps, kernel=lf2.LF2_KERNEL_SITE)
        got, ref = s.download(), t.download()
    assert np.array_equal(got[0], ref[0], equal_nan=True) and np.array_equal(got[1], ref[1], equal_nan=True)
    if steps > 1:
        return
    f = phi[..., 0]
    nbrs = [np.roll(f, sh, ax) for ax in range(3) for sh in (1, -1)]
    u, sub = Fraction(1, 2 ** 53), Fraction(1, 2 ** 1074)
    for at in np.ndindex(f.shape):
        c, nb = Fraction(f[at]), [Fraction(n[at]) for n in nbrs]
        scale, top = sum(map(abs, nb)) + 6 * abs(c), max(map(abs, nb))
        err = abs(Fraction(got[1][at][0]) - (sum(nb) - 6 * c))
        assert err <= 6 * u * scale + top / 2 ** 56 + 8 * sub, (at, float(err), float(scale))


def test_infinities_and_nan_reach_the_result(lf2):
    """As IEEE additions give them: an infinite neighbour makes pi' infinite, opposite infinities
    and NaN make it NaN (as does an infinite site itself: lambda phi^2 is 0 times infinity), the
    other sites stay finite."""
    phi = np.random.default_rng(6).standard_normal(SHAPE[::-1] + (1,))
    phi[0, 0, 0], phi[0, 0, 2], phi[3, 2, 4] = np.inf, -np.inf, np.nan
    f = phi[..., 0]
    with np.errstate(invalid="ignore"):
        want = sum(np.roll(f, sh, ax) for ax in range(3) for sh in (1, -1)) - (0.0 * f * f + 6) * f
    p = lf2.params(dx=1.0, dt=1.0, lam=0.0, eta=0.0, m2=0.0)
    with lf2.System(SHAPE, 1, "f64") as s:
        s.upload(phi, np.zeros_like(phi))
        lf2.lf2_leapfrog(s.phi, s.pi, p, 1)
        got = s.download()[1][..., 0]
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want))
    assert np.array_equal(got[np.isinf(got)], want[np.isinf(want)])
    fine = np.isfinite(want)
    assert np.allclose(got[fine], want[fine], rtol=1e-14, atol=1e-13)


@pytest.mark.parametrize("prec", ["f64", "f32k"])
@pytest.mark.parametrize("kind", ["near", "spread", "ties"])
def test_gradient_energy_differences_against_exact_rationals(lf2, kind, prec):
    """The forward differences, subtracted as integers, at the edges of their fast ranges: exponents
    7 to 11 (FP64) or 26 to 31 (FP32) binary orders apart, neighbours equal to the last bit, zeros.
    Bound: each difference is rounded once (u), squared and added in FP64: a sum of N terms, added
    in any order, is off by at most (N + 3) u of the sum of the (non-negative) terms."""
    rng = np.random.default_rng(8)
    n = SHAPE[::-1] + (1,)
    v = rng.standard_normal(n)
    if kind == "spread":
        span = (7, 12) if prec == "f64" else (26, 32)
        v = np.where(np.indices(n).sum(0) % 2 == 0, v, np.ldexp(v, -rng.integers(*span, n)))
    elif kind == "ties":
        v = np.where(rng.random(n) < 0.3, 0.0, 1.0) * (1.0 + 2.0 ** (-52 if prec == "f64" else -23) * rng.integers(-2, 3, n))
    if prec != "f64":
        v = v.astype(np.float32).astype(np.float64)
    p = lf2.params(dx=1.0, dt=0.1, lam=0.0, eta=0.0, m2=0.0)
    with lf2.System(SHAPE, 1, prec) as s:
        s.upload(v, np.zeros_like(v))
        e = lf2.lf2_energy(s.phi, s.pi, p, ncomp=1)
    f = v[..., 0]
    exact, terms = Fraction(0), 0
    for ax in range(3):
        up = np.roll(f, -1, ax)
        for at in np.ndindex(f.shape):
            exact += (Fraction(up[at]) - Fraction(f[at])) ** 2
            terms += 1
    got = 2 * Fraction(e["gradient"])
    assert abs(got - exact) <= (terms + 3) * Fraction(1, 2 ** 53) * exact, float(abs(got - exact) / exact)


@pytest.mark.parametrize("kernel", ["site", "stream", "tblock"])
def test_sums_of_signed_zeros_have_the_sign_of_ieee_additions(lf2, kernel):
    """A zero sum is -0 only if all six neighbours are.  It shows at a site of +0 with pi = -0: there
    pi' = nb + (-g phi + pi) is nb + -0."""
    rng = np.random.default_rng(9)
    phi = np.where(rng.random(SHAPE[::-1] + (1,)) < 0.08, 0.0, -0.0)
    pi = np.full_like(phi, -0.0)
    f = phi[..., 0]
    nbrs = [np.roll(f, sh, ax) for ax in range(3) for sh in (1, -1)]
    nb = reduce(np.add, nbrs)  # sum() would start from +0
    p = lf2.params(dx=1.0, dt=1.0, lam=0.0, eta=0.0, m2=0.0)
    with lf2.System(SHAPE, 1, "f64") as s, lf2.System(SHAPE, 1, "f64") as t:
        for q in (s, t):
            q.upload(phi, pi)
        steps, kw = {"site": (1, dict(kernel=1)), "stream": (1, dict(kernel=2)),
                     "tblock": (2, dict(kernel=3, depth=2, cx=1, tile_x=4, tile_y=4))}[kernel]
        lf2.lf2_leapfrog_ex(s.phi, s.pi, p, steps, **kw)
        lf2.lf2_leapfrog_ex(t.phi, t.pi, p, steps, kernel=lf2.LF2_KERNEL_SITE)
        got, ref = s.download(), t.download()
    for a, b in zip(got, ref):
        assert np.array_equal(a, b) and np.array_equal(np.signbit(a), np.signbit(b))
    if steps == 1:
        at = ~np.signbit(f)
        assert at.any() and np.array_equal(np.signbit(got[1][..., 0])[at], np.signbit(nb)[at])


@pytest.mark.parametrize("prec", ["f64", "f32k"])
@pytest.mark.parametrize("what", ["energy", "step"])
def test_zeros_cost_no_more_than_other_values(lf2, what, prec):
    """A field of zeros in one component, or in all of them, against one of Gaussian values, on a lattice
    that fills the GPU.  Nothing is added in FP64 for a zero that other values need not add, but the FP64
    energy subtracts zeros there: 27 FP64 instructions a site instead of 21.  (With the sums in FP64 too,
    1.55 and 1.7 times as long.)"""
    import torch
    n = (128, 128, 128)
    p = lf2.params(dx=1.0, dt=0.05, lam=1.0, eta=1.0, m2=0.0)
    rec = torch.zeros(16, dtype=torch.float64, device="cuda")
    full = np.random.default_rng(10).standard_normal(n[::-1] + (2,)) * 0.1
    times = []
    with lf2.System(n, 2, prec) as s:
        for zero in ([], [1], [0, 1]):
            phi = full.copy()
            phi[..., zero] = 0.0
            s.upload(phi, np.zeros_like(phi))
            lf2.lf2_leapfrog_init(s.phi, s.pi, p)
            best = 1e9
            for _ in range(8):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                for _ in range(4):
                    if what == "energy":
                        lf2.lf2_energy_device(s.phi, s.pi, p, rec.data_ptr())
                    else:
                        lf2.lf2_leapfrog_ex(s.phi, s.pi, p, 1, kernel=lf2.LF2_KERNEL_SITE)
                b.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b))
            times.append(best)
    assert max(times[1:]) <= (1.4 if (what, prec) == ("energy", "f64") else 1.25) * times[0], times
