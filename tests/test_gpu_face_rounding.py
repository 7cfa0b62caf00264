"""GPU: the face kernels' quotients at the operands where correct rounding is
hardest.  a/b lies next to a midpoint m of two doubles when a - m b is a small
multiple r of the last place of m b; for an odd mantissa B of b each r gives
one m (r/B modulo a power of two), so the hard numerators of a divisor are
listed, not searched.  Every pair is one face between two cells of its own."""
import math

import numpy as np
import pytest

from gpu_cases import bits, dev

pytestmark = pytest.mark.gpu


def hard_numerators(B):
    """The a in [1, 2) with a / (B 2^-52), B odd of 53 bits, within 9 units of the product's last place of a midpoint."""
    out = []
    for r in range(-9, 10, 2):
        for k in (53, 54):   # quotients in [1, 2) and in [1/2, 1)
            M = pow(B, -1, 1 << k) * r % (1 << k)
            M += (1 << 53) if k == 53 else 0
            A = (M * B - r) >> k
            if M >> 53 and 1 << 52 <= A < 1 << 53:
                out.append(A * 2.0 ** -52)
    return out


def face_coefficients(sf, d, gamma):
    """-upper of faces with area vectors sf, cell distances d and diffusivities gamma, a pair of cells each."""
    from paper_2512_22215_gb300 import LduMesh
    F = len(gamma)
    c = np.zeros((2 * F, 3))
    c[1::2] = d
    lo = np.arange(0, 2 * F, 2, dtype=np.int32)
    up, _ = LduMesh(lo, lo + 1, 2 * F).assemble_laplacian(dev(sf), dev(c), dev(gamma))
    return -up.cpu().numpy()


@pytest.mark.parametrize("divisors", ["below-two", "random"])
def test_hard_quotients(divisors):
    """|S| = n.S = 1, so a face's coefficient is gamma/d."""
    rng = np.random.default_rng(181)
    Bs = range(2 ** 53 - 8191, 2 ** 53, 2) if divisors == "below-two" else (rng.integers(2 ** 52, 2 ** 53, 6000) | 1).tolist()
    pairs = np.array([(a, B * 2.0 ** -52) for B in Bs for a in hard_numerators(B)])
    e = rng.integers(-30, 31, (len(pairs), 2))
    a, b = np.ldexp(pairs[:, 0], e[:, 0]), np.ldexp(pairs[:, 1], e[:, 1])
    unit = np.zeros((len(a), 3))
    unit[:, 0] = 1.0
    assert np.array_equal(bits(face_coefficients(unit, unit * b[:, None], a)), bits(a / b))


def squares_near_midpoints(count):
    """Doubles v in [1, 4) whose square root lies just above a midpoint m of two doubles: v = m^2 + j 2^-108 or so, j
    small (m^2 = -j modulo a power of two, solved bit by bit)."""
    out = []
    for r in range(-7, -8 * count, -8):
        for odd in (0, 1):
            k = 54 + odd
            x = 1
            for n in range(3, k):
                x += ((x * x - r) >> n & 1) << (n - 1)
            half = 1 << (k - 1)
            for M in {x % (2 * half), -x % (2 * half), (x + half) % (2 * half), (half - x) % (2 * half)}:
                V = (M * M - r) >> k
                if M >> 53 == 1 and V >> 52 == 1:
                    out.append(math.ldexp(V, odd - 52))
    return out


def test_hard_quotients_by_the_norm():
    """n.S = (S.d)/|S| next to a midpoint, where |S|^2 has a square root next to one too: what the square root leaves
    as 1/|S| has to be the reciprocal of the rounded root."""
    sf, d, num = [], [], []
    for v in squares_near_midpoints(800):
        mag = math.sqrt(v)
        B = int(mag * 2 ** 52)
        # S = (x, y, 0) with x^2 + y^2 = v as the kernels add it up
        x = math.nextafter(mag, 0.0)
        for _ in range(40):
            y = math.sqrt(v - x * x)
            if x * x + y * y == v:
                break
            x = math.nextafter(x, 0.0)
        if not B & 1 or x * x + y * y != v:
            continue
        for a in hard_numerators(B):
            for dx in (a / x, math.nextafter(a / x, 0.0), math.nextafter(a / x, 4.0)):
                if x * dx == a:
                    sf.append((x, y, 0.0))
                    d.append(dx)
                    num.append((a, mag))
                    break
    assert len(num) > 1500
    sf, d, (a, mag) = np.array(sf), np.array(d), np.array(num).T
    dist = np.zeros_like(sf)
    dist[:, 0] = d
    for gamma in (1.0, 1.25, 1.7):
        want = (gamma * mag) / (a / mag)      # n.S is far above 0.05 |d|
        assert np.array_equal(bits(face_coefficients(sf, dist, np.full(len(a), gamma))), bits(want))
