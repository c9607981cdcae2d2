"""The sliced FP64 product against the same 36 digit products in integers: what it returns is their sum, rounded once.

Reached through vtn_heff_apply with an identity core of local dimension 16 and one channel: the first product is
L theta with 256 chi_r columns, in so many tiles that its summation is not split over the CTAs, and the second one, with
R = I, is small enough for the FP64 units and exact."""
from fractions import Fraction

import numpy as np
import pytest

BIAS = sum(128 << (8 * i) for i in range(7))


def _digits(q):
    """Eight digits of a 64-bit fixed-point number, the leading one first: q = sum d_i 256^(7 - i)."""
    low = [(((q + BIAS) >> (8 * i)) & 255) - 128 for i in range(7)]
    return [(q - sum(d << (8 * i) for i, d in enumerate(low))) >> 56] + low[::-1]


def _biased(x):
    """Exponent fields of the larger component, 0 for zero."""
    m = np.maximum(np.abs(x.real), np.abs(x.imag))
    return np.where(m > 0, np.maximum(np.frexp(m)[1] + 1022, 1), 0)


def _fixed(x, e0, shift):
    """63-bit fixed point of x 2^-shift below exponent e0."""
    if x == 0.0:
        return 0
    f, e = np.frexp(abs(x))
    e, m = int(e) + 1022, int(f * 2.0 ** 53)
    if e < 1:
        m, e = m >> (1 - e), 1
    q = (m << 10) >> min(e0 - (e - shift), 64)
    return -q if x < 0 else q


class Restated:
    """Sums of the digit products of weight up to 7, for entries of A B."""

    def __init__(self, A, B):
        self.A, self.B = A, B
        ea, eb = _biased(A), _biased(B)
        x, y = ea.max(0), eb.max(1)
        self.scaled = x.max() + y.max() - (x + y)[(x > 0) & (y > 0)].max() > 4
        s = np.trunc((x - y) / 2).astype(int)
        s[(x == 0) & (y > 0)], s[(x > 0) & (y == 0)] = -4096, 4096
        self.s = s if self.scaled else 0 * s
        self.ra = np.where(ea > 0, ea - self.s[None, :], -10 ** 6).max(1)
        self.rb = np.where(eb > 0, eb + self.s[:, None], -10 ** 6).max(0)

    def entry(self, i, j, weights=8):
        e, f = int(self.ra[i]), int(self.rb[j])
        re = im = 0
        for k in range(self.A.shape[1]):
            a, b, s = complex(self.A[i, k]), complex(self.B[k, j]), int(self.s[k])
            ar, ai = (_digits(_fixed(v, e, s)) for v in (a.real, a.imag))
            br, bi = (_digits(_fixed(v, f, -s)) for v in (b.real, b.imag))
            for u in range(weights):
                for v in range(weights - u):
                    w = 8 * (14 - u - v)
                    re += (ar[u] * br[v] - ai[u] * bi[v]) << w
                    im += (ar[u] * bi[v] + ai[u] * br[v]) << w
        scale = Fraction(2) ** (e + f - 2170)
        return re * scale, im * scale

    def largest(self, i, j):
        """(largest component of the row) x (largest of the column), of the scaled operands."""
        top = lambda x, s: max(Fraction(float(max(abs(v.real), abs(v.imag)))) * Fraction(2) ** int(t) for v, t in zip(x, s))
        return top(self.A[i], -self.s) * top(self.B[:, j], self.s)


def _exact(A, B, i, j):
    re = im = Fraction(0)
    for a, b in zip(A[i], B[:, j]):
        ar, ai, br, bi = (Fraction(float(v)) for v in (a.real, a.imag, b.real, b.imag))
        re += ar * br - ai * bi
        im += ar * bi + ai * br
    return re, im


def _operands(kind, K, n):
    rng = np.random.default_rng(K)
    z = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    A, B = z(K, K), z(K, n)
    if kind == "graded":
        g = np.logspace(0, -28, K)
        A, B = A * g, B * g[::-1, None]
    elif kind == "mixed":  # gradings within the rows and columns that no scaling of the index removes
        A, B = (x * 2.0 ** rng.integers(-40, 1, x.shape) for x in (A, B))
    elif kind == "zeros":
        A[:, : K // 4] = 0
        B[: K // 4] *= 1e30
    elif kind == "largest":
        v = float.fromhex("0x1.fefefefefefefp0")
        A, B = np.full_like(A, complex(v, v)), np.full_like(B, complex(v, -v))
    return A, B


KINDS = ["normal", "graded", "mixed", "zeros", "largest"]


@pytest.mark.parametrize("kind", KINDS)
def test_digit_sums_are_within_their_bound_and_need_every_weight(kind):
    """The 28 pairs left out: at most 7.03 2^62 of 2^124 (the smallest product of two largest entries) a real product,
    and 2^64 for the cut of both operands to 63 bits; two real products a component: below 6 2^-60 a term."""
    A, B = _operands(kind, 60, 8)
    r = Restated(A, B)
    assert r.scaled == (kind in ("graded", "zeros"))
    seen = 0
    for i, j in [(0, 0), (59, 7), (17, 3)]:
        for s, x, t in zip(r.entry(i, j), _exact(A, B, i, j), r.entry(i, j, 7)):
            assert abs(s - x) <= 6 * 60 * Fraction(1, 2 ** 60) * r.largest(i, j)
            seen += abs(t - s) > Fraction(1, 2 ** 52) * abs(s)
    assert seen or kind == "largest"  # a sum without its last weight is told from a rounding


# summation lengths around the stages of 16 and the drains after 4, 5, 8 and 16 of them
@pytest.mark.gpu
@pytest.mark.parametrize("K,cr,kind", [(64, 15, "normal"), (65, 15, "largest"), (80, 15, "normal"), (81, 15, "normal"), (128, 8, "largest"),
                                       (129, 8, "normal"), (256, 8, "mixed"), (400, 4, "normal"), (400, 4, "graded"), (400, 4, "mixed"),
                                       (400, 4, "zeros"), (512, 4, "largest"), (1040, 2, "normal")])
def test_sliced_product_equals_its_digit_sums(ctx, K, cr, kind):
    import torch
    from paper_2410_18740_gb300 import vtn
    d, n = 16, 256 * cr
    A, B = _operands(kind, K, n)
    one = vtn.make_core(1, 1, d, [0], [0], np.eye(d, dtype=complex)[None])
    y = torch.empty(K, n, dtype=torch.complex128, device="cuda")
    vtn.vtn_heff_apply(ctx, one, one, K, cr, torch.from_numpy(A).cuda(), torch.eye(cr, dtype=torch.complex128, device="cuda"),
                       torch.from_numpy(B).cuda(), y)
    y, r, rng = y.cpu().numpy(), Restated(A, B), np.random.default_rng(cr)
    at = [(0, 0), (K - 1, n - 1)] + [(int(rng.integers(K)), int(rng.integers(n))) for _ in range(6 if K < 1000 else 2)]
    for i, j in at:
        for got, want in zip((y[i, j].real, y[i, j].imag), r.entry(i, j)):
            assert abs(Fraction(float(got)) - want) <= Fraction(1, 2 ** 53) * abs(want)  # one rounding to nearest
