"""FP64 GEMM on the tensor cores by exact integer slices (csrc/oz_gemm.cu) against exact rational sums.

Reached through vtn_heff_apply with one-channel identity cores of local dimension 1: y = L theta R.  With
R = I the second product is exact, so y is one product of the sizes asked for."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _product(ctx, L, th, R=None):
    import torch
    from paper_2410_18740_gb300 import vtn
    one = vtn.make_core(1, 1, 1, [0], [0], np.ones((1, 1, 1), complex))
    m, n = L.shape[0], th.shape[1]
    R = torch.eye(n, dtype=torch.complex128, device="cuda") if R is None else R
    y = torch.full((m, n), 7.0, dtype=torch.complex128, device="cuda")
    vtn.vtn_heff_apply(ctx, one, one, m, n, L, R, th, y)
    torch.cuda.synchronize()
    return y


def _randn(rng, *shape):
    import torch
    return torch.from_numpy(rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).cuda()


def _worst(L, th, y, rng, count=20):
    """Largest error of sampled entries over its bound: one rounding of the result and one of the second
    (exact) product, and the digit pairs left out: below 2^-61 (largest of the row) (largest of the column) a
    term, which the scaling keeps within 2^5 of the largest term of the sum."""
    L, th, y = (t.cpu().numpy() for t in (L, th, y))
    K = L.shape[1]
    term = float(np.max(np.abs(L.view(float)).reshape(L.shape + (2,)).max((0, 2)) * np.abs(th.view(float)).reshape(th.shape + (2,)).max((1, 2))))
    worst = 0.0
    at = [(0, 0), (L.shape[0] - 1, th.shape[1] - 1)] + [(int(rng.integers(L.shape[0])), int(rng.integers(th.shape[1]))) for _ in range(count)]
    for i, j in at:
        re = im = Fraction(0)
        for k in range(K):
            ar, ai, br, bi = (Fraction(float(v)) for v in (L[i, k].real, L[i, k].imag, th[k, j].real, th[k, j].imag))
            re += ar * br - ai * bi
            im += ar * bi + ai * br
        for got, want in ((y[i, j].real, re), (y[i, j].imag, im)):
            bound = 2.0 ** -52 * abs(float(want)) + 4 * K * 2.0 ** -56 * term
            worst = max(worst, abs(float(Fraction(float(got)) - want)) / bound)
    return worst


# rows, columns: around the 128 x 32 tiles, the 16-element summation stages, the drains after 4, 8 and 16
# stages, and a summation long enough to be split over the CTAs
@pytest.mark.parametrize("m,n", [(256, 129), (257, 128), (383, 65), (400, 33), (512, 31), (641, 32), (1040, 16), (2300, 3)])
def test_sliced_product_is_exact_to_one_rounding(ctx, m, n):
    rng = np.random.default_rng(m * 31 + n)
    L, th = _randn(rng, m, m), _randn(rng, m, n)
    assert _worst(L, th, _product(ctx, L, th), rng) <= 1.0


@pytest.mark.parametrize("value", [float.fromhex("0x1.fefefefefefefp0"), float.fromhex("0x1.ff7f7f7f7f7f7p0"),
                                   float.fromhex("0x1.0101010101010p0"), 2.0 - 2.0 ** -52, -1.0 / 3.0])
def test_sliced_product_with_the_largest_digits(ctx, value):
    """All terms of one sign and every digit as large as it gets: the FP32 partial sums reach 2^24."""
    import torch
    L = torch.full((1100, 1100), complex(value, value), dtype=torch.complex128, device="cuda")
    th = torch.full((1100, 40), complex(value, -value), dtype=torch.complex128, device="cuda")
    assert _worst(L, th, _product(ctx, L, th), np.random.default_rng(0), count=2) <= 1.0


@pytest.mark.parametrize("k", [64, 65, 80, 81, 128, 129])
def test_sliced_product_of_short_sums_with_the_largest_digits(ctx, k):
    """Four, five, six, eight and nine summation stages, every digit as large as it gets."""
    import torch
    v, n = float.fromhex("0x1.fefefefefefefp0"), 1300
    L = torch.full((k, k), complex(v, v), dtype=torch.complex128, device="cuda")
    th = torch.full((k, n), complex(v, -v), dtype=torch.complex128, device="cuda")
    assert _worst(L, th, _product(ctx, L, th), np.random.default_rng(k)) <= 1.0


def test_sliced_product_of_opposed_gradings(ctx):
    """Columns of the left and rows of the right operand graded against each other over 28 decades."""
    import torch
    rng = np.random.default_rng(5)
    g = torch.logspace(0, -28, 400, dtype=torch.float64, device="cuda")
    L, th = _randn(rng, 400, 400) * g[None, :], _randn(rng, 400, 64) * g.flip(0)[:, None]
    assert _worst(L, th, _product(ctx, L, th), rng) <= 1.0


@pytest.mark.parametrize("m,n,decades", [(64, 2300, 0), (33, 2275, 28)])
def test_sliced_product_with_several_row_tiles_a_block(ctx, m, n, decades):
    """The right operand's exponents taken by blocks of more than one tile of columns, with and without the
    scaling of the summation index: theta R, with L = I the exact product."""
    import torch
    rng = np.random.default_rng(n)
    g = torch.logspace(0, -decades, n, dtype=torch.float64, device="cuda")
    th, R = _randn(rng, m, n) * g[None, :], _randn(rng, n, n) * g.flip(0)[:, None]
    assert _worst(th, R, _product(ctx, torch.eye(m, dtype=torch.complex128, device="cuda"), th, R), rng) <= 1.0


def test_sliced_product_with_non_finite_rows_and_extreme_scales(ctx):
    import torch
    rng = np.random.default_rng(9)
    L, th = _randn(rng, 400, 400), _randn(rng, 400, 64)
    L[17] = 0
    clean = _product(ctx, L, th)
    bad = L.clone()
    bad[3, 5] = float("inf")
    bad[399, 7] = complex(0.0, float("nan"))
    got = _product(ctx, bad, th)
    rows = torch.ones(400, dtype=torch.bool)
    rows[[3, 399]] = False
    assert torch.equal(got[rows], clean[rows]) and bool((clean[17] == 0).all())
    assert not bool(torch.isfinite(torch.view_as_real(got[~rows])).all(-1).any())
    for s in (2.0 ** -600, 2.0 ** 500):  # powers of two: the same digits
        assert torch.equal(_product(ctx, L * s, th), clean * s)


def test_sliced_products_of_the_environment_updates(ctx):
    """Conjugated, batched and channel-shared operands, both sides, against plain FP64."""
    import torch
    from paper_2410_18740_gb300 import vtn
    rng = np.random.default_rng(11)
    w, d, cl, cr = 3, 2, 150, 171
    core = vtn.make_core(w, w, d, range(w), range(w), np.array([np.eye(d)] * w, complex))
    A = _randn(rng, cl, d, cr)
    for side, ci, co in ((0, cl, cr), (1, cr, cl)):
        E, out = _randn(rng, w, ci, ci), torch.empty(w, co, co, dtype=torch.complex128, device="cuda")
        vtn.vtn_env_update(ctx, core, side, cl, cr, E, A, out)
        ref = torch.einsum("itl,aij,jtk->alk", A.conj(), E, A) if side == 0 else torch.einsum("jtg,agp,itp->aji", A, E, A.conj())
        # two products of lengths ci and d * (the other): the reference's own rounding, u sqrt(K) each, with room
        assert float(torch.linalg.norm(out - ref) / torch.linalg.norm(ref)) <= 1e-14


def test_products_without_memory_for_the_digits(monkeypatch):
    """An allocator that refuses what the digits need: the FP64 kernel computes the product, the full reduction the
    truncation, and what the allocator gave is all given back."""
    import torch
    from paper_2410_18740_gb300 import vtn
    rng = np.random.default_rng(3)
    n, k, held, refused = 512, 64, {}, []

    def alloc(nbytes, user):
        if nbytes > 6 << 20:  # n x n complex numbers are 4 MiB, the digits of the two operands 8 and 16
            refused.append(nbytes)
            return None
        t = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    fields = vtn.vtn_allocator._fields_
    a = vtn.vtn_allocator(fields[0][1](alloc), fields[1][1](lambda p, user: (held.pop(p), None)[1]), None)
    monkeypatch.setattr(vtn, "_torch_allocator", lambda device: a)
    ctx = vtn.vtn_create(0)
    L, th = _randn(rng, n, n), _randn(rng, n, n)
    y = _product(ctx, L, th)
    # a sum of n products and the reference's: u sqrt(n) each, with room
    assert float(torch.linalg.norm(y - L @ th) / torch.linalg.norm(L @ th)) <= 1e-14
    left, right = _randn(rng, n, k), _randn(rng, k, n)
    _, lam, _ = vtn.vtn_truncate(ctx, n // 8, 8, 8, n // 8, 0, k, th, left, right)
    s = np.linalg.svd(th.cpu().numpy(), compute_uv=False)[:k] ** 2
    # n roundings of the largest eigenvalue
    assert np.abs(np.asarray(lam) - s).max() <= n * 2.0 ** -52 * s[0]
    assert refused and held
    vtn.vtn_destroy(ctx)
    assert not held


@pytest.mark.parametrize("decades", [6, 28])
def test_sliced_product_with_non_finite_entries_in_opposed_gradings(ctx, decades):
    """Non-finite entries beside operands whose summation index is scaled: they take no part in the scaling, so
    the outputs of the other rows and columns are those of the sum without them."""
    import torch
    rng = np.random.default_rng(decades)
    g = torch.logspace(0, -decades, 400, dtype=torch.float64, device="cuda")
    L, th = _randn(rng, 400, 400) * g[None, :], _randn(rng, 400, 64) * g.flip(0)[:, None]
    bad = L.clone()
    bad[3, 5] = float("inf")
    bad[399, 398] = complex(0.0, float("nan"))
    got = _product(ctx, bad, th)
    rows = torch.ones(400, dtype=torch.bool, device="cuda")
    rows[[3, 399]] = False
    assert _worst(L[rows], th, got[rows], rng) <= 1.0
    assert not bool(torch.isfinite(torch.view_as_real(got[~rows])).all(-1).any())
    # columns: theta R, with L = I the exact product
    th, R = _randn(rng, 64, 400) * g[None, :], _randn(rng, 400, 400) * g.flip(0)[:, None]
    bad = R.clone()
    bad[200, 63] = complex(float("nan"), 1.0)
    bad[5, 399] = float("-inf")
    got = _product(ctx, torch.eye(64, dtype=torch.complex128, device="cuda"), th, bad)
    cols = torch.ones(400, dtype=torch.bool, device="cuda")
    cols[[63, 399]] = False
    assert _worst(th, R[:, cols], got[:, cols], rng) <= 1.0
    assert not bool(torch.isfinite(torch.view_as_real(got[:, ~cols])).all(-1).any())


@pytest.mark.parametrize("side", [0, 1])
def test_sliced_product_with_indices_that_meet_only_zeros(ctx, side):
    """Summation indices whose entries are all zero in one operand and far above the rest in the other."""
    import torch
    rng = np.random.default_rng(side)
    L, th = _randn(rng, 400, 400), _randn(rng, 400, 64)
    L[:, 100:200] *= 0.0 if side == 0 else 1e30
    th[100:200] *= 1e30 if side == 0 else 0.0
    assert _worst(L, th, _product(ctx, L, th), rng) <= 1.0


@pytest.mark.parametrize("last", [float("inf"), float("-inf"), float("nan")])
def test_sliced_product_whose_last_term_is_not_finite(ctx, last):
    """Sums of 16384 terms whose last one is infinite or NaN in every column: more tiles than SMs, each summed term
    by term in its epilogue."""
    import torch
    from paper_2410_18740_gb300 import vtn
    rng = np.random.default_rng(2)
    w, m, n = 32, 2048, 512
    one = vtn.make_core(1, 1, 1, [0], [0], np.ones((1, 1, 1), complex))
    row = vtn.make_core(1, w, 1, [0] * w, range(w), np.ones((w, 1, 1), complex))
    L, th, R = torch.eye(m, dtype=torch.complex128, device="cuda"), _randn(rng, m, n), _randn(rng, w, n, n)
    R[w - 1, n - 1] = last
    y = torch.empty(m, n, dtype=torch.complex128, device="cuda")
    vtn.vtn_heff_apply(ctx, one, row, m, n, L, R, th, y)
    # (a + i b) (inf + 0 i) = a inf + i b inf beside finite terms
    want = torch.view_as_real(th[:, n - 1:]) * last
    assert torch.equal(torch.nan_to_num(torch.view_as_real(y)), torch.nan_to_num(want.expand(m, n, 2)))


def _recording_context(monkeypatch):
    """A context whose allocator notes the sizes that were asked for."""
    import torch
    from paper_2410_18740_gb300 import vtn
    sizes, held = [], {}

    def alloc(nbytes, user):
        sizes.append(nbytes)
        t = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    fields = vtn.vtn_allocator._fields_
    a = vtn.vtn_allocator(fields[0][1](alloc), fields[1][1](lambda p, user: (held.pop(p), None)[1]), None)
    monkeypatch.setattr(vtn, "_torch_allocator", lambda device: a)
    return vtn.vtn_create(0), sizes


# more than 1 GiB of digits: of the left operand's rows; of a summation that is split over the CTAs
@pytest.mark.parametrize("w_l,w_r,m,n", [(40, 1, 1024, 33), (1, 2049, 256, 64)])
def test_sliced_products_in_pieces(monkeypatch, w_l, w_r, m, n):
    import torch
    from paper_2410_18740_gb300 import vtn
    rng = np.random.default_rng(w_l)
    ctx, sizes = _recording_context(monkeypatch)
    Wi = vtn.make_core(w_l, 1, 1, range(w_l), [0] * w_l, np.ones((w_l, 1, 1), complex))
    Wj = vtn.make_core(1, w_r, 1, [0] * w_r, range(w_r), np.ones((w_r, 1, 1), complex))
    eye = lambda k: torch.eye(k, dtype=torch.complex128, device="cuda")[None]
    L, R = (eye(m), _randn(rng, w_r, n, n)) if w_l == 1 else (_randn(rng, w_l, m, m), eye(n))
    th, y = _randn(rng, m, n), torch.empty(m, n, dtype=torch.complex128, device="cuda")
    vtn.vtn_heff_apply(ctx, Wi, Wj, m, n, L, R, th, y)
    ref = L.sum(0) @ th @ R.sum(0)
    # the reference's sums over channels and products: u sqrt(terms) each, with room
    assert float(torch.linalg.norm(y - ref) / torch.linalg.norm(ref)) <= 2e-14
    assert max(sizes) <= 1 << 30
    vtn.vtn_destroy(ctx)


@pytest.mark.parametrize("direction", [0, 1])
def test_hermitian_sliced_product_in_pieces(monkeypatch, direction):
    """The density matrix of a tensor with exactly known factors (Hadamard blocks of 4096 and 256), 1.2 GB of digits."""
    import torch
    from paper_2410_18740_gb300 import vtn
    ctx, sizes = _recording_context(monkeypatch)

    def had(n):
        H = torch.ones(1, 1, dtype=torch.float64, device="cuda")
        while len(H) < n:
            H = torch.cat([torch.cat([H, H], 1), torch.cat([H, -H], 1)], 0)
        return H / n ** 0.5

    n1, n2, k = 4096, 256, 24
    n = n1 + n2
    U = torch.zeros(n, n, dtype=torch.complex128, device="cuda")
    U[:n1, :n1], U[n1:, n1:] = had(n1), 1j * had(n2)
    U = U[torch.randperm(n, generator=torch.Generator().manual_seed(1)).cuda()]
    S = torch.full((n,), 2.0 ** -10, dtype=torch.float64, device="cuda")
    top = torch.arange(k, device="cuda") * (n // k)  # in both blocks
    S[top] = torch.round(1024 * torch.linspace(1.0, 0.25, k, dtype=torch.float64, device="cuda")) / 1024
    T = (U * S) @ U.flip(0).conj().T
    left = torch.empty(n, k, dtype=torch.complex128, device="cuda")
    right = torch.empty(k, n, dtype=torch.complex128, device="cuda")
    _, lam, _ = vtn.vtn_truncate(ctx, n // 2, 2, 2, n // 2, direction, k, T, left, right)
    u = 2.0 ** -53
    assert np.abs(np.asarray(lam) - (S[top] ** 2).cpu().numpy()).max() <= 4 * n * u
    ref = (U[:, top] * S[top]) @ U.flip(0)[:, top].conj().T
    # gaps of about 1/16 between the kept part and the rest
    assert float(torch.linalg.norm(left @ right - ref)) <= 64 * n * u * k ** 0.5
    assert max(sizes) <= 1 << 30
    vtn.vtn_destroy(ctx)
