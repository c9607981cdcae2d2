"""Truncation of density matrices larger than 256 (Chebyshev-filtered subspace iteration, csrc/trunc_filter.cu)
against a singular value decomposition, with spectra it suits and spectra that go to the full reduction."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _tensor(rng, n1, n2, s):
    q = lambda n: np.linalg.qr(rng.standard_normal((n, len(s))) + 1j * rng.standard_normal((n, len(s))))[0]
    return (q(n1) * s) @ q(n2).conj().T


def _spectrum(kind, n, k):
    e = np.arange(n, dtype=float)
    if kind == "decaying":
        return np.exp(-9.0 * e / n)
    if kind == "flat":
        return np.exp(-1.0 * e / n)
    if kind == "degenerate top":
        return np.where(e < k // 2, 1.0, np.exp(-9.0 * e / n))
    if kind == "steep":  # squared Schmidt values below rounding inside the block
        return np.exp(-60.0 * e / n)
    if kind == "rank below k":
        return np.exp(-e[: k // 2] / n)
    assert kind == "degenerate at k"
    s = np.exp(-9.0 * e / n)
    s[k - 4:k + 2 * k] = s[k - 4]
    return s


# (chi_l, d1, d2, chi_r, k): just above the limit, a ragged block, unequal sides, a block of several tiles
@pytest.mark.parametrize("shape", [(52, 5, 5, 53, 20), (87, 6, 6, 91, 33), (65, 8, 8, 80, 64)])
@pytest.mark.parametrize("kind", ["decaying", "flat", "degenerate top", "steep", "rank below k", "degenerate at k"])
@pytest.mark.parametrize("direction", [0, 1])
def test_large_truncation_matches_the_svd(ctx, shape, kind, direction):
    import torch
    from paper_2410_18740_gb300 import vtn
    cl, d1, d2, cr, k = shape
    n1, n2 = cl * d1, d2 * cr
    rng = np.random.default_rng(n1 + 7 * n2 + direction)
    T = _tensor(rng, n1, n2, _spectrum(kind, min(n1, n2), k))
    th = torch.from_numpy(np.ascontiguousarray(T)).cuda()
    left = torch.empty(n1, k, dtype=torch.complex128, device="cuda")
    right = torch.empty(k, n2, dtype=torch.complex128, device="cuda")
    before = vtn.vtn_launch_count(ctx)
    kk, lam, disc = vtn.vtn_truncate(ctx, cl, d1, d2, cr, direction, k, th, left, right)
    launches = vtn.vtn_launch_count(ctx) - before
    U, S, Vh = np.linalg.svd(T, full_matrices=False)
    nrm2 = float((S ** 2).sum())
    n = n1 if direction == 0 else n2
    u = 2.0 ** -53
    # rounding of rho and of its eigenpairs: a small multiple of n u |rho| (as the bounds of the full reduction)
    assert kk == k and np.abs(lam - S[:k] ** 2).max() <= 4 * n * u * S[0] ** 2
    assert abs(disc - (1.0 - (S[:k] ** 2).sum() / nrm2)) <= 4 * n * u * k
    iso = left if direction == 0 else right.conj().T
    eye = torch.eye(k, dtype=torch.complex128, device="cuda")
    assert float((iso.conj().T @ iso - eye).abs().max()) <= 4 * n * u
    got = (left @ right).cpu().numpy()
    if kind in ("decaying", "flat", "degenerate top"):
        ref = (U[:, :k] * S[:k]) @ Vh[:k]
        gap = (S[k - 1] ** 2 - S[k] ** 2) / S[0] ** 2
        # subspace error: residual over gap, weighted by the boundary's Schmidt values
        assert np.linalg.norm(got - ref) <= (4 * n * u / gap * S[k - 1] + 4 * n * u * S[0]) * np.sqrt(k)
    # whatever was kept at a degenerate or noise-level boundary carries the largest weight there is
    assert np.linalg.norm(got) ** 2 >= (S[:k] ** 2).sum() - 8 * n * u * k * S[0] ** 2
    if kind == "decaying":
        assert launches > 120, launches  # the full reduction takes about 30


# one side of the tensor at most half of the other: the block is the tensor's own range
@pytest.mark.parametrize("shape,direction", [((8, 8, 8, 64, 64), 1), ((70, 5, 5, 11, 30), 0), ((1, 6, 6, 61, 6), 1)])
@pytest.mark.parametrize("decay", [0.0, 9.0, 60.0])  # the last is too ill-conditioned for it
def test_truncation_of_a_density_matrix_of_low_rank(ctx, shape, direction, decay):
    import torch
    from paper_2410_18740_gb300 import vtn
    cl, d1, d2, cr, k = shape
    n1, n2 = cl * d1, d2 * cr
    rng = np.random.default_rng(n1 + 3 * n2)
    r = min(n1, n2)
    T = _tensor(rng, n1, n2, np.exp(-decay * np.arange(r) / r))
    th = torch.from_numpy(np.ascontiguousarray(T)).cuda()
    left = torch.empty(n1, k, dtype=torch.complex128, device="cuda")
    right = torch.empty(k, n2, dtype=torch.complex128, device="cuda")
    kk, lam, disc = vtn.vtn_truncate(ctx, cl, d1, d2, cr, direction, k, th, left, right)
    U, S, Vh = np.linalg.svd(T, full_matrices=False)
    n, u = max(n1, n2), 2.0 ** -53
    assert kk == k and np.abs(lam - S[:k] ** 2).max() <= 4 * n * u * S[0] ** 2
    iso = left if direction == 0 else right.conj().T
    assert float((iso.conj().T @ iso - torch.eye(k, dtype=torch.complex128, device="cuda")).abs().max()) <= 4 * n * u
    got = (left @ right).cpu().numpy()
    assert np.linalg.norm(got) ** 2 >= (S[:k] ** 2).sum() - 8 * n * u * k * S[0] ** 2
    if k == r:
        assert np.linalg.norm(got - T) <= 4 * n * u * S[0] * np.sqrt(k)


# a density matrix larger than 4096 whose range is itself of a size that the filter takes (half of it, or nearly)
@pytest.mark.parametrize("shape,direction", [((300, 16, 8, 64, 32), 0), ((64, 8, 16, 300, 32), 1), ((260, 16, 13, 160, 90), 0)])
def test_truncation_whose_range_suits_the_filter(ctx, shape, direction):
    import torch
    from paper_2410_18740_gb300 import vtn
    cl, d1, d2, cr, k = shape
    n1, n2 = cl * d1, d2 * cr
    rng = np.random.default_rng(n1 + 5 * n2)
    r = min(n1, n2)
    S = np.exp(-9.0 * np.arange(r) / r)
    U, V = (np.linalg.qr(rng.standard_normal((n, r)) + 1j * rng.standard_normal((n, r)))[0] for n in (n1, n2))
    T = (U * S) @ V.conj().T
    left = torch.empty(n1, k, dtype=torch.complex128, device="cuda")
    right = torch.empty(k, n2, dtype=torch.complex128, device="cuda")
    kk, lam, disc = vtn.vtn_truncate(ctx, cl, d1, d2, cr, direction, k, torch.from_numpy(np.ascontiguousarray(T)).cuda(), left, right)
    n, u = max(n1, n2), 2.0 ** -53
    # the bounds of the tests above; T itself is the product of its factors to a rounding of r terms
    assert kk == k and np.abs(lam - S[:k] ** 2).max() <= 4 * n * u * S[0] ** 2
    assert abs(disc - (1.0 - (S[:k] ** 2).sum() / (S ** 2).sum())) <= 4 * n * u * k
    iso = left if direction == 0 else right.conj().T
    assert float((iso.conj().T @ iso - torch.eye(k, dtype=torch.complex128, device="cuda")).abs().max()) <= 4 * n * u
    ref = (U[:, :k] * S[:k]) @ V[:, :k].conj().T
    gap = (S[k - 1] ** 2 - S[k] ** 2) / S[0] ** 2
    assert np.linalg.norm((left @ right).cpu().numpy() - ref) <= (4 * n * u / gap * S[k - 1] + 4 * n * u * S[0]) * np.sqrt(k)


def _slices(a, axis):
    """Three parts of 19 bits below the largest entry along the axis: products of parts of two of them and their
    sums of up to 2^12 terms are exact in FP64."""
    import torch
    r = torch.view_as_real(a)
    e = torch.ceil(torch.log2(r.abs().amax((axis, 2), keepdim=True).clamp_min(1e-300))) + 1
    out = []
    for i in range(3):
        u = torch.exp2(e - 19 * (i + 1))
        s = torch.round(r / u) * u
        r = r - s
        out.append(torch.view_as_complex(s.contiguous()))
    return out


@pytest.mark.parametrize("n,d,k", [(512, 8, 64), (1024, 8, 128), (1024, 4, 100)])
@pytest.mark.parametrize("direction", [0, 1])
def test_large_truncation_is_as_accurate_as_its_roundings(ctx, n, d, k, direction):
    """A tensor whose entries and singular vectors are exact: permuted Hadamard matrices with phases 1, i, -1, -i
    and Schmidt values of 30 bits."""
    import torch
    from paper_2410_18740_gb300 import vtn
    rng = np.random.default_rng(n + k + direction)
    H = np.ones((1, 1))
    while len(H) < n:
        H = np.block([[H, H], [H, -H]])
    basis = lambda: (np.array([1, 1j, -1, -1j])[rng.integers(4, size=n)][:, None] * H)[rng.permutation(n)][:, rng.permutation(n)]
    U, V = basis(), basis()
    S = np.round(np.exp(-9.0 * np.arange(n) / n) * 2 ** 30) / 2 ** 30
    T, ref = (U * S) @ V.conj().T / n, (U[:, :k] * S[:k]) @ V[:, :k].conj().T / n
    left = torch.empty(n, k, dtype=torch.complex128, device="cuda")
    right = torch.empty(k, n, dtype=torch.complex128, device="cuda")
    _, lam, disc = vtn.vtn_truncate(ctx, n // d, d, d, n // d, direction, k, torch.from_numpy(T).cuda(), left, right)
    a, b, err = _slices(left, 1), _slices(right, 0), -torch.from_numpy(ref).cuda()
    for w in range(3):  # left right - ref, largest parts first: what is left after them is at rounding level
        for i in range(w + 1):
            err = err + a[i] @ b[w - i]
    u = 2.0 ** -53
    # theta: the basis, the projected tensor, the Ritz vectors on both sides and the two factors are rounded, at
    # most u of their norm each; as much again for what the products' sums and the first order leave out
    assert float(torch.linalg.norm(err)) <= 12 * u * np.linalg.norm(ref)
    # lam: a quotient of two sums whose roundings are below u each (a tree of a few levels), and one rounding
    assert np.linalg.norm(np.asarray(lam) - S[:k] ** 2) <= 2 * u * np.linalg.norm(S[:k] ** 2)
    assert abs(disc - (S[k:] ** 2).sum() / (S ** 2).sum()) <= 8 * u


@pytest.mark.parametrize("direction", [0, 1])
def test_eigenvalues_descend_where_many_are_equal(ctx, direction):
    import torch
    from paper_2410_18740_gb300 import vtn
    rng = np.random.default_rng(direction)
    T = _tensor(rng, 520, 512, _spectrum("degenerate top", 512, 64))
    left = torch.empty(520, 64, dtype=torch.complex128, device="cuda")
    right = torch.empty(64, 512, dtype=torch.complex128, device="cuda")
    _, lam, _ = vtn.vtn_truncate(ctx, 65, 8, 8, 64, direction, 64, torch.from_numpy(np.ascontiguousarray(T)).cuda(), left, right)
    assert (np.diff(np.asarray(lam)) <= 0).all()
