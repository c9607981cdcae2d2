"""Lanczos on vectors around the size where one CTA does a step's vector work (2048 elements), with more Krylov
vectors than one group of dot products (8), against the same recursion in numpy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _krylov_minimum(apply, x, K):
    V, al, be = [x / np.linalg.norm(x)], [], []
    for j in range(K):
        w = apply(V[j])
        for p in range(2):
            c = np.array(V).conj() @ w
            if p == 0:
                al.append(c[j].real)
            w = w - np.array(V).T @ c
        be.append(np.linalg.norm(w))
        if be[-1] < 1e-13:
            break
        V.append(w / be[-1])
    m = len(al)
    E, Y = np.linalg.eigh(np.diag(al) + np.diag(be[:m - 1], 1) + np.diag(be[:m - 1], -1))
    y = sum(Y[j, 0] * V[j] for j in range(m))
    return E[0], y / np.linalg.norm(y)


@pytest.mark.parametrize("cl,cr", [(3, 5), (32, 32), (25, 41), (64, 32), (50, 41), (90, 61)])
@pytest.mark.parametrize("K", [1, 8, 19])
def test_ritz_pair_after_a_fixed_number_of_steps(ctx, cl, cr, K):
    import torch
    from paper_2410_18740_gb300 import vtn
    rng = np.random.default_rng(cl * cr)
    herm = lambda n: (lambda a: (a + a.conj().T) / np.sqrt(8.0 * n))(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    L, R = herm(cl), herm(cr)
    x = rng.standard_normal((cl, cr)) + 1j * rng.standard_normal((cl, cr))
    K = min(K, cl * cr - 1)
    E0, v0 = _krylov_minimum(lambda v: (L @ v.reshape(cl, cr) @ R).reshape(-1), x.reshape(-1), K)
    one = vtn.make_core(1, 1, 1, [0], [0], np.ones((1, 1, 1), complex))
    th = torch.from_numpy(x).cuda()
    _, E, n_mv = vtn.vtn_heff_ground(ctx, one, one, cl, cr, torch.from_numpy(L).cuda(), torch.from_numpy(R).cuda(), th,
                                     tol=1e-15, krylov_max=K, max_restarts=0)
    # |H| <= about 2: rounding of K products and two orthogonalisations each, over the gap of the Ritz values
    assert n_mv == K and abs(E - E0) <= 1e-12
    v = th.cpu().numpy().reshape(-1)
    assert abs(abs(np.vdot(v0, v)) - 1.0) <= 1e-10 and abs(np.linalg.norm(v) - 1.0) <= 1e-13


@pytest.mark.parametrize("cl,cr", [(30, 40), (64, 64)])  # both forms of the vector work
@pytest.mark.parametrize("spread", [3e-5, 1e-5, 6e-6])
def test_long_runs_on_a_spectrum_narrow_against_its_shift(ctx, cl, cr, spread):
    """64 Krylov vectors of 1 + spread H, H's spectrum thin at its ends: a little below the lowest eigenvalue all 64
    pivots of the tridiagonal matrix are far below its norm, and their product is below the smallest double."""
    import torch
    from statistics import NormalDist
    from paper_2410_18740_gb300 import vtn
    rng = np.random.default_rng(cl)
    quantiles = lambda n: np.array([0.5 + 0.12 * NormalDist().inv_cdf((i + 0.5) / n) for i in range(n)])
    h, g = 1.0 + spread * quantiles(cl), 1.0 + spread / cl * quantiles(cr)
    q = lambda n: np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))[0]
    U, V = q(cl), q(cr)
    L, R = (U * h) @ U.conj().T, (V * g) @ V.conj().T
    x = rng.standard_normal((cl, cr)) + 1j * rng.standard_normal((cl, cr))
    one = vtn.make_core(1, 1, 1, [0], [0], np.ones((1, 1, 1), complex))
    th = torch.from_numpy(x).cuda()
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    _, E, n_mv = vtn.vtn_heff_ground(ctx, one, one, cl, cr, t(L), t(R), th, tol=1e-300, krylov_max=64, max_restarts=0)
    v = th.cpu().numpy()
    rq = np.vdot(v, L @ v @ R).real / np.vdot(v, v).real
    # a Ritz value lies within the spectrum and is its vector's Rayleigh quotient: 64 steps of roundings of |H| = 1
    assert n_mv == 64 and E >= (h[:, None] * g).min() - 64 * 2.0 ** -52 and abs(E - rq) <= 64 * 2.0 ** -52
