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
