"""FP64 core mixing from spelled-out terms: every kind of coefficient, empty channels, both directions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _core(rng, w_l, w_r, d):
    """Dense W[a, b, s', s] with pass-through, scaled, real, imaginary, complex and banded blocks; column w_r - 1
    and row w_l - 1 are empty."""
    W = np.zeros((w_l, w_r, d, d), complex)
    band = np.triu(np.tril(np.ones((d, d)), 1), -1) - np.eye(d)
    kinds = [np.eye(d), -1.75 * np.eye(d), band * rng.standard_normal((d, d)), 1j * band * rng.standard_normal((d, d)),
             rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d)), 1j * np.eye(d), np.diag(np.arange(d) + 1.0)]
    n = 0
    for a in range(w_l - 1):
        for b in range(w_r - 1):
            if a == b or rng.random() < 0.5:
                W[a, b] = kinds[n % len(kinds)]
                n += 1
    return W


@pytest.mark.parametrize("d,cl,cr", [(1, 5, 9), (2, 1, 1), (3, 17, 5), (6, 9, 31), (8, 16, 33), (16, 3, 4)])
def test_spelled_out_terms_match_the_dense_core(ctx, d, cl, cr):
    import torch
    from paper_2410_18740_gb300 import vtn
    rng = np.random.default_rng(100 * d + cl)
    wl, wm, wr = 4, 5, 3
    Wi, Wj = _core(rng, wl, wm, d), _core(rng, wm, wr, d)
    z = lambda *s: torch.from_numpy(rng.standard_normal(s) + 1j * rng.standard_normal(s)).cuda()
    t = lambda W: torch.from_numpy(W).cuda()
    L, R, th = z(wl, cl, cl), z(wr, cr, cr), z(cl, d, d, cr)
    y = torch.empty_like(th)
    vtn.vtn_heff_apply(ctx, vtn.core_from_dense(Wi), vtn.core_from_dense(Wj), cl, cr, L, R, th, y)
    T = torch.einsum("aij,jsvk->aisvk", L, th)
    T = torch.einsum("abts,aisvk->bitvk", t(Wi), T)
    T = torch.einsum("bcuv,bitvk->cituk", t(Wj), T)
    ref = torch.einsum("cituk,ckl->itul", T, R)
    # four contractions of at most w d chi terms, u sqrt(terms) each, with room
    assert float(torch.linalg.norm(y - ref)) <= 1e-14 * float(torch.linalg.norm(ref)) + 1e-300
    for side, ci, co, w_in, w_out in ((0, cl, cr, wl, wm), (1, cr, cl, wm, wl)):
        A, E = z(cl, d, cr), z(w_in, ci, ci)
        out = torch.empty(w_out, co, co, dtype=torch.complex128, device="cuda")
        vtn.vtn_env_update(ctx, vtn.core_from_dense(Wi), side, cl, cr, E, A, out)
        if side == 0:
            U = torch.einsum("abts,aisk->bitk", t(Wi), torch.einsum("aij,jsk->aisk", E, A))
            ref = torch.einsum("itl,bitk->blk", A.conj(), U)
            assert bool((out[-1] == 0).all())
        else:
            U = torch.einsum("abts,bjsp->ajtp", t(Wi), torch.einsum("jsg,bgp->bjsp", A, E))
            ref = torch.einsum("ajtp,itp->aji", U, A.conj())
            assert bool((out[-1] == 0).all())
        assert float(torch.linalg.norm(out - ref)) <= 1e-14 * float(torch.linalg.norm(ref)) + 1e-300


def test_channels_of_a_collapse_core_stay_apart_from_non_finite_ones(ctx):
    """Scaled identities between many channels, as one product on the tensor cores: an infinity in one channel reaches
    the channels that are coupled to it and no others, as term by term."""
    import torch
    from paper_2410_18740_gb300 import vtn
    rng = np.random.default_rng(8)
    w, d, cl, cr = 48, 4, 96, 96
    C = rng.standard_normal((w, w)) * (rng.random((w, w)) < 0.5)
    a, b = np.nonzero(C)
    core = vtn.make_core(w, w, d, a, b, C[a, b][:, None, None] * np.eye(d, dtype=complex))
    A = torch.from_numpy(rng.standard_normal((cl, d, cr)) + 1j * rng.standard_normal((cl, d, cr))).cuda()
    for side, ci, co in ((0, cl, cr), (1, cr, cl)):
        E = torch.from_numpy(rng.standard_normal((w, ci, ci)) + 1j * rng.standard_normal((w, ci, ci))).cuda()
        out, bad = (torch.empty(w, co, co, dtype=torch.complex128, device="cuda") for _ in range(2))
        vtn.vtn_env_update(ctx, core, side, cl, cr, E, A, out)
        E[7, 3, 5] = float("inf")
        vtn.vtn_env_update(ctx, core, side, cl, cr, E, A, bad)
        free = torch.from_numpy((C[7] if side == 0 else C[:, 7]) == 0).cuda()
        # the flagged elements are summed in FP64 instead of exactly: u sqrt(w) of a norm, with room
        assert float(torch.linalg.norm((bad - out)[free])) <= 1e-14 * float(torch.linalg.norm(out[free]))
        assert not bool(torch.isfinite(torch.view_as_real(bad[~free])).all((1, 2, 3)).any())


@pytest.mark.parametrize("side", [0, 1])
def test_collapse_core_on_the_tensor_cores_matches_the_dense_core(ctx, side):
    """Complex couplings between many channels at sizes where they are one sliced product, from either side."""
    import torch
    from paper_2410_18740_gb300 import vtn
    rng = np.random.default_rng(side)
    wl, wr, d, cl, cr = 40, 56, 4, 96, 91
    C = (rng.standard_normal((wl, wr)) + 1j * rng.standard_normal((wl, wr))) * (rng.random((wl, wr)) < 0.7)
    a, b = np.nonzero(C)
    core = vtn.make_core(wl, wr, d, a, b, C[a, b][:, None, None] * np.eye(d, dtype=complex))
    z = lambda *s: torch.from_numpy(rng.standard_normal(s) + 1j * rng.standard_normal(s)).cuda()
    A, W = z(cl, d, cr), torch.from_numpy(C).cuda()
    w_in, w_out, ci, co = (wl, wr, cl, cr) if side == 0 else (wr, wl, cr, cl)
    E, out = z(w_in, ci, ci), torch.empty(w_out, co, co, dtype=torch.complex128, device="cuda")
    vtn.vtn_env_update(ctx, core, side, cl, cr, E, A, out)
    if side == 0:
        ref = torch.einsum("itl,ab,aij,jtk->blk", A.conj(), W, E, A)
    else:
        ref = torch.einsum("jtg,ab,bgp,itp->aji", A, W, E, A.conj())
    # three contractions of at most 384 terms, u sqrt(terms) each, with room
    assert float(torch.linalg.norm(out - ref) / torch.linalg.norm(ref)) <= 1e-14
