"""Timed cases of the solver's main path, each through the public binding (``vtn``).

The sizes are those of the repository's three workload families (``inputs.workload``):

* ``plain`` -- M = 4 modes, d = D = 4, chi = 16: everything fits a few kilobytes, so a call costs its launches;
* ``split`` -- M = 24 modes, d = D = 8, chi up to 128;
* ``large`` -- M = 100 modes, Fock cutoff 24 rotated to d = 6, chi up to 512 (256 here, so that a pass of a
  windowed sweep stays well under two seconds and its 64-bit counterparts can be computed).

Bond dimensions between the powers of two stand for what sweeps meet at the chain's ends and while the bond
dimension grows.  Everything that runs in FP64 is the library's default precision; ``bf16x3`` is the
split-precision mode of the large workload, which is timed by its two products (H_eff psi and the environment
update) and by the truncation at its sizes: the states that whole split-precision sweeps end in are decided by
16-bit roundings, so that two exact truncations that differ in the last bit of an eigenvector lead to states
1e-4 apart.
"""
import math

import numpy as np
import torch

from paper_2410_18740_gb300 import inputs, vtn

PREC = {"f64": vtn.VTN_FP64, "bf16x3": vtn.VTN_BF16X3}
C128 = torch.complex128


# --------------------------------------------------------------------------- the cases
def listed():
    return [
        # one H_eff psi product of the smallest workload's size: what a short chain's Lanczos steps cost
        {"name": "heff_plain_f64", "kind": "heff", "family": "plain", "prec": "f64", "M": 8, "chi_l": 16, "chi_r": 16},
        # the hot product of a default-precision solve at its widest bond
        {"name": "heff_split_f64", "kind": "heff", "family": "split", "prec": "f64", "M": 24, "chi_l": 128, "chi_r": 128},
        # the hot product of the large workload's precision mode
        {"name": "heff_large_x3", "kind": "heff", "family": "large", "prec": "bf16x3", "M": 100, "chi_l": 256, "chi_r": 256},
        # environment update of a default-precision solve while the bond grows
        {"name": "env_left_f64", "kind": "env", "family": "split", "prec": "f64", "M": 24, "side": 0, "chi_l": 96, "chi_r": 121},
        # environment update of the large workload
        {"name": "env_right_x3", "kind": "env", "family": "large", "prec": "bf16x3", "M": 100, "side": 1, "chi_l": 384, "chi_r": 384},
        # truncation of a two-site tensor at the split workload's middle bonds
        {"name": "trunc_split", "kind": "trunc", "d": 8, "chi_l": 128, "chi_r": 128, "k": 128, "direction": 0},
        # truncation on the way to the large workload's bond dimension, sweeping left, ragged bonds
        {"name": "trunc_large", "kind": "trunc", "d": 6, "chi_l": 299, "chi_r": 305, "k": 300, "direction": 1},
        # one bond's Lanczos solve (12 Krylov steps, as a sweep with a fixed budget runs it)
        {"name": "ground_f64", "kind": "ground", "family": "split", "M": 24, "chi_l": 64, "chi_r": 64, "krylov": 12},
        # a whole solve of the smallest workload and its read-out
        {"name": "solve_plain", "kind": "solve", "solver": "two_site", "family": "plain", "M": 4, "d": 4, "chi": 16, "sweeps": 3},
        # a solve in the default precision on a chain of middling length, and its read-out
        {"name": "solve_split_f64", "kind": "solve", "solver": "two_site", "family": "split", "M": 10, "d": 8, "chi": 64, "sweeps": 2},
        # the single-site solver with subspace expansion on the same family, and its read-out
        {"name": "solve_single_site", "kind": "solve", "solver": "single_site", "family": "split", "M": 10, "d": 6, "chi": 40, "sweeps": 2},
        # read-out of a solved large chain: FP64 energy, every Fock marginal and photon-number samples
        {"name": "readout_large", "kind": "readout", "family": "large", "M": 100, "chi": 96, "samples": 64},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["heff", "heff", "env", "env", "trunc", "trunc", "ground", "solve", "solve", "readout"])
    if kind in ("heff", "env"):
        prec = rng.choice(["f64", "bf16x3"])
        if prec == "f64":
            c = {"kind": kind, "family": "split", "prec": prec, "M": rng.randint(8, 24)}
            c["chi_l"] = _log(rng, 12, 128)
        else:
            c = {"kind": kind, "family": "large", "prec": prec, "M": rng.randint(24, 100)}
            c["chi_l"] = _log(rng, 64, 256)
        c["chi_r"] = max(8, min(128 if prec == "f64" else 256, int(c["chi_l"] * rng.uniform(0.7, 1.4))))
        if kind == "env":
            c["side"] = rng.randint(0, 1)
        return c
    if kind == "trunc":
        chi = _log(rng, 16, 300)
        chi_r = max(8, min(305, int(chi * rng.uniform(0.8, 1.25))))
        return {"kind": "trunc", "d": rng.choice([4, 6]), "chi_l": chi, "chi_r": chi_r, "k": min(300, _log(rng, 16, 1.2 * chi)),
                "direction": rng.randint(0, 1)}
    if kind == "ground":
        chi = _log(rng, 12, 64)
        return {"kind": "ground", "family": "split", "M": rng.randint(8, 24), "chi_l": chi,
                "chi_r": max(8, min(64, int(chi * rng.uniform(0.7, 1.4)))), "krylov": rng.randint(6, 12)}
    if kind == "solve":
        return {"kind": "solve", "solver": rng.choice(["two_site", "single_site"]), "family": "split", "M": rng.randint(5, 10),
                "d": rng.randint(4, 6), "chi": _log(rng, 12, 48), "sweeps": rng.randint(1, 2)}
    return {"kind": "readout", "family": "large", "M": rng.randint(30, 100), "chi": _log(rng, 16, 96), "samples": _log(rng, 8, 64)}


# --------------------------------------------------------------------------- inputs
_ctx = None


def _context():
    """The one context a program creates at its start."""
    global _ctx
    if _ctx is None:
        _ctx = vtn.vtn_create(0)
    return _ctx


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 13)
    return g


def _randn(g, *shape):
    """Complex normals of unit variance."""
    return torch.view_as_complex(torch.randn(*shape, 2, dtype=torch.float64, device="cuda", generator=g) * math.sqrt(0.5))


def _workload(case, seed):
    """The instance: Haar interferometer and squeezing drawn from the seed.  Only the split family lets a case
    choose its local dimension (d = D, the Fock basis)."""
    over = {"M": case["M"]}
    if "d" in case and case["family"] != "large":
        over.update(D=case["d"], d=case["d"])
    return inputs.workload(case["family"], seed, **over)


def _middle_cores(case, seed, two):
    """Host copies of the MPO cores at the chain's middle: (w_l, w_r, rows, cols, ops) each."""
    w = _workload(case, seed)
    mpo = vtn.vtn_build_mpo(None, w.r, w.U, w.D, w.d)
    i = case["M"] // 2 - 1
    cores = [vtn.vtn_mpo_core(mpo, s) for s in ((i, i + 1) if two else (i,))]
    vtn.vtn_mpo_free(mpo)
    return cores, w.d


def _abi_core(core, d):
    return vtn.make_core(core[0], core[1], d, core[2], core[3], core[4])


def _environment(g, w, chi):
    """Channel blocks as a chain's middle has them: the identity of the untouched channel, Hermitian operator
    blocks of differing size for the pending ones, the accumulated Hamiltonian as the largest."""
    E = _randn(g, w, chi, chi)
    E = (E + E.conj().transpose(1, 2)) * (0.5 / math.sqrt(chi))
    size = torch.exp(torch.rand(w, dtype=torch.float64, device="cuda", generator=g) * math.log(20.0)) * 0.3
    size[-1] = 25.0
    E *= size.view(w, 1, 1)
    E[0] = torch.eye(chi, dtype=C128, device="cuda")
    return E.contiguous()


def _centre(g, rows, cols):
    """rows x cols two-site tensor with the decaying Schmidt spectrum of a solved bond, of unit norm."""
    r = min(rows, cols)
    s = torch.exp(-torch.linspace(0.0, 9.0, r, dtype=torch.float64, device="cuda"))
    T = (_randn(g, rows, r) * s.to(C128)) @ _randn(g, r, cols)
    return (T / torch.linalg.norm(T)).contiguous()


def _sites(case, seed, d):
    """Site tensors of a chain, nearly right-canonical (normals of that scale)."""
    M, chi = case["M"], case["chi"]
    dims = [min(chi, d ** min(s, 12), d ** min(M - s, 12)) for s in range(M + 1)]
    g = _gen(seed)
    return [(_randn(g, dims[s], d, dims[s + 1]) / math.sqrt(d * dims[s + 1])).cpu().numpy() for s in range(M)]


class State(dict):
    """What a program keeps between calls; handles are given back when it is dropped."""

    def __del__(self):
        for free, key in ((vtn.vtn_mps_free, "mps"), (vtn.vtn_mpo_free, "mpo")):
            if self.get(key) is not None:
                free(self[key])


def prepare(case, seed):
    ctx, kind = _context(), case["kind"]
    st = State(case=dict(case), kind=kind, ctx=ctx)
    if kind in ("heff", "ground", "env"):
        cores, d = _middle_cores(case, seed, kind != "env")
        st["cores"] = [_abi_core(c, d) for c in cores]
        cl, cr, g = case["chi_l"], case["chi_r"], _gen(seed)
        if kind == "env":
            left = case["side"] == 0
            st["env"] = _environment(g, cores[0][0] if left else cores[0][1], cl if left else cr)
            st["A"] = (_randn(g, cl, d, cr) / math.sqrt(d * max(cl, cr))).contiguous()
            st["out"] = torch.empty(cores[0][1] if left else cores[0][0], cr if left else cl, cr if left else cl, dtype=C128, device="cuda")
        else:
            st["L"], st["R"] = _environment(g, cores[0][0], cl), _environment(g, cores[1][1], cr)
            st["theta"] = _centre(g, cl * d, d * cr).reshape(cl, d, d, cr)
            st["y"] = torch.empty_like(st["theta"])
    elif kind == "trunc":
        d, cl, cr = case["d"], case["chi_l"], case["chi_r"]
        k = min(case["k"], cl * d, d * cr)
        st["theta"] = _centre(_gen(seed), cl * d, d * cr)
        st["left"] = torch.empty(cl * d, k, dtype=C128, device="cuda")
        st["right"] = torch.empty(k, d * cr, dtype=C128, device="cuda")
    else:
        w = _workload(case, seed)
        st["mpo"] = vtn.vtn_build_mpo(ctx, w.r, w.U, w.D, w.d)
        if kind == "readout":
            st["mps"] = vtn.vtn_mps_from_host(ctx, st["mpo"], _sites(case, seed, w.d))
        st["seed"] = int(seed)
    return st


# --------------------------------------------------------------------------- one pass
def run(st):
    case, kind, ctx = st["case"], st["kind"], st["ctx"]
    if kind == "heff":
        vtn.vtn_heff_apply(ctx, *st["cores"], case["chi_l"], case["chi_r"], st["L"], st["R"], st["theta"], st["y"], PREC[case["prec"]])
        return st["y"]
    if kind == "env":
        vtn.vtn_env_update(ctx, st["cores"][0], case["side"], case["chi_l"], case["chi_r"], st["env"], st["A"], st["out"], PREC[case["prec"]])
        return st["out"]
    if kind == "trunc":
        _, lam, disc = vtn.vtn_truncate(ctx, case["chi_l"], case["d"], case["d"], case["chi_r"], case["direction"], case["k"],
                                        st["theta"], st["left"], st["right"])
        # the two factors are defined up to a phase a kept vector; the compressed tensor is what the state becomes
        return {"lam": lam, "discarded": disc, "theta": st["left"] @ st["right"]}
    if kind == "ground":
        x = st["theta"].clone()
        _, E, _ = vtn.vtn_heff_ground(ctx, *st["cores"], case["chi_l"], case["chi_r"], st["L"], st["R"], x, tol=1e-12,
                                      krylov_max=case["krylov"], max_restarts=0)
        # an eigenvector's sign is free: the one with a positive overlap with the start
        ov = torch.vdot(st["theta"].reshape(-1), x.reshape(-1))
        return {"E": E, "theta": x * torch.where(ov.real < 0, -1.0, 1.0)}
    if kind == "solve":
        opts = vtn.vtn_sweep_opts_default(chi_max=case["chi"], n_sweeps=case["sweeps"], seed=st["seed"], lanczos_tol=1e-12,
                                          krylov_max=8, lanczos_max_restarts=0)
        sweep = vtn.vtn_sweep if case["solver"] == "two_site" else vtn.vtn_sweep_single_site
        _, mps, rep = sweep(ctx, st["mpo"], None, opts)
        P = vtn.vtn_marginals_all(ctx, st["mpo"], mps)
        vtn.vtn_mps_free(mps)
        return {"energy": np.array(rep["energy"]), "discarded": np.array(rep["max_discarded"]), "marginals": P}
    return {"energy": vtn.vtn_energy(ctx, st["mpo"], st["mps"]), "marginals": vtn.vtn_marginals_all(ctx, st["mpo"], st["mps"]),
            "samples": vtn.vtn_sample(ctx, st["mpo"], st["mps"], st["seed"], case["samples"])}


# --------------------------------------------------------------------------- what a pass cannot do without
def _widths(M):
    return [1 if s in (0, M) else 2 * min(s, M - s) + 2 for s in range(M + 1)]


def _heff_work(d, wl, wr, cl, cr):
    return (16 * (wl * cl * cl + wr * cr * cr + 2 * d * d * cl * cr), 8.0 * d * d * cl * cr * (wl * cl + wr * cr))


def _env_work(d, wi, wo, ci, co):
    return 16 * (wi * ci * ci + wo * co * co + d * ci * co), 8.0 * d * ci * co * (wi * ci + wo * co)


def _trunc_work(n1, n2, k, direction):
    n, m = (n1, n2) if direction == 0 else (n2, n1)
    # half of rho, its tridiagonal form, the back-transformation of k vectors, the product with the tensor
    return 16 * (n1 * n2 + k * (n1 + n2)) + 8 * k, 4.0 * n * n * m + 16.0 / 3 * n ** 3 + 8.0 * n * n * k + 8.0 * n * m * k


def work(case):
    kind = case["kind"]
    d = case.get("d") or {"plain": 4, "split": 8, "large": 6}[case["family"]]
    if kind == "trunc":
        b, f = _trunc_work(case["chi_l"] * d, d * case["chi_r"], min(case["k"], case["chi_l"] * d, d * case["chi_r"]), case["direction"])
        return {"bytes": b, "flops": f}
    M = case["M"]
    w, i = _widths(M), M // 2 - 1
    if kind in ("heff", "ground"):
        cl, cr = case["chi_l"], case["chi_r"]
        b, f = _heff_work(d, w[i], w[i + 2], cl, cr)
        if kind == "heff":
            return {"bytes": b, "flops": f}
        K, n = case["krylov"], d * d * cl * cr
        return {"bytes": b + 16 * n * K, "flops": f * K + 16.0 * n * K * (K + 1)}
    if kind == "env":
        ws = (w[i], w[i + 1]) if case["side"] == 0 else (w[i + 1], w[i])
        ch = (case["chi_l"], case["chi_r"]) if case["side"] == 0 else (case["chi_r"], case["chi_l"])
        b, f = _env_work(d, *ws, *ch)
        return {"bytes": b, "flops": f}
    dims = [min(case["chi"], d ** min(s, 12), d ** min(M - s, 12)) for s in range(M + 1)]
    env = [_env_work(d, w[s], w[s + 1], dims[s], dims[s + 1]) for s in range(M)]
    site_bytes = sum(16 * d * dims[s] * dims[s + 1] for s in range(M))
    if kind == "readout":
        D = 24 if case["family"] == "large" else d
        b, f = site_bytes + 8 * M * D + 4 * M * case["samples"], sum(e[1] for e in env)
        for s in range(M):
            a, c = dims[s], dims[s + 1]
            # right environments, the density of each mode, one conditional step a sample and mode
            f += 8.0 * d * a * c * (a + c) + 8.0 * d * d * a * c + 8.0 * case["samples"] * D * a * c
        return {"bytes": b, "flops": f}
    b, f = site_bytes, sum(e[1] for e in env)
    for s in range(M - 1):
        h = 8 * _heff_work(d, w[s], w[s + 2], dims[s], dims[s + 2])[1]
        t = _trunc_work(dims[s] * d, d * dims[s + 2], dims[s + 1], 0)[1]
        if case["solver"] == "single_site":
            h, t = h / d, _trunc_work(dims[s] * d, dims[s + 1], dims[s + 1], 0)[1]
        f += 2 * case["sweeps"] * (h + t + env[s][1])
    return {"bytes": b, "flops": f}


# --------------------------------------------------------------------------- the same in plain 64 bits
def _dense(core, d):
    wl, wr, rows, cols, ops = core
    W = torch.zeros(wl, wr, d, d, dtype=C128)
    for a, b, o in zip(rows, cols, ops):
        W[int(a), int(b)] += torch.from_numpy(np.ascontiguousarray(o))
    return W.cuda()


def _mix(W, X):
    """Y[b, i, t, q] = sum W[a, b, t, s] X[a, i, s, q]"""
    a, i, s, q = X.shape
    m = W.permute(1, 2, 0, 3).reshape(-1, a * s)
    Y = m @ X.permute(0, 2, 1, 3).reshape(a * s, i * q)
    return Y.reshape(W.shape[1], W.shape[2], i, q).permute(0, 2, 1, 3).contiguous()


def _apply(Wi, Wj, L, R, x):
    cl, d, _, cr = x.shape
    wl, wm, wr = Wi.shape[0], Wi.shape[1], Wj.shape[1]
    T = (L.reshape(wl * cl, cl) @ x.reshape(cl, -1)).reshape(wl, cl, d, d * cr)
    T = _mix(Wi, T).reshape(wm, cl * d, d, cr)
    T = _mix(Wj, T).reshape(wr, cl * d * d, cr)
    y = torch.zeros(cl * d * d, cr, dtype=C128, device="cuda")
    for c in range(wr):
        y += T[c] @ R[c]
    return y.reshape(cl, d, d, cr)


def _lanczos(apply, x0, K):
    V, al, be = [x0.reshape(-1) / torch.linalg.norm(x0)], [], []
    for j in range(K):
        w = apply(V[j].reshape(x0.shape)).reshape(-1)
        for p in range(2):
            B = torch.stack(V)
            c = B.conj() @ w
            if p == 0:
                al.append(float(c[j].real))
            w = w - B.T @ c
        be.append(float(torch.linalg.norm(w)))
        V.append(w / be[-1])
    E, Y = np.linalg.eigh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))
    x = sum(float(Y[j, 0]) * V[j] for j in range(K))
    return float(E[0]), (x / torch.linalg.norm(x)).reshape(x0.shape)


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        return None
    if kind == "trunc":
        d, cl, cr = case["d"], case["chi_l"], case["chi_r"]
        k = min(case["k"], cl * d, d * cr)
        T = _centre(_gen(seed), cl * d, d * cr)
        rho = T @ T.conj().T if case["direction"] == 0 else T.conj().T @ T
        lam, U = torch.linalg.eigh(rho)
        lam, U = lam.flip(0)[:k], U.flip(1)[:, :k]
        theta = U @ (U.conj().T @ T) if case["direction"] == 0 else (T @ U) @ U.conj().T
        return {"lam": lam, "discarded": float(1 - lam.sum() / torch.linalg.norm(T) ** 2), "theta": theta}
    if kind == "readout":
        return _exact_readout(case, seed)
    cores, d = _middle_cores(case, seed, kind != "env")
    W = [_dense(c, d) for c in cores]
    cl, cr, g = case["chi_l"], case["chi_r"], _gen(seed)
    if kind == "env":
        W, left = W[0], case["side"] == 0
        wl, wr = W.shape[:2]
        E = _environment(g, wl if left else wr, cl if left else cr)
        A = _randn(g, cl, d, cr) / math.sqrt(d * max(cl, cr))
        if left:
            T = _mix(W, (E.reshape(wl * cl, cl) @ A.reshape(cl, -1)).reshape(wl, cl, d, cr))
            return torch.matmul(A.reshape(cl * d, cr).conj().T, T.reshape(wr, cl * d, cr))
        T = torch.matmul(A.reshape(1, cl * d, cr), E).reshape(wr, cl, d, cr)
        T = _mix(W.transpose(0, 1), T)
        return torch.matmul(T.reshape(wl, cl, d * cr), A.reshape(cl, d * cr).conj().T)
    L, R = _environment(g, W[0].shape[0], cl), _environment(g, W[1].shape[1], cr)
    x = _centre(g, cl * d, d * cr).reshape(cl, d, d, cr)
    if kind == "heff":
        return _apply(W[0], W[1], L, R, x)
    E, v = _lanczos(lambda t: _apply(W[0], W[1], L, R, t), x, case["krylov"])
    ov = torch.vdot(x.reshape(-1), v.reshape(-1))
    return {"E": E, "theta": v * (-1.0 if ov.real < 0 else 1.0)}


def _exact_readout(case, seed):
    w = _workload(case, seed)
    mpo = vtn.vtn_build_mpo(None, w.r, w.U, w.D, w.d)  # its cores and isometries are inputs here
    M, d = w.M, w.d
    A = [torch.from_numpy(a).cuda() for a in _sites(case, seed, d)]
    one = torch.ones(1, 1, dtype=C128, device="cuda")
    R, L, H = [None] * M + [one], one, one.reshape(1, 1, 1)
    for s in range(M - 1, -1, -1):
        R[s] = torch.einsum("asg,gh,bsh->ab", A[s], R[s + 1], A[s].conj())  # [ket][bra]
    P = []
    for s in range(M):
        X = torch.einsum("ij,jtk->itk", L, A[s])  # L[bra][ket]
        rho = torch.einsum("isb,ab,ita->st", torch.einsum("jsk,kb->jsb", X, R[s + 1]), torch.eye(R[s + 1].shape[0], dtype=C128, device="cuda"), A[s].conj())
        V = torch.from_numpy(np.ascontiguousarray(vtn.vtn_mpo_isometry(mpo, s))).cuda()
        P.append(torch.einsum("ns,st,nt->n", V, rho, V.conj()).real)
        L = torch.einsum("itl,itk->lk", A[s].conj(), X)
        W = _dense(vtn.vtn_mpo_core(mpo, s), d)
        T = _mix(W, torch.matmul(H, A[s].reshape(1, A[s].shape[0], -1)).reshape(H.shape[0], H.shape[1], d, -1))
        H = torch.matmul(A[s].reshape(-1, A[s].shape[2]).conj().T, T.reshape(T.shape[0], -1, T.shape[3]))
    vtn.vtn_mpo_free(mpo)
    norm = float(L[0, 0].real)
    return {"energy": float(H[0, 0, 0].real) / norm, "marginals": (torch.stack(P) / norm).cpu().numpy(), "samples": None}
