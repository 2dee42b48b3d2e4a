"""The work that programs have this library do, as cases that can be timed and compared.

A case is a dict of plain values: the entry point it calls (`call`), the compute
path, and the sizes.  prepare() makes what a program holds before the call (a
THC Hamiltonian and states on the GPU, drawn from the seed), run() is one call
of the entry point.  A result state is returned as its coefficients over all
determinants of its particle-number sector (the CI vector), because the site
tensors themselves are only defined up to an orthogonal rotation of every bond:
two right answers can differ in every site tensor and in no coefficient.

Where the cut of a truncation falls between two nearby singular values, the
result depends on rounding far more than any kernel does, and in float32 a few
hundred such cuts decide every digit that is compared.  So the float32 and TF32
cases truncate states whose Schmidt spectrum is prescribed (compress), or keep
everything (D_max at the rank); the float64 cases truncate freely.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2409_12708_gb300 import binding as B
from paper_2409_12708_gb300.workloads import full_bond_profile, sector_mps, thc_hamiltonian

DTYPE = {"fp64": torch.float64, "fp32": torch.float32, "tf32": torch.float32}


# ---------------------------------------------------------------------- the cases
def listed():
    return [
        # a scalar product of two small states: the shortest call, many times per Krylov step
        dict(name="inner L6 D16 f64", call="inner", path="fp64", L=6, D=16, D2=16),
        # one ladder layer on the test-sized state: launches and latency only
        dict(name="layer L6 D16 f64", call="layer", path="fp64", L=6, D=16, D_max=16, sigma=1, dagger=1),
        # a small truncation by tolerance, float32 storage
        dict(name="compress L8 64-16 f32", call="compress", path="fp32", L=8, D=64, D_max=16, tol=1e-3),
        # one truncation of a long state back to the working bond, odd input bond
        dict(name="compress L12 255-128 tf32", call="compress", path="tf32", L=12, D=255, D_max=128, tol=0.0),
        # one ladder layer at the flagship's bond (128, expanded to 256), kept whole
        dict(name="layer L12 128-256 tf32", call="layer", path="tf32", L=12, D=128, D_max=256, sigma=0, dagger=1),
        # the largest bond supported
        dict(name="layer L10 256-512 f32", call="layer", path="fp32", L=10, D=256, D_max=512, sigma=0, dagger=0),
        # a Gram-Schmidt sum or the combination of Krylov vectors
        dict(name="add n8 L8 D256 tf32", call="add", path="tf32", L=8, D=256, D_max=256, n=8),
        # H|psi> of the small Krylov configuration, every term, truncated
        dict(name="H L6 N12 D16 f64", call="apply", path="fp64", L=6, N=12, D=16, terms=588, merge=False),
        # a share of H|psi> that fills the GPU with terms, at bond 256
        dict(name="H L8 N24 D256 tf32", call="apply", path="tf32", L=8, N=24, D=256, terms=608, merge=False),
        # the same path in its small form: every term of a six-site problem
        dict(name="H L6 N12 D64 f32", call="apply", path="fp32", L=6, N=12, D=64, terms=588, merge=False),
        # the derivatives of <phi|H|psi> in t, chi, zeta and psi
        dict(name="grad L10 N30 D64 f32", call="grad", path="fp32", L=10, N=30, D=64, terms=1024),
        # one time step of a complex state
        dict(name="step L5 N10 D16 c64", call="expm", path="fp32", L=5, N=10, D=16, K=3),
    ]


def draw(rng):
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    call = rng.choice(["inner", "layer", "layer", "compress", "compress", "add", "apply", "apply", "apply", "batched",
                       "grad", "lanczos", "expm"])
    path = rng.choice(["fp64", "fp32", "tf32"])
    wide = path != "fp64"
    if call == "inner":
        return dict(call=call, path=rng.choice(["fp64", "fp32"]), L=rng.randint(4, 12), D=log(4, 256), D2=log(4, 256))
    if call == "layer":
        L, D = (rng.randint(4, 12), log(6, 128)) if wide else (rng.randint(4, 10), log(4, 64))
        return dict(call=call, path=path, L=L, D=D, D_max=2 * D if wide else max(2, D - rng.randint(0, 3)),
                    sigma=rng.randint(0, 1), dagger=rng.randint(0, 1))
    if call == "compress":
        L, D = rng.randint(6, 12), log(16, 256 if wide else 64)
        return dict(call=call, path=path, L=L, D=D, D_max=max(4, int(D * rng.uniform(0.3, 0.8))),
                    tol=rng.choice([0.0, 0.0, 1e-3]))
    if call == "add":
        L = rng.randint(4, 8)
        D = 4 ** (L // 2) if wide else log(6, 24)
        return dict(call=call, path=path, L=L, D=D, D_max=D, n=rng.randint(2, 10))
    if call == "apply":
        L = rng.randint(4, 8 if wide else 6)
        N = rng.randint(L, 3 * L)
        most = 4 * N * N + 2 * L
        D = 4 ** (L // 2) if wide else log(5, 16)
        merge = (not wide) and rng.random() < 0.5
        return dict(call=call, path=path, L=L, N=N, D=D, merge=merge,
                    terms=3 * N * N + 2 * L if merge else min(most, log(2 * N, 608)))
    if call == "batched":
        return dict(call=call, path=path, n=rng.randint(2, 6), L=4, L2=rng.randint(5, 6), D=64 if wide else log(5, 16))
    if call == "grad":
        L = rng.randint(4, 10)
        N = rng.randint(L, 3 * L)
        return dict(call=call, path=rng.choice(["fp64", "fp32"]), L=L, N=N, D=log(4, 48),
                    terms=min(4 * N * N + 2 * L, log(2 * N, 1024)))
    L = rng.randint(4, 5)
    return dict(call=call, path="fp64" if call == "lanczos" else rng.choice(["fp64", "fp32"]), L=L,
                N=rng.randint(L, 2 * L), D=16, K=rng.randint(2, 4))


# ---------------------------------------------------------------------- inputs
def _decay(D):  # the flagship's spectrum, exp(-k / 12) at bond 128, for any bond
    return max(2.0, 12.0 * D / 128.0)


def _state(L, D, seed, bond=None):
    return sector_mps(L, L // 2, L - L // 2, D, seed, decay=_decay(bond or D))


def _dev(arrays, dtype=torch.float64):
    return [torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype) for a in arrays]


def _sector(L, n_up, n_dn):
    """Indices of the determinants with n_up, n_dn electrons in the 4^L vector."""
    code = torch.arange(4 ** L, device="cuda")
    up, dn = torch.zeros_like(code), torch.zeros_like(code)
    for i in range(L):
        up += (code >> (2 * i + 1)) & 1
        dn += (code >> (2 * i)) & 1
    return torch.nonzero((up == n_up) & (dn == n_dn))[:, 0]


def _out_sector(case):
    L = case["L"]
    up, dn = L // 2, L - L // 2
    if case["call"] == "layer":
        step = 1 if case["dagger"] else -1
        up, dn = (up + step, dn) if case["sigma"] == 0 else (up, dn + step)
    return up, dn


def _inputs(case, seed):
    """The seeded host inputs (float64 numpy) of a case."""
    call, rng = case["call"], np.random.default_rng(seed)
    s = lambda: int(rng.integers(1 << 31))  # noqa: E731
    if call == "batched":
        Ls = [case["L"] + (case["L2"] - case["L"]) * i // max(1, case["n"] - 1) for i in range(case["n"])]
        return {"Ls": Ls, "hams": [thc_hamiltonian(L, L, s()) for L in Ls],
                "psis": [_state(L, case["D"], s()) for L in Ls]}
    L, D = case["L"], case["D"]
    # a state to be compressed has the spectrum of the working bond
    x = {"psi": _state(L, D, s(), case["D_max"] if call == "compress" else None)}
    if call == "inner":
        x["phi"] = _state(L, case["D2"], s())
    elif call == "layer":
        x["coef"] = rng.standard_normal(L) / math.sqrt(L)
    elif call == "add":
        x["xs"] = [x["psi"]] + [_state(L, D, s()) for _ in range(case["n"] - 1)]
        x["coef"] = rng.standard_normal(case["n"])
    elif call in ("apply", "grad", "lanczos", "expm"):
        x["ham"] = thc_hamiltonian(L, case["N"], s())
        if call == "grad":
            x["phi"] = _state(L, D, s())
    return x


def prepare(case, seed):
    x, dt = _inputs(case, seed), DTYPE[case["path"]]
    st = {"case": case}
    if case["call"] == "batched":
        st["hams"] = [tuple(_dev(h)) for h in x["hams"]]
        st["psis"] = [_dev(p, dt) for p in x["psis"]]
        st["sectors"] = [_sector(L, L // 2, L - L // 2) for L in x["Ls"]]
        return st
    st["psi"] = _dev(x["psi"], dt)
    if "phi" in x:
        st["phi"] = _dev(x["phi"], dt)
    if "xs" in x:
        st["xs"], st["coef"] = [_dev(p, dt) for p in x["xs"]], [float(c) for c in x["coef"]]
    elif "coef" in x:
        st["coef"] = _dev([x["coef"]])[0]
    if "ham" in x:
        st["ham"] = tuple(_dev(x["ham"]))
    if case["call"] not in ("inner", "grad"):
        st["sector"] = _sector(case["L"], *_out_sector(case))
        if case["call"] == "lanczos":
            st["psi_ci"] = _ci(st["psi"], st["sector"])
    return st


# ---------------------------------------------------------------------- one call
def _dense(sites):
    """All 4^L coefficients of an MPS: the two halves contracted, then multiplied."""
    half = len(sites) // 2
    left = sites[0].reshape(4, -1)
    for a in sites[1:half]:
        left = (left @ a.reshape(a.shape[0], -1)).reshape(-1, a.shape[2])
    right = sites[-1].reshape(-1, 4)
    for a in reversed(sites[half:-1]):
        right = (a.reshape(-1, a.shape[2]) @ right).reshape(a.shape[0], -1)
    return (left @ right).reshape(-1)


def _ci(sites, sector):
    return _dense(sites)[sector]


def run(st):
    c = st["case"]
    call, path = c["call"], c["path"]
    if call == "inner":
        return B.mps_inner(st["phi"], st["psi"])
    if call == "layer":
        return _ci(B.thc_layer_apply(st["psi"], st["coef"], c["sigma"], c["dagger"], D_max=c["D_max"], path=path),
                   st["sector"])
    if call == "compress":
        return _ci(B.thc_compress(st["psi"], D_max=c["D_max"], tol=c["tol"], path=path), st["sector"])
    if call == "add":
        return _ci(B.mps_add_compress(st["coef"], st["xs"], D_max=c["D_max"], path=path), st["sector"])
    if call == "apply":
        return _ci(B.thc_apply_H(*st["ham"], st["psi"], D_max=c["D"], path=path, term_begin=0, term_end=c["terms"],
                                 merge_spin=c["merge"]), st["sector"])
    if call == "batched":
        outs = B.thc_apply_H_batched(st["hams"], st["psis"], D_max=c["D"], path=path)
        return [_ci(o, s) for o, s in zip(outs, st["sectors"])]
    if call == "grad":
        e, dt, dchi, dzeta, dpsi = B.thc_expect_grad(*st["ham"], st["phi"], st["psi"], path=path, term_begin=0,
                                                     term_end=c["terms"])
        return {"value": e, "t": dt, "chi": dchi, "zeta": dzeta, "psi": dpsi}
    if call == "lanczos":
        e, ritz, ground = B.krylov_lanczos_ground(*st["ham"], st["psi"], c["K"], D_max=c["D"], path=path,
                                                  want_ground=True)
        g = _ci(ground, st["sector"])  # the eigenvector's sign: towards the start vector
        return {"energy": e, "ritz": np.array(ritz), "ground": g * torch.sign(g @ st["psi_ci"])}
    out, lost = B.krylov_expm_apply(*st["ham"], st["psi"], 0.05, c["K"], D_max=c["D"], path=path)
    return {"state": _ci(out, st["sector"])}


# ---------------------------------------------------------------------- what a call cannot do without
def _compress_flops(bonds, D):
    """QR sweep and SVD sweep of one compression (Golub & Van Loan counts): R and
    the site it is absorbed by, then singular values and right vectors."""
    L, f = len(bonds) - 1, 0.0
    k = list(bonds)
    for s in range(L - 1, 0, -1):
        m, n = 4 * k[s + 1], bonds[s]
        k[s] = min(n, m)
        q = min(m, n)
        f += 2.0 * m * n * q - q * q * (m + n) + 2.0 * q ** 3 / 3 + 8.0 * bonds[s - 1] * n * q
    left = 1
    for s in range(L - 1):
        m, n = 4 * left, k[s + 1]
        out = min(D, m, n)
        f += 4.0 * max(m, n) * min(m, n) ** 2 + 8.0 * min(m, n) ** 3 + 8.0 * out * n * k[min(s + 2, L)]
        left = out
    return f


def _mps_values(L, D):
    b = full_bond_profile(L, D)
    return sum(4 * b[i] * b[i + 1] for i in range(L))


def work(case):
    call, size = case["call"], 8 if case["path"] == "fp64" else 4
    if call == "batched":
        x = [dict(case, call="apply", L=L, N=L, terms=4 * L * L + 2 * L) for L in (case["L"], case["L2"])]
        w = [work(y) for y in x]
        return {k: case["n"] * (w[0][k] + w[1][k]) / 2 for k in ("bytes", "flops")}
    L, D = case["L"], case["D"]
    b = full_bond_profile(L, D)
    vals = _mps_values(L, D)
    if call == "inner":
        b2 = full_bond_profile(L, case["D2"])
        f = sum(8.0 * b[i] * b2[i] * b2[i + 1] + 8.0 * b[i] * b[i + 1] * b2[i + 1] for i in range(L))
        return {"bytes": size * (vals + _mps_values(L, case["D2"])), "flops": f}
    dbl = [1] + [2 * v for v in b[1:-1]] + [1]
    if call == "layer":
        return {"bytes": size * (vals + _mps_values(L, case["D_max"])), "flops": _compress_flops(dbl, case["D_max"])}
    if call == "compress":
        return {"bytes": size * (vals + _mps_values(L, case["D_max"])), "flops": _compress_flops(b, case["D_max"])}
    one = _compress_flops(dbl, D)
    if call == "add":
        return {"bytes": size * (case["n"] + 1) * vals, "flops": (case["n"] - 1) * one}
    N = case["N"]
    ham = 8.0 * (L * L + L * N + N * N)
    if call == "grad":
        f = case["terms"] * sum(8.0 * 16 * b[i] * b[i + 1] * (b[i] + b[i + 1]) * 3 for i in range(L))
        return {"bytes": 2 * ham + size * 3 * vals, "flops": f}
    terms = case.get("terms", 4 * N * N + 2 * L)
    slots = -(-terms // (2 * N))
    f = (2 * terms + 2 * min(2 * N, slots) + terms - 1) * one
    steps = case.get("K", 1) * (4 if call == "expm" else 1)
    return {"bytes": ham + size * 2 * vals, "flops": steps * f}


# ---------------------------------------------------------------------- the same in 64 bits
# Untruncated results: ladder operators on the dense 4^L vector.
def _ladder(v, coef, sigma, dagger):
    """sum_s coef_s a_{s sigma} v (or the creation operators), Jordan-Wigner order
    site-major with spin up first; local index 2 n_up + n_dn."""
    L = len(coef)
    pairs = (((0, 2, 1.0), (1, 3, 1.0)), ((0, 1, 1.0), (2, 3, -1.0)))[sigma]  # (to, from, sign) of a
    sign = torch.ones(1, dtype=torch.float64, device=v.device)
    out = torch.zeros_like(v)
    for s in range(L):
        x, y = v.view(4 ** s, 4, -1), out.view(4 ** s, 4, -1)
        if float(coef[s]) != 0.0:
            for to, fr, g in pairs:
                i, j = (fr, to) if dagger else (to, fr)
                y[:, i] += (g * float(coef[s]) * sign)[:, None] * x[:, j]
        sign = torch.kron(sign, torch.tensor([1.0, -1.0, -1.0, 1.0], dtype=torch.float64, device=v.device))
    return out


def _one_body(v, m, sigma):
    """sum_pq m_pq a+_p a_q v"""
    out = torch.zeros_like(v)
    for p in range(m.shape[0]):
        e = np.zeros(m.shape[0])
        e[p] = 1.0
        out += _ladder(_ladder(v, m[p], sigma, False), e, sigma, True)
    return out


def _apply_dense(v, ham, terms):
    """The first `terms` terms of H on a dense vector, in the term order of the
    library: Coulomb ((s' N + nu) 2 + s) N + mu, then kinetic s L + i."""
    t, chi, zeta = ham
    L, N = chi.shape
    out = torch.zeros_like(v)
    for blk in range(min(2 * N, -(-terms // (2 * N)))):
        sp, nu = divmod(blk, N)
        phi = _ladder(_ladder(v, chi[:, nu], sp, False), chi[:, nu], sp, True)
        for s in range(2):
            n = min(N, terms - (blk * 2 + s) * N)
            if n > 0:
                out += _one_body(phi, (chi[:, :n] * (0.5 * zeta[:n, nu])) @ chi[:, :n].T, s)
    lam, u = np.linalg.eigh(t)
    for s in range(2):
        n = min(L, terms - 4 * N * N - s * L)
        if n > 0:
            out += _one_body(v, (u[:, :n] * lam[:n]) @ u[:, :n].T, s)
    return out


# Truncated results: the compression and the pairwise tree on numpy MPS.
def _np_compress(A, D, tol=0.0):
    A, L = [a.copy() for a in A], len(A)
    for i in range(L - 1, 0, -1):
        q, r = np.linalg.qr(A[i].reshape(A[i].shape[0], -1).T)
        A[i] = q.T.reshape(-1, 4, A[i].shape[2])
        A[i - 1] = np.tensordot(A[i - 1], r.T, axes=(2, 0))
    for i in range(L - 1):
        l = A[i].shape[0]
        u, s, vh = np.linalg.svd(A[i].reshape(4 * l, -1), full_matrices=False)
        k = min(D, len(s))
        if tol > 0.0:
            tail = np.append(np.cumsum((s ** 2)[::-1])[::-1], 0.0)
            k = max(1, min(k, int(np.argmax(tail <= tol * tol * tail[0]))))
        A[i] = u[:, :k].reshape(l, 4, k)
        A[i + 1] = np.tensordot(s[:k, None] * vh[:k], A[i + 1], axes=(1, 0))
    return A


_LOCAL = {}
for _sig, _b in enumerate((np.kron([[0.0, 1.0], [0.0, 0.0]], np.eye(2)),
                           np.kron(np.diag([1.0, -1.0]), [[0.0, 1.0], [0.0, 0.0]]))):
    _LOCAL[_sig, False], _LOCAL[_sig, True] = _b, _b.T


def _np_layer(A, coef, sigma, dagger, D, tol=0.0):
    L, out = len(A), []
    par = np.array([1.0, -1.0, -1.0, 1.0])[None, :, None]
    for s, a in enumerate(A):
        l, _, r = a.shape
        x = np.zeros((2, l, 4, 2, r))
        x[0, :, :, 0] = par * a
        x[0, :, :, 1] = coef[s] * np.einsum("mn,lnr->lmr", _LOCAL[sigma, dagger], a)
        x[1, :, :, 1] = a
        x = x[:1] if s == 0 else x
        x = x[:, :, :, 1:] if s == L - 1 else x
        out.append(x.reshape(x.shape[0] * l, 4, -1))
    return _np_compress(out, D, tol)


def _np_sum(items, D):
    def pair(a, b):
        out = []
        for i, (x, y) in enumerate(zip(a, b)):
            if i == 0:
                out.append(np.concatenate([x, y], axis=2))
            elif i == len(a) - 1:
                out.append(np.concatenate([x, y], axis=0))
            else:
                z = np.zeros((x.shape[0] + y.shape[0], 4, x.shape[2] + y.shape[2]))
                z[:x.shape[0], :, :x.shape[2]], z[x.shape[0]:, :, x.shape[2]:] = x, y
                out.append(z)
        return _np_compress(out, D)
    while len(items) > 1:
        items = [pair(items[i], items[i + 1]) if i + 1 < len(items) else items[i] for i in range(0, len(items), 2)]
    return items[0]


def _np_apply(psi, ham, D, terms, merge):
    t, chi, zeta = ham
    L, N = chi.shape
    if merge:
        todo = [(nu, 0, mu, 0, 1.0) for nu in range(N) for mu in range(N)]
        todo += [(nu, 1, mu, s, 2.0 - s) for nu in range(N) for s in range(2) for mu in range(N)]
    else:
        todo = [(nu, sp, mu, s, 1.0) for sp in range(2) for nu in range(N) for s in range(2) for mu in range(N)]
    lam, u = np.linalg.eigh(t)
    both = lambda x, c1, c2, s: _np_layer(_np_layer(x, c1, s, False, D), c2, s, True, D)  # noqa: E731
    reuse, out = {}, []
    for nu, sp, mu, s, f in todo[:terms]:
        if (nu, sp) not in reuse:
            reuse[nu, sp] = both(psi, chi[:, nu], chi[:, nu], sp)
        out.append(both(reuse[nu, sp], 0.5 * f * zeta[mu, nu] * chi[:, mu], chi[:, mu], s))
    for k in range(max(0, terms - len(todo))):
        s, i = divmod(k, L)
        out.append(both(psi, lam[i] * u[:, i], u[:, i], s))
    return _np_sum(out, D)


def _krylov(v, ham, K):
    """Orthonormal Krylov basis of a dense vector and H projected on it."""
    L, N = ham[1].shape
    basis, images = [v / v.norm()], []
    for k in range(K):
        w = _apply_dense(basis[k], ham, 4 * N * N + 2 * L)
        images.append(w)
        for _ in range(2):
            w = w - sum((b @ w) * b for b in basis)
        if k + 1 < K:
            basis.append(w / w.norm())
    V = torch.stack(basis)
    h = V @ torch.stack(images).T
    return V, ((h + h.T) / 2).cpu().numpy()


def _grad_exact(x, terms):
    """E = <phi|H|psi> over the first `terms` terms and its derivatives: the
    amplitudes <a+_q a_p phi | a+_r a_s psi> once, the factors by autograd."""
    t, chi, zeta = (torch.from_numpy(a).cuda().requires_grad_() for a in x["ham"])
    L, N = chi.shape
    sites = [a.requires_grad_() for a in _dev(x["psi"])]
    psi, phi = _dense(sites), _dense(_dev(x["phi"]))
    unit = np.eye(L)

    def bilinears(v):  # a+_p a_q v for all (sigma, p, q)
        low = [[_ladder(v, unit[q], s, False) for q in range(L)] for s in range(2)]
        return [[[_ladder(low[s][q], unit[p], s, True) for q in range(L)] for p in range(L)] for s in range(2)]

    bra, ket = bilinears(phi), bilinears(psi.detach())
    rows = torch.stack([torch.stack([torch.stack(r) for r in m]) for m in bra]).reshape(2 * L * L, -1)
    cols = torch.stack([torch.stack([torch.stack(r) for r in m]) for m in ket]).reshape(2 * L * L, -1)
    amp = (rows @ cols.T).reshape(2, L, L, 2, L, L)  # <a+_p a_q phi | a+_r a_s psi>
    index = torch.arange(4 * N * N, device="cuda").reshape(2, N, 2, N)  # s', nu, s, mu
    mask = (index < terms).double()
    pair = torch.einsum("pm,qm->mpq", chi, chi)
    inner = torch.einsum("apqbrs,npq,mrs->bman", amp, pair, pair)  # s' nu of the ket, s mu of the bra
    e = 0.5 * torch.einsum("bman,bman,nm->", mask, inner, zeta)
    kin = torch.arange(2 * L, device="cuda").reshape(2, L) + 4 * N * N < terms
    rows = rows.reshape(2, L, L, -1)
    gamma = rows @ psi.detach()  # [s, q, p]: <a+_q a_p phi|psi> = <phi|a+_p a_q psi>
    e = e + torch.einsum("pq,sqp,sq->", t, gamma, kin.double())
    e.backward()
    with torch.no_grad():  # dE/dpsi as a dense vector: sum of the terms' transposes on phi
        w = torch.einsum("bman,npq,nm->bmapq", mask, pair, 0.5 * zeta)
        g = torch.zeros_like(phi)
        acc = torch.einsum("bmapq,apqx->bmx", w, rows)
        for s in range(2):
            for m in range(N):
                if bool(mask[s, m].any()):
                    c = x["ham"][1][:, m]
                    g += _ladder(_ladder(acc[s, m], c, s, False), c, s, True)
        g += torch.einsum("pq,sq,sqpx->x", t, kin.double(), rows)
    (g @ _dense(sites)).backward()
    return {"value": float(e), "t": t.grad, "chi": chi.grad, "zeta": zeta.grad, "psi": [a.grad for a in sites]}


def exact(case, seed):
    """What run() returns, in 64 bits."""
    x, call, L = _inputs(case, seed), case["call"], case["L"]
    f64, dt = case["path"] == "fp64", DTYPE[case["path"]]
    given = lambda p: _dev([a.double().cpu().numpy() for a in _dev(p, dt)])  # noqa: E731 (as stored by the path)
    host = lambda p: [a.cpu().numpy() for a in given(p)]  # noqa: E731
    if call == "batched":
        out = []
        for l, ham, psi in zip(x["Ls"], x["hams"], x["psis"]):
            sector, terms = _sector(l, l // 2, l - l // 2), 4 * l * l + 2 * l
            out.append(_ci(_dev(_np_apply(psi, ham, case["D"], terms, False)), sector) if f64
                       else _apply_dense(_dense(given(psi)), ham, terms)[sector])
        return out
    if call == "inner":
        return float(_dense(given(x["phi"])) @ _dense(given(x["psi"])))
    if call == "grad":
        x["psi"], x["phi"] = host(x["psi"]), host(x["phi"])
        return _grad_exact(x, case["terms"])
    sector = _sector(L, *_out_sector(case))
    if call == "compress":
        return _ci(_dev(_np_compress(host(x["psi"]), case["D_max"], case["tol"])), sector)
    if call == "layer":
        if f64:
            return _ci(_dev(_np_layer(host(x["psi"]), x["coef"], case["sigma"], bool(case["dagger"]), case["D_max"])),
                       sector)
        return _ladder(_dense(given(x["psi"])), x["coef"], case["sigma"], bool(case["dagger"]))[sector]
    if call == "add":
        if f64:
            return _ci(_dev(_np_sum([[*p[:-1], p[-1] * c] for p, c in zip(x["xs"], x["coef"])], case["D_max"])), sector)
        return sum(c * _dense(given(p)) for p, c in zip(x["xs"], x["coef"]))[sector]
    if call == "apply":
        if f64:
            return _ci(_dev(_np_apply(x["psi"], x["ham"], case["D"], case["terms"], case["merge"])), sector)
        return _apply_dense(_dense(given(x["psi"])), x["ham"], case["terms"])[sector]
    v = _dense(given(x["psi"]))
    V, h = _krylov(v, x["ham"], case["K"])
    lam, y = np.linalg.eigh(h)
    if call == "lanczos":
        g = torch.from_numpy(y[:, 0]).cuda() @ V
        g = (g * torch.sign(g @ v))[sector]
        return {"energy": float(lam[0]), "ritz": lam, "ground": g}
    a = (y * np.exp(-0.05j * lam)) @ y[0]
    out = torch.from_numpy(a).cuda() @ V.to(torch.complex128)
    return {"state": (out * float(v.norm()) / out.norm())[sector]}
