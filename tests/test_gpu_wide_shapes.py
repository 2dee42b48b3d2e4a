"""What the launch rules pick at large bonds: the 32-wide tiles of the 64-bit GEMM
(taken once 32 x 32 tiles alone give two CTAs a SM), through mps_inner at odd and
round bonds near 300, and the QR's launch shapes of 4, 8 and 16 warps a quad in
the complex types, through compressions that keep a complex state whole.

Bounds.  Inner product: as at the small tiles, 1e-13 of the norms (float64 sums of
at most 4 D terms an entry).  Compression: 2 L orthogonal factors, each off by
about 4 roundings of the state's norm: 8 L u, u = 2^-24 (1.2e-13 would be 8 L u at
twice the length in 64 bits; 1e-12 there, the bound of the other compressions)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2409_12708_gb300.workloads import random_mps  # noqa: E402


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_12708_gb300 import binding
    return binding


def on_gpu(sites, dtype):
    return [torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype) for a in sites]


def complex_mps(L, D, seed):
    parts = zip(random_mps(L, D, seed=seed), random_mps(L, D, seed=seed + 1000))
    return [(a + 1j * b) / np.sqrt(8.0 * a.shape[0]) for a, b in parts]  # norm of order one


def inner(a, b):
    E = torch.ones(1, 1, dtype=a[0].dtype, device="cuda")
    for x, y in zip(a, b):
        E = torch.einsum("anb,anc->bc", x.conj(), torch.einsum("ab,bnc->anc", E, y))
    return E[0, 0]


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.complex128, torch.complex64])
@pytest.mark.parametrize("Da,Db", [(320, 320), (289, 353), (511, 305)])
def test_inner_with_32_wide_tiles(B, dtype, Da, Db):
    L = 10
    make = complex_mps if dtype.is_complex else lambda L, D, seed: random_mps(L, D, seed=seed)  # noqa: E731
    a, b = on_gpu(make(L, Da, Da), dtype), on_gpu(make(L, Db, 7 * Db), dtype)
    # the largest product is Da x 4 Db: the rule's threshold is 304 tiles of 32
    assert -(-Da // 32) * -(-4 * Db // 32) >= 304
    up = torch.complex128 if dtype.is_complex else torch.float64
    na, nb = [x.to(up) for x in a], [x.to(up) for x in b]
    norms = (inner(na, na).real * inner(nb, nb).real).sqrt().item()
    assert abs(B.mps_inner(a, b) - inner(na, nb).item()) <= 1e-13 * norms


def dense(sites):
    half = len(sites) // 2
    left = sites[0].reshape(4, -1)
    for a in sites[1:half]:
        left = (left @ a.reshape(a.shape[0], -1)).reshape(-1, a.shape[2])
    right = sites[-1].reshape(-1, 4)
    for a in reversed(sites[half:-1]):
        right = (a.reshape(-1, a.shape[2]) @ right).reshape(a.shape[0], -1)
    return (left @ right).reshape(-1)


# rows m = 4 D of X^T: complex64 516 and 1028 (4 and 8 warps a quad), complex128 516 and
# 1028 (8 and 16); bond 257 is a state of rank 256 (D_max = 256 is the complex types'
# largest) in a basis of 257 vectors
@pytest.mark.parametrize("path,dtype", [("fp32", torch.complex64), ("fp64", torch.complex128)])
@pytest.mark.parametrize("L,D", [(10, 129), (12, 257)])
def test_complex_compression_at_wide_quads(B, path, dtype, L, D):
    rank = min(D, 256)
    psi = complex_mps(L, rank, D)
    rng = np.random.default_rng(D)
    if D > rank:
        for s in range(L - 1):
            if psi[s].shape[2] == rank and 4 ** min(s + 1, L - s - 1) > rank:
                G = np.linalg.qr(rng.standard_normal((D, rank)))[0]
                psi[s] = np.einsum("anb,cb->anc", psi[s], G)
                psi[s + 1] = np.einsum("cb,bnd->cnd", G, psi[s + 1])
    assert max(a.shape[0] for a in psi) == D and sum(a.shape[0] == D for a in psi) >= 2
    psi = on_gpu(psi, dtype)
    out = B.thc_compress(psi, D_max=rank if D > rank else 2 * D - 2, path=path)
    up = torch.complex128
    want, got = dense([a.to(up) for a in psi]), dense([a.to(up) for a in out])
    tol = 8 * L * 2.0 ** -24 if path == "fp32" else 1e-12
    assert ((got - want).norm() <= tol * want.norm()).item()
