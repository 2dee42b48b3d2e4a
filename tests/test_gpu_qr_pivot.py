"""Pivoting inside a panel of the QR: every step takes the column with the
largest remaining norm, also where the norms have fallen far below their value at
the start of the panel (graded spectra over more than eight decades, rank-deficient
matrices), whose order a metric that is only ever reduced by the rows found so far
no longer knows.  The remaining norms follow from the kernel's own R (reflectors
keep a column's norm to rounding).  Bound: the metric is measured again once it has
lost half the digits, so it is within 80 roundings over sqrt(eps) of the norm, 2 % in
32 bits; a taken column has at least 0.9 of the largest squared norm."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from kernel_harness import compile_kernels, pointer  # noqa: E402

# (scalar, panel width, warps per quad, chunks): one and several warps per quad
SHAPES = {"f32_1": ("float", 32, 1, 2), "f32_2": ("float", 32, 2, 4), "f32_8": ("float", 8, 8, 4),
          "f64_1": ("double", 32, 1, 2), "f64_2": ("double", 16, 2, 4), "f64_h": ("double", 16, 2, 2), "c64_1": ("cplx<float>", 32, 1, 2)}
SOURCE = r"""
#include "qr.cuh"
using namespace thc;
template <class T, int NB, int S, int NQ>
static int run(int B, int m, int n, void* A, void* R, int* order) {
    QRJob<T> job{};
    job.A = (T*)A;
    job.strideA = (long)m * n;
    job.m = job.ld = m;
    job.n = n;
    job.out = (T*)R;
    job.strideOut = (long)n * n;
    job.mode = QR_R_ROWS;
    job.colmap = order;
    const size_t smem = qr_smem_bytes<T>(QrShape{NB, S, NQ}, m, n, true);
    auto* k = k_qr<T, NB, S, NQ, true>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return -1;
    k<<<B, 32 * S * NB / QR_NC, smem>>>(job);
    return (int)cudaDeviceSynchronize();
}
""" + "".join('extern "C" int %s(int B, int m, int n, void* A, void* R, int* order) '
              "{ return run<%s, %d, %d, %d>(B, m, n, A, R, order); }\n" % (k, *v) for k, v in SHAPES.items())
DTYPE = {"f32": torch.float32, "f64": torch.float64, "c64": torch.complex64}


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return compile_kernels(tmp_path_factory.mktemp("qr_pivot"), SOURCE)


def spectrum(kind, n, scalar):
    digits = 16 if scalar == "f64" else 7
    k = np.arange(n)
    if kind == "graded":  # over half as many decades again as the storage holds
        return 10.0 ** (-1.5 * digits * k / (n - 1))
    if kind == "deficient":  # a quarter of full rank, the rest rounding noise
        return np.where(k < n // 4, 1.0, 0.0)
    if kind == "step":  # two clusters, the lower one well above the noise
        return np.where(k < n // 4, 1.0, 10.0 ** (-0.7 * digits)) * 0.99 ** k
    return np.exp(-k / 8.0)


@pytest.mark.parametrize("kind", ["graded", "deficient", "step", "mild"])
@pytest.mark.parametrize("shape,m,n", [("f32_1", 64, 32), ("f32_1", 256, 47), ("f32_2", 512, 40), ("f32_8", 400, 24),
                                       ("f64_1", 128, 40), ("f64_2", 500, 70), ("f64_h", 256, 52), ("c64_1", 128, 32)])
def test_each_step_takes_the_largest_remaining_column(lib, kind, shape, m, n):
    scalar, nb, B = shape[:3], SHAPES[shape][1], 6
    rng = np.random.default_rng(m + n)
    cplx = scalar == "c64"
    draw = lambda *s: rng.standard_normal(s) + (1j * rng.standard_normal(s) if cplx else 0.0)  # noqa: E731
    mats = []
    for _ in range(B):
        U, W = np.linalg.qr(draw(m, n))[0], np.linalg.qr(draw(n, n))[0]
        mats.append((U * spectrum(kind, n, scalar)) @ W)
    # column-major matrices
    A0 = torch.from_numpy(np.stack([a.T.copy() for a in mats])).to("cuda", DTYPE[scalar])
    A, R = A0.clone(), torch.empty(B, n, n, dtype=DTYPE[scalar], device="cuda")
    order = torch.empty(B, n, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    f = getattr(lib, shape)
    assert f(ctypes.c_int(B), ctypes.c_int(m), ctypes.c_int(n), pointer(A), pointer(R), pointer(order)) == 0
    up = torch.complex128 if cplx else torch.float64
    R, P, order = R.to(up), A0.to(up), order.long()
    eps = 1.2e-16 if scalar == "f64" else 6e-8
    for b in range(B):
        assert sorted(order[b].tolist()) == list(range(n))
        C, r = P[b][order[b]], R[b]  # the matrix's columns (as rows) in the order taken
        # R^H R = C^H C: m products and 2 n reflectors, each a rounding of the norm
        gram = C.conj() @ C.T
        assert ((r.conj().T @ r - gram).abs().max() <= 8 * (n + np.sqrt(m)) * eps * gram.abs().max()).item()
        tail = torch.flip(torch.cumsum(torch.flip(r.abs() ** 2, [0]), 0), [0])  # [j, c]: norm^2 of column c below row j
        for j in range(n):
            end = min(n, j // nb * nb + nb)  # the panel's columns
            assert (tail[j, j] >= 0.9 * tail[j, j:end].max()).item(), (b, j, tail[j, j:end])


# Whole compressions of such states: Schmidt values exp(-k / decay), over 1e8 within a
# panel at decay 1, and a state of rank 8 in bonds of 64.  Nothing is cut; the bounds are
# those of the other untruncated compressions.  An exhausted Jacobi budget is counted only.
@pytest.mark.parametrize("path,dtype,tol", [("fp32", torch.float32, 2e-6), ("fp64", torch.float64, 1e-12)])
@pytest.mark.parametrize("rank,decay", [(64, 1.0), (64, 3.0), (8, 8.0)])
def test_steep_and_deficient_states_compress(path, dtype, tol, rank, decay):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import mps as OM
    from paper_2409_12708_gb300 import binding as B
    from paper_2409_12708_gb300.workloads import sector_mps
    rng = np.random.default_rng(rank)
    psi = sector_mps(8, 4, 4, rank, seed=rank, decay=decay)
    for s in range(7):  # into bonds of 64
        have = psi[s].shape[2]
        want = min(64, 4 ** (s + 1), 4 ** (7 - s))
        if have < want:
            G = np.linalg.qr(rng.standard_normal((want, have)))[0]
            psi[s] = np.einsum("anb,cb->anc", psi[s], G)
            psi[s + 1] = np.einsum("cb,bnd->cnd", G, psi[s + 1])
    psi = [torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype) for a in psi]
    B.profile_read()
    out = B.thc_compress(psi, D_max=64, path=path)
    assert "jacobi_budget_exhausted" not in B.profile_read()
    want, got = (OM.to_dense([a.double().cpu().numpy() for a in s]) for s in (psi, out))
    assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)
