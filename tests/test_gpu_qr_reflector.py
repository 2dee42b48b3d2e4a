"""The reflector's scalars (qr_scalars, qr_root, qr_recip: hardware reciprocal and
reciprocal square root in 32 bits, then Newton and Halley steps) against the
correctly rounded values, over the range the kernel sends to them, and whole
reflectors on both sides of the switches to the library's square root and
division (1e-30 in 32 bits, 2^-100 and 2^100 in 64 bits).

Bounds, u = 2^-24 or 2^-53.  sqrt(a2): its last step adds to a value right to a few
u a correction right to a few u, so one rounding of the result and one of the
residual: 2 u.  1 / sqrt(a2): one step less, 4 u.  d = |x| + sqrt(a2): 2 u + u.
1 / d: 3 u from d and 2 u of its own step, 5 u.  d / sqrt(a2): 3 u + 2 u from its
two arguments and 2 u of its own step, 7 u.  1 / d alone: 2 u."""
import ctypes
from fractions import Fraction as Fr  # exact arithmetic: no host type is wide enough

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from kernel_harness import compile_kernels, pointer  # noqa: E402

SOURCE = r"""
#include "qr.cuh"
using namespace thc;
template <class T>
__global__ void scalars(int n, const T* a2, const T* ax, T* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    qr_scalars(a2[i], ax[i], out[i], out[n + i], out[2 * n + i]);
    if constexpr (sizeof(T) == 8) {
        out[3 * n + i] = qr_root(a2[i], out[4 * n + i]);
        out[5 * n + i] = qr_recip(a2[i]);
    }
}
extern "C" int scalars_f32(int n, const float* a2, const float* ax, float* out) {
    scalars<<<(n + 255) / 256, 256>>>(n, a2, ax, out);
    return (int)cudaDeviceSynchronize();
}
extern "C" int scalars_f64(int n, const double* a2, const double* ax, double* out) {
    scalars<<<(n + 255) / 256, 256>>>(n, a2, ax, out);
    return (int)cudaDeviceSynchronize();
}
template <class T>
static int column(int B, int m, void* A, void* L, void* Tw) {  // B matrices of one column
    QRJob<T> job{};
    job.A = (T*)A;
    job.strideA = job.m = job.ld = m;
    job.n = 1;
    job.Tw = (T*)Tw;
    job.strideT = 32 * 32;
    job.out = (T*)L;
    job.strideOut = 1;
    job.mode = QR_L_AND_Q;
    const size_t smem = qr_smem_bytes<T>(QrShape{32, 1, 2}, m, 1, false);
    auto* k = k_qr<T, 32, 1, 2, false>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return -1;
    k<<<B, 256, smem>>>(job);
    return (int)cudaDeviceSynchronize();
}
extern "C" int column_f32(int B, int m, void* A, void* L, void* Tw) { return column<float>(B, m, A, L, Tw); }
extern "C" int column_f64(int B, int m, void* A, void* L, void* Tw) { return column<double>(B, m, A, L, Tw); }
extern "C" int column_c64(int B, int m, void* A, void* L, void* Tw) { return column<cplx<float>>(B, m, A, L, Tw); }
extern "C" int column_c128(int B, int m, void* A, void* L, void* Tw) { return column<cplx<double>>(B, m, A, L, Tw); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return compile_kernels(tmp_path_factory.mktemp("qr_reflector"), SOURCE)


@pytest.mark.parametrize("dtype,lo,hi", [(torch.float32, 1e-30, 3e38), (torch.float64, 2.0 ** -100, 2.0 ** 100)])
def test_scalars_against_exact_values(lib, dtype, lo, hi):
    rng = np.random.default_rng(3)
    n = 20000
    a2 = np.exp(rng.uniform(np.log(lo), np.log(hi), n))
    a2[:4] = lo, hi, 1.0, np.nextafter(1.0, 2.0)
    ax = np.sqrt(a2) * np.where(rng.random(n) < 0.2, 1.0 - 1e-7 * rng.random(n), 10.0 ** rng.uniform(-12, 0, n))
    ax[4:8] = 0.0
    a2, ax = (torch.from_numpy(v).to(dtype) for v in (a2, ax))
    out = torch.zeros(6, n, dtype=dtype, device="cuda")
    a2d, axd = a2.cuda(), ax.cuda()
    f = lib.scalars_f32 if dtype == torch.float32 else lib.scalars_f64
    torch.cuda.synchronize()
    assert f(ctypes.c_int(n), pointer(a2d), pointer(axd), pointer(out)) == 0
    u = 2.0 ** -24 if dtype == torch.float32 else 2.0 ** -53
    o = out.cpu().double().numpy()
    a2, ax = a2.double().numpy(), ax.double().numpy()
    worst = np.zeros(6)
    for i in range(0, n, 1 if dtype == torch.float32 else 4):
        A, x, s = Fr(a2[i]), Fr(ax[i]), Fr(np.sqrt(a2[i]))
        s = (s + A / s) / 2  # one Newton step from the correctly rounded root: exact to u^2
        d = x + s
        want = [s, d / s, 1 / d, s, 1 / s, 1 / A]
        for k in range(3 if dtype == torch.float32 else 6):
            worst[k] = max(worst[k], abs(float((Fr(o[k, i]) - want[k]) / want[k])))
    print("worst in units of u:", worst / u)
    assert (worst <= np.array([2, 7, 5, 2, 4, 2]) * u).all()


@pytest.mark.parametrize("name,dtype", [("f32", torch.float32), ("f64", torch.float64), ("c64", torch.complex64),
                                        ("c128", torch.complex128)])
def test_reflectors_across_the_switches(lib, name, dtype):
    m = 64
    wide = dtype in (torch.float64, torch.complex128)
    edges = (2.0 ** -100, 2.0 ** 100) if wide else (1e-30,)
    # squared norms from far below to far above each switch, and just beside it
    sq = np.concatenate([np.geomspace(1e-250 if wide else 1e-44, 1e250 if wide else 1e34, 61)]
                        + [e * np.array([0.5, 0.999, 1.0, 1.001, 2.0, 8.0]) for e in edges])
    # the part below the diagonal relative to the diagonal entry
    ratio = np.array([1e-6, 1e-3, 1.0, 1e3, 1e6, np.inf])
    B = sq.size * ratio.size
    rng = np.random.default_rng(9)
    a = rng.standard_normal((B, m)) + (1j * rng.standard_normal((B, m)) if dtype.is_complex else 0.0)
    below = np.linalg.norm(a[:, 1:], axis=1)
    r = np.tile(ratio, sq.size)
    a[:, 1:] *= np.where(np.isinf(r), 1.0, r)[:, None] / below[:, None]
    a[:, 0] = np.where(np.isinf(r), 0.0, a[:, 0] / np.abs(a[:, 0]))
    a *= (np.sqrt(np.repeat(sq, ratio.size)) / np.linalg.norm(a, axis=1))[:, None]
    A0 = torch.from_numpy(a).to(dtype).cuda()
    A, Lo = A0.clone(), torch.zeros(B, dtype=dtype, device="cuda")
    Tw = torch.zeros(B, 32 * 32, dtype=dtype, device="cuda")
    torch.cuda.synchronize()
    assert getattr(lib, "column_" + name)(ctypes.c_int(B), ctypes.c_int(m), pointer(A), pointer(Lo), pointer(Tw)) == 0
    up = torch.complex128 if dtype.is_complex else torch.float64
    x, q, l = A0.to(up), A.to(up), Lo.to(up)  # x = q l
    u = 2.0 ** -53 if wide else 2.0 ** -24
    scale = x.abs().max(dim=1, keepdim=True).values  # squares stay in range
    x, l = x / scale, l / scale[:, 0]
    norm = torch.linalg.vector_norm(x, dim=1)
    # |l| = |x|: 64 squares (exact to u^2 in 32 bits, 64 u / sqrt(64) in 64 bits), 2 u of the
    # root, one rounding each of the sum and the store; entries below 1e-38 have fewer bits
    fine = (scale[:, 0] > 1e-30) | wide
    assert (((l.abs() - norm).abs() / norm)[fine].max() <= 16 * u).item()
    # q = e_1 - tau conj(v_1) v: tau to 7 u, v to 6 u, the products to 2 u
    assert ((torch.linalg.vector_norm(q, dim=1) - 1.0).abs()[fine].max() <= 32 * u).item()
    assert (torch.linalg.vector_norm(x - q * l[:, None], dim=1)[fine] <= 48 * u * norm[fine]).all().item()
