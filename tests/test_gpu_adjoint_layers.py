"""The adjoint's transposed layers on one site block: an infinity reaches only the
entries that the ladder operators connect it to.  A zero coefficient has to leave
its entry alone (0 times infinity is a NaN).  Every single infinite entry of every
pair of operators, against the operators' matrices written out here (App. C)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from kernel_harness import compile_kernels, pointer  # noqa: E402

SOURCE = r"""
#include "engine.cuh"
#include "adjoint.cuh"
using namespace thc;
template <class T>
static int run(int B, const int* op, const T* coef, const T* Q, const T* X, T* P, T* Y, double* g) {
    const AdjTerms<T> tm{op, coef, 2, 1};
    k_adj_bwd<T, 2><<<dim3(1, B), 256>>>(1, 1, 16, Q, P, X, g, tm, 0);
    k_adj_fwd<T, 2><<<dim3(1, B), 256>>>(1, 1, 16, X, Y, tm, 0);
    return (int)cudaDeviceSynchronize();
}
extern "C" int layers_f32(int B, const int* op, const float* c, const float* Q, const float* X, float* P, float* Y,
                          double* g) { return run(B, op, c, Q, X, P, Y, g); }
extern "C" int layers_f64(int B, const int* op, const double* c, const double* Q, const double* X, double* P, double* Y,
                          double* g) { return run(B, op, c, Q, X, P, Y, g); }
"""

B_UP = np.zeros((4, 4))
B_UP[0, 2] = B_UP[1, 3] = 1.0
B_DN = np.zeros((4, 4))
B_DN[0, 1], B_DN[2, 3] = 1.0, -1.0
OPS = [B_UP, B_DN, B_UP.T, B_DN.T]
PAR = np.diag([1.0, -1.0, -1.0, 1.0])


def times(M, v):
    """M v where a zero entry of M adds nothing."""
    out = np.zeros(4)
    for i in range(4):
        for j in range(4):
            if M[i, j] != 0.0:
                out[i] += M[i, j] * v[j]
    return out


def forward(Z, ops, c):  # Z[w][n], bit l of w = layer l's bond
    for l in range(2):
        for w in range(4):
            if not w >> l & 1:
                Z[w | 1 << l] = Z[w | 1 << l] + c[l] * times(OPS[ops[l]], Z[w])
                Z[w] = times(PAR, Z[w])
    return Z


def backward(Z, ops, c):
    for l in (1, 0):
        for w in range(4):
            if not w >> l & 1:
                Z[w] = times(PAR, Z[w]) + c[l] * times(OPS[ops[l]].T, Z[w | 1 << l])
    return Z


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return compile_kernels(tmp_path_factory.mktemp("adjoint_layers"), SOURCE)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_an_infinity_stays_where_the_operators_take_it(lib, dtype):
    rng = np.random.default_rng(5)
    cases = [(o0, o1, e) for o0 in range(4) for o1 in range(4) for e in range(-1, 16)]
    n = len(cases)
    X, Q = rng.uniform(0.5, 1.5, (2, n, 4, 4))
    coef = rng.uniform(0.5, 1.5, (n, 2))
    for i, (_, _, e) in enumerate(cases):
        if e >= 0:
            X[i].flat[e] = Q[i].flat[e] = np.inf
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype)  # noqa: E731
    X, Q, coef = dev(X), dev(Q), dev(coef)
    Qk = Q.transpose(1, 2).contiguous()  # the kernel's order [n'][w']
    op = torch.tensor([c[:2] for c in cases], dtype=torch.int32, device="cuda")
    P, Y = torch.empty_like(X), torch.empty_like(X)
    g = torch.zeros(n, 2, dtype=torch.float64, device="cuda")
    f = lib.layers_f32 if dtype == torch.float32 else lib.layers_f64
    torch.cuda.synchronize()
    assert f(ctypes.c_int(n), pointer(op), pointer(coef), pointer(Qk), pointer(X), pointer(P), pointer(Y), pointer(g)) == 0
    Xn, Qn, cn = (t.double().cpu().numpy() for t in (X, Q, coef))
    for i, (o0, o1, _) in enumerate(cases):
        with np.errstate(invalid="ignore"):
            want = (backward(Qn[i].copy(), (o0, o1), cn[i]), forward(Xn[i].copy(), (o0, o1), cn[i]).T)
        for got, ref in zip((P[i], Y[i]), want):
            got = got.double().cpu().numpy().reshape(4, 4)
            # sums of at most four products of values below 2: 32 roundings of 2^4
            tol = 32 * 16 * (6e-8 if dtype == torch.float32 else 1.2e-16)
            assert (np.isfinite(got) == np.isfinite(ref)).all(), (cases[i], got, ref)
            assert np.abs(got - ref)[np.isfinite(ref)].max(initial=0.0) <= tol
