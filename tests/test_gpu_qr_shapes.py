"""The QR kernel's launch shapes: a compression that truncates nothing returns
the same state, at bonds on both sides of the rows every shape covers (m = 4 D
rows of X^T; float32 256 / 512 / 1024, float64 and complex64 128 / 256 / 512,
complex128 64 / 128 / 256), odd bonds and the smallest ones.  Bounds: those of
the untruncated layer tests (2e-6 in 32 bits, 1e-12 in 64 bits: a chain of
orthogonal factors, each off by a few roundings of its norm)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2409_12708_gb300.workloads import random_mps  # noqa: E402

CASES = [("fp32", torch.float32, D) for D in (1, 5, 16, 63, 64, 65, 127, 129, 255, 257)] \
    + [("fp64", torch.float64, D) for D in (7, 32, 33, 65, 129)] \
    + [("fp32", torch.complex64, D) for D in (5, 31, 33, 65)] \
    + [("fp64", torch.complex128, D) for D in (15, 17, 33, 65)]


def dense(sites):
    half = len(sites) // 2
    up = torch.complex128 if sites[0].is_complex() else torch.float64
    left = sites[0].to(up).reshape(4, -1)
    for a in sites[1:half]:
        left = (left @ a.to(up).reshape(a.shape[0], -1)).reshape(-1, a.shape[2])
    right = sites[-1].to(up).reshape(-1, 4)
    for a in reversed(sites[half:-1]):
        right = (a.to(up).reshape(-1, a.shape[2]) @ right).reshape(a.shape[0], -1)
    return (left @ right).reshape(-1)


@pytest.mark.parametrize("path,dtype,D", CASES)
def test_untruncated_compression_keeps_the_state(path, dtype, D):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_12708_gb300 import binding as B
    L = 10 if D > 64 else 8
    psi = random_mps(L, D, seed=D)
    if dtype.is_complex:
        psi = [a + 1j * b for a, b in zip(psi, random_mps(L, D, seed=1000 + D))]
    psi = [torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype) for a in psi]
    out = B.thc_compress(psi, D_max=min(2 * D, 512 if not dtype.is_complex else 256), path=path)
    want = dense(psi)
    tol = 2e-6 if path == "fp32" else 1e-12
    assert ((dense(out) - want).norm() <= tol * want.norm()).item()
