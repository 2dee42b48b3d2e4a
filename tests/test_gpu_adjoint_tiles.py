"""The float32 GEMM's tile shapes through the adjoint, whose products have every
pairing of a bond (rows) with a bond or four bonds (columns): bonds 4, 16, D at the
outer sites and up to D inside, at and beside the 32-, 64- and 128-wide tiles.
Against the float64 adjoint of the same float32 values, relative 1e-5: the bound
of the float32 adjoint test (sums of at most 4 D = 520 rounded products a site)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2409_12708_gb300.workloads import random_mps, thc_hamiltonian  # noqa: E402


@pytest.mark.parametrize("D", [33, 64, 65, 127, 128, 130])
def test_adjoint_at_tile_edges(D):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_12708_gb300 import binding as B
    L, N = 8, 3
    h32 = [torch.from_numpy(np.ascontiguousarray(a)).to("cuda", torch.float32).double()
           for a in thc_hamiltonian(L, N, seed=D)]
    psi = [torch.from_numpy(np.ascontiguousarray(a)).to("cuda", torch.float32) for a in random_mps(L, D, seed=D)]
    up = [a.double() for a in psi]
    r64 = B.thc_expect_grad(*h32, up, up)
    r32 = B.thc_expect_grad(*h32, psi, psi, path="fp32")
    rel = lambda a, b: ((a.double() - b).norm() / b.norm()).item()  # noqa: E731
    assert abs(r32[0] - r64[0]) <= 1e-5 * abs(r64[0])
    assert max(rel(a, b) for a, b in zip(list(r32[1:4]) + list(r32[4]), list(r64[1:4]) + list(r64[4]))) <= 1e-5
