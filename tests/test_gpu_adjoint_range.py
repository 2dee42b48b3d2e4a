"""The float32 adjoint's coefficient gradients are sums of float64 range and
precision: with phi scaled at the left end and psi at the right end by the same
factor, the blocks that are multiplied stay well inside float32 (1e-20 or 1e20)
and their products do not.  Against the float64 adjoint of the same values,
relative 1e-5 (the bound of the float32 adjoint test), at the inner sites: at the
two ends one block carries both factors and leaves float32 by itself."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2409_12708_gb300.workloads import sector_mps, thc_hamiltonian  # noqa: E402


@pytest.mark.parametrize("scale", [1e-20, 1e-12, 1.0, 1e12, 1e20])
def test_coefficient_gradients_of_scaled_states(scale):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_12708_gb300 import binding as B
    L, N, D = 6, 5, 16
    dev = lambda a, dt=torch.float32: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)  # noqa: E731
    ham = [dev(a).double() for a in thc_hamiltonian(L, N, seed=11)]
    phi = [dev(a) for a in sector_mps(L, 3, 3, D, seed=12)]
    psi = [dev(a) for a in sector_mps(L, 3, 3, D, seed=13)]
    phi[0] = phi[0] * scale
    psi[-1] = psi[-1] * scale
    r32 = B.thc_expect_grad(*ham, phi, psi, path="fp32")
    r64 = B.thc_expect_grad(*ham, [a.double() for a in phi], [a.double() for a in psi])
    for got, want in zip(r32[1:3], r64[1:3]):  # dt, dchi
        got, want = got[1:-1], want[1:-1]
        assert ((got - want).norm() <= 1e-5 * want.norm()).item()
