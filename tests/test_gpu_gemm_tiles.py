"""The small-tile GEMM through mps_inner, whose products take every tile size:
bonds at the edges of the 16- and 32-wide tiles, odd ones, 1, and beyond, real
and complex, against numpy.  Bound: a float64 sum of 4 D terms per entry and L
sites in either order, 1e-13 of the norms (float32 storage is exact input)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import mps as OM  # noqa: E402
from paper_2409_12708_gb300.workloads import random_mps  # noqa: E402


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.complex128, torch.complex64])
@pytest.mark.parametrize("Da,Db", [(1, 1), (3, 17), (15, 16), (16, 33), (31, 32), (33, 5), (40, 64)])
def test_inner_at_tile_edges(dtype, Da, Db):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_12708_gb300 import binding as B
    a, b = random_mps(7, Da, seed=Da), random_mps(7, Db, seed=100 + Db)
    if dtype.is_complex:
        a = [x + 1j * y for x, y in zip(a, random_mps(7, Da, seed=200 + Da))]
        b = [x + 1j * y for x, y in zip(b, random_mps(7, Db, seed=300 + Db))]
    a = [torch.from_numpy(np.ascontiguousarray(x)).to("cuda", dtype) for x in a]
    b = [torch.from_numpy(np.ascontiguousarray(x)).to("cuda", dtype) for x in b]
    up = lambda s: [x.to(torch.complex128 if dtype.is_complex else torch.float64).cpu().numpy() for x in s]  # noqa: E731
    na, nb = up(a), up(b)
    assert abs(B.mps_inner(a, b) - OM.inner(na, nb)) <= 1e-13 * OM.norm(na) * OM.norm(nb)
