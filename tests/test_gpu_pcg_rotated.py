"""The Poisson solve of grid maps that are not axis-parallel.  A corner of such
a map meets the interior by its cell's diagonal alone, whose weight is 0 in
exact arithmetic and rounding noise (1e-18 .. 1e-15) when the map is rotated:
a column whose right-hand side is that small has to converge like the others,
relative to its own size, in as many iterations.  Tolerance: each entry of P
within FP32 rounding of the oracle's value plus 1e-12, as the solve promises."""
import numpy as np
import pytest

from oracle.poisson import PoissonOracle
from synthetic import workloads
from tests._gpu import ctx_and_lib

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,n_obst", [(24, 0), (40, 0), (140, 5)])
@pytest.mark.parametrize("degrees", [17, 30, 64])
def test_rotated_grid(N, n_obst, degrees):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dd, ctx = ctx_and_lib()
    try:
        mesh = workloads.small_grid(N, n_obst, T=1, S=0).mesh
        c, s = np.cos(np.deg2rad(degrees)), np.sin(np.deg2rad(degrees))
        xy = np.ascontiguousarray(mesh.xy @ np.array([[c, s], [-s, c]]))
        idx, off = mesh.loop_arrays()
        mid = dd.dd_load_mesh(ctx, xy, mesh.tri, idx, off)
        iters, resid = dd.dd_poisson_kernel(ctx, mid, 1e-15, 200)
        P = PoissonOracle(xy, mesh.tri, mesh.loops).full()
        out = torch.empty(P.shape, dtype=torch.float32, device="cuda")
        dd.dd_get_poisson_kernel(ctx, mid, out)
        dd.dd_sync(ctx)
        got = out.cpu().numpy().astype(np.float64)
        assert resid <= 1e-15 and iters <= 64
        assert np.all(np.abs(got - P) <= 2.0 ** -24 * np.abs(P) * 1.001 + 1e-12)
    finally:
        dd.dd_destroy(ctx)
