"""The Poisson solve (multigrid cycle in pairs of floats, two columns a
thread) at the edges of its blocks: column counts around the 64 pairs of a
CTA, interior counts from the smallest that takes the cycle, two to four
levels.  Tolerance: each entry of P within FP32 rounding of the oracle's
value plus 1e-12, as the solve promises."""
import numpy as np
import pytest

from oracle.poisson import PoissonOracle
from synthetic import workloads
from synthetic.meshes import disk_rings
from tests._gpu import ctx_and_lib, load

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

MESHES = {
    "grid17": lambda: workloads.small_grid(17, 0, T=1, S=1).mesh,          # m = 256, k = 68
    "grid31": lambda: workloads.small_grid(31, 0, T=1, S=1).mesh,          # k = 124
    "grid33": lambda: workloads.small_grid(33, 0, T=1, S=1).mesh,          # k = 132
    "disk7x129": lambda: disk_rings(7, 129),                               # k = 129, a centre of 129 triangles
    "grid60": lambda: workloads.small_grid(60, 3, T=1, S=1, seed=60).mesh,
}


@pytest.mark.parametrize("name", list(MESHES))
def test_poisson_kernel_sizes(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dd, ctx = ctx_and_lib()
    try:
        mesh = MESHES[name]()
        mid = load(dd, ctx, mesh)
        iters, resid = dd.dd_poisson_kernel(ctx, mid, 1e-15, 20000)
        P = PoissonOracle(mesh.xy, mesh.tri, mesh.loops).full()
        out = torch.empty(P.shape, dtype=torch.float32, device="cuda")
        dd.dd_get_poisson_kernel(ctx, mid, out)
        dd.dd_sync(ctx)
        got = out.cpu().numpy().astype(np.float64)
        assert resid <= 1e-15 and iters <= 64
        assert np.all(np.abs(got - P) <= 2.0 ** -24 * P * 1.001 + 1e-12)
    finally:
        dd.dd_destroy(ctx)
