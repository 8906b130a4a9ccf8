"""The multigrid-preconditioned solve on grid maps that are not axis-parallel
(host check, no GPU): a corner's column meets the interior by a weight that is
rounding noise, 1e-18 .. 1e-15, and has to converge relative to that size as
the others do (the V-cycle takes its residual in pairs of floats)."""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

from oracle.laplacian import cotan_laplacian
from oracle.topology import split_boundary
from synthetic import workloads


@pytest.fixture(scope="module")
def dd():
    from paper_1708_02845_gb300.build import build
    build()
    from paper_1708_02845_gb300 import dd as mod
    return mod


@pytest.mark.parametrize("N", [24, 60])
@pytest.mark.parametrize("radians", [0.3, 0.7, 1.1])
def test_columns_of_rounding_noise(dd, N, radians):
    mesh = workloads.small_grid(N, 0, T=1, S=0).mesh
    c, s = np.cos(radians), np.sin(radians)
    L = cotan_laplacian(mesh.xy @ np.array([[c, s], [-s, c]]), mesh.tri).tocsr()
    B, I = split_boundary(mesh.n_v, mesh.tri, mesh.loops)
    A = (-L[I][:, I]).tocsr()
    A.sort_indices()
    rhs = L[I][:, B].toarray()
    norms = np.linalg.norm(rhs, axis=0)
    tiny = np.nonzero((norms > 0) & (norms < 1e-13))[0]
    assert len(tiny)
    lu = spla.splu(A.tocsc())
    for j in list(tiny) + [int(norms.argmax())]:
        b = rhs[:, j]
        x, it, _ = dd.dd_multigrid_check(A.indptr, A.indices, A.data, b, rtol=1e-14, max_iter=200)
        ref = lu.solve(b)
        assert it <= 40
        assert np.abs(x - ref).max() <= 1e-10 * np.abs(ref).max()
