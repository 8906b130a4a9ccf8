"""The tensor-core KL where it replaces the exact form's recompute of the FP32
tile (0.07 to 0.25): no further from 64 bits than that recompute is (8e-8 to
1.6e-7 in the root mean square on these kernels).

The hardest kernels are target rows of equal entries: what the three slices of
their log2 P leave does not average out over a row.  The logs are sliced less a
whole number in the middle of their chunk's, so below 1/2 in magnitude, and the
slices leave at most 2^-28 of them, ln2 * 2^-28 = 2.6e-9 of the KL and 3.7e-8 of
0.07; the chunk of the one larger entry (below 8 from the middle, a tenth to a
sixth of a row's sum) leaves 2^-24 of a sixth, 6.9e-9 and 9.8e-8 at the most,
uniform and so 5.7e-8 in the root mean square at 0.07 and 2.7e-8 at 0.15, about
where the values lie.  The last three roundings add 2^-24 / sqrt(3) = 3.5e-8 at
the most.  Together about 5e-8; the test allows 8e-8."""
import numpy as np
import pytest

from synthetic import workloads
from tests._gpu import ctx_and_lib, load

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N", [66, 100])      # 398 and 606 columns: the chunks' sums fit the last chunk's rest, or in part
@pytest.mark.parametrize("T", [7, 40, 130])
def test_error_against_64_bits(N, T):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dd, ctx = ctx_and_lib()
    try:
        mesh = workloads.small_grid(N, 4 if N == 66 else 5, T=1, S=0, seed=66).mesh
        mid = load(dd, ctx, mesh)
        info = dd.dd_mesh_info(ctx, mid)
        n, k = info["n_v"], info["k"]
        assert n * info["k_pad"] >= 1 << 20
        rng = np.random.default_rng(N + T)
        targets = rng.choice(np.nonzero(~mesh.boundary_flags())[0], T, replace=False).astype(np.int32)
        P = np.exp(rng.uniform(0.3, 0.6, n)[:, None] * rng.standard_normal((n, k)))
        P /= P.sum(1, keepdims=True)
        eps = rng.uniform(0.0, 0.1, T)
        P[targets] = ((1 - eps) / k)[:, None]
        P[targets, 0] += eps
        dd.dd_set_poisson_kernel(ctx, mid, P)
        P = P.astype(np.float32).astype(np.float64)
        out = torch.full((1, T, n), float("nan"), dtype=torch.float32, device="cuda")
        dd.dd_distance(ctx, mid, targets, dd.DD_F_KL, dd.DD_PREC_FP32, out)
        dd.dd_sync(ctx)
        got = out[0].cpu().numpy().astype(np.float64)
        L = np.log(P)
        ref = (P * L).sum(1)[None] - L[targets] @ P.T
        rel = (got / np.where(ref > 0, ref, 1.0) - 1.0)[(ref > 0.07) & (ref < 0.25)]
        assert len(rel) > 1000
        assert np.sqrt((rel * rel).mean()) <= 8e-8
    finally:
        dd.dd_destroy(ctx)


@pytest.mark.parametrize("k", [4300, 4352])       # 68 chunks: their sums take two more, one shared with P's columns or none
@pytest.mark.parametrize("T", [3, 70])
def test_more_chunks_than_one_holds_sums_of(k, T):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from synthetic.meshes import disk_rings
    dd, ctx = ctx_and_lib()
    try:
        mid = load(dd, ctx, disk_rings(1, k))         # one interior vertex
        n = k + 1
        rng = np.random.default_rng(k)
        P = np.exp(rng.uniform(0.3, 0.6, n)[:, None] * rng.standard_normal((n, k)))
        P[0] = 1.0
        P /= P.sum(1, keepdims=True)
        dd.dd_set_poisson_kernel(ctx, mid, P)
        P = P.astype(np.float32).astype(np.float64)
        out = torch.full((1, T, n), float("nan"), dtype=torch.float32, device="cuda")
        dd.dd_distance(ctx, mid, np.zeros(T, np.int32), dd.DD_F_KL, dd.DD_PREC_FP32, out)
        dd.dd_sync(ctx)
        got = out[0].cpu().numpy().astype(np.float64)
        L = np.log(P)
        ref = (P * L).sum(1) - P @ L[0]
        assert np.array_equal(got, np.broadcast_to(got[0], got.shape)) and got[0, 0] == 0.0
        rel = (got[0] / np.where(ref > 0, ref, 1.0) - 1.0)[(ref > 0.07) & (ref < 0.25)]
        assert len(rel) > 1000 and np.sqrt((rel * rel).mean()) <= 8e-8
    finally:
        dd.dd_destroy(ctx)
