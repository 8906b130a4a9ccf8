"""Sparse fields of a map whose copy is large enough (2^22 kept entries) for KLT
to run beside KL and TV on a second stream: the same bits as with everything on
the caller's stream (its per-kernel timing on), as in calls of their own, and
with another context's timing on, for a context on a stream of its own."""
import numpy as np
import pytest

from synthetic import workloads
from tests._gpu import ctx_and_lib, load

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("T", [1, 3])
def test_klt_beside_kl_and_tv(T):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        dd, ctx = ctx_and_lib()
    other = dd.dd_create(0, torch.cuda.current_stream().cuda_stream)
    try:
        mesh = workloads.small_grid(170, 5, T=1, S=0, seed=170).mesh
        mid = load(dd, ctx, mesh)
        dd.dd_poisson_kernel(ctx, mid, 1e-15, 20000)
        kept, _ = dd.dd_sparsify(ctx, mid)
        assert kept >= 1 << 22
        n = mesh.n_v
        targets = np.nonzero(~mesh.boundary_flags())[0][[900, 7000, 20000][:T]].astype(np.int32)
        KL, TV, KLT = dd.DD_F_KL, dd.DD_F_TV, dd.DD_F_KLT

        def fields(mask):
            with torch.cuda.stream(stream):
                out = torch.full((bin(mask).count("1"), T, n), float("nan"), dtype=torch.float32, device="cuda")
                dd.dd_distance(ctx, mid, targets, mask, dd.DD_PREC_SPARSE, out)
            dd.dd_sync(ctx)
            return out.cpu()

        for _ in range(3):
            beside = fields(KL | TV | KLT)
        apart = torch.cat([fields(KL), fields(TV), fields(KLT)])
        assert torch.equal(beside, apart)
        assert torch.equal(fields(KL | KLT), apart[[0, 2]]) and torch.equal(fields(TV | KLT), apart[[1, 2]])
        dd.dd_kernel_timing(other, 1)
        assert torch.equal(fields(KL | TV | KLT), apart)
        dd.dd_kernel_timing(other, 0)
        dd.dd_kernel_timing(ctx, 1)
        assert torch.equal(fields(KL | TV | KLT), apart)
        dd.dd_kernel_timing(ctx, 0)
    finally:
        dd.dd_destroy(other)
        dd.dd_destroy(ctx)
