"""Paths on more fields than a launch grid has rows for (65,535 groups of four
at a vertex with a wide fan): the last fields' paths are those of a call with
these fields alone, bit for bit."""
import numpy as np
import pytest

from synthetic.meshes import disk_rings
from tests._gpu import ctx_and_lib, load

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_more_fields_than_grid_rows():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dd, ctx = ctx_and_lib()
    try:
        mesh = disk_rings(4, 32)                       # a centre of 32 triangles
        n, S, mp, few, T = mesh.n_v, 128, 8, 24, 4 * 65536 + 24
        mid = load(dd, ctx, mesh)
        dd.dd_poisson_kernel(ctx, mid, 1e-15, 20000)
        inner = np.nonzero(~mesh.boundary_flags())[0].astype(np.int32)
        targets = inner[np.arange(few) * 4 + 1]
        f = torch.empty((1, few, n), dtype=torch.float32, device="cuda")
        dd.dd_distance(ctx, mid, targets, dd.DD_F_KL, dd.DD_PREC_FP32, f)
        dd.dd_sync(ctx)
        sources = np.resize(np.arange(n, dtype=np.int32), S)      # the centre first

        def paths(reps):
            t = np.tile(targets, reps)
            xy = torch.zeros((len(t), S, mp, 2), dtype=torch.float32, device="cuda")
            ln = torch.zeros((len(t), S), dtype=torch.int32, device="cuda")
            st = torch.zeros((len(t), S), dtype=torch.int32, device="cuda")
            fields = f[0].repeat(reps, 1)
            dd.dd_trace_fields(ctx, mid, fields, t, np.tile(sources, (len(t), 1)), mp, xy, ln, st)
            dd.dd_sync(ctx)
            xy, ln = xy[-few:], ln[-few:]
            return torch.where(torch.arange(mp, device="cuda")[:, None] < ln[..., None, None], xy, 0), ln, st[-few:]

        for got, ref in zip(paths(T // few + 1), paths(5)):       # both with stored decisions
            assert torch.equal(got, ref)
    finally:
        dd.dd_destroy(ctx)
