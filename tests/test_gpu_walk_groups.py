"""The walk with a warp, four lanes and one lane a path (chosen by the number
of paths), with and without stored vertex decisions: the same paths bit for
bit, on a disk whose centre has a fan of 128 triangles (sources at and around
it, targets beside it) and on a grid with obstacles (boundary sources too)."""
import numpy as np
import pytest

from synthetic import workloads
from tests._gpu import ctx_and_lib, load

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("name", ["disk", "grid24"])
def test_groups_give_the_same_paths(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dd, ctx = ctx_and_lib()
    try:
        wl = workloads.disk() if name == "disk" else workloads.small_grid(24, 2, T=5, S=8)
        n, mp = wl.mesh.n_v, 512
        mid = load(dd, ctx, wl.mesh)
        dd.dd_poisson_kernel(ctx, mid, 1e-15, 20000)
        inner = np.nonzero(~wl.mesh.boundary_flags())[0].astype(np.int32)
        targets = inner[[1, len(inner) // 3, len(inner) - 2]]
        T = len(targets)
        f = torch.empty((1, T, n), dtype=torch.float32, device="cuda")
        dd.dd_distance(ctx, mid, targets, dd.DD_F_KL, dd.DD_PREC_FP32, f)

        def paths(S, sources):
            xy = torch.zeros((T * S, mp, 2), dtype=torch.float32, device="cuda")
            ln = torch.zeros(T * S, dtype=torch.int32, device="cuda")
            st = torch.zeros(T * S, dtype=torch.int32, device="cuda")
            dd.dd_trace_fields(ctx, mid, f[0], targets, sources, mp, xy, ln, st)
            dd.dd_sync(ctx)
            xy = torch.where(torch.arange(mp, device="cuda")[None, :, None] < ln[:, None, None], xy, 0)
            return xy.reshape(T, S, mp, 2), ln.reshape(T, S), st.reshape(T, S)

        # 811 paths a target: four lanes a path (2,433 in all); 810 and below: a warp each
        base = np.resize(np.arange(n, dtype=np.int32), 811)
        src = np.tile(base, (T, 1))
        four = paths(811, src)
        parts = [paths(len(c), np.tile(c, (T, 1))) for c in np.array_split(base, 2)]
        for got, ref in zip(four, zip(*parts)):
            assert torch.equal(got, torch.cat(ref, 1))
        few = paths(100, src[:, :100])                      # no stored decisions, a warp each
        one = paths(811 * 16, np.tile(base, (T, 16)))       # one lane a path (38,928)
        for a in range(3):
            assert torch.equal(few[a], four[a][:, :100])
            assert torch.equal(one[a][:, :811], four[a]) and torch.equal(one[a][:, -811:], four[a])
    finally:
        dd.dd_destroy(ctx)
