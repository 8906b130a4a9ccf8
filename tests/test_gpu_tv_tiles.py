"""The pipelined TV pass in every tile its launch rule chooses (152 SMs): 128, 64
or 32 rows by 64 targets, and a last target tile of at most 32 or 16 targets in
a launch of its own, the first or a later tile.  Vertex counts are chosen so that
the rule takes each; rows and targets are ragged.  The sums are the staged
shapes' bit for bit, and one field is the oracle's (1e-5 relative)."""
import numpy as np
import pytest

from oracle.divergence import tv_field
from synthetic.meshes import disk_rings
from tests._gpu import TOL_FP32, ctx_and_lib, field_error, load

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SEGS = 70
CASES = [                    # rings, T, launches
    (82, 333, 2),            # 64 x 64, 128 x 16 at tile 5
    (98, 333, 2),            # 128 x 64, 128 x 16
    (82, 3, 1),              # 128 x 16 alone
    (175, 90, 2),            # 32 x 64, 128 x 32
    (141, 17, 1),            # 128 x 32 alone
    (303, 150, 2),           # 32 x 64, 256 x 32 at tile 2
    (383, 150, 2),           # 128 x 64, 256 x 32
    (279, 17, 1),            # 256 x 32 alone
    (835, 70, 2),            # 32 x 64, 512 x 16 at tile 1
    (835, 136, 2),           # 64 x 64, 512 x 16
    (835, 3, 1),             # 512 x 16 alone
]


@pytest.mark.parametrize("rings,T,launches", CASES)
def test_tiles_have_the_staged_sums(monkeypatch, rings, T, launches):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dd, ctx = ctx_and_lib()
    try:
        mesh = disk_rings(rings, SEGS)
        n = mesh.n_v
        mid = load(dd, ctx, mesh)
        P = np.random.default_rng(rings).random((n, SEGS)) ** 4
        P /= P.sum(1, keepdims=True)
        dd.dd_set_poisson_kernel(ctx, mid, P)
        inner = np.nonzero(~mesh.boundary_flags())[0]
        targets = inner[(np.arange(T) * 911 + 5) % len(inner)].astype(np.int32)
        got = []
        for shape in ("0", "3"):
            monkeypatch.setenv("DD_TILE_SHAPE", shape)
            out = torch.full((1, T, n), float("nan"), dtype=torch.float32, device="cuda")
            dd.dd_kernel_timing(ctx, 1)
            dd.dd_distance(ctx, mid, targets, dd.DD_F_TV, dd.DD_PREC_FP32, out)
            dd.dd_sync(ctx)
            marks = dd.dd_kernel_timing(ctx, 0)
            got.append(out[0])
        assert torch.equal(got[0], got[1])
        if torch.cuda.get_device_properties(0).multi_processor_count == 152:
            assert marks["field_tile_kernel"][0] == launches
        a = T - 1
        assert field_error(got[1][a].cpu().numpy(), tv_field(P, P[targets[a]])) <= TOL_FP32
    finally:
        dd.dd_destroy(ctx)
