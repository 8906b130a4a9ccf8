"""The tensor-core KL of many targets (maps from 2^20 entries of P on) against
the FP64 oracle at the edges of its tiles, and its routes: KL alone and with
TV, a batch of maps, and a P whose rows it does not cover (their sums exceed
1.01), which keeps the FP32 tile kernels.

Tolerance: the FP32 path's 1e-5 relative.  The kernel's own bound is far
inside it: slices to 2^-33 of a chunk's largest entry times its largest log,
below 1e-7 absolute over 64 columns, against 7e-7 at its exact-recompute
threshold of 0.07.
"""
import numpy as np
import pytest

from oracle.divergence import kl_field_fast, tv_field
from oracle.poisson import PoissonOracle
from synthetic import workloads
from tests._gpu import TOL_FP32, ctx_and_lib, field_error, load

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dd, ctx = ctx_and_lib()
    wl = workloads.small_grid(66, 4, T=4, S=1, seed=66)
    mesh = wl.mesh
    po = PoissonOracle(mesh.xy, mesh.tri, mesh.loops)
    P = po.full()
    assert P.size >= 1 << 20 and mesh.n_v % 128 and P.shape[1] % 64
    mid = load(dd, ctx, mesh)
    dd.dd_set_poisson_kernel(ctx, mid, P)
    yield dd, ctx, mesh, po, P, mid
    dd.dd_destroy(ctx)


def targets_of(po, T):
    return [int(po.I[(i * 7919 + 13) % po.m]) for i in range(T)]


def fields(dd, ctx, mid, n_v, targets, mask):
    out = torch.full((2 if mask == 3 else 1, len(targets), n_v), float("nan"), dtype=torch.float32, device="cuda")
    dd.dd_distance(ctx, mid, targets, mask, dd.DD_PREC_FP32, out)
    dd.dd_sync(ctx)
    return out.cpu().numpy()


@pytest.mark.parametrize("T", [3, 16, 17, 64, 65, 128, 130])
def test_tile_edges(env, T):
    dd, ctx, mesh, po, P, mid = env
    targets = targets_of(po, T)
    both = fields(dd, ctx, mid, mesh.n_v, targets, dd.DD_F_KL | dd.DD_F_TV)
    alone = fields(dd, ctx, mid, mesh.n_v, targets, dd.DD_F_KL)
    assert np.array_equal(both[0], alone[0])
    for a in sorted({0, 1, 15, 16, 63, 64, 127, 128, T - 1} & set(range(T))):
        t = targets[a]
        assert field_error(both[0, a], kl_field_fast(P, P[t])) <= TOL_FP32
        assert field_error(both[1, a], tv_field(P, P[t])) <= TOL_FP32
        assert both[0, a, t] == 0.0 and both[1, a, t] == 0.0
    # a target's field does not depend on the tile and column it falls in (up to
    # 64 targets share one order of the small products, more another)
    few = targets[:3] if T <= 64 else targets[:65]
    single = fields(dd, ctx, mid, mesh.n_v, few, dd.DD_F_KL)
    assert np.array_equal(single[0], both[0, :len(few)])


def test_batch_has_the_fields_of_single_calls(env, monkeypatch):
    dd, ctx, mesh, po, P, mid = env
    Ts = [5, 70]
    targets = [targets_of(po, T) for T in Ts]
    n = mesh.n_v
    ref = np.concatenate([fields(dd, ctx, mid, n, t, 3).reshape(-1) for t in targets])
    for pipe in ("0", "1"):
        monkeypatch.setenv("DD_BATCH_PIPE", pipe)
        out = torch.full((sum(2 * T * n for T in Ts),), float("nan"), dtype=torch.float32, device="cuda")
        dd.dd_query_batch(ctx, [mid, mid], Ts, np.concatenate(targets).astype(np.int32), None, 0, 3, 1, 2, out)
        dd.dd_sync(ctx)
        assert np.array_equal(out.cpu().numpy(), ref)


@pytest.mark.parametrize("scale", [1.0, 1.5])
def test_replaced_kernel(env, scale):
    """A new P replaces the operands; rows that sum to 1.5 take the FP32 tile."""
    dd, ctx, mesh, po, P, mid = env
    P2 = np.ascontiguousarray(scale * 0.5 * (P + P[:, ::-1]))
    dd.dd_set_poisson_kernel(ctx, mid, P2)
    targets = targets_of(po, 20)
    out = fields(dd, ctx, mid, mesh.n_v, targets, 3)
    dd.dd_set_poisson_kernel(ctx, mid, P)
    for a in (0, 7, 19):
        assert field_error(out[0, a], kl_field_fast(P2, P2[targets[a]])) <= TOL_FP32
        assert field_error(out[1, a], tv_field(P2, P2[targets[a]])) <= TOL_FP32


@pytest.mark.parametrize("T", [7, 16, 17, 32, 33, 72, 96])
def test_tv_pass_of_narrow_last_tiles(env, monkeypatch, T):
    """The pipelined TV pass (every shape of its last target tile) has the
    staged shapes' sums bit for bit, alone and in a batch."""
    dd, ctx, mesh, po, P, mid = env
    targets = targets_of(po, T)
    ref = None
    for shape in ("0", "3"):
        monkeypatch.setenv("DD_TILE_SHAPE", shape)
        got = fields(dd, ctx, mid, mesh.n_v, targets, dd.DD_F_TV)[0]
        ref = got if ref is None else ref
        assert np.array_equal(got, ref)
    monkeypatch.delenv("DD_TILE_SHAPE")
    n = mesh.n_v
    both = fields(dd, ctx, mid, n, targets, 3)
    for pipe in ("0", "1"):
        monkeypatch.setenv("DD_BATCH_PIPE", pipe)
        out = torch.full((2 * (T + 64) * n,), float("nan"), dtype=torch.float32, device="cuda")
        dd.dd_query_batch(ctx, [mid, mid], [T, 64], np.concatenate([targets, targets_of(po, 64)]).astype(np.int32),
                          None, 0, 3, 1, 2, out)
        dd.dd_sync(ctx)
        assert np.array_equal(out[:2 * T * n].reshape(2, T, n).cpu().numpy(), both)
