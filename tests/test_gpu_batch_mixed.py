"""A batch of maps of both kinds -- KL from the tensor cores and from the FP32
tile (fewer than 2^20 entries of P, or row sums it does not cover) -- has the
fields of single calls, bit for bit: an item's result does not depend on the
other items' maps.  Paths of the batch are those of single calls too."""
import numpy as np
import pytest

from synthetic import workloads
from tests._gpu import ctx_and_lib, load

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dd, ctx = ctx_and_lib()
    meshes = [workloads.small_grid(66, 4, T=1, S=0, seed=66).mesh, workloads.small_grid(24, 2, T=1, S=0).mesh,
              workloads.small_grid(70, 2, T=1, S=0, seed=70).mesh]
    mids = [load(dd, ctx, m) for m in meshes]
    for mid in mids:
        dd.dd_poisson_kernel(ctx, mid, 1e-15, 20000)
    info = dd.dd_mesh_info(ctx, mids[2])            # the third: rows that sum to 1.5
    P = torch.empty((info["n_v"], info["k"]), dtype=torch.float32, device="cuda")
    dd.dd_get_poisson_kernel(ctx, mids[2], P)
    dd.dd_sync(ctx)
    dd.dd_set_poisson_kernel(ctx, mids[2], 1.5 * P.cpu().numpy())
    yield dd, ctx, meshes, mids
    dd.dd_destroy(ctx)


@pytest.mark.parametrize("mask", [1, 2, 3])
@pytest.mark.parametrize("order", [(0, 1, 0), (1, 0), (2, 1, 0, 1), (2, 0)])
def test_fields_of_single_calls(env, monkeypatch, mask, order):
    dd, ctx, meshes, mids = env
    Ts = [(70, 5, 64, 19)[j] for j in range(len(order))]
    inner = [np.nonzero(~meshes[i].boundary_flags())[0] for i in order]
    targets = [v[(np.arange(T) * 37 + 11) % len(v)].astype(np.int32) for v, T in zip(inner, Ts)]
    ref = []
    for i, t in zip(order, targets):
        out = torch.empty((bin(mask).count("1"), len(t), meshes[i].n_v), dtype=torch.float32, device="cuda")
        dd.dd_distance(ctx, mids[i], t, mask, dd.DD_PREC_FP32, out)
        ref.append(out.reshape(-1))
    ref = torch.cat(ref)
    for pipe in ("0", "1"):
        monkeypatch.setenv("DD_BATCH_PIPE", pipe)
        out = torch.full_like(ref, float("nan"))
        dd.dd_query_batch(ctx, [mids[i] for i in order], Ts, np.concatenate(targets), None, 0, mask, mask & -mask, 2,
                          out)
        dd.dd_sync(ctx)
        assert torch.equal(out, ref)


def test_paths_of_single_calls(env):
    dd, ctx, meshes, mids = env
    order, Ts, S, mp = (1, 0, 2), (6, 4, 3), 9, 600
    inner = [np.nonzero(~meshes[i].boundary_flags())[0] for i in order]
    targets = [v[(np.arange(T) * 53 + 7) % len(v)].astype(np.int32) for v, T in zip(inner, Ts)]
    sources = [v[(np.arange(T * S) * 29 + 3) % len(v)].astype(np.int32).reshape(T, S) for v, T in zip(inner, Ts)]

    def outputs(n):
        return (torch.zeros((n, mp, 2), dtype=torch.float32, device="cuda"),
                torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda"))

    def prefix(xy, ln):
        return torch.where(torch.arange(mp, device="cuda")[None, :, None] < ln[:, None, None], xy, 0)

    fields = torch.zeros(sum(T * meshes[i].n_v for i, T in zip(order, Ts)), device="cuda")
    xy, ln, st = outputs(sum(Ts) * S)
    dd.dd_query_batch(ctx, [mids[i] for i in order], Ts, np.concatenate(targets),
                      np.concatenate([s.reshape(-1) for s in sources]), S, 1, 1, mp, fields, xy, ln, st)
    dd.dd_sync(ctx)
    at = f0 = 0
    for i, t, s in zip(order, targets, sources):
        n = meshes[i].n_v
        f = fields[f0:f0 + len(t) * n].reshape(len(t), n)
        a, b, c = outputs(len(t) * S)
        dd.dd_trace_fields(ctx, mids[i], f, t, s, mp, a, b, c)
        dd.dd_sync(ctx)
        rows = slice(at, at + len(t) * S)
        assert torch.equal(ln[rows], b) and torch.equal(st[rows], c)
        assert torch.equal(prefix(xy[rows], ln[rows]), prefix(a, b))
        at += len(t) * S
        f0 += len(t) * n
