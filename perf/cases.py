"""The work that users of the library have it do, as measurable cases.

A planner loads a map (a triangle mesh with obstacles), solves for its Poisson
kernel once, and then asks for divergence fields and paths, many times, for
targets that it has not asked for before.  The cases go through the public
entry points of ``paper_1708_02845_gb300.dd`` for one such request each:

  query    dd_query: one robot asks for a target's fields and the paths from
           its candidate sources (device or pinned host outputs)
  fields   dd_distance: the KL and / or TV fields of T targets (FP32, split
           BF16, or the sparse fields)
  diverge  dd_divergence: another f-divergence's field
  batch    dd_query_batch without paths: targets on several uneven maps
  paths    dd_trace_fields: paths on fields that the program already has
  poisson  dd_poisson_kernel: the solve for a new map

Maps are the unit square cut into N x N cells with rectangular obstacles (the
sizes of the configurations grid140, grid450 and batch64) or the unit disk;
a case's sizes fix its map, the seed draws targets and sources.
"""

import functools
import math
import random

import numpy as np
import torch

from paper_1708_02845_gb300 import dd

KL, TV, KLT = dd.DD_F_KL, dd.DD_F_TV, dd.DD_F_KLT
FLT_MIN = float(np.finfo(np.float32).tiny)


def listed():
    return [
        # the smallest call: one target and 32 paths on the 2,049-vertex disk; launches and latency count
        dict(name="query_disk", kind="query", rings=16, segs=128, T=1, S=32, host=False),
        # one robot's request on a room-sized map, results read back into the planner's pinned host buffers
        dict(name="query_room_host", kind="query", N=140, obst=8, T=1, S=256, host=True),
        # one target's KL and TV fields on the largest configured map: P is read once
        dict(name="field_one_large", kind="fields", N=450, obst=24, T=1, mask=KL | TV, prec=dd.DD_PREC_FP32),
        # a handful of targets, KL alone, odd sizes: more than the one-target pass takes, fewer than fill a tile
        dict(name="fields_few_kl", kind="fields", N=201, obst=5, T=7, mask=KL, prec=dd.DD_PREC_FP32),
        # the room-sized map's usual batch of 64 targets
        dict(name="fields_room", kind="fields", N=140, obst=8, T=64, mask=KL | TV, prec=dd.DD_PREC_FP32),
        # the largest: 1,024 targets on the largest configured map
        dict(name="fields_large", kind="fields", N=450, obst=24, T=1024, mask=KL | TV, prec=dd.DD_PREC_FP32),
        # the split-BF16 KL with FP32 TV, ragged target count
        dict(name="fields_bf16", kind="fields", N=300, obst=16, T=333, mask=KL | TV, prec=dd.DD_PREC_BF16X3),
        # the sparse fields (all three) of one target on a large map
        dict(name="fields_sparse", kind="fields", N=300, obst=16, T=1, mask=KL | TV | KLT, prec=dd.DD_PREC_SPARSE),
        # an alpha-divergence of two targets
        dict(name="alpha_two", kind="diverge", N=300, obst=16, T=2, family=dd.DD_DIV_ALPHA, param=0.5),
        # targets on twelve uneven maps in one call
        dict(name="batch_uneven", kind="batch", domains=12, n_lo=70, n_hi=170, t_lo=16, t_hi=256, draw=1),
        # 64 targets x 256 paths on ready-made fields (the walk and its decisions alone)
        dict(name="paths_many", kind="paths", rings=140, segs=512, T=64, S=256),
        # a new map: the solve for its Poisson kernel
        dict(name="poisson_room", kind="poisson", N=140, obst=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "fields", "fields", "fields", "diverge", "batch", "paths", "poisson"])
    if kind == "query":
        if rng.random() < 0.5:
            return dict(kind=kind, rings=rng.randint(9, 40), segs=rng.randint(64, 200), T=rng.randint(1, 2),
                        S=_log_int(rng, 1, 300), host=rng.random() < 0.5)
        return dict(kind=kind, N=rng.randint(40, 140), obst=rng.randint(0, 8), T=rng.randint(1, 2),
                    S=_log_int(rng, 1, 300), host=rng.random() < 0.5)
    if kind == "fields":
        N = _log_int(rng, 40, 300)
        prec = rng.choice([dd.DD_PREC_FP32, dd.DD_PREC_FP32, dd.DD_PREC_FP32, dd.DD_PREC_BF16X3, dd.DD_PREC_SPARSE])
        if prec == dd.DD_PREC_SPARSE:
            return dict(kind=kind, N=N, obst=rng.randint(1, 16), T=rng.randint(1, 4), mask=rng.randint(1, 7), prec=prec)
        mask = rng.choice([KL, TV, KL | TV, KL | TV, KL | TV])
        return dict(kind=kind, N=N, obst=rng.randint(0, 16) if N > 100 else rng.randint(0, 4), T=_log_int(rng, 1, 700),
                    mask=(mask | KL) if prec == dd.DD_PREC_BF16X3 else mask, prec=prec)
    if kind == "diverge":
        family, param = rng.choice([(dd.DD_DIV_CHI2, 0.0), (dd.DD_DIV_HELLINGER, 0.0), (dd.DD_DIV_POWER, 2.5),
                                    (dd.DD_DIV_ALPHA, 0.5), (dd.DD_DIV_ALPHA, -0.5), (dd.DD_DIV_KL_REVERSE, 0.0)])
        return dict(kind=kind, N=_log_int(rng, 60, 300), obst=rng.randint(0, 8), T=rng.randint(1, 5), family=family,
                    param=param)
    if kind == "batch":
        return dict(kind=kind, domains=rng.randint(2, 12), n_lo=70, n_hi=rng.randint(90, 170), t_lo=rng.randint(3, 16),
                    t_hi=rng.randint(17, 256), draw=rng.randint(2, 10 ** 6))
    if kind == "paths":
        return dict(kind=kind, rings=rng.randint(30, 140), segs=rng.randint(100, 512), T=rng.randint(1, 64),
                    S=_log_int(rng, 4, 256))
    return dict(kind=kind, N=rng.randint(40, 140), obst=rng.randint(0, 8))


# ---- maps -----------------------------------------------------------------

def _blocks(N, count, key):
    """count rectangles (i, j, w, h) of whole cells, a free cell between any two and around the edge."""
    rng, got = random.Random(key), []
    lo, hi = max(2, N // 50), max(3, N // 12)
    for _ in range(100000):
        if len(got) == count:
            break
        w, h = rng.randint(lo, hi), rng.randint(lo, hi)
        i, j = rng.randint(1, N - 1 - w), rng.randint(1, N - 1 - h)
        if all(i > a + c or a > i + w or j > b + d or b > j + h for a, b, c, d in got):
            got.append((i, j, w, h))
    return got


@functools.lru_cache(maxsize=24)
def _square(N, count, key=""):
    """(xy, triangles, loop vertex ids, loop offsets) of the square with obstacles."""
    solid = np.zeros((N + 1, N + 1), bool)
    free = np.ones((N, N), bool)
    blocks = _blocks(N, count, "%d/%d/%s" % (N, count, key))
    for i, j, w, h in blocks:
        solid[j + 1:j + h, i + 1:i + w] = True
        free[j:j + h, i:i + w] = False
    ids = np.cumsum(~solid).reshape(solid.shape) - 1
    y, x = np.nonzero(~solid)
    j, i = np.nonzero(free)
    a, b, c, d = ids[j, i], ids[j, i + 1], ids[j + 1, i + 1], ids[j + 1, i]
    tri = np.stack([np.stack([a, b, c], 1), np.stack([a, c, d], 1)], 1).reshape(-1, 3)

    def ring(i, j, w, h):        # around a rectangle, counter-clockwise
        r, s = np.arange(w), np.arange(h)
        return np.concatenate([ids[j, i + r], ids[j + s, i + w], ids[j + h, i + w - r], ids[j + h - s, i]])

    loops = [ring(0, 0, N, N)] + [ring(*q)[::-1] for q in blocks]
    off = np.cumsum([0] + [len(q) for q in loops]).astype(np.int64)
    return np.stack([x, y], 1) / N, tri.astype(np.int32), np.concatenate(loops).astype(np.int32), off


@functools.lru_cache(maxsize=24)
def _disk(rings, segs):
    """The unit disk: a centre and `rings` rings of `segs` vertices."""
    ang = 2 * np.pi * np.arange(segs) / segs
    rad = np.arange(1, rings + 1) / rings
    xy = np.concatenate([np.zeros((1, 2)), np.stack([np.outer(rad, np.cos(ang)), np.outer(rad, np.sin(ang))], 2).reshape(-1, 2)])
    i, nxt = np.arange(segs), (np.arange(segs) + 1) % segs
    fan = np.stack([np.zeros(segs, int), 1 + i, 1 + nxt], 1)
    base = 1 + segs * np.arange(rings - 1)[:, None]
    a, b, c, d = base + i, base + segs + i, base + segs + nxt, base + nxt
    quads = np.stack([np.stack([a, b, c], 2), np.stack([a, c, d], 2)], 2).reshape(-1, 3)
    return xy, np.concatenate([fan, quads]).astype(np.int32), (1 + segs * (rings - 1) + i).astype(np.int32), np.array([0, segs], np.int64)


def _map(case):
    return _disk(case["rings"], case["segs"]) if "rings" in case else _square(case["N"], case["obst"])


def _interior(m):
    flag = np.ones(len(m[0]), bool)
    flag[m[2]] = False
    return np.nonzero(flag)[0]


def _domains(case):
    """The maps and target counts of a batch: vertex counts spread over their logarithm."""
    rng = random.Random("batch/%d" % case["draw"])
    return [(_square(_log_int(rng, case["n_lo"], case["n_hi"]), rng.randint(0, 8), "b%d" % d),
             rng.randint(case["t_lo"], case["t_hi"])) for d in range(case["domains"])]


# ---- states ---------------------------------------------------------------

class _State:
    """A context on torch's stream with its maps loaded, and the request."""

    def __init__(self, case):
        self.case = case
        self.ctx = dd.dd_create(torch.cuda.current_device(), torch.cuda.current_stream().cuda_stream)

    def load(self, m, solve=True):
        mid = dd.dd_load_mesh(self.ctx, *m)
        if solve:
            dd.dd_poisson_kernel(self.ctx, mid)
        return mid

    def __del__(self):
        torch.cuda.synchronize()
        dd.dd_destroy(self.ctx)


def _nf(mask):
    return bin(mask).count("1")


def _max_pts(m):
    return min(4096, 16 * int(math.sqrt(len(m[0]))) + 64)


def _draws(case, seed, inner):
    """Targets and, where the case has paths, sources, all interior."""
    rng = np.random.default_rng(seed)
    T = case["T"]
    targets = rng.choice(inner, T, replace=T > len(inner)).astype(np.int32)
    return targets, rng.choice(inner, (T, case.get("S", 1))).astype(np.int32)


def _disk_fields(m, targets):
    """The disk's KL fields in closed form, -log(1 - |C_t(x)|^2), float32 [T, n]; the boundary as its discrete rows."""
    z = torch.complex(*(torch.as_tensor(m[0][:, q].copy(), device="cuda") for q in (0, 1)))
    t = z[torch.as_tensor(targets, dtype=torch.long, device="cuda")][:, None]
    f = -torch.log1p(-((z - t).abs() / (1 - z * t.conj()).abs()).square().clamp(max=1 - 1e-12))
    b = torch.as_tensor(m[2], dtype=torch.long, device="cuda")
    f[:, b] = -torch.log((1 - t.abs().square()) / (z[b] - t).abs().square() / len(m[2]))
    return f.float().contiguous()


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    if kind == "batch":
        rng = np.random.default_rng(seed)
        doms = _domains(case)
        s.mids = [s.load(m) for m, _ in doms]
        s.Ts = [T for _, T in doms]
        s.targets = np.concatenate([rng.choice(_interior(m), T).astype(np.int32) for m, T in doms])
        s.sizes = [(2, T, len(m[0])) for m, T in doms]
        s.out = torch.zeros(sum(math.prod(q) for q in s.sizes), device="cuda")
        return s
    m = _map(case)
    n = len(m[0])
    if kind == "poisson":
        # a map of the case's sizes, its corner moved by the seed (the kernel is a map's own)
        xy = m[0] * (1.0 + 0.25 * np.random.default_rng(seed).random(2))
        s.mid = s.load((xy,) + m[1:], solve=False)
        s.out = torch.zeros((n, len(m[2])), device="cuda")
        return s
    s.mid = s.load(m, solve=kind != "paths")
    s.targets, s.sources = _draws(case, seed, _interior(m))
    T, S = case["T"], case.get("S", 0)
    if kind == "paths":
        s.fields = _disk_fields(m, s.targets)
    elif kind == "fields" and case["prec"] == dd.DD_PREC_SPARSE:
        dd.dd_sparsify(s.ctx, s.mid)
    host = case.get("host", False)

    def buffer(shape, dtype=torch.float32):
        return torch.zeros(shape, dtype=dtype).pin_memory() if host else torch.zeros(shape, dtype=dtype, device="cuda")

    if kind in ("query", "fields"):
        s.out = buffer((2 if kind == "query" else _nf(case["mask"]), T, n))
    elif kind == "diverge":
        s.out = buffer((T, n))
    if kind in ("query", "paths"):
        s.max_pts = _max_pts(m)
        s.xy, s.len, s.status = buffer((T * S, s.max_pts, 2)), buffer(T * S, torch.int32), buffer(T * S, torch.int32)
    return s


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "query":
        dd.dd_query(s.ctx, s.mid, s.targets, s.sources, KL | TV, dd.DD_PREC_FP32, KL, s.max_pts, s.out, s.xy, s.len, s.status)
        return {"fields": s.out, "xy": s.xy, "len": s.len, "status": s.status}
    if kind == "fields":
        dd.dd_distance(s.ctx, s.mid, s.targets, case["mask"], case["prec"], s.out)
        return {"fields": list(s.out)}
    if kind == "diverge":
        dd.dd_divergence(s.ctx, s.mid, s.targets, case["family"], case["param"], s.out)
        return {"fields": s.out}
    if kind == "batch":
        dd.dd_query_batch(s.ctx, s.mids, s.Ts, s.targets, None, 0, KL | TV, KL, 2, s.out)
        return {"fields": s.out}
    if kind == "paths":
        dd.dd_trace_fields(s.ctx, s.mid, s.fields, s.targets, s.sources, s.max_pts, s.xy, s.len, s.status)
        return {"xy": s.xy, "len": s.len, "status": s.status}
    dd.dd_poisson_kernel(s.ctx, s.mid)
    dd.dd_get_poisson_kernel(s.ctx, s.mid, s.out)
    return {"P": s.out}


def work(case):
    """P read once and every field written once; two operations a (vertex, column, target) term of a field."""
    kind = case["kind"]
    if kind == "batch":
        got = [(len(m[0]), len(m[2]), T) for m, T in _domains(case)]
        return {"bytes": sum(4.0 * n * k + 8.0 * T * n for n, k, T in got), "flops": sum(4.0 * n * k * T for n, k, T in got)}
    m = _map(case)
    n, k, T = float(len(m[0])), float(len(m[2])), case.get("T", 1)
    paths = 0.0
    if kind in ("query", "paths"):
        # about one point per crossed edge, two edges a cell, half the map's width on average: a point
        # written, and three field values, ids and positions read for it
        paths = T * case["S"] * math.sqrt(n) * (8.0 + 3 * 4.0 + 64.0)
    if kind == "paths":
        return {"bytes": paths, "flops": paths / 4}
    if kind == "poisson":
        # P written, and per entry one product with the matrix's five entries a row
        return {"bytes": 4.0 * n * k, "flops": 10.0 * n * k}
    if kind == "diverge":
        return {"bytes": 4.0 * n * k + 4.0 * T * n, "flops": 2.0 * n * k * T}
    nf = 2 if kind == "query" else _nf(case["mask"])
    kept = 0.25 if case.get("prec") == dd.DD_PREC_SPARSE else 1.0      # about what the threshold keeps, with its columns
    return {"bytes": kept * 4.0 * n * k + 4.0 * nf * T * n + paths, "flops": kept * 2.0 * nf * n * k * T}


# ---- what the outputs are in 64 bits ---------------------------------------

def _exact_kernel(m, xy=None):
    """P = [-L_II^-1 L_IB; I] of the cotangent Laplacian by a dense factorisation."""
    xy = torch.as_tensor(m[0] if xy is None else xy, dtype=torch.float64, device="cuda")
    tri = torch.as_tensor(m[1], dtype=torch.long, device="cuda")
    n, k = len(m[0]), len(m[2])
    A = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    for a in range(3):
        o, p, q = tri[:, a], tri[:, (a + 1) % 3], tri[:, (a + 2) % 3]
        u, v = xy[p] - xy[o], xy[q] - xy[o]
        w = (u * v).sum(1) / (u[:, 0] * v[:, 1] - u[:, 1] * v[:, 0]) / 2
        A.index_put_((p, q), -w, accumulate=True)
        A.index_put_((q, p), -w, accumulate=True)
    A.diagonal().copy_(-A.sum(1))
    inner, outer = torch.as_tensor(_interior(m), device="cuda"), torch.as_tensor(m[2], dtype=torch.long, device="cuda")
    B = -A[inner][:, outer]
    A = A[inner][:, inner]
    P = torch.zeros((n, k), dtype=torch.float64, device="cuda")
    P[inner] = torch.cholesky_solve(B, torch.linalg.cholesky(A)).clamp(min=0)
    P[outer, torch.arange(k, device="cuda")] = 1.0
    return P


def _xlogy(p, q):
    """p log(p / q) with 0 log 0 = 0 and logarithms taken of no less than float32's smallest normal number."""
    return torch.where(p > 0, p * (p.clamp(min=FLT_MIN).log() - q.clamp(min=FLT_MIN).log()), torch.zeros_like(p))


def _exact_fields(P, targets, mask, sparse=False):
    n = len(P)
    if sparse:
        # the threshold is a float32 product on the float32 kernel
        P32 = P.float()
        kept = (P32 >= torch.tensor(1.0 / math.sqrt(n), device="cuda").float() * P32.amax(1, keepdim=True)) & (P32 > 0)
        Q = torch.where(kept, P, torch.zeros_like(P))
    else:
        Q = P
    step = max(1, (1 << 27) // P.shape[1])
    out = []
    for bit in (KL, TV, KLT):
        if not mask & bit:
            continue
        f = torch.empty((len(targets), n), dtype=torch.float64, device="cuda")
        for a, t in enumerate(targets.tolist()):
            for r in range(0, n, step):
                x, qx = P[r:r + step], Q[r:r + step]
                if bit == KL:
                    d = _xlogy(qx, P[t].expand_as(x))
                elif bit == TV:
                    d = (qx - Q[t]).abs()
                else:
                    d = _xlogy(Q[t].expand_as(x), x)
                f[a, r:r + step] = d.sum(1)
        out.append(f)
    return out


def _exact_divergence(P, targets, family, a):
    out = torch.empty((len(targets), len(P)), dtype=torch.float64, device="cuda")
    for i, t in enumerate(targets.tolist()):
        q = P[t]
        if family == dd.DD_DIV_KL_REVERSE:
            out[i] = _xlogy(q.expand_as(P), P).sum(1)
        elif family == dd.DD_DIV_HELLINGER:
            out[i] = (q.sqrt() - P.sqrt()).square().sum(1)
        else:
            out[i] = (4 / (1 - a * a) * (P - P.pow((1 - a) / 2) * q.pow((1 + a) / 2)) + 2 / (1 - a) * (q - P)).sum(1)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("paths", "batch"):
        return None                     # decisions on float32 fields; many factorisations
    m = _map(case)
    if len(m[0]) > 24000:
        return None                     # a dense factorisation takes too long
    if kind == "poisson":
        xy = m[0] * (1.0 + 0.25 * np.random.default_rng(seed).random(2))
        return {"P": _exact_kernel(m, xy)}
    targets, _ = _draws(case, seed, _interior(m))
    if kind == "diverge":
        if case["family"] in (dd.DD_DIV_CHI2, dd.DD_DIV_POWER) or case["param"] < 0:
            return None                 # infinite on boundary rows, or a kernel entry's reciprocal
        return {"fields": _exact_divergence(_exact_kernel(m), targets, case["family"], case["param"])}
    if kind == "query":
        return {"fields": torch.stack(_exact_fields(_exact_kernel(m), targets, KL | TV)), "xy": None, "len": None, "status": None}
    if case["T"] * len(m[0]) * len(m[2]) > 1.5e10:
        return None
    return {"fields": _exact_fields(_exact_kernel(m), targets, case["mask"], case["prec"] == dd.DD_PREC_SPARSE)}
