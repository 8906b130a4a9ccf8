// Triangle-based gradient-descent path tracing, Section IV ("Gradient-descent
// path generation"), one thread per (target, source) pair.
//
// The field is piecewise linear, so triangle tau has the constant gradient
// g = (f0 - f2) grad(phi_0) + (f1 - f2) grad(phi_1) and the path follows -g.
// The walk, made precise from the paper's prose:
//  * vertex v: stop at the target; if v neighbours the target, the path lies
//    on an edge incident on it: append the target and stop.  Otherwise follow
//    the steepest incident triangle whose descent direction enters it from v
//    (inside the corner wedge; ties to the lowest triangle id) to the opposite
//    edge.  With no such triangle take the incident edge of largest positive
//    slope (f_v - f_u)/|v - u| to its other end; none means a local minimum.
//  * edge (a, b) left from triangle tau: an edge incident on the target ends
//    the path at the target.  Otherwise enter the triangle across; if its
//    descent direction points into it, cross to the exit edge; if not (valley
//    edge) or there is no triangle across (boundary edge), slide along the
//    edge to its lower endpoint (ties to the lower id).
//  * an exit whose barycentric coordinate is <= kEpsBary lands on the vertex.
// Geometry and gradients are FP32; the hat-function gradients are computed in
// FP64 on the host and rounded once.
//
// Work split for latency.  What a vertex state decides depends only on the
// field and the vertex (the best triangle is the steepest, ties by id, so the
// order in which the incident triangles are examined does not matter).  Where
// many paths share a field it is computed for every vertex of every field
// before the walk (vertex_decision_kernel; wide fans in wide_decision_kernel),
// from the fields vertex by vertex (fields_by_vertex_kernel), into decisions
// stored [vertex][field]: a warp of the decision kernel handles one vertex for
// 32 fields, so the triangle records it reads are shared by all its lanes and
// the values it reads are contiguous.
// The walk (walk_path) then does one thing per iteration: cross one triangle
// from an edge, apply one vertex decision, or slide along a valley or
// boundary edge.  Batches of several maps walk one path per thread on stored
// rates (trace_path).
//
// Measured, longest path 436 points: grid140, one target, 256 paths 279 -> 119
// us (a call with its fields, results in host buffers, 362 -> 222 us); 142
// points, 32 paths on the 2,049-vertex disk 250 -> 47 us (a call 240 -> 68 us);
// 941 points, 64 x 256 paths on the 71,681-vertex disk 953 -> 476 us and the
// decisions 778 -> 221 us (a call 1,749 -> 689 us).
#include <cfloat>
#include <cstring>
#include <cstdlib>
#include <algorithm>
#include <cmath>
#include <random>
#include <vector>

#include "dd_internal.h"

namespace {

constexpr float kEpsBary = 1e-6f;    // barycentric snap to a vertex
constexpr float kEpsWedge = 1e-6f;   // relative tolerance of the wedge / entry tests
constexpr int kWideFan = kWideFanTriangles;
constexpr int64_t kWarpPaths = 2432;      // 16 a SM
constexpr int32_t kDenseMinPaths = 128;   // paths per field from which decisions are precomputed

// Triangle record (64 bytes): vertex ids, the ids of the triangles across the
// edges opposite each vertex (-1 on the boundary), the squared norms q_i of
// the hat gradients, and the vertex positions.
struct Tri {
    int v0, v1, v2, n0, n1, n2;
    float q0, q1, q2;
    float2 p0, p1, p2;
};

__device__ __forceinline__ Tri load_tri(const int4 *__restrict__ rec, int t) {
    const int4 a = __ldg(rec + 4 * t), b = __ldg(rec + 4 * t + 1);
    const float4 c = __ldg(reinterpret_cast<const float4 *>(rec) + 4 * t + 2);
    const float4 d = __ldg(reinterpret_cast<const float4 *>(rec) + 4 * t + 3);
    Tri T;
    T.v0 = a.x;
    T.v1 = a.y;
    T.v2 = a.z;
    T.n0 = a.w;
    T.n1 = b.x;
    T.n2 = b.y;
    T.q0 = __int_as_float(b.z);
    T.q1 = __int_as_float(b.w);
    T.q2 = c.x;
    T.p0 = make_float2(c.z, c.w);
    T.p1 = make_float2(d.x, d.y);
    T.p2 = make_float2(d.z, d.w);
    return T;
}

__device__ __forceinline__ int vid(const Tri &T, int i) { return i == 0 ? T.v0 : (i == 1 ? T.v1 : T.v2); }
__device__ __forceinline__ float2 pos(const Tri &T, int i) { return i == 0 ? T.p0 : (i == 1 ? T.p1 : T.p2); }
__device__ __forceinline__ int local_of(const Tri &T, int x) { return T.v0 == x ? 0 : (T.v1 == x ? 1 : 2); }
__device__ __forceinline__ float sel3f(int i, float a, float b, float c) { return i == 0 ? a : (i == 1 ? b : c); }
__device__ __forceinline__ int sel3i(int i, int a, int b, int c) { return i == 0 ? a : (i == 1 ? b : c); }

// Per (field, triangle): (r0, r1, r2, |g|^2) with r_i = -grad(phi_i) . g the
// rate of change of barycentric coordinate i along the descent direction -g.
// g = f0 grad(phi_0) + f1 grad(phi_1) + f2 grad(phi_2) = (f0 - f2) g0 + (f1 - f2) g1.
// h: (g0x, g0y, g1x, g1y)
__device__ __forceinline__ float4 rates_of(const float4 &h, float f0, float f1, float f2) {
    const float d0 = f0 - f2, d1 = f1 - f2;
    const float gx = d0 * h.x + d1 * h.z, gy = d0 * h.y + d1 * h.w;
    const float r0 = -(h.x * gx + h.y * gy), r1 = -(h.z * gx + h.w * gy);
    return make_float4(r0, r1, -(r0 + r1), gx * gx + gy * gy);
}
__device__ __forceinline__ float4 tri_rates(const float4 *__restrict__ gphi, const int4 *__restrict__ rec, int64_t t,
                                            const float *__restrict__ f) {
    const int4 a = __ldg(rec + 4 * t);
    return rates_of(__ldg(gphi + 2 * t), f[a.x], f[a.y], f[a.z]);
}

// ft[v * T + a] = field a at vertex v: the fields vertex by vertex, so that a
// warp of the decision kernel reads 32 fields of a vertex at once
__global__ void __launch_bounds__(256) fields_by_vertex_kernel(const float *__restrict__ fields, int64_t field_stride,
                                                               int64_t n_v, int32_t T, int32_t first,
                                                               float *__restrict__ ft) {
    __shared__ float tile[32][33];
    const int64_t v0 = (int64_t)blockIdx.x * 32;
    const int a0 = first + blockIdx.y * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
    for (int i = ty; i < 32; i += 8)
        if (a0 + i < T && v0 + tx < n_v) tile[i][tx] = fields[(int64_t)(a0 + i) * field_stride + v0 + tx];
    __syncthreads();
#pragma unroll
    for (int i = ty; i < 32; i += 8)
        if (v0 + i < n_v && a0 + tx < T) ft[(v0 + i) * T + a0 + tx] = tile[tx][i];
}

// What the walk does at a vertex (32 bytes)
enum { kVCross = 0, kVVertex = 1, kVAdjacent = 2, kVStuck = 3 };
struct VDec {
    int4 h;      // kind, then: cross (ea, eb, t_next) | vertex (u, -, -) | adjacent (target, -, -)
    float4 w;    // cross (la, lb, point) | vertex, adjacent (position, -, -)
};

struct TraceDom {
    const int4 *rec, *hrec;
    const float4 *gphi;
    const float2 *xy;
    const int32_t *vt_off, *vt;
    int64_t n_t, n_v;
};

// The vertex state at v, one incident triangle at a time: add() examines a
// triangle of v's fan, finish() turns the fan's best candidate into the
// decision.  Both the decision kernel (a whole fan in one call) and the walk
// without precomputed decisions (one triangle per iteration) use it, so the
// two give the same decision bit for bit.
struct FanScan {
    bool adj;
    int best, b_vj, b_vk, b_next;
    float best_g2, baj, bak;
    float2 b_pj, b_pk;

    __device__ __forceinline__ void begin() {
        adj = false;
        best = -1;
        b_vj = b_vk = 0;
        b_next = -1;
        best_g2 = baj = bak = 0.f;
        b_pj = b_pk = make_float2(0.f, 0.f);
    }

    // triangle tl (record T, rates R of the field), v its local vertex L, then X
    // and Y counter-clockwise (rates rX, rY; vertices and positions): the exit
    // edge is X-Y
    __device__ __forceinline__ void consider(int target, int tl, float rX, float rY, float qX, float qY, float gg, int vX,
                                             int vY, float2 pX, float2 pY, int next) {
        const float eps2 = kEpsWedge * kEpsWedge;
        adj |= (vX == target) | (vY == target);
        const float tol2 = eps2 * gg * fmaxf(qX, qY);
        const bool in_x = rX >= 0.f || rX * rX <= tol2;
        const bool in_y = rY >= 0.f || rY * rY <= tol2;
        if (gg > 0.f && in_x && in_y && rX + rY > 0.f && (gg > best_g2 || (gg == best_g2 && tl < best))) {
            best = tl;
            best_g2 = gg;
            baj = fmaxf(rX, 0.f);
            bak = fmaxf(rY, 0.f);
            b_vj = vX;
            b_vk = vY;
            b_pj = pX;
            b_pk = pY;
            b_next = next;
        }
    }

    // triangle tl (record T, rates R of the field) incident on v
    __device__ __forceinline__ void add(int v, int target, int tl, const Tri &T, const float4 &R) {
        const int L = local_of(T, v), X = L == 2 ? 0 : L + 1, Y = L == 0 ? 2 : L - 1;
        consider(target, tl, sel3f(X, R.x, R.y, R.z), sel3f(Y, R.x, R.y, R.z), sel3f(X, T.q0, T.q1, T.q2),
                 sel3f(Y, T.q0, T.q1, T.q2), R.w, sel3i(X, T.v0, T.v1, T.v2), sel3i(Y, T.v0, T.v1, T.v2), pos(T, X),
                 pos(T, Y), sel3i(L, T.n0, T.n1, T.n2));
    }
    // the same where the whole warp looks at one triangle and vertex: a branch
    // on the local vertex instead of a choice for every operand
    __device__ __forceinline__ void add_same(int v, int target, int tl, const Tri &T, const float4 &R) {
        if (T.v0 == v)
            consider(target, tl, R.y, R.z, T.q1, T.q2, R.w, T.v1, T.v2, T.p1, T.p2, T.n0);
        else if (T.v1 == v)
            consider(target, tl, R.z, R.x, T.q2, T.q0, R.w, T.v2, T.v0, T.p2, T.p0, T.n1);
        else
            consider(target, tl, R.x, R.y, T.q0, T.q1, R.w, T.v0, T.v1, T.p0, T.p1, T.n2);
    }

    // (G lanes of `mask` hold the same scan and share the fallback's fan)
    template <int G>
    __device__ __forceinline__ VDec finish(const TraceDom &p, const float *__restrict__ f, int target, int v,
                                           unsigned mask = 0) const {
        VDec d;
        if (adj) {                                   // v lies on an edge incident on the target
            const float2 pt = p.xy[target];
            d.h = make_int4(kVAdjacent, target, 0, 0);
            d.w = make_float4(pt.x, pt.y, 0.f, 0.f);
            return d;
        }
        if (best >= 0) {
            const float s = __fdividef(1.0f, baj + bak);
            const float lj = s * baj, lk = s * bak;
            if (lj <= kEpsBary) {
                d.h = make_int4(kVVertex, b_vk, 0, 0);
                d.w = make_float4(b_pk.x, b_pk.y, 0.f, 0.f);
            } else if (lk <= kEpsBary) {
                d.h = make_int4(kVVertex, b_vj, 0, 0);
                d.w = make_float4(b_pj.x, b_pj.y, 0.f, 0.f);
            } else {
                d.h = make_int4(kVCross, b_vj, b_vk, b_next);
                d.w = make_float4(lj, lk, lj * b_pj.x + lk * b_pk.x, lj * b_pj.y + lk * b_pk.y);
            }
            return d;
        }
        // no descending triangle: the incident edge of largest positive slope (ties to the
        // lower id), the fan over the G lanes of the group
        int best_u = -1;
        float best_s = 0.f;
        float2 best_p = make_float2(0.f, 0.f);
        const float fv = f[v];
        const float2 pv = p.xy[v];
        for (int q = p.vt_off[v] + (threadIdx.x & (G - 1)); q < p.vt_off[v + 1]; q += G) {
            const Tri Q = load_tri(p.rec, p.vt[q]);
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                const int u = vid(Q, e);
                if (u == v) continue;
                const float2 pu = pos(Q, e);
                const float dx = pv.x - pu.x, dy = pv.y - pu.y;
                const float slope = (fv - f[u]) / sqrtf(dx * dx + dy * dy);
                if (slope > 0.f && (slope > best_s || (slope == best_s && u < best_u))) {
                    best_s = slope;
                    best_u = u;
                    best_p = pu;
                }
            }
        }
        if (G > 1) {
            __syncwarp(mask);
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) {
                const float s2 = __shfl_xor_sync(mask, best_s, o);
                const int u2 = __shfl_xor_sync(mask, best_u, o);
                const float px = __shfl_xor_sync(mask, best_p.x, o), py = __shfl_xor_sync(mask, best_p.y, o);
                if (u2 >= 0 && (s2 > best_s || (s2 == best_s && u2 < best_u))) {
                    best_s = s2;
                    best_u = u2;
                    best_p = make_float2(px, py);
                }
            }
        }
        if (best_u < 0) {
            d.h = make_int4(kVStuck, 0, 0, 0);
            d.w = make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
            d.h = make_int4(kVVertex, best_u, 0, 0);
            d.w = make_float4(best_p.x, best_p.y, 0.f, 0.f);
        }
        return d;
    }
};

// The best triangle of a fan whose triangles were dealt to the G lanes of a
// group (aligned, all of them in `mask`): the steepest, ties to the lowest id
// -- what one lane scanning the whole fan finds, in any order.
template <int G>
__device__ __forceinline__ void fan_reduce(FanScan &fs, unsigned mask) {
    int from = threadIdx.x & 31, adj = fs.adj;
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        adj |= __shfl_xor_sync(mask, adj, o);
        const float g2 = __shfl_xor_sync(mask, fs.best_g2, o);
        const int tl = __shfl_xor_sync(mask, fs.best, o), at = __shfl_xor_sync(mask, from, o);
        if (g2 > fs.best_g2 || (g2 == fs.best_g2 && tl < fs.best)) {
            fs.best_g2 = g2;
            fs.best = tl;
            from = at;
        }
    }
    fs.adj = adj != 0;
    fs.baj = __shfl_sync(mask, fs.baj, from);
    fs.bak = __shfl_sync(mask, fs.bak, from);
    fs.b_vj = __shfl_sync(mask, fs.b_vj, from);
    fs.b_vk = __shfl_sync(mask, fs.b_vk, from);
    fs.b_next = __shfl_sync(mask, fs.b_next, from);
    fs.b_pj.x = __shfl_sync(mask, fs.b_pj.x, from);
    fs.b_pj.y = __shfl_sync(mask, fs.b_pj.y, from);
    fs.b_pk.x = __shfl_sync(mask, fs.b_pk.x, from);
    fs.b_pk.y = __shfl_sync(mask, fs.b_pk.y, from);
}

// one warp per vertex and 32 fields (blockIdx.y, from field `first` on), lane = field: dec[v * T + a];
// vertices of more than kWideFan triangles are left to wide_decision_kernel.
// The rates of a fan's triangles are formed here from the fields by vertex:
// 64 fields of 71,681 vertices, the rates of every triangle stored first (147
// MB written, read three times) took 68 + 230 us, this 8 + 183 (216 with a
// choice among the local vertices for every operand).
__global__ void __launch_bounds__(128) vertex_decision_kernel(const TraceDom p, int32_t T, int32_t first,
                                                              const float *__restrict__ fields, int64_t field_stride,
                                                              const float *__restrict__ ft,
                                                              const int32_t *__restrict__ targets,
                                                              VDec *__restrict__ dec) {
    const int64_t v = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    const int a = first + blockIdx.y * 32 + (threadIdx.x & 31);
    if (v >= p.n_v || a >= T) return;
    const int q0 = p.vt_off[v], q1 = p.vt_off[v + 1];
    if (q1 - q0 > kWideFan) return;
    const int target = targets[a];
    FanScan fs;
    fs.begin();
    for (int q = q0; q < q1; ++q) {
        const int tl = p.vt[q];
        const Tri t = load_tri(p.rec, tl);
        const float4 r = rates_of(__ldg(p.gphi + 2 * (int64_t)tl), ft[(int64_t)t.v0 * T + a], ft[(int64_t)t.v1 * T + a],
                                  ft[(int64_t)t.v2 * T + a]);
        fs.add_same((int)v, target, tl, t, r);
    }
    dec[v * T + a] = fs.finish<1>(p, fields + (int64_t)a * field_stride, target, (int)v);
}

// The vertices with wide fans (a disk's centre: as many triangles as the disk
// has sectors), one warp per (vertex, field), the fan over the lanes.  With
// one lane scanning it the 512 triangles of one centre were a chain of 0.65
// ms, all of the decision pass but 0.12 ms (71,681 vertices, 64 fields).
__global__ void wide_decision_kernel(const TraceDom p, const int32_t *__restrict__ wide, int32_t T, int32_t first,
                                     const float *__restrict__ fields, int64_t field_stride,
                                     const int32_t *__restrict__ targets, VDec *__restrict__ dec) {
    const int v = wide[blockIdx.x], lane = threadIdx.x & 31;
    const int a = first + blockIdx.y * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (a >= T) return;
    const float *f = fields + (int64_t)a * field_stride;
    FanScan fs;
    fs.begin();
    for (int q = p.vt_off[v] + lane, q1 = p.vt_off[v + 1]; q < q1; q += 32) {
        const int tl = p.vt[q];
        fs.add(v, targets[a], tl, load_tri(p.rec, tl), tri_rates(p.gphi, p.rec, tl, f));
    }
    __syncwarp();
    fan_reduce<32>(fs, 0xffffffffu);
    const VDec d = fs.finish<32>(p, f, targets[a], v, 0xffffffffu);
    if (lane == 0) dec[(int64_t)v * T + a] = d;
}

// One path: walk from `source` to `target` on field f, with that field's
// triangle rates.  The warp votes at the top of every
// iteration, so its threads reconverge once per step; finished threads (and
// padding lanes) idle there until the last path of the warp ends.
// (rates of this field start at `rates`, one entry per triangle; a vertex
// state computes its decision itself, from the same functions as the decision
// kernels, so with the same result.)  One thread a path: for batches of maps,
// whose hundreds of thousands of paths fill the GPU.
__device__ __forceinline__ void trace_path(const TraceDom &p, const float *__restrict__ f,
                                           const float4 *__restrict__ rates, int target, int source,
                                           float2 *__restrict__ out, int32_t max_pts, int32_t max_steps,
                                           int32_t *len_out, int32_t *status_out, bool active) {
    const float eps2 = kEpsWedge * kEpsWedge;
    int len = 0;
    int status = DD_TRACE_STEP_LIMIT;
    int states = 1;                // vertex and edge states entered (the step cap counts these)
    bool fin = !active;
    bool at_vertex = true;
    int v = source;
    // fan scan of the current vertex: one
    // incident triangle (from the vertex's triangle list) per iteration
    FanScan fs;
    fs.begin();
    int scan_q = 0, scan_end = 0;
    if (active) {
        scan_q = p.vt_off[v];
        scan_end = p.vt_off[v + 1];
    }
    // edge state: the path sits on edge (ea, eb) at weights (la, lb) and enters
    // t_next (the triangle across that edge, -1 on the boundary)
    int t_next = -1, ea = 0, eb = 0;
    float la = 0.f, lb = 0.f;
    float2 pa = make_float2(0.f, 0.f), pb = pa;
    if (active) {
        out[len++] = p.xy[v];
        if (v == target) {
            status = DD_TRACE_OK;
            fin = true;
        }
    }

// The macros end the current iteration with `continue` when the path ends;
// they are used as statements inside braces (no do-while wrapper, so that
// `continue` reaches the walk loop).
#define DD_PUSH(pt)                              \
    if (len >= max_pts) {                        \
        status = DD_TRACE_TRUNCATED;             \
        fin = true;                              \
        continue;                                \
    }                                            \
    out[len++] = (pt);
#define DD_ENTER_VERTEX(vert)                    \
    v = (vert);                                  \
    at_vertex = true;                            \
    fs.begin();                                  \
    scan_q = p.vt_off[v];                        \
    scan_end = p.vt_off[v + 1];                  \
    if (++states > max_steps) {                  \
        fin = true;                              \
        continue;                                \
    }                                            \
    if (v == target) {                           \
        status = DD_TRACE_OK;                    \
        fin = true;                              \
        continue;                                \
    }
#define DD_SLIDE()                                                     \
    {                                                                  \
        const float fa = f[ea], fb = f[eb];                            \
        const bool a_low = fa < fb || (fa == fb && ea < eb);           \
        DD_PUSH(a_low ? pa : pb);                                      \
        DD_ENTER_VERTEX(a_low ? ea : eb);                              \
    }

    const int64_t iter_cap = 4LL * max_steps + 16;
    for (int64_t iter = 0;; ++iter) {
        if (!fin && iter >= iter_cap) fin = true;
        if (!__any_sync(0xffffffffu, !fin)) break;
        if (fin) continue;
        if (at_vertex) {
            // ---- vertex state: scan one incident triangle per iteration (so the warp's
            // other lanes wait little), then apply the decision
            if (scan_q < scan_end) {
                const int tl = p.vt[scan_q++];
                fs.add(v, target, tl, load_tri(p.rec, tl), __ldg(rates + tl));
                continue;
            }
            const VDec own = fs.finish<1>(p, f, target, v);
            const int4 h = own.h;
            const float4 w = own.w;
            const int kind = h.x;
            if (kind == kVStuck) {
                status = DD_TRACE_STUCK;
                fin = true;
                continue;
            }
            const bool cross = kind == kVCross;
            DD_PUSH(make_float2(cross ? w.z : w.x, cross ? w.w : w.y));
            if (kind == kVAdjacent) {
                status = DD_TRACE_OK;
                fin = true;
                continue;
            }
            if (!cross) {
                DD_ENTER_VERTEX(h.y);
                continue;
            }
            at_vertex = false;
            ea = h.y;
            eb = h.z;
            t_next = h.w;
            la = w.x;
            lb = w.y;
            pa = fs.b_pj;
            pb = fs.b_pk;
            if (++states > max_steps) fin = true;
            continue;
        }
        if (t_next < 0) {                // boundary edge: slide to the lower endpoint
            DD_SLIDE();
            continue;
        }
        // ---- edge state: entering T across (ea, eb); in T's counter-clockwise order
        // eb is local vertex L, ea is X, and the opposite vertex is Y
        const int tl = t_next;
        const Tri T = load_tri(p.rec, tl);
        const float4 Rt = __ldg(rates + tl);
        const int L = local_of(T, eb), X = L == 2 ? 0 : L + 1, Y = L == 0 ? 2 : L - 1;
        const float ra = sel3f(X, Rt.x, Rt.y, Rt.z), rb = sel3f(L, Rt.x, Rt.y, Rt.z), rc = sel3f(Y, Rt.x, Rt.y, Rt.z);
        const float qY = sel3f(Y, T.q0, T.q1, T.q2);
        const bool enters = rc > 0.f && rc * rc > eps2 * Rt.w * qY;
        const float sa = ra < 0.f ? __fdividef(la, -ra) : INFINITY;
        const float sb = rb < 0.f ? __fdividef(lb, -rb) : INFINITY;
        if (!enters || !(fminf(sa, sb) < INFINITY)) {   // valley edge (or no exit): lower endpoint
            DD_SLIDE();
            continue;
        }
        const int vY = sel3i(Y, T.v0, T.v1, T.v2);
        const float2 pY = pos(T, Y);
        const bool via_a = sa <= sb;                      // exit through the edge opposite a (the Y-R edge)
        const float s = via_a ? sa : sb;
        float lkeep = fmaxf(via_a ? lb + s * rb : la + s * ra, 0.f);
        float lc2 = fmaxf(s * rc, 0.f);
        const float inv = __fdividef(1.0f, lkeep + lc2);
        lkeep *= inv;
        lc2 *= inv;
        const int keep_v = via_a ? eb : ea;
        const float2 keep_p = via_a ? pb : pa;
        if (lkeep <= kEpsBary) {
            DD_PUSH(pY);
            DD_ENTER_VERTEX(vY);
            continue;
        }
        if (lc2 <= kEpsBary) {
            DD_PUSH(keep_p);
            DD_ENTER_VERTEX(keep_v);
            continue;
        }
        DD_PUSH(make_float2(lkeep * keep_p.x + lc2 * pY.x, lkeep * keep_p.y + lc2 * pY.y));
        // new edge in T's counter-clockwise order: via a -> (Y, R) = (c, b); via b -> (X, Y) = (a, c)
        if (via_a) {
            t_next = sel3i(X, T.n0, T.n1, T.n2);
            ea = vY;
            eb = keep_v;
            pa = pY;
            pb = keep_p;
            la = lc2;
            lb = lkeep;
        } else {
            t_next = sel3i(L, T.n0, T.n1, T.n2);
            ea = keep_v;
            eb = vY;
            pa = keep_p;
            pb = pY;
            la = lkeep;
            lb = lc2;
        }
        if (++states > max_steps) {
            fin = true;
            continue;
        }
        if (ea == target || eb == target) {   // an edge incident on the target
            DD_PUSH(p.xy[target]);
            status = DD_TRACE_OK;
            fin = true;
            continue;
        }
    }
#undef DD_PUSH
#undef DD_ENTER_VERTEX
#undef DD_SLIDE
    if (active) {
        *len_out = len;
        *status_out = status;
    }
}

// A crossing as the walk meets it, 48 bytes for each triangle and entry edge
// (4 t + L, L the local vertex that is the entry edge's second end b; a is the
// next vertex counter-clockwise and Y the one across): no choice among local
// vertices is left but the order in which the rates are formed.
//   (g0x, g0y, g1x, g1y)  (Y, position of Y, |grad phi_Y|^2)
//   (na, nb, oa, ob): the crossing after leaving through the edge opposite a
//   or b (-1 on the boundary) and the vertex beyond that edge
__global__ void crossings_kernel(const int4 *__restrict__ rec, const float4 *__restrict__ gphi, int64_t n_t,
                                 int4 *__restrict__ hrec) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t t = i >> 2;
    const int L = (int)(i & 3);
    if (t >= n_t) return;
    int4 *h = hrec + 3 * i;
    if (L == 3) {
        h[0] = h[1] = h[2] = make_int4(0, 0, 0, 0);
        return;
    }
    const Tri T = load_tri(rec, (int)t);
    const int X = L == 2 ? 0 : L + 1, Y = L == 0 ? 2 : L - 1;
    const int vb = vid(T, L), vY = vid(T, Y);
    const float2 pY = pos(T, Y);
    // through the edge opposite a = (Y, b): b stays second; opposite b = (a, Y): Y is
    auto next = [&](int tn, int second, int &n, int &o) {
        n = -1;
        o = -1;
        if (tn < 0) return;
        const Tri Q = load_tri(rec, tn);
        const int l = local_of(Q, second);
        n = 4 * tn + l;
        o = vid(Q, l == 0 ? 2 : l - 1);
    };
    int4 w;
    next(sel3i(X, T.n0, T.n1, T.n2), vb, w.x, w.z);
    next(sel3i(L, T.n0, T.n1, T.n2), vY, w.y, w.w);
    const float4 g = gphi[2 * t];
    h[0] = make_int4(__float_as_int(g.x), __float_as_int(g.y), __float_as_int(g.z), __float_as_int(g.w));
    h[1] = make_int4(vY, __float_as_int(pY.x), __float_as_int(pY.y), __float_as_int(sel3f(Y, T.q0, T.q1, T.q2)));
    h[2] = w;
}

// One path, walked by a group of G lanes (aligned within the warp, `mask`).
// The walk is trace_path's, decision by decision and operation by operation;
// what differs is what a step costs and when things are read, for a step's
// chain is what a path waits for:
//  * crossings come ready-made (crossings_kernel): a step took 300
//    instructions on triangle records, most of them choosing among local
//    vertices;
//  * at the start of a crossing the two that can follow it and the field at
//    the vertices beyond are read, and arrive while it is decided; with the
//    edge's field values carried along, no read of a step waits for another;
//  * every lane of the group carries the whole state (reads of one address by
//    a group are one access) and its first lane writes the points;
//  * a vertex state without precomputed decisions deals the fan's triangles
//    to the lanes.
// Fewer paths to a warp also mean fewer of them waiting for another's branch.
template <int G>
__device__ __forceinline__ void walk_path(const TraceDom &p, const float *__restrict__ f,
                                          const VDec *__restrict__ dec, int64_t dstride, int target, int source,
                                          float2 *__restrict__ out, int32_t max_pts, int32_t max_steps,
                                          int32_t *len_out, int32_t *status_out, bool active, unsigned mask) {
    const float eps2 = kEpsWedge * kEpsWedge;
    const int gl = threadIdx.x & (G - 1);
    struct Crossing {
        float4 g, y;
        int4 n;
    };
    auto read = [&](int h) {
        Crossing c;
        const int4 *r = p.hrec + 3 * (int64_t)h;
        c.g = __ldg(reinterpret_cast<const float4 *>(r));
        c.y = __ldg(reinterpret_cast<const float4 *>(r + 1));
        c.n = __ldg(r + 2);
        return c;
    };
    int len = 0;
    int status = DD_TRACE_STEP_LIMIT;
    int states = 1;
    bool fin = !active;
    bool at_vertex = true;
    int v = source;
    // edge state: edge (ea, eb) at weights (la, lb), its ends' field values and
    // positions; the crossing h (4 t + L, -1 on the boundary) and the field at its Y
    int h = -1, ea = 0, eb = 0;
    float la = 0.f, lb = 0.f, fa = 0.f, fb = 0.f, fc = 0.f;
    float2 pa = make_float2(0.f, 0.f), pb = pa;
    Crossing c = {};
    if (active) {
        if (gl == 0) out[len] = p.xy[v];
        ++len;
        if (v == target) {
            status = DD_TRACE_OK;
            fin = true;
        }
    }
#define DD_PUSH(pt)                              \
    if (len >= max_pts) {                        \
        status = DD_TRACE_TRUNCATED;             \
        fin = true;                              \
        continue;                                \
    }                                            \
    if (gl == 0) out[len] = (pt);                \
    ++len;
#define DD_ENTER_VERTEX(vert)                    \
    v = (vert);                                  \
    at_vertex = true;                            \
    if (++states > max_steps) {                  \
        fin = true;                              \
        continue;                                \
    }                                            \
    if (v == target) {                           \
        status = DD_TRACE_OK;                    \
        fin = true;                              \
        continue;                                \
    }
#define DD_SLIDE()                                                     \
    {                                                                  \
        const bool a_low = fa < fb || (fa == fb && ea < eb);           \
        DD_PUSH(a_low ? pa : pb);                                      \
        DD_ENTER_VERTEX(a_low ? ea : eb);                              \
    }

    for (;;) {
        // (one path to a warp: its lanes agree)
        if (G == 32 ? fin : !__any_sync(0xffffffffu, !fin)) break;
        if (fin) continue;
        if (at_vertex) {
            VDec d;
            if (dec) {
                const VDec *dv = dec + (int64_t)v * dstride;
                d.h = __ldg(&dv->h);
                d.w = __ldg(&dv->w);
            } else {
                FanScan fs;
                fs.begin();
                for (int q = p.vt_off[v] + gl, q1 = p.vt_off[v + 1]; q < q1; q += G) {
                    const int tl = p.vt[q];
                    fs.add(v, target, tl, load_tri(p.rec, tl), tri_rates(p.gphi, p.rec, tl, f));
                }
                if (G > 1) {
                    __syncwarp(mask);
                    fan_reduce<G>(fs, mask);
                }
                d = fs.finish<G>(p, f, target, v, mask);
            }
            const int kind = d.h.x;
            if (kind == kVStuck) {
                status = DD_TRACE_STUCK;
                fin = true;
                continue;
            }
            const bool cross = kind == kVCross;
            DD_PUSH(make_float2(cross ? d.w.z : d.w.x, cross ? d.w.w : d.w.y));
            if (kind == kVAdjacent) {
                status = DD_TRACE_OK;
                fin = true;
                continue;
            }
            if (!cross) {
                DD_ENTER_VERTEX(d.h.y);
                continue;
            }
            at_vertex = false;
            ea = d.h.y;
            eb = d.h.z;
            la = d.w.x;
            lb = d.w.y;
            pa = p.xy[ea];
            pb = p.xy[eb];
            fa = f[ea];
            fb = f[eb];
            h = -1;
            if (d.h.w >= 0) {
                const int4 q = __ldg(p.rec + 4 * (int64_t)d.h.w);
                h = 4 * d.h.w + (q.x == eb ? 0 : (q.y == eb ? 1 : 2));
                c = read(h);
                fc = f[__float_as_int(c.y.x)];
            }
            if (++states > max_steps) fin = true;
            continue;
        }
        if (h < 0) {                     // boundary edge: slide to the lower endpoint
            DD_SLIDE();
            continue;
        }
        // edge state: crossing the triangle from (ea, eb) to one of its other edges
        const int ha = c.n.x, hb = c.n.y;
        const float foa = f[max(c.n.z, 0)], fob = f[max(c.n.w, 0)];
        const Crossing ca = read(max(ha, 0)), cb = read(max(hb, 0));
        const bool l0 = (h & 3) == 0, l1 = (h & 3) == 1;       // b is local vertex 0, 1 (or 2)
        const float4 Rt = rates_of(c.g, l0 ? fb : (l1 ? fc : fa), l0 ? fa : (l1 ? fb : fc), l0 ? fc : (l1 ? fa : fb));
        const float ra = l0 ? Rt.y : (l1 ? Rt.z : Rt.x), rb = l0 ? Rt.x : (l1 ? Rt.y : Rt.z),
                    rc = l0 ? Rt.z : (l1 ? Rt.x : Rt.y);
        const bool enters = rc > 0.f && rc * rc > eps2 * Rt.w * c.y.w;
        const float sa = ra < 0.f ? __fdividef(la, -ra) : INFINITY;
        const float sb = rb < 0.f ? __fdividef(lb, -rb) : INFINITY;
        if (!enters || !(fminf(sa, sb) < INFINITY)) {   // valley edge (or no exit): lower endpoint
            DD_SLIDE();
            continue;
        }
        const int vY = __float_as_int(c.y.x);
        const float2 pY = make_float2(c.y.y, c.y.z);
        const bool via_a = sa <= sb;                      // exit through the edge opposite a (the Y-b edge)
        const float s = via_a ? sa : sb;
        float lkeep = fmaxf(via_a ? lb + s * rb : la + s * ra, 0.f);
        float lc2 = fmaxf(s * rc, 0.f);
        const float inv = __fdividef(1.0f, lkeep + lc2);
        lkeep *= inv;
        lc2 *= inv;
        const int keep_v = via_a ? eb : ea;
        const float2 keep_p = via_a ? pb : pa;
        if (lkeep <= kEpsBary) {
            DD_PUSH(pY);
            DD_ENTER_VERTEX(vY);
            continue;
        }
        if (lc2 <= kEpsBary) {
            DD_PUSH(keep_p);
            DD_ENTER_VERTEX(keep_v);
            continue;
        }
        DD_PUSH(make_float2(lkeep * keep_p.x + lc2 * pY.x, lkeep * keep_p.y + lc2 * pY.y));
        // new edge, counter-clockwise: via a -> (Y, b); via b -> (a, Y)
        if (via_a) {
            h = ha;
            c = ca;
            ea = vY;
            pa = pY;
            fa = fc;
            fc = foa;
            la = lc2;
            lb = lkeep;
        } else {
            h = hb;
            c = cb;
            eb = vY;
            pb = pY;
            fb = fc;
            fc = fob;
            la = lkeep;
            lb = lc2;
        }
        if (++states > max_steps) {
            fin = true;
            continue;
        }
        if (vY == target || keep_v == target) {   // an edge incident on the target
            DD_PUSH(p.xy[target]);
            status = DD_TRACE_OK;
            fin = true;
            continue;
        }
    }
#undef DD_PUSH
#undef DD_ENTER_VERTEX
#undef DD_SLIDE
    if (active && gl == 0) {
        *len_out = len;
        *status_out = status;
    }
}

struct TraceParams {
    TraceDom d;
    const VDec *dec;               // [n_v][T]
    const float *fields;
    int64_t field_stride;
    const int32_t *targets, *sources;
    int64_t total;
    int32_t S, max_pts, max_steps, T;
    float2 *out_xy;
    int32_t *out_len, *out_status;
};

// G lanes a path
template <int G>
__global__ void __launch_bounds__(64) trace_group_kernel(const TraceParams p) {
    const int64_t gid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const bool active = gid < p.total;
    const int64_t id = active ? gid : 0;
    const int a = (int)(id / p.S);
    const unsigned mask = G == 32 ? 0xffffffffu : (((1u << (G & 31)) - 1u) << (threadIdx.x & 31 & ~(G - 1)));
    walk_path<G>(p.d, p.fields + (int64_t)a * p.field_stride, p.dec ? p.dec + a : nullptr, p.T, p.targets[a],
                 p.sources[id], p.out_xy + id * p.max_pts, p.max_pts, p.max_steps, p.out_len + id, p.out_status + id,
                 active, mask);
}

// ---- several meshes in one launch: global target g belongs to domain tdom[g] (local index tloc[g])
struct BatchTraceDom {
    TraceDom d;
    const float *fields;      // [T_d][n_v]
    float4 *rates;            // [T_d][n_t] (decisions are computed by the walk itself)
    int32_t max_steps, T;
};

__global__ void batch_rates_kernel(const BatchTraceDom *__restrict__ doms, const int32_t *__restrict__ tdom,
                                   const int32_t *__restrict__ tloc) {
    const int g = blockIdx.y;
    const BatchTraceDom q = doms[tdom[g]];
    const int a = tloc[g];
    const float *f = q.fields + (int64_t)a * q.d.n_v;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < q.d.n_t; t += (int64_t)gridDim.x * blockDim.x)
        q.rates[(int64_t)a * q.d.n_t + t] = tri_rates(q.d.gphi, q.d.rec, t, f);
}

// path id -> global target: id / S, or path_target[id] when sources per target vary
__global__ void __launch_bounds__(64) batch_trace_kernel(const BatchTraceDom *__restrict__ doms,
                                                        const int32_t *__restrict__ tdom,
                                                        const int32_t *__restrict__ tloc,
                                                        const int32_t *__restrict__ targets,
                                                        const int32_t *__restrict__ sources,
                                                        const int32_t *__restrict__ path_target, int64_t total,
                                                        int32_t S, int32_t max_pts, float2 *__restrict__ out_xy,
                                                        int32_t *__restrict__ out_len, int32_t *__restrict__ out_status) {
    const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool active = gid < total;         // padding lanes stay in the warp's walk loop, idle
    const int64_t id = active ? gid : 0;
    const int g = path_target ? path_target[id] : (int)(id / S);
    const BatchTraceDom q = doms[tdom[g]];
    const int a = tloc[g];
    trace_path(q.d, q.fields + (int64_t)a * q.d.n_v, q.rates + (int64_t)a * q.d.n_t, targets[g], sources[id],
               out_xy + id * max_pts, max_pts, q.max_steps, out_len + id, out_status + id, active);
}

TraceDom make_dom(const DevMesh &m) {
    TraceDom d;
    d.rec = m.trec;
    d.hrec = m.hrec;
    d.gphi = m.gphi;
    d.xy = m.xy;
    d.vt_off = m.vt_off;
    d.vt = m.vt;
    d.n_t = m.n_t;
    d.n_v = m.n_v;
    return d;
}

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

int32_t step_cap(const DevMesh &m) {
    const int64_t cap = 4 * m.n_t;
    return cap > (int64_t)INT32_MAX ? INT32_MAX : (int32_t)cap;
}

}  // namespace

size_t trace_scratch_bytes(const DevMesh &m, int32_t T, bool decisions) {
    return decisions ? align256((size_t)T * m.n_v * sizeof(float)) + align256((size_t)T * m.n_v * sizeof(VDec))
                     : align256((size_t)T * m.n_t * sizeof(float4));
}

// Vertex decisions for every (field, vertex) before the walk pay off when
// many paths share a field (they are reused) and share warps (a group that
// scans a fan holds up the others of its warp); with few each vertex state
// computes its own.  grid140, one target, 256 paths: the walk takes 119 us
// either way and the two passes 24; 71,681 vertices, 64 x 256 paths: 476 + 340
// us against 1,155.  DD_TRACE_DECISIONS=dense|lazy overrides the choice (for
// measurements).
bool trace_dense_decisions(int32_t T, int32_t S) {
    static int mode = -1;
    if (mode < 0) {
        const char *e = getenv("DD_TRACE_DECISIONS");
        mode = (e && !strcmp(e, "dense")) ? 1 : (e && !strcmp(e, "lazy")) ? 0 : 2;
    }
    return mode == 2 ? S >= kDenseMinPaths && (int64_t)T * S > kWarpPaths : mode == 1;
}

void launch_trace(const DevMesh &m, const float *fields, int64_t field_stride, const int32_t *targets,
                  const int32_t *sources, int32_t T, int32_t S, int32_t max_pts, float2 *out_xy, int32_t *out_len,
                  int32_t *out_status, void *scratch, cudaStream_t s) {
    const bool dense = trace_dense_decisions(T, S);
    TraceParams p;
    float *ft = dense ? reinterpret_cast<float *>(scratch) : nullptr;
    VDec *dec = dense ? reinterpret_cast<VDec *>(reinterpret_cast<char *>(scratch) +
                                                 align256((size_t)T * m.n_v * sizeof(float)))
                      : nullptr;
    p.d = make_dom(m);
    p.dec = dec;
    p.fields = fields;
    p.field_stride = field_stride;
    p.targets = targets;
    p.sources = sources;
    p.total = (int64_t)T * S;
    p.S = S;
    p.max_pts = max_pts;
    p.max_steps = step_cap(m);
    p.T = T;
    p.out_xy = out_xy;
    p.out_len = out_len;
    p.out_status = out_status;
    if (p.total == 0) return;
    if (dense) {
        // (a grid has at most 65,535 rows; here each has up to 65,504 groups of fields)
        auto by_fields = [&](int per_group, auto launch) {
            constexpr int64_t kRows = 65504;
            for (int64_t first = 0; first < T; first += kRows * per_group)
                launch((int32_t)first, (unsigned)std::min<int64_t>(kRows, (T - first + per_group - 1) / per_group));
        };
        by_fields(32, [&](int32_t first, unsigned rows) {
            KMark km_("fields_by_vertex_kernel", s);
            fields_by_vertex_kernel<<<dim3((unsigned)((m.n_v + 31) / 32), rows), 256, 0, s>>>(fields, field_stride,
                                                                                             m.n_v, T, first, ft);
        });
        by_fields(32, [&](int32_t first, unsigned rows) {
            KMark km_("vertex_decision_kernel", s);
            vertex_decision_kernel<<<dim3((unsigned)((m.n_v + 3) / 4), rows), 128, 0, s>>>(
                p.d, T, first, fields, field_stride, ft, targets, dec);
        });
        if (m.n_wide > 0)
            by_fields(4, [&](int32_t first, unsigned rows) {
                KMark km_("wide_decision_kernel", s);
                wide_decision_kernel<<<dim3((unsigned)m.n_wide, rows), 128, 0, s>>>(p.d, m.wide, T, first, fields,
                                                                                   field_stride, targets, dec);
            });
    }
    auto groups = [&](auto kern, int G) {
        KMark km_("trace_kernel", s);
        kern<<<(unsigned)((p.total * G + 63) / 64), 64, 0, s>>>(p);
    };
    // Lanes a path: a warp each while that leaves every scheduler at most four
    // warps (a path alone in its warp never waits for another's branch: 256
    // paths of grid140 119 us, against 134 with eight lanes and 153 with one),
    // then four (16,384 paths: 476 us; 1,340 with a warp each, issue-bound;
    // 493 with one lane), one where there are warps enough without
    if (p.total <= kWarpPaths)
        groups(trace_group_kernel<32>, 32);
    else if (p.total <= 16 * kWarpPaths)
        groups(trace_group_kernel<4>, 4);
    else
        groups(trace_group_kernel<1>, 1);
}

void launch_crossings(const DevMesh &m, cudaStream_t s) {
    if (m.n_t > 0) crossings_kernel<<<(unsigned)((4 * m.n_t + 255) / 256), 256, 0, s>>>(m.trec, m.gphi, m.n_t, m.hrec);
}

size_t batch_trace_dom_bytes() { return sizeof(BatchTraceDom); }

// host-side builder of one domain descriptor (into a byte buffer uploaded by the
// caller); scratch: trace_scratch_bytes(m, T) bytes of device memory
void fill_batch_trace_dom(void *dst, const DevMesh &m, const float *fields, int32_t T, void *scratch) {
    BatchTraceDom q;
    q.d = make_dom(m);
    q.fields = fields;
    q.rates = reinterpret_cast<float4 *>(scratch);
    q.max_steps = step_cap(m);
    q.T = T;
    std::memcpy(dst, &q, sizeof q);
}

void launch_batch_trace(const void *d_doms, const int32_t *d_tdom, const int32_t *d_tloc, const int32_t *d_targets,
                        const int32_t *d_sources, int32_t n_targets, int32_t S, int64_t max_nt, int64_t max_nv,
                        int32_t max_pts, float2 *out_xy, int32_t *out_len, int32_t *out_status, cudaStream_t s,
                        const int32_t *d_path_target, int64_t n_paths) {
    if (n_targets <= 0) return;
    const BatchTraceDom *doms = reinterpret_cast<const BatchTraceDom *>(d_doms);
    const int64_t total = d_path_target ? n_paths : (int64_t)n_targets * S;
    if (total == 0) return;
    dim3 gr((unsigned)std::max<int64_t>(1, std::min<int64_t>(64, (max_nt + 255) / 256)), (unsigned)n_targets);
    {
        KMark km_("batch_rates_kernel", s);
        batch_rates_kernel<<<gr, 256, 0, s>>>(doms, d_tdom, d_tloc);
    }
    (void)max_nv;
    {
        KMark km_("batch_trace_kernel", s);
        batch_trace_kernel<<<(unsigned)((total + 63) / 64), 64, 0, s>>>(doms, d_tdom, d_tloc, d_targets, d_sources,
                                                                        d_path_target, total, S, max_pts, out_xy, out_len,
                                                                        out_status);
    }
}

namespace {
// one warp per path: its first len points.  MODE 2: point pairs as 16-byte
// stores (rows 16-byte aligned at both ends); 1: one point (8 bytes) per
// store; 0: one float per store (any 4-byte aligned buffer).
template <int MODE>
__global__ void copy_paths_kernel(const float2 *__restrict__ src, const int32_t *__restrict__ len, int64_t n,
                                  int32_t max_pts, float2 *__restrict__ dst) {
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= n) return;
    const int L = min(max(len[w], 0), max_pts);
    const float2 *a = src + w * (int64_t)max_pts;
    float2 *b = dst + w * (int64_t)max_pts;
    if (MODE == 2) {
        const float4 *a4 = reinterpret_cast<const float4 *>(a);
        float4 *b4 = reinterpret_cast<float4 *>(b);
        for (int i = lane; 2 * i + 1 < L; i += 32) b4[i] = __ldcs(a4 + i);
        if ((L & 1) && lane == 0) b[L - 1] = a[L - 1];
    } else if (MODE == 1) {
        for (int i = lane; i < L; i += 32) b[i] = a[i];
    } else {
        const float *af = reinterpret_cast<const float *>(a);
        float *bf = reinterpret_cast<float *>(b);
        for (int i = lane; i < 2 * L; i += 32) bf[i] = af[i];
    }
}
}  // namespace

void launch_copy_paths(const float2 *src, const int32_t *len, int64_t n, int32_t max_pts, float2 *dst,
                       cudaStream_t s) {
    if (n <= 0) return;
    const uintptr_t d = reinterpret_cast<uintptr_t>(dst);
    const unsigned grid = (unsigned)((n + 7) / 8);
    KMark km_("copy_paths_kernel", s);
    if ((max_pts & 1) == 0 && (d & 15) == 0)
        copy_paths_kernel<2><<<grid, 256, 0, s>>>(src, len, n, max_pts, dst);
    else if ((d & 7) == 0)
        copy_paths_kernel<1><<<grid, 256, 0, s>>>(src, len, n, max_pts, dst);
    else
        copy_paths_kernel<0><<<grid, 256, 0, s>>>(src, len, n, max_pts, dst);
}

// ------------------------------------------------------------------ dependent-load latency
// The walk's floor is a chain of dependent gathers.  This measures the
// latency of one such gather: one thread follows a random cycle through a
// buffer, one 4-byte index at the head of every 128-byte line, each load's
// address the value of the one before (loads at L2, bypassing L1).
namespace {
// steps loads from the position *pos, which is left where the chase ended
__global__ void load_chase_kernel(const int32_t *__restrict__ a, int64_t steps, int32_t *__restrict__ pos) {
    int32_t j = *pos;
    for (int64_t i = 0; i < steps; ++i) j = __ldcg(a + j);
    *pos = j;
}
}  // namespace

dd_status measure_load_latency(int64_t bytes, int32_t steps, cudaStream_t s, double *ns, std::string &err) {
    const int64_t n = bytes / 128;            // lines
    // a single cycle over all lines in a seeded random order
    std::vector<int64_t> perm((size_t)n);
    for (int64_t i = 0; i < n; ++i) perm[(size_t)i] = i;
    std::mt19937_64 rng(0x5eedULL);
    for (int64_t i = n - 1; i > 0; --i) {
        const int64_t j = (int64_t)(rng() % (uint64_t)(i + 1));
        std::swap(perm[(size_t)i], perm[(size_t)j]);
    }
    std::vector<int32_t> next((size_t)n);
    for (int64_t i = 0; i < n; ++i) next[(size_t)perm[(size_t)i]] = (int32_t)(perm[(size_t)((i + 1) % n)] * 32);
    int32_t *d = nullptr, *sink = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    dd_status st = DD_OK;
    auto fail = [&](dd_status code, const char *what) {
        cudaGetLastError();
        err = what;
        st = code;
    };
    if (cudaMalloc(&d, (size_t)n * 128) != cudaSuccess || cudaMalloc(&sink, sizeof(int32_t)) != cudaSuccess) {
        fail(DD_ENOMEM, "allocation of the latency buffer failed");
    } else if (cudaMemcpy2DAsync(d, 128, next.data(), sizeof(int32_t), sizeof(int32_t), (size_t)n,
                                 cudaMemcpyHostToDevice, s) != cudaSuccess ||
               cudaMemsetAsync(sink, 0, sizeof(int32_t), s) != cudaSuccess ||
               cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        fail(DD_ECUDA, "latency buffer set-up failed");
    } else {
        // warm-up: the whole cycle when it is short (the timed loads then hit
        // L2), else its first 2^18 lines (the timed loads go on to lines not
        // yet visited)
        load_chase_kernel<<<1, 1, 0, s>>>(d, std::min<int64_t>(n, 1 << 18), sink);
        cudaEventRecord(e0, s);
        load_chase_kernel<<<1, 1, 0, s>>>(d, steps, sink);
        cudaEventRecord(e1, s);
        float ms = 0.f;
        if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess)
            fail(DD_ECUDA, "latency kernel failed");
        else
            *ns = (double)ms * 1e6 / steps;
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (d) cudaFree(d);
    if (sink) cudaFree(sink);
    return st;
}
