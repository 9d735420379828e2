// closestPoint and adjacentHyperplane for sm_103a (arXiv 2411.13507,
// Algorithm 2; Sec. III-D: the separating hyperplane between an MPC node and
// an obstacle).
//
// For a point v outside a convex obstacle O = {z : A z <= b} the closest
// point (the Euclidean projection onto O) lies in the relative interior of a
// face, on an edge, or at a vertex.  A prep step computes, in FP64 once per
// obstacle, every facet's unit normal and offset and every edge of O as a
// segment: a base point, a unit direction and the parameter interval the
// other facets leave (a facet or pair of facets with an empty interval is not
// a face or an edge; an unbounded edge keeps an infinite end).  Per (point,
// obstacle), in FP32: inside O (every row <= 0) -> distance 0; otherwise the
// nearest of the projections onto the faces that land inside O (m = 3; in 2-D
// the faces are the edges) and of the closest points of the edge segments
// (parameter clamped to its interval, which also covers the vertices).  Every
// candidate is a point of O, so the nearest one is the projection.  The
// segments come rounded from FP64, so the FP32 error does not grow with how
// sharp a vertex is (no linear solve happens per pair).  The plane:
// h = (v - z) / |v - z|, l = h . z.
#include <cuda_runtime.h>

#include <cstdint>

#include "plan_internal.h"

namespace plan {

namespace {

#define PDEV __device__ __forceinline__

constexpr float U32P = 5.9604644775390625e-08f;  // 2^-24
constexpr int EDGE_F4 = 4;  // float4 per edge record

PDEV void p_status(DevInfo* info, int code, int detail) {
    if (atomicCAS(&info->status, 0, code) == 0) atomicExch(&info->detail, detail);
}
PDEV bool p_failed(const DevInfo* info) { return *((volatile const int*)&info->status) != 0; }
PDEV float pld32(const void* p, long long i, int f32) {
    return f32 ? ((const float*)p)[i] : (float)((const double*)p)[i];
}

// Obstacle rows in 3-D as {A_0, A_1, A_2, b} (FP32, for the inside test),
// max_orows per obstacle, with row-count checks.
__global__ void k_planes_prep(PlanesParams Q) {
    after_stream<true>();
    const long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= (long long)Q.n_obst * Q.max_orows) return;
    const int o = (int)(u / Q.max_orows), k = (int)(u % Q.max_orows);
    const int r0 = Q.obst_off[o], nr = Q.obst_off[o + 1] - r0;
    if (nr < 0 || nr > Q.max_orows || r0 < 0 || (nr > 0 && (!Q.A || !Q.b))) {
        if (k == 0) p_status(Q.info, nr > Q.max_orows ? PLAN_ERR_UNSUPPORTED : PLAN_ERR_INVALID_ARG, DET_ROWS);
        if (k == 0) Q.ocount[o] = 0;
        return;
    }
    if (k == 0) Q.ocount[o] = nr;
    if (k < nr) {
        const long long r = r0 + k;
        float4 f;
        f.x = pld32(Q.A, r * 3, Q.in_f32);
        f.y = pld32(Q.A, r * 3 + 1, Q.in_f32);
        f.z = pld32(Q.A, r * 3 + 2, Q.in_f32);
        f.w = pld32(Q.b, r, Q.in_f32);
        reinterpret_cast<float4*>(Q.orow)[u] = f;
    }
}

PDEV double pld64(const void* p, long long i, int f32) {
    return f32 ? (double)((const float*)p)[i] : ((const double*)p)[i];
}

// The interval of t along z0 + t d in 3-D that every row leaves (t_lo > t_hi: none).
PDEV void clip_line(const PlanesParams& Q, int r0, int nr, const double* z0, const double* d, double& tlo, double& thi) {
    const double inf = __longlong_as_double(0x7FF0000000000000ll);
    tlo = -inf;
    thi = inf;
    for (int r = 0; r < nr; ++r) {
        double ad = 0.0, az = 0.0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double A = pld64(Q.A, (long long)(r0 + r) * 3 + a, Q.in_f32);
            ad = fma(A, d[a], ad);
            az = fma(A, z0[a], az);
        }
        const double slack = pld64(Q.b, r0 + r, Q.in_f32) - az;
        const double scale = fabs(pld64(Q.b, r0 + r, Q.in_f32)) + 1.0;
        if (fabs(ad) <= 1e-12) {
            if (slack < -1e-12 * scale) {  // parallel to the line and excluding it
                tlo = inf;
                thi = -inf;
            }
        } else if (ad > 0.0) {
            if (slack / ad < thi) thi = slack / ad;
        } else {
            if (slack / ad > tlo) tlo = slack / ad;
        }
    }
}

// Unit normal and offset of row r (FP64).
template <int M>
PDEV void unit_row(const PlanesParams& Q, int r0, int r, double* n, double& c) {
    double n2 = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) n[a] = 0.0;
#pragma unroll
    for (int a = 0; a < M; ++a) {
        n[a] = pld64(Q.A, (long long)(r0 + r) * M + a, Q.in_f32);
        n2 = fma(n[a], n[a], n2);
    }
    const double rn = n2 > 0.0 ? 1.0 / sqrt(n2) : 0.0;
#pragma unroll
    for (int a = 0; a < M; ++a) n[a] *= rn;
    c = pld64(Q.b, r0 + r, Q.in_f32) * rn;
}

// One warp per obstacle (3-D): faces (unit normal, offset) and edges,
// compacted; FP64, rounded to FP32 at the end.  Edge record (4 float4): base point and
// t_lo; unit direction and t_hi; the unit normals of its two facets.
__global__ void __launch_bounds__(128) k_planes_geom(PlanesParams Q) {
    after_stream<true>();
    constexpr int M = 3;
    const int lane = threadIdx.x & 31;
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long o = gw; o < Q.n_obst; o += nw) {
        const int r0 = Q.obst_off[o];
        int nr = Q.obst_off[o + 1] - r0;
        if (nr < 0 || nr > Q.max_orows || r0 < 0 || (nr > 0 && (!Q.A || !Q.b))) nr = 0;
        float4* face = reinterpret_cast<float4*>(Q.face) + o * Q.max_orows;
        float4* edge = reinterpret_cast<float4*>(Q.edge) + EDGE_F4 * o * Q.max_edges;
        // faces
        for (int r = lane; r < Q.max_orows; r += 32) {
            float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r < nr) {
                double A[3] = {0.0, 0.0, 0.0}, n2 = 0.0;
#pragma unroll
                for (int a = 0; a < M; ++a) {
                    A[a] = pld64(Q.A, (long long)(r0 + r) * M + a, Q.in_f32);
                    n2 = fma(A[a], A[a], n2);
                }
                const double rn = n2 > 0.0 ? 1.0 / sqrt(n2) : 0.0;
                f = make_float4((float)(A[0] * rn), (float)(A[1] * rn), (float)(A[2] * rn),
                                (float)(pld64(Q.b, r0 + r, Q.in_f32) * rn));
            }
            face[r] = f;
        }
        // edges: a pair of facets' line
        const int ncand = nr * nr;
        int count = 0;
        for (int c0 = 0; c0 < ncand; c0 += 32) {
            const int c = c0 + lane;
            bool ok = false;
            double z0[3] = {0.0, 0.0, 0.0}, d[3] = {0.0, 0.0, 0.0}, tlo = 0.0, thi = 0.0;
            int ra = -1, rb = -1;  // the edge's own facets
            if (c < ncand) {
                const int r1 = c / nr, r2 = c - r1 * nr;
                if (r1 < r2) {
                    double a[3], bq[3], b1, b2;
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        a[k] = pld64(Q.A, (long long)(r0 + r1) * 3 + k, Q.in_f32);
                        bq[k] = pld64(Q.A, (long long)(r0 + r2) * 3 + k, Q.in_f32);
                    }
                    b1 = pld64(Q.b, r0 + r1, Q.in_f32);
                    b2 = pld64(Q.b, r0 + r2, Q.in_f32);
                    double x[3] = {a[1] * bq[2] - a[2] * bq[1], a[2] * bq[0] - a[0] * bq[2], a[0] * bq[1] - a[1] * bq[0]};
                    const double xx = x[0] * x[0] + x[1] * x[1] + x[2] * x[2];
                    const double aa = a[0] * a[0] + a[1] * a[1] + a[2] * a[2];
                    const double bbq = bq[0] * bq[0] + bq[1] * bq[1] + bq[2] * bq[2];
                    if (xx > 1e-20 * aa * bbq) {
                        // z0 = alpha a + beta bq with a . z0 = b1, bq . z0 = b2
                        const double ab = a[0] * bq[0] + a[1] * bq[1] + a[2] * bq[2];
                        const double det = aa * bbq - ab * ab;
                        const double al = (b1 * bbq - b2 * ab) / det, be = (b2 * aa - b1 * ab) / det;
                        const double rx = 1.0 / sqrt(xx);
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            z0[k] = al * a[k] + be * bq[k];
                            d[k] = x[k] * rx;
                        }
                        ra = r1;
                        rb = r2;
                        ok = true;
                    }
                }
                if (ok) {
                    clip_line(Q, r0, nr, z0, d, tlo, thi);
                    ok = tlo <= thi;
                }
            }
            const unsigned bal = __ballot_sync(0xffffffffu, ok);
            const int slot = count + __popc(bal & ((1u << lane) - 1u));
            if (ok && slot < Q.max_edges) {
                float4* ed = edge + EDGE_F4 * slot;
                ed[0] = make_float4((float)z0[0], (float)z0[1], (float)z0[2], __double2float_rd(tlo));
                ed[1] = make_float4((float)d[0], (float)d[1], (float)d[2], __double2float_ru(thi));
                double na[3], nb[3], ca = 0.0, cb = 0.0;
                unit_row<M>(Q, r0, ra, na, ca);
                unit_row<M>(Q, r0, rb, nb, cb);
                ed[2] = make_float4((float)na[0], (float)na[1], (float)na[2], 0.f);
                ed[3] = make_float4((float)nb[0], (float)nb[1], (float)nb[2], 0.f);
            }
            count += __popc(bal);
        }
        if (lane == 0) {
            Q.nedge[o] = count < Q.max_edges ? count : Q.max_edges;
            if (count > Q.max_edges) p_status(Q.info, PLAN_ERR_UNSUPPORTED, DET_ROWS);
        }
    }
}

// The turn from an edge's normal a to the normal n of the row that ends it: its
// sign, or NaN where they do not span a cone (no row there, or parallel).
PDEV float turn(float ax, float ay, float nx, float ny) {
    const float kk = ax * ny - ay * nx;
    return kk > 0.f ? 1.f : (kk < 0.f ? -1.f : __int_as_float(0x7fc00000));
}

// The 2-D form of k_planes_prep and k_planes_geom in one launch: one warp per
// obstacle, four lanes per row (its line's clipping against the other rows and
// the three unit normals split over them), eight rows at a time.  A chain of
// FP64 instructions on a pipe that takes about 64 cycles for each of a warp's,
// so what counts is their number a lane: divisions by 2 rows instead of 7,
// one root instead of three (500 obstacles: 2.6 + 19 -> 12 us).  Edge record (4
// float4): base point, turn and t_lo; unit direction, turn and t_hi; the unit
// normals of the rows that end the segment at t_lo and t_hi (zero at an infinite
// end); the edge's own unit normal and offset.
__global__ void __launch_bounds__(128) k_planes_geom2(PlanesParams Q) {
    after_stream<true>();
    const int lane = threadIdx.x & 31, rs = lane & 3;
    const double inf = __longlong_as_double(0x7FF0000000000000ll);
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long o = gw; o < Q.n_obst; o += nw) {
        const int r0 = Q.obst_off[o];
        int nr = Q.obst_off[o + 1] - r0;
        if (nr < 0 || nr > Q.max_orows || r0 < 0 || (nr > 0 && (!Q.A || !Q.b))) {
            if (lane == 0) p_status(Q.info, nr > Q.max_orows ? PLAN_ERR_UNSUPPORTED : PLAN_ERR_INVALID_ARG, DET_ROWS);
            nr = 0;
        }
        float4* row = reinterpret_cast<float4*>(Q.orow) + o * Q.max_orows;
        float4* face = reinterpret_cast<float4*>(Q.face) + o * Q.max_orows;
        float4* edge = reinterpret_cast<float4*>(Q.edge) + EDGE_F4 * o * Q.max_edges;
        for (int r = nr + lane; r < Q.max_orows; r += 32) face[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        int count = 0;
        for (int c0 = 0; c0 < nr; c0 += 8) {
            const int c = c0 + (lane >> 2);
            bool ok = false;
            double z0[2] = {0.0, 0.0}, d[2] = {0.0, 0.0}, tlo = -inf, thi = inf;
            int rlo = -1, rhi = -1;
            if (c < nr) {
                const double a0 = pld64(Q.A, (long long)(r0 + c) * 2, Q.in_f32);
                const double a1 = pld64(Q.A, (long long)(r0 + c) * 2 + 1, Q.in_f32);
                const double n2 = a0 * a0 + a1 * a1;
                if (rs == 0)
                    row[c] = make_float4(pld32(Q.A, (long long)(r0 + c) * 2, Q.in_f32),
                                         pld32(Q.A, (long long)(r0 + c) * 2 + 1, Q.in_f32), 0.f, pld32(Q.b, r0 + c, Q.in_f32));
                if (n2 > 0.0) {
                    const double rn = 1.0 / sqrt(n2), bb = pld64(Q.b, r0 + c, Q.in_f32);
                    d[0] = -a1 * rn;
                    d[1] = a0 * rn;
                    z0[0] = a0 * bb / n2;   // the line's point nearest the origin
                    z0[1] = a1 * bb / n2;
                    ok = true;
                    for (int r = rs; r < nr; r += 4) {
                        double ad = 0.0, az = 0.0;
#pragma unroll
                        for (int a = 0; a < 2; ++a) {
                            const double A = pld64(Q.A, (long long)(r0 + r) * 2 + a, Q.in_f32);
                            ad = fma(A, d[a], ad);
                            az = fma(A, z0[a], az);
                        }
                        const double b = pld64(Q.b, r0 + r, Q.in_f32), slack = b - az;
                        if (fabs(ad) <= 1e-12) {
                            if (slack < -1e-12 * (fabs(b) + 1.0)) {  // parallel to the line and excluding it
                                tlo = inf;
                                thi = -inf;
                            }
                        } else {
                            const double t = slack / ad;
                            if (ad > 0.0) {
                                if (t < thi) {
                                    thi = t;
                                    rhi = r;
                                }
                            } else if (t > tlo) {
                                tlo = t;
                                rlo = r;
                            }
                        }
                    }
                }
            }
#pragma unroll
            for (int of = 1; of < 4; of <<= 1) {  // the four lanes' intervals; ties to the lower row, as in row order
                const double l2 = __shfl_xor_sync(0xffffffffu, tlo, of), h2 = __shfl_xor_sync(0xffffffffu, thi, of);
                const int rl2 = __shfl_xor_sync(0xffffffffu, rlo, of), rh2 = __shfl_xor_sync(0xffffffffu, rhi, of);
                if (l2 > tlo || (l2 == tlo && (unsigned)rl2 < (unsigned)rlo)) {
                    tlo = l2;
                    rlo = rl2;
                }
                if (h2 < thi || (h2 == thi && (unsigned)rh2 < (unsigned)rhi)) {
                    thi = h2;
                    rhi = rh2;
                }
            }
            ok = ok && tlo <= thi;
            const unsigned bal = __ballot_sync(0xffffffffu, ok && rs == 0);
            const int slot = count + __popc(bal & ((1u << (lane & ~3)) - 1u));
            // unit normals: lane 0 of the four the row's own, 1 and 2 of the rows at its ends (zero at an infinite end)
            double n[3] = {0.0, 0.0, 0.0}, cn = 0.0;
            const int rn_ = rs == 0 ? c : (rs == 1 ? rlo : rhi);
            if (c < nr && rs < 3 && rn_ >= 0) unit_row<2>(Q, r0, rn_, n, cn);
            const float nx = (float)n[0], ny = (float)n[1];
            const float hx = __shfl_down_sync(0xffffffffu, nx, 1), hy = __shfl_down_sync(0xffffffffu, ny, 1);
            const float lx = hx, ly = hy;  // in lane 0 of the four: the normals at t_lo, t_hi
            const float gx = __shfl_down_sync(0xffffffffu, nx, 2), gy = __shfl_down_sync(0xffffffffu, ny, 2);
            if (c < nr && rs == 0) face[c] = make_float4(nx, ny, 0.f, (float)cn);
            if (ok && slot < Q.max_edges) {
                float4* ed = edge + EDGE_F4 * slot;
                if (rs == 0) {
                    ed[0] = make_float4((float)z0[0], (float)z0[1], turn(nx, ny, lx, ly), __double2float_rd(tlo));
                    ed[1] = make_float4((float)d[0], (float)d[1], turn(nx, ny, gx, gy), __double2float_ru(thi));
                    ed[3] = make_float4(nx, ny, (float)cn, 0.f);
                } else if (rs == 1) {
                    ed[2] = make_float4(nx, ny, hx, hy);
                }
            }
            count += __popc(bal);
        }
        if (lane == 0) {
            Q.ocount[o] = nr;
            Q.nedge[o] = count < Q.max_edges ? count : Q.max_edges;
            if (count > Q.max_edges) p_status(Q.info, PLAN_ERR_UNSUPPORTED, DET_ROWS);
        }
    }
}

template <int M>
PDEV float pdot(const float4& f, const float* z) {
    float s = f.x * z[0];
    s = fmaf(f.y, z[1], s);
    if (M == 3) s = fmaf(f.z, z[2], s);
    return s;
}

// Nearest-only mode, pass A: per point an upper bound of its nearest
// obstacle's distance -- the distance to one vertex (the first edge's start)
// of every obstacle, min-reduced (non-negative floats order as their bits).
template <int M>
__global__ void __launch_bounds__(256) k_planes_ub(PlanesParams Q) {
    after_stream<false>();
    const long long total = (long long)Q.P * Q.n_obst;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    for (long long base = (long long)blockIdx.x * blockDim.x; base < total; base += stride) {
        const long long k = base + threadIdx.x;
        const bool act = k < total;
        long long p = 0;
        unsigned ub = 0x7f7f7f7fu;
        if (act) {
            p = k / Q.n_obst;
            const int o = (int)(k - p * Q.n_obst);
            const float4* ew = reinterpret_cast<const float4*>(Q.edge) + EDGE_F4 * (long long)o * Q.max_edges;
            if (Q.nedge[o] >= 1) {
                const float4 e0 = __ldg(ew), e1 = __ldg(ew + 1);
                if (fabsf(e0.w) < 3.0e38f) {   // an unbounded edge has no start vertex
                    float d2 = 0.f;
#pragma unroll
                    for (int a = 0; a < M; ++a) {
                        const float c = fmaf(e0.w, a == 0 ? e1.x : (a == 1 ? e1.y : e1.z),
                                             a == 0 ? e0.x : (a == 1 ? e0.y : e0.z));
                        const float t = pld32(Q.points, p * M + a, Q.in_f32) - c;
                        d2 = fmaf(t, t, d2);
                    }
                    ub = __float_as_uint(sqrtf(d2));
                }
            }
        }
        // lanes of one point are consecutive obstacles: one atomic per run
        const long long p0 = __shfl_sync(0xffffffffu, p, 0), p31 = __shfl_sync(0xffffffffu, p, 31);
        if (p0 == p31 && __all_sync(0xffffffffu, act)) {
            for (int of = 16; of > 0; of >>= 1) ub = min(ub, __shfl_xor_sync(0xffffffffu, ub, of));
            if (lane == 0) atomicMin(reinterpret_cast<unsigned*>(Q.ub) + p, ub);
        } else if (act && ub != 0x7f7f7f7fu) {
            atomicMin(reinterpret_cast<unsigned*>(Q.ub) + p, ub);
        }
    }
}

// One obstacle's rows, faces and edges: in global memory, or (SH) in shared
// memory with `stride` float4 from one entry of an obstacle to its next.
template <bool SH>
struct Geom {
    const float4 *rows, *faces, *edges;
    int stride, nr, ne;
    PDEV float4 at(const float4* p, int i) const { return SH ? p[i * stride] : __ldg(p + i); }
    PDEV float4 row(int r) const { return at(rows, r); }
    PDEV float4 face_of(int r) const { return at(faces, r); }
    PDEV float4 edge_of(int e, int i) const { return at(edges, EDGE_F4 * e + i); }
};

// The point z of a 2-D obstacle nearest to each of NP points v, and its
// squared distance (0 and v itself inside; infinite without an edge): the
// first edge segment that holds it by sign tests, else the nearest candidate.
// A segment whose parameter needs no clamping and whose facet v lies outside of
// holds the projection; a vertex does when v - vertex lies in the cone of its
// two facet normals.  Without a branch: the lanes of a warp (one obstacle
// each) settle on different edges, so every edge is run anyway.
template <bool SH, int NP>
PDEV void closest_2d(const float (&v)[NP][2], const Geom<SH>& geo, float (&z)[NP][2], float (&d2)[NP]) {
    const float inf = __int_as_float(0x7f800000);
    bool in[NP], found[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) in[i] = true;
    for (int r = 0; r < geo.nr; ++r) {
        const float4 f = geo.row(r);
#pragma unroll
        for (int i = 0; i < NP; ++i) in[i] = in[i] & (pdot<2>(f, v[i]) - f.w <= 0.f);
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        z[i][0] = v[i][0];
        z[i][1] = v[i][1];
        d2[i] = in[i] ? 0.f : inf;
        found[i] = in[i];
    }
    for (int e = 0; e < geo.ne; ++e) {
        const float4 e0 = geo.edge_of(e, 0), e1 = geo.edge_of(e, 1), e2 = geo.edge_of(e, 2), e3 = geo.edge_of(e, 3);
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            float t = e1.x * (v[i][0] - e0.x);
            t = fmaf(e1.y, v[i][1] - e0.y, t);
            const float tc = fminf(fmaxf(t, e0.w), e1.w);
            const float cx = fmaf(tc, e1.x, e0.x), cy = fmaf(tc, e1.y, e0.y);
            const float wx = v[i][0] - cx, wy = v[i][1] - cy;
            const float dd = fmaf(wy, wy, wx * wx);
            const float sd = fmaf(e3.y, v[i][1], e3.x * v[i][0]) - e3.z;  // outside this facet?
            // a clamped end: v - c in the cone of the two normals, whose turn sg is (NaN: no vertex there)
            const bool lo = t < e0.w;
            const float nx = lo ? e2.x : e2.z, ny = lo ? e2.y : e2.w, sg = lo ? e0.z : e1.z;
            const bool cone = ((e3.x * wy - e3.y * wx) * sg >= 0.f) & ((wx * ny - wy * nx) * sg >= 0.f);
            const bool hit = tc == t ? sd > 0.f : cone;
            const bool take = !found[i] & (hit | (dd < d2[i]));
            found[i] |= hit;
            if (take) {
                d2[i] = dd;
                z[i][0] = cx;
                z[i][1] = cy;
            }
        }
    }
}

// The point z of a 3-D obstacle nearest to v and its squared distance (0 and v
// itself inside; infinite for an obstacle without a face or an edge).
PDEV void closest_3d(const float (&v)[3], const Geom<false>& geo, float (&z)[3], float& d2) {
    const float inf = __int_as_float(0x7f800000);
    const int nr = geo.nr;
    bool in = true;
    for (int r = 0; r < nr; ++r) {
        const float4 f = geo.row(r);
        in = in & (pdot<3>(f, v) - f.w <= 0.f);
    }
    d2 = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) z[a] = v[a];
    if (in) return;
    d2 = inf;
    for (int r = 0; r < nr; ++r) {  // faces whose projection lands inside the obstacle
        const float4 f = geo.face_of(r);
        const float sd = pdot<3>(f, v) - f.w;
        if (!(sd > 0.f) || sd * sd >= d2) continue;
        float c[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) c[a] = fmaf(-sd, a == 0 ? f.x : (a == 1 ? f.y : f.z), v[a]);
        bool ok = true;
        for (int q = 0; q < nr; ++q) {
            if (q == r) continue;
            const float4 g = geo.row(q);
            const float sv = pdot<3>(g, c) - g.w;
            const float mag = fabsf(g.x * c[0]) + fabsf(g.y * c[1]) + fabsf(g.z * c[2]) + fabsf(g.w);
            ok = ok && sv <= 8.f * U32P * mag;
        }
        if (ok) {
            d2 = sd * sd;
#pragma unroll
            for (int a = 0; a < 3; ++a) z[a] = c[a];
        }
    }
    // edge segments (and their end points, the vertices).  The
    // candidate is chosen by sign tests, not by comparing nearly
    // equal distances: a segment whose parameter needs no clamping
    // holds the projection.  The nearest candidate is the fallback
    // for what rounding leaves undecided.
    const int ne = geo.ne;
    bool found = false;
    float fb_d2 = inf, fb[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) fb[a] = v[a];
    for (int e = 0; e < ne && !found && !(d2 < inf); ++e) {
        const float4 e0 = geo.edge_of(e, 0), e1 = geo.edge_of(e, 1);
        const float w[3] = {v[0] - e0.x, v[1] - e0.y, v[2] - e0.z};
        float t = e1.x * w[0];
        t = fmaf(e1.y, w[1], t);
        t = fmaf(e1.z, w[2], t);
        const float tc = fminf(fmaxf(t, e0.w), e1.w);
        float c[3], dd = 0.f;
        c[0] = fmaf(tc, e1.x, e0.x);
        c[1] = fmaf(tc, e1.y, e0.y);
        c[2] = fmaf(tc, e1.z, e0.z);
#pragma unroll
        for (int a = 0; a < 3; ++a) dd = fmaf(v[a] - c[a], v[a] - c[a], dd);
        // an unclamped point of an edge whose two facet normals span v - c
        bool hit = false;
        if (tc == t) {
            const float4 e2 = geo.edge_of(e, 2), e3 = geo.edge_of(e, 3);
            const float wx = v[0] - c[0], wy = v[1] - c[1], wz = v[2] - c[2];
            // signs of (n_a x w) . d, (w x n_b) . d and (n_a x n_b) . d
            const float k1 = (e2.y * wz - e2.z * wy) * e1.x + (e2.z * wx - e2.x * wz) * e1.y +
                             (e2.x * wy - e2.y * wx) * e1.z;
            const float k2 = (wy * e3.z - wz * e3.y) * e1.x + (wz * e3.x - wx * e3.z) * e1.y +
                             (wx * e3.y - wy * e3.x) * e1.z;
            float kk = (e2.y * e3.z - e2.z * e3.y) * e1.x + (e2.z * e3.x - e2.x * e3.z) * e1.y +
                       (e2.x * e3.y - e2.y * e3.x) * e1.z;
            float s1 = k1, s2 = k2;
            if (kk < 0.f) {
                s1 = -s1;
                s2 = -s2;
                kk = -kk;
            }
            hit = kk > 0.f && s1 >= 0.f && s2 >= 0.f;
        }
        if (hit) {
            found = true;
            d2 = dd;
#pragma unroll
            for (int a = 0; a < 3; ++a) z[a] = c[a];
        } else if (dd < fb_d2) {
            fb_d2 = dd;
#pragma unroll
            for (int a = 0; a < 3; ++a) fb[a] = c[a];
        }
    }
    if (!found && fb_d2 < d2) {
        d2 = fb_d2;
#pragma unroll
        for (int a = 0; a < 3; ++a) z[a] = fb[a];
    }
}

// Either dimension, one point, from global memory.
template <int M>
PDEV void pair_closest(const float (&v)[M], const Geom<false>& geo, float (&z)[M], float& d2) {
    if constexpr (M == 2) {
        const float v1[1][2] = {{v[0], v[1]}};
        float z1[1][2], d1[1];
        closest_2d<false, 1>(v1, geo, z1, d1);
        z[0] = z1[0][0];
        z[1] = z1[0][1];
        d2 = d1[0];
    } else {
        closest_3d(v, geo, z, d2);
    }
}

// One thread per (point, obstacle), the obstacle index fastest (coalesced
// stores of the point-major outputs); per point the nearest obstacle as a
// 64-bit key (distance bits << 32 | obstacle), min-reduced per warp first.
template <int M>
__global__ void __launch_bounds__(256) k_planes(PlanesParams Q) {
    after_stream<false>();
    __shared__ int s_fail;
    if (threadIdx.x == 0) s_fail = p_failed(Q.info);
    __syncthreads();
    if (s_fail) return;
    const long long total = Q.pair_obst ? (long long)Q.P : (long long)Q.P * Q.n_obst;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    const float inf = __int_as_float(0x7f800000);
    for (long long base = (long long)blockIdx.x * blockDim.x; base < total; base += stride) {
        const long long k = base + threadIdx.x;
        const bool act = k < total;
        long long p = 0;
        int o = 0;
        unsigned long long key = ~0ull;
        if (act && Q.pair_obst) {  // pair mode (no keys): the given obstacle of point k
            p = k;
            o = Q.pair_obst[k];
            if (o < 0 || o >= Q.n_obst) {
                if (Q.plane)
                    for (int a = 0; a <= M; ++a) Q.plane[k * (M + 1) + a] = 0.f;
                if (Q.dist) Q.dist[k] = inf;
                continue;
            }
        } else if (act) {
            p = k / Q.n_obst;
            o = (int)(k - p * Q.n_obst);
        }
        bool pruned = false;
        if (act && Q.ub) {
            // nearest-only mode: an obstacle whose distance lower bound (the
            // largest signed distance to one of its facet planes) exceeds the
            // point's upper bound (with room for float rounding) cannot be
            // the nearest, nor tie with it
            float v[M], vs = 1.f;
#pragma unroll
            for (int a = 0; a < M; ++a) {
                v[a] = pld32(Q.points, p * M + a, Q.in_f32);
                vs += fabsf(v[a]);
            }
            const int nr = Q.ocount[o];
            const float4* fw = reinterpret_cast<const float4*>(Q.face) + (long long)o * Q.max_orows;
            float lb = -inf;
            for (int r = 0; r < nr; ++r) {
                const float4 f = __ldg(fw + r);
                lb = fmaxf(lb, pdot<M>(f, v) - f.w);
            }
            const float ub = Q.ub[p];
            pruned = lb > fmaf(ub, 1.00001f, 1e-5f * vs);
        }
        if (act && !pruned) {
            float v[M];
#pragma unroll
            for (int a = 0; a < M; ++a) v[a] = pld32(Q.points, p * M + a, Q.in_f32);
            const long long oo = o;
            const Geom<false> geo = {reinterpret_cast<const float4*>(Q.orow) + oo * Q.max_orows,
                                     reinterpret_cast<const float4*>(Q.face) + oo * Q.max_orows,
                                     reinterpret_cast<const float4*>(Q.edge) + EDGE_F4 * oo * Q.max_edges,
                                     1, Q.ocount[o], Q.nedge[o]};
            float z[M], d2;
            pair_closest<M>(v, geo, z, d2);
            const float d = sqrtf(d2);
            if (Q.closest)
#pragma unroll
                for (int a = 0; a < M; ++a) Q.closest[k * M + a] = d2 < inf ? z[a] : __int_as_float(0x7fc00000);
            if (Q.dist) Q.dist[k] = d;
            if (Q.plane) {
                const float rdn = (d > 0.f && d < inf) ? 1.f / d : 0.f;
                float l = 0.f;
#pragma unroll
                for (int a = 0; a < M; ++a) {
                    const float h = (v[a] - z[a]) * rdn;
                    Q.plane[k * (M + 1) + a] = h;
                    l = fmaf(h, z[a], l);
                }
                Q.plane[k * (M + 1) + M] = l;
            }
            key = ((unsigned long long)__float_as_uint(d) << 32) | (unsigned)o;
        }
        if (Q.keys) {
            // lanes of one point are consecutive obstacles: reduce runs of the same point
            const long long p0 = __shfl_sync(0xffffffffu, p, 0), p31 = __shfl_sync(0xffffffffu, p, 31);
            if (p0 == p31 && __all_sync(0xffffffffu, act)) {
                unsigned long long kk = key;
                for (int of = 16; of > 0; of >>= 1) {
                    const unsigned long long ok = __shfl_xor_sync(0xffffffffu, kk, of);
                    kk = ok < kk ? ok : kk;
                }
                if (lane == 0) atomicMin(Q.keys + p, kk);
            } else if (act && !pruned) {
                atomicMin(Q.keys + p, key);
            }
        }
    }
}

// All pairs in 2-D, by blocks of up to 128 obstacles whose geometry stays in
// shared memory while groups of as many threads take the points of a chunk in
// turn (one thread an obstacle, so a point's outputs are stored coalesced).
// Read per pair from global memory, the 32 obstacles of a warp take 32 lines
// a load, and those loads bounded the kernel (5000 points x 500 obstacles:
// 71 us); from shared memory, laid out [entry][obstacle] with one float4 of
// padding, a load is conflict-free: 53 us, bound by issue (43.8 M warp
// instructions, 560 a warp of pairs; 70% issue active, 32% of the warps).  Same
// arithmetic and results.
constexpr int PL_THREADS = 384, PL_NP = 4;

__global__ void __launch_bounds__(PL_THREADS, 2) k_planes_all(PlanesParams Q, int ob, int chunk) {
    after_stream<false>();
    extern __shared__ float4 geo_sm[];
    __shared__ int s_fail;
    const int tid = threadIdx.x, lane = tid & 31, stride = ob + 1, n4 = Q.max_orows + EDGE_F4 * Q.max_edges;
    if (tid == 0) s_fail = p_failed(Q.info);
    const int o0 = blockIdx.x * ob, nob = min(ob, Q.n_obst - o0);
    const float4* rw = reinterpret_cast<const float4*>(Q.orow) + (long long)o0 * Q.max_orows;
    const float4* ew = reinterpret_cast<const float4*>(Q.edge) + EDGE_F4 * (long long)o0 * Q.max_edges;
    for (int u = tid; u < nob * n4; u += PL_THREADS) {
        const int lo = u / n4, j = u - lo * n4, e = j - Q.max_orows;
        geo_sm[j * stride + lo] = e < 0 ? rw[lo * Q.max_orows + j] : ew[lo * EDGE_F4 * Q.max_edges + e];
    }
    const int groups = PL_THREADS / ob, g = tid / ob, lo = tid - g * ob, o = o0 + lo;
    const bool act = lo < nob && g < groups;
    Geom<true> geo = {geo_sm + lo, nullptr, geo_sm + Q.max_orows * stride + lo, stride, 0, 0};
    if (act) {
        geo.nr = Q.ocount[o];
        geo.ne = Q.nedge[o];
    }
    __syncthreads();
    if (s_fail || g >= groups) return;  // whole warps: ob is a multiple of 32
    const float inf = __int_as_float(0x7f800000);
    const bool pair_aligned = ((uintptr_t)Q.closest & 7) == 0, whole = __all_sync(0xffffffffu, act);
    const int p1 = (int)min((long long)Q.P, ((long long)blockIdx.y + 1) * chunk);
    for (int pb = blockIdx.y * chunk + g; pb < p1; pb += groups * PL_NP) {
        float v[PL_NP][2], z[PL_NP][2], d2[PL_NP];
#pragma unroll
        for (int i = 0; i < PL_NP; ++i) {
            const long long p = min(pb + i * groups, p1 - 1);
            v[i][0] = pld32(Q.points, p * 2, Q.in_f32);
            v[i][1] = pld32(Q.points, p * 2 + 1, Q.in_f32);
        }
        if (act) closest_2d<true, PL_NP>(v, geo, z, d2);
#pragma unroll
        for (int i = 0; i < PL_NP; ++i) {
            const int p = pb + i * groups;
            if (p >= p1) break;  // warp-uniform
            const long long k = (long long)p * Q.n_obst + o;
            unsigned bits = 0xffffffffu;
            float h[2] = {0.f, 0.f}, l = 0.f;
            if (act) {
                const float d = sqrtf(d2[i]);
                if (Q.closest) {
                    const float nan = __int_as_float(0x7fc00000);
                    const float2 c = d2[i] < inf ? make_float2(z[i][0], z[i][1]) : make_float2(nan, nan);
                    if (pair_aligned) {
                        reinterpret_cast<float2*>(Q.closest)[k] = c;
                    } else {
                        Q.closest[2 * k] = c.x;
                        Q.closest[2 * k + 1] = c.y;
                    }
                }
                if (Q.dist) Q.dist[k] = d;
                const float rdn = (d > 0.f && d < inf) ? 1.f / d : 0.f;
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    h[a] = (v[i][a] - z[i][a]) * rdn;
                    l = fmaf(h[a], z[i][a], l);
                }
                bits = __float_as_uint(d);
            }
            if (Q.plane) {
                if (whole) {  // 96 words of the warp, exchanged for coalesced stores
                    float* out = Q.plane + 3 * (k - lane);
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        const int w = 32 * q + lane, src = w / 3, c = w - 3 * src;
                        const float x0 = __shfl_sync(0xffffffffu, h[0], src), x1 = __shfl_sync(0xffffffffu, h[1], src);
                        const float x2 = __shfl_sync(0xffffffffu, l, src);
                        out[w] = c == 0 ? x0 : (c == 1 ? x1 : x2);
                    }
                } else if (act) {
                    Q.plane[3 * k] = h[0];
                    Q.plane[3 * k + 1] = h[1];
                    Q.plane[3 * k + 2] = l;
                }
            }
            if (Q.keys) {
                const unsigned mn = __reduce_min_sync(0xffffffffu, bits);
                const unsigned who = __ballot_sync(0xffffffffu, act && bits == mn);  // the lowest lane is the lowest obstacle
                if (who && lane == __ffs(who) - 1) atomicMin(Q.keys + p, ((unsigned long long)mn << 32) | (unsigned)o);
            }
        }
    }
}

__global__ void k_planes_nearest(PlanesParams Q) {
    after_stream<true>();
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= Q.P || p_failed(Q.info)) return;
    const unsigned long long key = Q.keys[p];
    const bool none = key == ~0ull;
    if (Q.nearest) Q.nearest[p] = none ? -1 : (int32_t)(key & 0xffffffffu);
    if (Q.nearest_dist) Q.nearest_dist[p] = none ? __int_as_float(0x7f800000) : __uint_as_float((unsigned)(key >> 32));
}

}  // namespace

int launch_planes(const PlanesParams& Q, void* stream, int num_sms, int* launches) {
    cudaStream_t st = (cudaStream_t)stream;
    const long long orows = (long long)Q.n_obst * Q.max_orows;
    if (orows > 0) {
        if (Q.m == 2) {
            launch_next(k_planes_geom2, dim3((Q.n_obst + 3) / 4), dim3(128), 0, st, Q);
        } else {
            launch_next(k_planes_prep, dim3((int)((orows + 255) / 256)), dim3(256), 0, st, Q);
            launch_next(k_planes_geom, dim3((Q.n_obst + 3) / 4), dim3(128), 0, st, Q);
            ++*launches;
        }
        ++*launches;
    }
    const long long total = (long long)Q.P * Q.n_obst;
    if (total > 0) {
        long long grid = (total + 255) / 256;
        if (grid > (long long)num_sms * 16) grid = (long long)num_sms * 16;
        if (Q.ub) {
            if (Q.m == 2) launch_next(k_planes_ub<2>, dim3((int)grid), dim3(256), 0, st, Q);
            else launch_next(k_planes_ub<3>, dim3((int)grid), dim3(256), 0, st, Q);
            ++*launches;
        }
        // all pairs in 2-D: obstacles in blocks of whole warps, and as many
        // chunks of points as fill the GPU once.  Not where a block would be
        // alone on an SM (the most rows) or a warp mostly empty (few obstacles).
        const int ob = Q.n_obst >= 128 ? 128 : (Q.n_obst + 31) & ~31;
        const size_t smem = sizeof(float4) * (size_t)(ob + 1) * (Q.max_orows + EDGE_F4 * Q.max_edges);
        const int fit = (int)(220 * 1024 / (smem + 2 * 1024));
        if (Q.m == 2 && !Q.ub && Q.n_obst >= 24 && fit >= 2) {
            const cudaError_t ea = allow_shared<k_planes_all>();
            if (ea != cudaSuccess) return (int)ea;
            const int nb = (Q.n_obst + ob - 1) / ob, groups = PL_THREADS / ob;
            long long chunks = (2LL * num_sms + nb - 1) / nb;
            const long long most = (Q.P + groups * PL_NP - 1) / (groups * PL_NP);
            if (chunks > most) chunks = most;
            if (chunks > 65535) chunks = 65535;
            const int chunk = (int)((Q.P + chunks - 1) / chunks);
            launch_next(k_planes_all, dim3((unsigned)nb, (unsigned)((Q.P + chunk - 1) / chunk)), dim3(PL_THREADS), smem, st, Q, ob, chunk);
        } else if (Q.m == 2) {
            launch_next(k_planes<2>, dim3((int)grid), dim3(256), 0, st, Q);
        } else {
            launch_next(k_planes<3>, dim3((int)grid), dim3(256), 0, st, Q);
        }
        ++*launches;
    }
    if (Q.P > 0 && (Q.nearest || Q.nearest_dist)) {
        launch_next(k_planes_nearest, dim3((int)((Q.P + 255) / 256)), dim3(256), 0, st, Q);
        ++*launches;
    }
    if (Q.P > 0 && Q.nearest_plane && Q.nearest) {
        // the plane of each point's nearest obstacle: the same per-pair work
        // for the pairs (p, nearest[p]) only
        PlanesParams Q2 = Q;
        Q2.pair_obst = Q.nearest;
        Q2.closest = nullptr;
        Q2.dist = nullptr;
        Q2.plane = Q.nearest_plane;
        Q2.keys = nullptr;
        Q2.ub = nullptr;
        Q2.nearest = nullptr;
        Q2.nearest_dist = nullptr;
        long long grid = (Q.P + 255) / 256;
        if (grid > (long long)num_sms * 16) grid = (long long)num_sms * 16;
        if (Q.m == 2) launch_next(k_planes<2>, dim3((int)grid), dim3(256), 0, st, Q2);
        else launch_next(k_planes<3>, dim3((int)grid), dim3(256), 0, st, Q2);
        ++*launches;
    }
    return (int)cudaGetLastError();
}

}  // namespace plan
