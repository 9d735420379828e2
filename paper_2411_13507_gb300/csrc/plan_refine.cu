// Differentiable refinement objective for sm_103a: M threads per Bezier
// segment (one an axis of the reach margins and the snap energy, and two of
// the interior control points of the free margins), forward (loss) and
// hand-written backward (d loss / d control points and d loss / d T) of
//
//   loss = w_snap J_snap + mu sum_r phi_delta(margin_r)
//
// with the reach margins c_k -/+ Q^(k)_j (Theorem 1 read per axis on the
// hodograph control points Q^(k)_j = p!/(p-k)! T^-k Delta^k P_j), the free
// margins b_r - A_r P_l of the interior control points (Property 1), the
// relaxed log-barrier phi_delta (-log m above delta, its C^2 quadratic
// extension below) and the snap energy
//   J_snap = (p!/(p-4)!)^2 T^-7 sum_jl G_jl <Delta^4 P_j, Delta^4 P_l>,
//   G_jl = C(q,j) C(q,l) / ((2q+1) C(2q,j+l)),  q = p-4,
// the exact integral of ||b''''||^2 over [0, T].  The backward pass applies
// the adjoint of the forward-difference operator (x_l = g_{l-1} - g_l) to the
// margin and snap gradients.
#include <cuda_runtime.h>

#include <cstdint>

#include "plan_internal.h"

namespace plan {

#define DEVI __device__ __forceinline__

namespace {

// The relaxed barrier's constants: value and slope of the quadratic below delta.
struct Barrier {
    float delta, inv, off;  // delta, 1 / delta, -log delta - 1/2
};

// phi(m) and, with GRAD, phi'(m) of one margin.
template <bool GRAD>
DEVI float phi_one(const Barrier& B, float m, float& slope) {
    const bool in = m >= B.delta;
    const float z = (m - 2.f * B.delta) * B.inv;
    if (GRAD) slope = in ? -1.f / m : z * B.inv;  // not / delta^2, which underflows first
    return in ? -logf(m) : fmaf(0.5f * z, z, B.off);
}

// phi(c - Q) + phi(c + Q) and its derivative in Q.  Both margins in the
// logarithm share one root of work: log m1 + log m2 = log(m1 m2), and the two
// reciprocals come from one.  m1 + m2 = 2 c and both are at least delta, so the
// product lies between c delta and c^2: in range for bounds below 2^60 with
// c delta above 2^-125; others take the margins one by one.
template <bool GRAD>
DEVI float phi_pair(const Barrier& B, float c, float Q, float& slope) {
    const float m1 = c - Q, m2 = c + Q;
    if (c > 1.152921504606847e18f || c * B.delta < 2.350988701644575e-38f) {
        float s1 = 0.f, s2 = 0.f;
        const float v = phi_one<GRAD>(B, m1, s1) + phi_one<GRAD>(B, m2, s2);
        if (GRAD) slope = s2 - s1;
        return v;
    }
    const bool in1 = m1 >= B.delta, in2 = m2 >= B.delta;
    const float u1 = in1 ? m1 : 1.f, u2 = in2 ? m2 : 1.f, pr = u1 * u2;
    const float z1 = (m1 - 2.f * B.delta) * B.inv, z2 = (m2 - 2.f * B.delta) * B.inv;
    float v = -logf(pr);
    v += in1 ? 0.f : fmaf(0.5f * z1, z1, B.off);
    v += in2 ? 0.f : fmaf(0.5f * z2, z2, B.off);
    if (GRAD) {
        const float r = 1.f / pr;
        const float s1 = in1 ? -r * u2 : z1 * B.inv, s2 = in2 ? -r * u1 : z2 * B.inv;
        slope = s2 - s1;
    }
    return v;
}

// Constants of degree PD, formed at compile time: kept as an object, because a
// constexpr function called in an unrolled loop is compiled as a call.
template <int PD>
struct RefineConst {
    float scale[5];               // p! / (p-k)!, k = 0 .. 4
    float gram[PD - 3][PD - 3];   // C(q,j) C(q,l) / ((2q+1) C(2q,j+l)), q = PD - 4
};
template <int PD>
constexpr RefineConst<PD> refine_const() {
    RefineConst<PD> c{};
    c.scale[0] = 1.f;
    for (int k = 1; k <= 4; ++k) c.scale[k] = c.scale[k - 1] * (float)(PD - k + 1);
    constexpr int q = PD - 4;
    long long C[2 * q + 1][2 * q + 1] = {};
    for (int n = 0; n <= 2 * q; ++n)
        for (int k = 0; k <= n; ++k) C[n][k] = (k == 0 || k == n) ? 1 : C[n - 1][k - 1] + C[n - 1][k];
    for (int j = 0; j <= q; ++j)
        for (int l = 0; l <= q; ++l) c.gram[j][l] = (float)(C[q][j] * C[q][l]) / (float)((2 * q + 1) * C[2 * q][j + l]);
    return c;
}

template <int L>
DEVI void fwd_diff(float (&d)[L], int len) {  // d[0..len-2] = d[j+1] - d[j]
#pragma unroll
    for (int j = 0; j < L - 1; ++j)
        if (j < len - 1) d[j] = d[j + 1] - d[j];
}

// adjoint of the forward difference: g has `len` entries -> len+1 entries
template <int L>
DEVI void adj_diff(float (&g)[L], int len) {
    float prev = 0.f;
#pragma unroll
    for (int l = 0; l < L; ++l)
        if (l <= len) {
            const float cur = l < len ? g[l] : 0.f;
            g[l] = prev - cur;
            prev = cur;
        }
}

}  // namespace

// A CTA takes RF_SEGS consecutive segments: their control points, rows and
// bounds come in coalesced (each a contiguous run of the input), and the
// gradients go out the same way, all through shared memory (per-segment
// strides odd, so that threads of different segments hit different banks).
//
// One thread a segment took 59 us forward and 80 us backward for 65,536 3-D
// segments: 2048 warps waited for strided loads, and the snap energy's
// binomials were formed by recursive calls at run time (a third of all
// instructions and most of the memory traffic, to the call stack).  M threads a
// segment balance (18 reach rows and 2 of 6 interior points' rows each), have no
// global load inside the loops and share one logarithm and one reciprocal
// between the two margins of a reach row: 21 and 30 us, bound by issue.
constexpr int RF_SEGS = 64;
constexpr int RF_ROWS = 16;  // polytope rows staged at a time

template <int M, int G, int PD, bool GRAD>
__global__ void __launch_bounds__(RF_SEGS * M) k_refine(RefineParams R) {
    constexpr int L = PD + 1, NT = RF_SEGS * M, PS = (L * M) | 1, AS = (RF_ROWS * M) | 1, BS = RF_ROWS | 1;
    static_assert(PD - 1 == 2 * M, "two interior control points a thread");
    constexpr RefineConst<PD> K = refine_const<PD>();
    __shared__ float sP[RF_SEGS * PS];                // [segment][PS] control points
    __shared__ float sG[GRAD ? RF_SEGS * PS : 1];     // their gradient
    __shared__ float sA[RF_SEGS * AS], sB[RF_SEGS * BS];  // [segment][rows of a chunk]
    __shared__ float s_red[2][NT];                    // loss and dT parts
    const int tid = threadIdx.x, rmax = R.rmax;
    const long long s0 = (long long)blockIdx.x * RF_SEGS;
    const int ns = (int)min((long long)RF_SEGS, R.S - s0);
    auto stage_rows = [&](int c0) {  // rows c0 .. c0 + RF_ROWS of every segment
        const int rc = min(RF_ROWS, rmax - c0);
        for (int u = tid; u < ns * rc * M; u += NT) {
            const int sg = u / (rc * M), x = u - sg * rc * M;
            sA[sg * AS + x] = R.A[((s0 + sg) * rmax + c0) * M + x];
        }
        for (int u = tid; u < ns * rc; u += NT) {
            const int sg = u / rc, x = u - sg * rc;
            sB[sg * BS + x] = R.b[(s0 + sg) * rmax + c0 + x];
        }
    };
    for (int u = tid; u < ns * L * M; u += NT) sP[u / (L * M) * PS + u % (L * M)] = R.P[s0 * L * M + u];
    if (rmax > 0) stage_rows(0);
    const int q = tid / M, a = tid - q * M;  // segment of the block, axis
    const bool act = q < ns;
    const float T = act ? R.T[s0 + q] : 1.f, up = GRAD && act ? R.grad_loss[s0 + q] : 1.f;
    const int nr = act ? min(R.nrows[s0 + q], rmax) : 0;
    __syncthreads();
    const float mu = R.mu, ws = R.w_snap, Ti = 1.f / T;
    const Barrier B = {R.delta, 1.f / R.delta, -logf(R.delta) - 0.5f};
    float loss = 0.f, dT = 0.f;
    if (act) {
        // reach margins and snap energy of axis a (Theorem 1 per axis; the snap
        // integral is the sum of the axes' integrals)
        float Pa[L], ga[L];
#pragma unroll
        for (int l = 0; l < L; ++l) {
            Pa[l] = sP[q * PS + l * M + a];
            ga[l] = 0.f;
        }
        float d[L], pk = 1.f;
#pragma unroll
        for (int l = 0; l < L; ++l) d[l] = Pa[l];
#pragma unroll
        for (int k = 1; k <= G; ++k) {
            fwd_diff<L>(d, L - k + 1);  // the k-th differences
            pk *= Ti;
            const float sk = K.scale[k] * pk, ck = R.bound[k - 1];
            float g[L], dk = 0.f;
#pragma unroll
            for (int j = 0; j < L; ++j) {
                g[j] = 0.f;
                if (j < L - k) {
                    const float Q = sk * d[j];
                    float sl = 0.f;
                    loss += phi_pair<GRAD>(B, ck, Q, sl);
                    if (GRAD) {
                        g[j] = sl * sk;
                        dk = fmaf(sl, Q, dk);
                    }
                }
            }
            if (GRAD) {
                dT = fmaf(-(float)k, dk, dT);
#pragma unroll
                for (int it = k; it >= 1; --it) adj_diff<L>(g, L - it);
#pragma unroll
                for (int l = 0; l < L; ++l) ga[l] += g[l];
            }
        }
        loss *= mu;
        dT *= mu * Ti;
        {
            constexpr int qd = PD - 4;
#pragma unroll
            for (int it = G; it < 4; ++it) fwd_diff<L>(d, L - it);
            float c = K.scale[4] * K.scale[4];
            float t7 = Ti * Ti * Ti;
            t7 = t7 * t7 * Ti;
            c *= t7;
            float quad = 0.f, gd[L];
#pragma unroll
            for (int j = 0; j < L; ++j) gd[j] = 0.f;
#pragma unroll
            for (int j = 0; j <= qd; ++j)
#pragma unroll
                for (int l = 0; l <= qd; ++l) {
                    const float Gjl = K.gram[j][l];
                    quad = fmaf(Gjl * d[j], d[l], quad);
                    if (GRAD) gd[j] = fmaf(Gjl, d[l], gd[j]);
                }
            const float J = c * quad;
            loss += ws * J;
            if (GRAD) {
                const float f = ws * c * 2.f;
#pragma unroll
                for (int it = 4; it >= 1; --it) adj_diff<L>(gd, L - it);
#pragma unroll
                for (int l = 0; l < L; ++l) sG[q * PS + l * M + a] = fmaf(f, gd[l], mu * ga[l]) * up;
                dT += ws * (-7.f) * J * Ti;
            }
        }
    }
    // free margins of control points 2a+1 and 2a+2
    float fl = 0.f, P2[2][M], df[2][M];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int c = 0; c < M; ++c) {
            P2[i][c] = act ? sP[q * PS + (2 * a + 1 + i) * M + c] : 0.f;
            df[i][c] = 0.f;
        }
    for (int c0 = 0; c0 < rmax; c0 += RF_ROWS) {
        if (c0 > 0) {
            __syncthreads();
            stage_rows(c0);
            __syncthreads();
        }
        const int n = min(nr - c0, RF_ROWS);
        for (int r = 0; r < n; ++r) {
            float Ar[M];
#pragma unroll
            for (int c = 0; c < M; ++c) Ar[c] = sA[q * AS + r * M + c];
            const float br = sB[q * BS + r];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                float dot = 0.f;
#pragma unroll
                for (int c = 0; c < M; ++c) dot = fmaf(Ar[c], P2[i][c], dot);
                float sl = 0.f;
                fl += phi_one<GRAD>(B, br - dot, sl);
                if (GRAD) {
#pragma unroll
                    for (int c = 0; c < M; ++c) df[i][c] = fmaf(-sl, Ar[c], df[i][c]);
                }
            }
        }
    }
    s_red[0][tid] = fmaf(mu, fl, loss);
    s_red[1][tid] = dT;
    __syncthreads();
    if (act) {
        if (GRAD) {  // each interior point by one thread
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int c = 0; c < M; ++c) sG[q * PS + (2 * a + 1 + i) * M + c] += df[i][c] * (mu * up);
        }
        if (a == 0) {
            float v = 0.f, w = 0.f;
#pragma unroll
            for (int c = 0; c < M; ++c) {
                v += s_red[0][tid + c];
                w += s_red[1][tid + c];
            }
            if (R.loss) R.loss[s0 + q] = v;
            if (GRAD) R.dT[s0 + q] = w * up;
        }
    }
    if (GRAD) {
        __syncthreads();
        for (int u = tid; u < ns * L * M; u += NT) R.dP[s0 * L * M + u] = sG[u / (L * M) * PS + u % (L * M)];
    }
}

bool refine_supported(int m, int g, int p) { return (m == 3 && g == 3 && p == 7) || (m == 2 && g == 2 && p == 5); }

int launch_refine(const RefineParams& R, void* stream, int* launches) {
    cudaStream_t st = (cudaStream_t)stream;
    const unsigned nb = (unsigned)((R.S + RF_SEGS - 1) / RF_SEGS);
    if (R.S == 0) return 0;
    const bool grad = R.grad_loss != nullptr;
    if (R.m == 3 && R.g == 3 && R.p == 7) {
        if (grad) k_refine<3, 3, 7, true><<<nb, RF_SEGS * 3, 0, st>>>(R);
        else k_refine<3, 3, 7, false><<<nb, RF_SEGS * 3, 0, st>>>(R);
    } else if (R.m == 2 && R.g == 2 && R.p == 5) {
        if (grad) k_refine<2, 2, 5, true><<<nb, RF_SEGS * 2, 0, st>>>(R);
        else k_refine<2, 2, 5, false><<<nb, RF_SEGS * 2, 0, st>>>(R);
    } else {
        return (int)cudaErrorInvalidValue;
    }
    ++*launches;
    return (int)cudaGetLastError();
}

}  // namespace plan
