// Device pieces shared by the per-agent kernels of the J-update (lm.cu, jupdate.cu): 2x2 blocks in
// registers, CTA-wide sums, the block-Jacobi preconditioner, the penalty of Eq. sumtrace2 and the
// gauge terms (see lm.cu for the method).
#pragma once

#include <math.h>

#include "calib_internal.cuh"
#include "df.cuh"

namespace calib {
namespace {

constexpr double TCG_KAPPA = 0.1;   // residual test ||r|| <= ||r0|| min(||r0||, kappa)
constexpr double RTR_ACCEPT = 0.1;  // a step is accepted when its ratio exceeds this
struct Blk { float v[8]; };

__device__ __forceinline__ Blk ld_blk(const float* base, int blk) {
    const float4* q = reinterpret_cast<const float4*>(base) + 2 * (size_t)blk;
    const float4 a0 = q[0], a1 = q[1];
    return Blk{{a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w}};
}
__device__ __forceinline__ void st_blk(float* base, int blk, const Blk& b) {
    float4* q = reinterpret_cast<float4*>(base) + 2 * (size_t)blk;
    q[0] = make_float4(b.v[0], b.v[1], b.v[2], b.v[3]);
    q[1] = make_float4(b.v[4], b.v[5], b.v[6], b.v[7]);
}
__device__ __forceinline__ Blk zero_blk() { return Blk{{0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}}; }
__device__ __forceinline__ float dot8(const Blk& a, const Blk& b) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) s = fmaf(a.v[i], b.v[i], s);
    return s;
}

// Sum over the CTA of each v[i]; every thread gets the same totals. red: NV*32 floats owned by
// this call site (no barrier is needed before the next call site writes its own).
template <int NV>
__device__ __forceinline__ void block_sum(float (&v)[NV], float* red) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
        if (lane == 0) red[i * 32 + w] = v[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        float s = 0.f;
        for (int k = 0; k < nw; ++k) s += red[i * 32 + k];
        v[i] = s;
    }
}
__device__ __forceinline__ float block_max(float v, float* red) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) red[w] = v;
    __syncthreads();
    float m = red[0];
    for (int k = 1; k < nw; ++k) m = fmaxf(m, red[k]);
    return m;
}
// (G + lam I)^-1 of a Hermitian G (g00, g11, re g01, im g01), in the same form.
__device__ __forceinline__ float4 precond_inverse(const float (&G)[4], float lam) {
    const float a = G[0] + lam, c = G[1] + lam, br = G[2], bi = G[3];
    const float id = 1.f / (a * c - (br * br + bi * bi));
    // id * [[c, -b], [-conj(b), a]]
    return make_float4(c * id, a * id, -br * id, -bi * id);
}
// x M for a 2x2 complex block x (row-major re,im pairs) and M as precond_inverse gives it.
__device__ __forceinline__ Blk precond_apply(const Blk& x, float4 M) {
    const float m00 = M.x, m11 = M.y, m01r = M.z, m01i = M.w, m10r = M.z, m10i = -M.w;
    Blk z;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const float x0r = x.v[r * 4 + 0], x0i = x.v[r * 4 + 1], x1r = x.v[r * 4 + 2], x1i = x.v[r * 4 + 3];
        // z[r][0] = x[r][0] m00 + x[r][1] m10 ; z[r][1] = x[r][0] m01 + x[r][1] m11
        z.v[r * 4 + 0] = x0r * m00 + x1r * m10r - x1i * m10i;
        z.v[r * 4 + 1] = x0i * m00 + x1r * m10i + x1i * m10r;
        z.v[r * 4 + 2] = x0r * m01r - x0i * m01i + x1r * m11;
        z.v[r * 4 + 3] = x0r * m01i + x0i * m01r + x1i * m11;
    }
    return z;
}
__device__ __forceinline__ Blk precond(const Blk& x, const float (&G)[4], float lam) { return precond_apply(x, precond_inverse(G, lam)); }

__device__ __forceinline__ int n_parts(const LMArgs& a, int agent) { return a.part_n ? a.part_n[agent] : a.part_stride; }

// Sum of the partial station sums of a sweep, fixed piece order.
__device__ __forceinline__ Blk sum_parts(const LMArgs& a, int agent, int blk, int KN) {
    const float* base = a.part + (size_t)agent * a.part_stride * KN * 8;
    Blk s = ld_blk(base, blk);
    const int np = n_parts(a, agent);
    for (int ch = 1; ch < np; ++ch) {
        const Blk q = ld_blk(base + (size_t)ch * KN * 8, blk);
#pragma unroll
        for (int i = 0; i < 8; ++i) s.v[i] += q.v[i];
    }
    return s;
}

// Penalty Re tr(Y^H D) + rho/2 ||D||^2 of one block, D = J - BZ (Eq. sumtrace2).
__device__ __forceinline__ float penalty_blk(const Blk& j, const Blk& y, const Blk& bz, float rk) {
    float yd = 0.f, dd = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float d = j.v[i] - bz.v[i];
        yd = fmaf(y.v[i], d, yd);
        dd = fmaf(d, d, dd);
    }
    return yd + 0.5f * rk * dd;
}
// pen(J) - pen(Jt) = -(Re tr(Y^H x) + rho Re tr(D^H x) + rho/2 ||x||^2), D = J - BZ, x = Jt - J, of one
// block. Formed from the small x, so it is accurate relative to the decrease itself.
__device__ __forceinline__ float penalty_decrease_blk(const Blk& j, const Blk& jt, const Blk& y, const Blk& bz, float rk) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float x = jt.v[i] - j.v[i];  // exact: Jt = J + x was rounded once
        const float d = j.v[i] - bz.v[i];
        s -= fmaf(y.v[i], x, rk * fmaf(0.5f * x, x, d * x));
    }
    return s;
}

// ---- gauge projection
// g is invariant under J_k -> J_k U (C = c I_2, Eq. coh), so the exact data gradient has no
// component along the gauge orbit {J_k A : A anti-Hermitian}: the anti-Hermitian part of
// J_k^H G_k vanishes. Float32 residuals leave round-off there, which would otherwise steer the
// weakly determined gauge mode (curved only by the rho/2 penalty). With S = J^H J, solve
// (S A + A S)/2 = skew(J^H G) for A = [[i a, b + i c], [-b + i c, i d]] and set G <- G - J A (the
// h-orthogonal projection); exact arithmetic leaves G unchanged. The skew part is a small
// difference of large station terms, so its sums carry about 48 bits: double-float accumulation
// built from error-free float32 transformations (the exact product error by FMA, Dekker 1971;
// the exact sum error by TwoSum, Knuth TAOCP vol. 2, 4.2.2). The 4x4 system is well conditioned
// (S is the Gram matrix of J_k) and is solved in float32 in closed form.
constexpr int GT = 12;  // per-block gauge terms: 4 double-float (t0, t1, 2 t2, 2 t3) and s0, s1, u, w

// This block's terms of skew(J^H G) and J^H J. Row m, column c of a block: v[m*4 + c*2 + (0 re, 1 im)].
__device__ __forceinline__ void gauge_terms(const Blk& j, const Blk& g, float* out) {
    DF t0{0.f, 0.f}, t1{0.f, 0.f}, t2{0.f, 0.f}, t3{0.f, 0.f};
    float s0 = 0.f, s1 = 0.f, u = 0.f, w = 0.f;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        const float a0r = j.v[m * 4 + 0], a0i = j.v[m * 4 + 1], a1r = j.v[m * 4 + 2], a1i = j.v[m * 4 + 3];
        const float g0r = g.v[m * 4 + 0], g0i = g.v[m * 4 + 1], g1r = g.v[m * 4 + 2], g1i = g.v[m * 4 + 3];
        // t0 = Im M00, t1 = Im M11 with M = J^H G
        df_add_prod(t0, a0r, g0i);
        df_add_prod(t0, -a0i, g0r);
        df_add_prod(t1, a1r, g1i);
        df_add_prod(t1, -a1i, g1r);
        // 2 t2 = Re M01 - Re M10,  2 t3 = Im M01 + Im M10
        df_add_prod(t2, a0r, g1r);
        df_add_prod(t2, a0i, g1i);
        df_add_prod(t2, -a1r, g0r);
        df_add_prod(t2, -a1i, g0i);
        df_add_prod(t3, a0r, g1i);
        df_add_prod(t3, -a0i, g1r);
        df_add_prod(t3, a1r, g0i);
        df_add_prod(t3, -a1i, g0r);
        s0 = fmaf(a0r, a0r, fmaf(a0i, a0i, s0));
        s1 = fmaf(a1r, a1r, fmaf(a1i, a1i, s1));
        u = fmaf(a0r, a1r, fmaf(a0i, a1i, u));
        w = fmaf(a0r, a1i, fmaf(-a0i, a1r, w));
    }
    out[0] = t0.hi; out[1] = t0.lo; out[2] = t1.hi; out[3] = t1.lo;
    out[4] = t2.hi; out[5] = t2.lo; out[6] = t3.hi; out[7] = t3.lo;
    out[8] = s0; out[9] = s1; out[10] = u; out[11] = w;
}

// Solve the gauge system of one direction from its summed terms; A = (a, d, b, c).
// Eliminating b and c (rows 3 and 4) leaves two scalar equations in a and d whose sum gives
// e = a + d with the determinant of S as denominator.
__device__ __forceinline__ float4 gauge_solve(const float (&tt)[GT]) {
    const float t0 = tt[0] + tt[1], t1 = tt[2] + tt[3], T2 = tt[4] + tt[5], T3 = tt[6] + tt[7];
    const float s0 = tt[8], s1 = tt[9], u = tt[10], w = tt[11];
    const float sig = s0 + s1, uw = u * u + w * w;
    const float det = s0 * s1 - uw;
    if (!(sig > 0.f) || !(det > 1e-12f * sig * sig) || !isfinite(T2 + T3 + t0 + t1)) return make_float4(0.f, 0.f, 0.f, 0.f);
    const float h = (u * T3 - w * T2) / sig, q = uw / sig;
    const float e = ((t0 - h) * s1 + (t1 - h) * s0) / det;
    return make_float4((t0 - h + q * e) / s0, (t1 - h + q * e) / s1, (T2 + w * e) / sig, (T3 - u * e) / sig);
}

// One warp's sums of a direction's gauge terms (sm: [N][GT]) over its stations, in every lane.
__device__ __forceinline__ void gauge_sums(const float* sm, int N, int lane, DF (&t)[4], float (&s)[4]) {
    for (int p = lane; p < N; p += 32) {
        const float* q = sm + (size_t)p * GT;
#pragma unroll
        for (int i = 0; i < 4; ++i) t[i] = df_add(t[i], DF{q[2 * i], q[2 * i + 1]});
#pragma unroll
        for (int i = 0; i < 4; ++i) s[i] += q[8 + i];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const DF other{__shfl_xor_sync(0xffffffffu, t[i].hi, o), __shfl_xor_sync(0xffffffffu, t[i].lo, o)};
            t[i] = df_add(t[i], other);
            s[i] += __shfl_xor_sync(0xffffffffu, s[i], o);
        }
    }
}

// g <- g - j A for one block, A as gauge_solve gives it.
__device__ __forceinline__ void remove_gauge(const Blk& j, float4 Asol, Blk& g) {
    const float a = Asol.x, d = Asol.y, b = Asol.z, c = Asol.w;
    // A = [[i a, b + i c], [-b + i c, i d]]
    const float A00r = 0.f, A00i = a, A01r = b, A01i = c, A10r = -b, A10i = c, A11r = 0.f, A11i = d;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const float jr0 = j.v[r * 4 + 0], ji0 = j.v[r * 4 + 1], jr1 = j.v[r * 4 + 2], ji1 = j.v[r * 4 + 3];
        // (J A)[r][0] = J[r][0] A00 + J[r][1] A10 ; (J A)[r][1] = J[r][0] A01 + J[r][1] A11
        g.v[r * 4 + 0] -= jr0 * A00r - ji0 * A00i + jr1 * A10r - ji1 * A10i;
        g.v[r * 4 + 1] -= jr0 * A00i + ji0 * A00r + jr1 * A10i + ji1 * A10r;
        g.v[r * 4 + 2] -= jr0 * A01r - ji0 * A01i + jr1 * A11r - ji1 * A11i;
        g.v[r * 4 + 3] -= jr0 * A01i + ji0 * A01r + jr1 * A11i + ji1 * A11r;
    }
}

// Project the gauge component out of this CTA's data-gradient blocks g (held by their threads).
// sm: KN*GT floats; Asol: 4*K floats.
template <int BPT>
__device__ void project_out_gauge(const Blk (&j)[BPT], Blk (&g)[BPT], int K, int N, float* sm, float* Asol) {
    const int T = blockDim.x, KN = K * N;
#pragma unroll
    for (int i = 0; i < BPT; ++i) {
        const int blk = threadIdx.x + i * T;
        if (blk < KN) gauge_terms(j[i], g[i], sm + (size_t)blk * GT);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = T >> 5;
    for (int k = warp; k < K; k += nw) {
        DF t[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
        float s[4] = {0.f, 0.f, 0.f, 0.f};
        gauge_sums(sm + (size_t)k * N * GT, N, lane, t, s);
        if (lane == 0) {
            const float tt[GT] = {t[0].hi, t[0].lo, t[1].hi, t[1].lo, t[2].hi, t[2].lo, t[3].hi, t[3].lo,
                                  s[0], s[1], s[2], s[3]};
            const float4 A = gauge_solve(tt);
            Asol[k * 4 + 0] = A.x;
            Asol[k * 4 + 1] = A.y;
            Asol[k * 4 + 2] = A.z;
            Asol[k * 4 + 3] = A.w;
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < BPT; ++i) {
        const int blk = threadIdx.x + i * T;
        if (blk >= KN) continue;
        const int k = blk / N;
        remove_gauge(j[i], make_float4(Asol[k * 4 + 0], Asol[k * 4 + 1], Asol[k * 4 + 2], Asol[k * 4 + 3]), g[i]);
    }
}

// Jacobi blocks G_pk = sum_o s_(p,o)k J_ok^H J_ok at the CTA's J (held by the threads), from the
// dense weights gw (all loads independent) and the
// products J_ok^H J_ok staged in sm (KN*4 floats).
template <int BPT>
__device__ void gram_blocks(const LMArgs& a, int agent, const Blk (&j)[BPT], float* sm, float (&G)[BPT][4]) {
    const int T = blockDim.x, N = a.N, K = a.K, KN = K * N;
#pragma unroll
    for (int i = 0; i < BPT; ++i) {
        const int blk = threadIdx.x + i * T;
        if (blk >= KN) continue;
        const float* v = j[i].v;
        // J^H J: x00 = |J00|^2 + |J10|^2, x11 = |J01|^2 + |J11|^2, x01 = conj(J00) J01 + conj(J10) J11
        reinterpret_cast<float4*>(sm)[blk] = make_float4(
            v[0] * v[0] + v[1] * v[1] + v[4] * v[4] + v[5] * v[5],
            v[2] * v[2] + v[3] * v[3] + v[6] * v[6] + v[7] * v[7],
            v[0] * v[2] + v[1] * v[3] + v[4] * v[6] + v[5] * v[7],
            v[0] * v[3] - v[1] * v[2] + v[4] * v[7] - v[5] * v[6]);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < BPT; ++i) {
        const int blk = threadIdx.x + i * T;
        G[i][0] = G[i][1] = G[i][2] = G[i][3] = 0.f;
        if (blk >= KN) continue;
        const int k = blk / N, p = blk - k * N;
        // the weights are symmetric: read along a row, consecutive threads read consecutive words
        const int NW = (N + 3) / 4 * 4;
        const float* W = a.gw + ((size_t)agent * K + k) * N * NW + p;
        const float4* X = reinterpret_cast<const float4*>(sm) + k * N;
        float g0 = 0.f, g1 = 0.f, g2 = 0.f, g3 = 0.f;
#pragma unroll 16
        for (int o = 0; o < N; ++o) {
            const float w = __ldg(W + (size_t)o * NW);
            const float4 x = X[o];
            g0 = fmaf(w, x.x, g0);
            g1 = fmaf(w, x.y, g1);
            g2 = fmaf(w, x.z, g2);
            g3 = fmaf(w, x.w, g3);
        }
        G[i][0] = g0; G[i][1] = g1; G[i][2] = g2; G[i][3] = g3;
        reinterpret_cast<float4*>(a.Gm + (size_t)agent * KN * 4)[blk] = make_float4(g0, g1, g2, g3);
    }
}

}  // namespace
}  // namespace calib
