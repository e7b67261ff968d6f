// Data ingestion and coherency prediction.
//
// Ingestion moves user-layout visibilities [A][B][T_a][2][2] and coherencies [A][B][T_a][K] into
// the circulant-diagonal layout used by the sweeps (see calib_internal.cuh); a pair held reversed
// gets V^H and conj(c), which is the same measurement seen from the other station (Eq. vispq).
//
// Prediction (Eq. coh): c_pq = sum_s I_s(f) exp(i phi_pq,s) with phi = -2 pi (f/c)
// (u_pq l + v_pq m + w_pq (n - 1)) and (u,v,w)_pq = (u,v,w)_p - (u,v,w)_q. The phase splits into
// station phasors E_ps = exp(-2 pi i turns_ps), turns_ps = (f/c)(u_p l + v_p m + w_p (n-1)), so
// c_pq = sum_s I_s E_ps conj(E_qs). Turns are formed in float64 and reduced to [-1/2, 1/2)
// before the float32 sincospi, so the phase error does not grow with baseline length.
#include <math.h>

#include <algorithm>

#include "calib_internal.cuh"
#include "tma.cuh"

namespace calib {
namespace {

constexpr double C_LIGHT = 299792458.0;

// Every value that is moved is checked: non-finite ones set STATUS_NONFINITE.
__device__ __forceinline__ void report_nonfinite(bool bad, int* status) {
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(status, STATUS_NONFINITE);
}

// Visibilities: one CTA per (diagonal, agent), two threads per slot (one per row of the 2x2 blocks) looping over
// the samples, so that a thread's 16-byte accesses are independent and the four samples of a 128-byte line
// of the source are read one after the other. A reversed pair's V^H takes one entry of each row from the other
// thread. VEC: the source is 16-byte aligned (else two 8-byte loads). Bound by HBM: 62 stations, 320 agents of 10 samples
// (388 MB) 66 us with the checks, against 112 + 34 us for an element a thread and a separate pass of checks.
constexpr int INGEST_THREADS = 128;

template <bool VEC>
__global__ void __launch_bounds__(INGEST_THREADS) k_ingest_vis(const IngestArgs a) {
    const int d = blockIdx.x, agent = blockIdx.y, h = threadIdx.x & 1;
    const DiagDesc dsc = a.desc[(size_t)agent * a.D + d];
    const int Ta = a.T[agent];
    const float2* src = a.src + a.src_off[agent];
    bool bad = false;
    for (int g0 = 0; g0 < dsc.n_pad; g0 += INGEST_THREADS / 2) {  // the same trips in every thread (shuffles)
        const int g = g0 + (threadIdx.x >> 1);
        const bool on = g < dsc.n;
        const int sl = on ? a.slot[dsc.slot_off + g] : 0;
        const bool rev = (sl >> 16) & 1;
        const float2* s = src + (on ? (long long)a.slot_b[dsc.slot_off + g] * Ta * 4 + 2 * h : 0);
        float4* o = reinterpret_cast<float4*>(a.dst + dsc.voff) + 2 * (size_t)g + h;
#pragma unroll 5
        for (int t = 0; t < Ta; ++t) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (on) {
                if (VEC) {
                    v = __ldg(reinterpret_cast<const float4*>(s + 4 * t));
                } else {
                    const float2 u = __ldg(s + 4 * t), w = __ldg(s + 4 * t + 1);
                    v = make_float4(u.x, u.y, w.x, w.y);
                }
            }
            bad |= !(isfinite(v.x) && isfinite(v.y) && isfinite(v.z) && isfinite(v.w));
            // row h of V^H = (conj V[0][h], conj V[1][h]); the other thread has V[1 - h][h]
            const float2 other = make_float2(__shfl_xor_sync(0xffffffffu, h ? v.x : v.z, 1), __shfl_xor_sync(0xffffffffu, h ? v.y : v.w, 1));
            if (rev) v = h ? make_float4(other.x, -other.y, v.z, -v.w) : make_float4(v.x, -v.y, other.x, -other.y);
            if (g < dsc.n_pad) o[(size_t)t * dsc.n_pad * 2] = v;
        }
    }
    report_nonfinite(bad, a.status);
}

// Coherencies: one thread per (slot, direction) looping over the samples; OUT: back into the user layout.
template <bool OUT>
__global__ void __launch_bounds__(512) k_ingest_coh(const IngestArgs a, float2* out) {
    const int d = blockIdx.x, agent = blockIdx.y, K = a.K;
    const DiagDesc dsc = a.desc[(size_t)agent * a.D + d];
    const int Ta = a.T[agent], np = dsc.n_pad;
    const float2* src = a.src + a.src_off[agent];
    bool bad = false;
    for (int it = threadIdx.x; it < (OUT ? dsc.n : np) * K; it += blockDim.x) {
        const int g = it / K, k = it - g * K;
        float2* in = a.dst + dsc.coff + it;  // internal entry (t, g, k) at t np K + g K + k
        const bool on = g < dsc.n;
        const float sg = on && ((a.slot[dsc.slot_off + g] >> 16) & 1) ? -1.f : 1.f;
        const size_t u = on ? (size_t)a.slot_b[dsc.slot_off + g] * Ta * K + k : 0;
        if (OUT) {
            float2* o = out + a.src_off[agent] + u;
#pragma unroll 5
            for (int t = 0; t < Ta; ++t) {
                const float2 v = in[(size_t)t * np * K];
                o[(size_t)t * K] = make_float2(v.x, sg * v.y);
            }
        } else {
            const float2* s = src + u;
#pragma unroll 5
            for (int t = 0; t < Ta; ++t) {
                const float2 v = on ? __ldg(s + (size_t)t * K) : make_float2(0.f, 0.f);
                bad |= !(isfinite(v.x) && isfinite(v.y));
                in[(size_t)t * np * K] = make_float2(v.x, sg * v.y);
            }
        }
    }
    if (!OUT) report_nonfinite(bad, a.status);
}

// Flagged baselines have no slot. One warp each: their data are checked all the same (ZERO false: src), or the
// user-layout output of a call is zeroed there (ZERO).
template <bool ZERO>
__global__ void __launch_bounds__(128) k_flagged(const int2* list, int n, const long long* off, const int* T, int w, const float2* src,
                                                 float2* out, int* status) {
    bool bad = false;
    for (int i = blockIdx.x * 4 + (threadIdx.x >> 5); i < n; i += gridDim.x * 4) {
        const int2 ab = list[i];  // (agent, baseline)
        const long long m = (long long)T[ab.x] * w, o = off[ab.x] + ab.y * m;
        for (long long e = threadIdx.x & 31; e < m; e += 32) {
            if (ZERO) {
                out[o + e] = make_float2(0.f, 0.f);
            } else {
                const float2 v = src[o + e];
                bad |= !(isfinite(v.x) && isfinite(v.y));
            }
        }
    }
    if (!ZERO) report_nonfinite(bad, status);
}

// Residual visibilities (Section 2: the solutions correct the data, and the residual is the data
// minus the predicted model). In the layout's station order (i, j), where the data are V_ij and the
// coherencies c_ij: R = V_ij - sum_{k in mask} c_ij,k J_ik J_jk^H, then, with a correction
// direction k0, R <- J_i,k0^-1 R J_j,k0^-H. A pair held reversed is written back as R^H, which is
// the user-order residual (and correction) of the same baseline. Reads V and C
// once and writes each residual once; each M_k = J_ik J_jk^H is formed once per slot, not once per sample.
struct cf { float x, y; };
__device__ __forceinline__ cf cmulf(cf a, cf b) { return cf{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
__device__ __forceinline__ cf cmulcf(cf a, cf b) { return cf{a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x}; }  // conj(a) b
__device__ __forceinline__ cf caddf(cf a, cf b) { return cf{a.x + b.x, a.y + b.y}; }
struct m22 { cf e[2][2]; };
__device__ __forceinline__ m22 ld_m22(const float4* rows) {
    const float4 r0 = __ldg(rows), r1 = __ldg(rows + 1);
    return m22{{{cf{r0.x, r0.y}, cf{r0.z, r0.w}}, {cf{r1.x, r1.y}, cf{r1.z, r1.w}}}};
}
// A B
__device__ __forceinline__ m22 mmul(const m22& A, const m22& B) {
    m22 o;
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) o.e[r][c] = caddf(cmulf(A.e[r][0], B.e[0][c]), cmulf(A.e[r][1], B.e[1][c]));
    return o;
}
// A^-1 by the adjugate: [[a11, -a01], [-a10, a00]] / (a00 a11 - a01 a10)
__device__ __forceinline__ m22 minv(const m22& A) {
    const cf a = cmulf(A.e[0][0], A.e[1][1]), b = cmulf(A.e[0][1], A.e[1][0]);
    const cf det{a.x - b.x, a.y - b.y};
    const float s = 1.f / (det.x * det.x + det.y * det.y);
    const cf id{det.x * s, -det.y * s};  // 1 / det
    m22 o;
    o.e[0][0] = cmulf(A.e[1][1], id);
    o.e[1][1] = cmulf(A.e[0][0], id);
    o.e[0][1] = cmulf(cf{-A.e[0][1].x, -A.e[0][1].y}, id);
    o.e[1][0] = cmulf(cf{-A.e[1][0].x, -A.e[1][0].y}, id);
    return o;
}
__device__ __forceinline__ m22 mherm(const m22& A) {
    m22 o;
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) o.e[r][c] = cf{A.e[c][r].x, -A.e[c][r].y};
    return o;
}

constexpr int RES_THREADS = 128, RES_SLOTS = 64, RES_T = 2;  // RES_T: samples a warp takes at a time

// One CTA per (diagonal, agent), RES_SLOTS slots at a time: first every slot's model matrices M_k = J_ik J_jk^H of the
// masked directions into shared memory (Ms: [K][2 rows][RES_SLOTS] float4), then the samples, a warp taking
// 16 slots x 2 samples: 512 contiguous bytes of V a sample and 64 of the output a slot. Bound by HBM: 629 MB
// (62 stations, K = 5, 320 agents of 10 samples) in 136 us, against 205 us with one thread per slot.
// VEC: the caller's array is 16-byte aligned (else 8-byte stores, which any complex64 array takes).
template <bool VEC>
__global__ void __launch_bounds__(RES_THREADS) k_residual(const ResidualArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    float4* Ms = reinterpret_cast<float4*>(smem);
    const int d = blockIdx.x, agent = blockIdx.y, tid = threadIdx.x;
    const DiagDesc dsc = a.desc[(size_t)agent * a.D + d];
    const int Ta = a.T[agent], K = a.K, N = a.N;
    const float4* __restrict__ J = reinterpret_cast<const float4*>(a.J) + (size_t)agent * K * N * 2;  // [K][N][2 rows]
    const float4* __restrict__ V = reinterpret_cast<const float4*>(a.V + dsc.voff);                 // [T][n_pad][2 rows]
    const float2* __restrict__ C = a.C + dsc.coff;                                                   // [T][n_pad][K]
    float2* __restrict__ out = a.out + a.vis_off[agent];                                            // [B][T_a][2][2]
    for (int g0 = 0; g0 < dsc.n; g0 += RES_SLOTS) {
        const int ng = min(RES_SLOTS, dsc.n - g0);
        __syncthreads();  // the matrices of the slots before are read
        for (int it = tid; it < K * RES_SLOTS; it += RES_THREADS) {
            const int k = it / RES_SLOTS, s = it - k * RES_SLOTS;
            if (s >= ng || !((a.mask >> k) & 1u)) continue;
            const int sl = a.slot[dsc.slot_off + g0 + s];
            const m22 Ji = ld_m22(J + ((size_t)k * N + (sl & 0xff)) * 2), Jj = ld_m22(J + ((size_t)k * N + ((sl >> 8) & 0xff)) * 2);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                // (J_i J_j^H)[r][cc] = J_i[r][0] conj(J_j[cc][0]) + J_i[r][1] conj(J_j[cc][1])
                const cf m0 = caddf(cmulcf(Jj.e[0][0], Ji.e[r][0]), cmulcf(Jj.e[0][1], Ji.e[r][1]));
                const cf m1 = caddf(cmulcf(Jj.e[1][0], Ji.e[r][0]), cmulcf(Jj.e[1][1], Ji.e[r][1]));
                Ms[(k * 2 + r) * RES_SLOTS + s] = make_float4(m0.x, m0.y, m1.x, m1.y);
            }
        }
        __syncthreads();
        constexpr int WS = 32 / RES_T;  // slots of a warp
        const int s = (tid >> 5) * WS + tid % WS, t0 = (tid & 31) / WS, g = g0 + s;
        if (s >= ng) continue;
        const int sl = a.slot[dsc.slot_off + g];
        const int i = sl & 0xff, j = (sl >> 8) & 0xff, rev = (sl >> 16) & 1;
        const long long b = a.slot_b[dsc.slot_off + g];
        m22 Li{}, Rj{};
        if (a.correct >= 0) {
            Li = minv(ld_m22(J + ((size_t)a.correct * N + i) * 2));
            Rj = mherm(minv(ld_m22(J + ((size_t)a.correct * N + j) * 2)));
        }
#pragma unroll 3
        for (int t = t0; t < Ta; t += RES_T) {
            const size_t pos = (size_t)t * dsc.n_pad + g;
            m22 R = ld_m22(V + pos * 2);
            for (int k = 0; k < K; ++k) {
                if (!((a.mask >> k) & 1u)) continue;
                const float2 c2 = __ldg(C + pos * K + k);
                const cf c{c2.x, c2.y};
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const float4 q = Ms[(k * 2 + r) * RES_SLOTS + s];
                    const cf m[2] = {cf{q.x, q.y}, cf{q.z, q.w}};
#pragma unroll
                    for (int cc = 0; cc < 2; ++cc) {
                        const cf cm = cmulf(c, m[cc]);
                        R.e[r][cc] = cf{R.e[r][cc].x - cm.x, R.e[r][cc].y - cm.y};
                    }
                }
            }
            if (a.correct >= 0) R = mmul(mmul(Li, R), Rj);
            if (rev) R = mherm(R);
            float2* o = out + ((size_t)b * Ta + t) * 4;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const cf u = R.e[r][0], w = R.e[r][1];
                if (VEC) {
                    *reinterpret_cast<float4*>(o + 2 * r) = make_float4(u.x, u.y, w.x, w.y);
                } else {
                    o[2 * r] = make_float2(u.x, u.y);
                    o[2 * r + 1] = make_float2(w.x, w.y);
                }
            }
        }
    }
}

// ---- prediction
//
// What does not depend on the sample is formed once per call: flux and direction (l, m, n - 1) f / c of every
// source at every frequency, in float64 (k_predict_sources). A table larger than the context keeps is not
// built; the values are then formed where they are used.
__device__ __forceinline__ float predict_flux(const double* src, double f, double f0) { return (float)(src[2] * pow(f / f0, src[3])); }
__device__ __forceinline__ void predict_direction(const double* src, double fc, double (&d)[3]) {
    const double l = src[0], m = src[1];
    const double r2 = l * l + m * m;
    d[0] = fc * l;
    d[1] = fc * m;
    d[2] = fc * (-r2 / (1.0 + sqrt(1.0 - r2)));  // sqrt(1 - l^2 - m^2) - 1, cancellation-free
}
__global__ void __launch_bounds__(128) k_predict_sources(const PredictArgs a) {
    const int KS = a.K * a.S;
    const long long n = (long long)a.P * KS;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double f = a.freqs[i / KS];
        const double* src = a.sky + (size_t)(i % KS) * 4;
        double d[3];
        predict_direction(src, f / C_LIGHT, d);
        double* o = a.sources + i * 4;
        o[0] = d[0];
        o[1] = d[1];
        o[2] = d[2];
        o[3] = (double)predict_flux(src, f, a.f0);
    }
}

// turns - rint(turns) in float32. The float64 rate is low on this GPU, so the fraction is cut out of the
// mantissa with integer instructions (64 fractional bits: the same float32 as by rint) from 2^-12 turns on
// while it has bits there; the rest by rint, in a call, so that it is not executed beside the usual case.
__device__ __noinline__ float predict_rint_fraction(double turns) { return (float)(turns - rint(turns)); }
__device__ __forceinline__ float predict_fraction(double turns) {
    const long long bits = __double_as_longlong(turns);
    const int shift = (int)((bits >> 52) & 0x7ff) - 1011;  // |turns| = mantissa 2^(shift - 64)
    if ((unsigned)shift >= 64u) return predict_rint_fraction(turns);
    const long long frac = (long long)((((unsigned long long)bits & 0xfffffffffffffull) | 0x10000000000000ull) << shift);
    const float fr = __ll2float_rn(frac) * 5.421010862427522e-20f;  // 2^-64
    return bits < 0 ? -fr : fr;  // (the integer of one half exactly has no negative)
}

// One CTA per (sample, agent) and group of directions. The sums c_pq = sum_s I_s E_ps conj(E_qs) are products
// of a station x source matrix with its conjugate transpose: a thread holds a 4 x 4 tile of station pairs
// (first station in block bp, second in block bq) of one direction, so that a source costs four 16-byte shared loads for
// 96 arithmetic instructions (one pair a thread: two 8-byte loads for 6). Phasors of one chunk of sources are formed while the
// chunk before is summed (two buffers, one barrier a chunk). The sums go through shared memory into the
// slot layout, so that a slot's directions are written together; long sums are cut into parts there.
// Measured: 62 stations, 5 directions of 100 sources, 640 (sample, agent)s: 418 us against 795 us with one pair a
// thread (465 us with one CTA of 736 threads an SM, all directions in one group, instead of three CTAs of at most 288).
// No pipe bounds it (float64 46 % busy, FP32 38 %, issue 62 %): every warp forms phasors and sums in turn, with one CTA
// barrier a chunk, half of the shared wavefronts are bank conflicts, and at 72 registers (three CTAs an SM) 88 bytes
// a thread are spilled.
constexpr int PRED_THREADS_SMALL = 288;  // up to 288 tiles a direction (62 stations: 144, two directions at a time)
constexpr int PRED_THREADS = 736;        // more tiles, at most 561 (128 stations); 80 registers, 48 spilled bytes
// Tiles of station blocks delta apart: with the lower block first where some pair of theirs is at most N / 2
// apart (held in station order), with the higher block first where some pair is further apart.
__host__ __device__ inline int predict_tile_fwd(int N, int delta) { return 2 * (delta == 0 ? 1 : 4 * delta - 3) <= N; }
__host__ __device__ inline int predict_tile_rev(int N, int delta) { return delta > 0 && 2 * (4 * delta + 3) > N; }  // (delta 0: both orders in one tile)
__host__ __device__ inline int predict_tiles(int N) {
    const int nb = (N + 3) / 4;
    int n = 0;
    for (int delta = 0; delta < nb; ++delta) n += (nb - delta) * (predict_tile_fwd(N, delta) + predict_tile_rev(N, delta));
    return n;
}
constexpr int PRED_SMEM_MAX = 200 * 1024;
constexpr int PRED_PHASORS = 56 * 1024;  // bytes of the two phasor buffers

template <int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) k_predict(const PredictArgs a, const int KG, const int chunk, const int part) {
    extern __shared__ __align__(128) unsigned char smem[];  // one declaration for the file's kernels
    const int N = a.N, K = a.K, S = a.S, N4 = (N + 3) / 4 * 4, nb = N4 / 4, tiles = predict_tiles(N);
    const int iv = blockIdx.y / a.P, fi = blockIdx.y - iv * a.P, agent = blockIdx.y, t = blockIdx.x, k0 = blockIdx.z * KG;
    if (t >= a.T[agent]) return;
    const int kg = min(KG, K - k0), tid = threadIdx.x, nthr = blockDim.x;
    const double f = a.freqs[fi], fc = f / C_LIGHT;
    const double* uvw = a.uvw + (((size_t)iv * a.Tmax + t) * N) * 3;
    const double* sources = a.sources ? a.sources + (size_t)fi * K * S * 4 : nullptr;
    const int bufn = KG * chunk * N4;
    float2* E = reinterpret_cast<float2*>(smem);                             // [2][KG][chunk][N4]
    float* fx = reinterpret_cast<float*>(smem + (size_t)2 * bufn * 8);       // [2][KG][chunk]
    float2* cs = reinterpret_cast<float2*>(smem + (size_t)2 * KG * chunk * (N4 * 8 + 4) / 16 * 16 + 16);  // [D * N][KG] sums

    // this thread's tile: direction kk, first and second station blocks bp, bq
    const int kk = tid / tiles;
    int bp = 0, bq = 0;
    for (int w = tid - kk * tiles, delta = 0; delta < nb; ++delta) {
        const int fwd = predict_tile_fwd(N, delta), rev = predict_tile_rev(N, delta), n = nb - delta;
        if (w < n * (fwd + rev)) {
            const bool swap = w >= n * fwd;
            const int b = swap ? w - n * fwd : w;
            bp = swap ? b + delta : b;
            bq = swap ? b : b + delta;
            break;
        }
        w -= n * (fwd + rev);
    }
    const bool on = kk < kg;
    float2 acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);

    // Phasors of the sources s0 .. s0 + ns into buffer b, as two planes of station pairs: station p at float4
    // plane (p >> 1) & 1, block p >> 2, so that consecutive blocks are consecutive 16-byte words. A thread keeps its station.
    const int rows = nthr / N4, fp = tid % N4, fr0 = tid / N4;
    const double u0 = fp < N ? uvw[fp * 3] : 0.0, u1 = fp < N ? uvw[fp * 3 + 1] : 0.0, u2 = fp < N ? uvw[fp * 3 + 2] : 0.0;
    auto form = [&](int s0, int ns, int b) {
        float2* Eb = E + (size_t)b * bufn + (fp >> 2) * 2 + (fp & 1) + ((fp >> 1) & 1) * (N4 / 2);
        if (fr0 >= rows) return;
        int k = fr0 / ns, s = fr0 - k * ns;
        while (k < kg) {
            const int src = (k0 + k) * S + s0 + s;
            double dir[3], w;
            if (sources) {
                const double2 u = *reinterpret_cast<const double2*>(sources + (size_t)src * 4), v = *reinterpret_cast<const double2*>(sources + (size_t)src * 4 + 2);
                dir[0] = u.x;
                dir[1] = u.y;
                dir[2] = v.x;
                w = v.y;
            } else {
                predict_direction(a.sky + (size_t)src * 4, fc, dir);
                w = fp == 0 ? (double)predict_flux(a.sky + (size_t)src * 4, f, a.f0) : 0.0;
            }
            float2 e = make_float2(0.f, 0.f);
            if (fp < N) {
                const double turns = u0 * dir[0] + u1 * dir[1] + u2 * dir[2];
                float sn, c;
                sincospif(2.0f * predict_fraction(turns), &sn, &c);
                e = make_float2(c, -sn);  // exp(-2 pi i turns)
            }
            Eb[(k * chunk + s) * N4] = e;
            if (fp == 0) fx[b * KG * chunk + k * chunk + s] = (float)w;
            for (s += rows; s >= ns; s -= ns) ++k;
        }
    };
    // sources of the chunk from s0 on: a chunk ends where a part of the sum ends
    auto count = [&](int s0) { return min(min(chunk, S - s0), part - s0 % part); };
    const bool early = (tid >> 5) & 1;
    form(0, count(0), 0);
    __syncthreads();
    for (int s0 = 0, b = 0, ns = 0; s0 < S; s0 += ns, b ^= 1) {
        ns = count(s0);
        // Half of the warps form the next phasors before they sum, the others after: the float64 and
        // transcendental latency of the one runs beside the FMAs of the other.
        if (early && s0 + ns < S) form(s0 + ns, count(s0 + ns), b ^ 1);
        if (on) {
            const float4* Ek = reinterpret_cast<const float4*>(E + (size_t)b * bufn + (size_t)kk * chunk * N4);
            const float* fk = fx + b * KG * chunk + kk * chunk;
#pragma unroll 2
            for (int s = 0; s < ns; ++s) {
                const float4* Es = Ek + (size_t)s * (N4 / 2);
                const float4 p01 = Es[bp], p23 = Es[nb + bp], q01 = Es[bq], q23 = Es[nb + bq];
                const float w = fk[s];
                const float2 p[4] = {make_float2(p01.x, p01.y), make_float2(p01.z, p01.w), make_float2(p23.x, p23.y), make_float2(p23.z, p23.w)};
                const float2 q[4] = {make_float2(q01.x, q01.y), make_float2(q01.z, q01.w), make_float2(q23.x, q23.y), make_float2(q23.z, q23.w)};
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {  // I_s E_p conj(E_q): the product rounded before the sum's FMA
                        const float re = p[i].x * q[j].x + p[i].y * q[j].y;
                        const float im = p[i].y * q[j].x - p[i].x * q[j].y;
                        acc[i][j].x = fmaf(w, re, acc[i][j].x);
                        acc[i][j].y = fmaf(w, im, acc[i][j].y);
                    }
            }
        }
        // End of a part: its sums to shared memory, position p of diagonal d (each entry by its own thread).
        if (on && ((s0 + ns) % part == 0 || s0 + ns == S)) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int p = bp * 4 + i, q = bq * 4 + j;
                    const int d = q >= p ? q - p : q - p + N;  // the pair's diagonal with p as its first station
                    if (p < N && q < N && p != q && (2 * d < N || (2 * d == N && p < q))) {
                        float2* c = cs + ((size_t)(d - 1) * N + p) * KG + kk;
                        const float2 v = acc[i][j];
                        *c = s0 + ns <= part ? v : make_float2(c->x + v.x, c->y + v.y);
                    }
                    acc[i][j] = make_float2(0.f, 0.f);
                }
        }
        if (!early && s0 + ns < S) form(s0 + ns, count(s0 + ns), b ^ 1);
        __syncthreads();
    }
    const DiagDesc* dsc_agent = a.desc + (size_t)agent * a.D;
    for (int d = tid >> 5; d < a.D; d += nthr >> 5) {
        const DiagDesc dsc = dsc_agent[d];
        float2* out = a.C + dsc.coff + (size_t)t * dsc.n_pad * K + k0;
        for (int i = tid & 31; i < dsc.n_pad * kg; i += 32) {
            const int g = i / kg, k = i - g * kg;
            out[(size_t)g * K + k] = g < dsc.n ? cs[((size_t)d * N + (a.slot[dsc.slot_off + g] & 0xff)) * KG + k] : make_float2(0.f, 0.f);
        }
    }
}

// Jacobi weights of one agent (the direct form; the statistics pass writes them itself): gw[k][o][p] = gw[k][p][o] = s_bk = sum_t |c_btk|^2 for the baseline
// b = (p, o), zero for flagged baselines and o = p (fixed for the whole calibration). Each entry is
// written by the one slot that holds its station pair: no atomics.
// One CTA per (diagonal, agent); the entries no slot writes (the diagonal p = o, flagged pairs,
// the row padding) are zeroed by the launcher first.
__global__ void k_gram_weights(const float2* C, const DiagDesc* desc, const int* slot, const int* T, float* gw,
                               int D, int K, int N) {
    const int d = blockIdx.x, agent = blockIdx.y;
    const int NW = (N + 3) / 4 * 4;  // row stride: 16-byte rows
    float* W = gw + (size_t)agent * K * N * NW;
    const int Ta = T[agent];
    const DiagDesc dsc = desc[(size_t)agent * D + d];
    for (int it = threadIdx.x; it < dsc.n * K; it += blockDim.x) {
        const int g = it / K, k = it - g * K;
        float s = 0.f;
        for (int t = 0; t < Ta; ++t) {
            const float2 c = __ldg(C + dsc.coff + ((size_t)t * dsc.n_pad + g) * K + k);
            s = fmaf(c.x, c.x, fmaf(c.y, c.y, s));
        }
        const int sl = slot[dsc.slot_off + g];
        const int f = sl & 0xff, sc = (sl >> 8) & 0xff;
        W[((size_t)k * N + f) * NW + sc] = s;
        W[((size_t)k * N + sc) * NW + f] = s;
    }
}

// Sufficient statistics per (agent, diagonal), one pass over its visibilities and coherencies:
// U_k[e] = sum_t conj(c_tk) V_t[e] and the packed S_kl = sum_t conj(c_tk) c_tl (l >= k). Thread
// (slot g, direction k) accumulates U_k (4 entries) and row k of S over the samples (the threads of
// one slot share the loads of V_t and of the slot's K coherencies). STAGED: the CTA's whole V and C
// block (contiguous, [T_a][n_pad][4] and [T_a][n_pad][K]) arrives in shared memory by two bulk
// copies on one mbarrier, so every CTA has its bytes in flight at once; otherwise the samples are
// read from global memory, two in flight per thread. Written into the full circulant layout:
// compacted slot g goes to position i = its first station. Positions of flagged baselines are
// never written (they hold the zeros set when the layout was built). KB >= K: register bucket. WEIGHTS: the Jacobi
// weights too (new coherencies).
// Largest V + C block staged whole in shared memory; even one CTA per SM keeps far more bytes in
// flight than the streaming loop.
constexpr size_t SS_STATS_STAGED_MAX = 200 * 1024;

template <int KB, bool STAGED, bool WEIGHTS>
__global__ void __launch_bounds__(512, KB > 8 ? 1 : 2) k_ss_stats(const float2* __restrict__ V, const float2* __restrict__ C,
                                                                   float2* __restrict__ U, float2* __restrict__ S,
                                                                   float* __restrict__ gw, int N, const DiagDesc* desc, const int* slot, const int* T,
                                                                   int D, int K, int NP, int* status) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar;
    const int d = blockIdx.x, agent = blockIdx.y;
    const DiagDesc dsc = desc[(size_t)agent * D + d];
    if (dsc.n == 0) return;
    const int Ta = T[agent];
    const int KK = K * (K + 1) / 2;
    const size_t blk = ((size_t)agent * D + d) * NP;  // first position of this (agent, diagonal)
    const uint32_t vbytes = (uint32_t)Ta * dsc.n_pad * 32, cbytes = (uint32_t)Ta * dsc.n_pad * K * 8;
    const float4* Vb = reinterpret_cast<const float4*>(V + dsc.voff);
    const float2* Cb = C + dsc.coff;
    if (STAGED) {
        if (threadIdx.x == 0) {
            mbar_init(&bar, 1);
            fence_mbar_init();
            mbar_expect_tx(&bar, vbytes + cbytes);
            bulk_g2s(smem, Vb, vbytes, &bar);
            bulk_g2s(smem + vbytes, Cb, cbytes, &bar);
        }
        __syncthreads();
        const bool ok = mbar_wait_bounded(&bar, 0);
        if (__syncthreads_or(!ok)) {
            if (threadIdx.x == 0) {
                atomicOr(status, STATUS_TIMEOUT);
                mbar_wait_bounded(&bar, 0);  // the copies in flight still target this CTA's memory
            }
            return;
        }
        Vb = reinterpret_cast<const float4*>(smem);
        Cb = reinterpret_cast<const float2*>(smem + vbytes);
    }
    auto ld4 = [](const float4* p) { return STAGED ? *p : __ldg(p); };
    auto ld2 = [](const float2* p) { return STAGED ? *p : __ldg(p); };
    for (int it = threadIdx.x; it < dsc.n * K; it += blockDim.x) {
        const int g = it / K, k = it - g * K;
        float2 u[4], srow[KB];
#pragma unroll
        for (int e = 0; e < 4; ++e) u[e] = make_float2(0.f, 0.f);
#pragma unroll
        for (int l = 0; l < KB; ++l) srow[l] = make_float2(0.f, 0.f);
        const float4* vp = Vb + (size_t)g * 2;
        const float2* cp = Cb + (size_t)g * K;
        const size_t vstride = (size_t)dsc.n_pad * 2, cstride = (size_t)dsc.n_pad * K;
        auto accumulate = [&](float4 v0, float4 v1, const float2* c) {
            const float2 ck = ld2(c + k);
            const float2 vv[4] = {make_float2(v0.x, v0.y), make_float2(v0.z, v0.w), make_float2(v1.x, v1.y),
                                  make_float2(v1.z, v1.w)};
#pragma unroll
            for (int e = 0; e < 4; ++e) {  // conj(c_k) V
                u[e].x = fmaf(ck.x, vv[e].x, fmaf(ck.y, vv[e].y, u[e].x));
                u[e].y = fmaf(ck.x, vv[e].y, fmaf(-ck.y, vv[e].x, u[e].y));
            }
#pragma unroll
            for (int l = 0; l < KB; ++l) {  // conj(c_k) c_l, l >= k
                if (l < k || l >= K) continue;
                const float2 cl = ld2(c + l);
                srow[l].x = fmaf(ck.x, cl.x, fmaf(ck.y, cl.y, srow[l].x));
                srow[l].y = fmaf(ck.x, cl.y, fmaf(-ck.y, cl.x, srow[l].y));
            }
        };
        int t = 0;
        for (; t + 1 < Ta; t += 2) {
            const float4 a0 = ld4(vp + t * vstride), a1 = ld4(vp + t * vstride + 1);
            const float4 b0 = ld4(vp + (t + 1) * vstride), b1 = ld4(vp + (t + 1) * vstride + 1);
            accumulate(a0, a1, cp + t * cstride);
            accumulate(b0, b1, cp + (t + 1) * cstride);
        }
        if (t < Ta) accumulate(ld4(vp + t * vstride), ld4(vp + t * vstride + 1), cp + t * cstride);
        const size_t pos = blk + (slot[dsc.slot_off + g] & 0xff);
        float4* uo = reinterpret_cast<float4*>(U + (pos * K + k) * 4);
        uo[0] = make_float4(u[0].x, u[0].y, u[1].x, u[1].y);
        uo[1] = make_float4(u[2].x, u[2].y, u[3].x, u[3].y);
        float2* so = S + pos * KK + (size_t)k * K - k * (k - 1) / 2;  // entry (k, l) at so[l - k]
#pragma unroll
        for (int l = 0; l < KB; ++l)
            if (l >= k && l < K) so[l - k] = srow[l];
        if (WEIGHTS) {  // S_kk is the Jacobi weight of the baseline (see k_gram_weights), at both of its stations
            float skk = 0.f;
#pragma unroll
            for (int l = 0; l < KB; ++l)
                if (l == k) skk = srow[l].x;
            const int sl = slot[dsc.slot_off + g], f = sl & 0xff, sc = (sl >> 8) & 0xff;
            float* W = gw + ((size_t)agent * K + k) * N * NP;
            W[(size_t)f * NP + sc] = skk;
            W[(size_t)sc * NP + f] = skk;
        }
    }
}

}  // namespace

cudaError_t prepare_data_kernels() {
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const int st = (int)SS_STATS_STAGED_MAX;
    cudaError_t e = cudaFuncSetAttribute(k_predict<PRED_THREADS, 1>, attr, PRED_SMEM_MAX);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_predict<PRED_THREADS_SMALL, 3>, attr, PRED_SMEM_MAX);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_ss_stats<4, true, true>, attr, st);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_ss_stats<8, true, true>, attr, st);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_ss_stats<MAX_K, true, true>, attr, st);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_ss_stats<4, true, false>, attr, st);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_ss_stats<8, true, false>, attr, st);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_ss_stats<MAX_K, true, false>, attr, st);
    return e;
}

// Equal passes of at most 512 threads over a diagonal's (slot, direction)s.
int coh_threads(const IngestArgs& a) {
    const int m = std::max(1, a.slots_max * a.K), passes = (m + 511) / 512;
    return ((m + passes - 1) / passes + 31) / 32 * 32;
}
cudaError_t launch_ingest(const IngestArgs& a, cudaStream_t s) {
    const dim3 grid(a.D, a.A);
    if (!a.is_vis)
        k_ingest_coh<false><<<grid, coh_threads(a), 0, s>>>(a, nullptr);
    else if ((reinterpret_cast<uintptr_t>(a.src) & 15) == 0)
        k_ingest_vis<true><<<grid, INGEST_THREADS, 0, s>>>(a);
    else
        k_ingest_vis<false><<<grid, INGEST_THREADS, 0, s>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || a.n_flagged == 0) return e;
    k_flagged<false><<<std::min(1024, (a.n_flagged + 3) / 4), 128, 0, s>>>(a.flagged, a.n_flagged, a.src_off, a.T, a.is_vis ? 4 : a.K, a.src, nullptr,
                                                                         a.status);
    return cudaGetLastError();
}
cudaError_t launch_zero_flagged(const int2* flagged, int n, const long long* off, const int* T, int w, float2* out, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_flagged<true><<<std::min(1024, (n + 3) / 4), 128, 0, s>>>(flagged, n, off, T, w, nullptr, out, nullptr);
    return cudaGetLastError();
}
cudaError_t launch_extract_coh(const IngestArgs& a, float2* user_dst, cudaStream_t s) {
    k_ingest_coh<true><<<dim3(a.D, a.A), coh_threads(a), 0, s>>>(a, user_dst);
    return cudaGetLastError();
}
cudaError_t launch_residual(const ResidualArgs& a, cudaStream_t s) {
    const dim3 grid(a.D, a.A);
    const size_t smem = (size_t)a.K * 2 * RES_SLOTS * sizeof(float4);
    if ((reinterpret_cast<uintptr_t>(a.out) & 15) == 0)
        k_residual<true><<<grid, RES_THREADS, smem, s>>>(a);
    else
        k_residual<false><<<grid, RES_THREADS, smem, s>>>(a);
    return cudaGetLastError();
}
// Directions and sources at a time: as many directions as have tiles for the threads, sources to fill the
// phasor buffers; the sums of a group have their own shared memory behind them.
size_t predict_smem(int N, int KG, int chunk) {
    const size_t N4 = (N + 3) / 4 * 4;
    return (size_t)2 * KG * chunk * (N4 * 8 + 4) / 16 * 16 + 16 + (size_t)(N / 2) * N * KG * 8;
}
cudaError_t launch_predict(const PredictArgs& a, cudaStream_t s) {
    const int N4 = (a.N + 3) / 4 * 4, tiles = predict_tiles(a.N);
    // all tiles of a direction have to have a thread: at most 561 (N = 128)
    const bool small = tiles <= PRED_THREADS_SMALL;
    int KG = std::max(1, std::min(a.K, (small ? PRED_THREADS_SMALL : PRED_THREADS) / tiles));
    while (KG > 1 && predict_smem(a.N, KG, 1) > PRED_SMEM_MAX) --KG;
    const int groups = (a.K + KG - 1) / KG;
    KG = (a.K + groups - 1) / groups;
    const int chunk = std::max(1, std::min(a.S, (small ? PRED_PHASORS / 2 : PRED_PHASORS) / (2 * KG * (N4 * 8 + 4))));
    if (a.sources) {
        const long long n = (long long)a.P * a.K * a.S;
        k_predict_sources<<<(unsigned)std::min<long long>((n + 127) / 128, 4096), 128, 0, s>>>(a);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const int threads = std::max(64, (KG * tiles + 31) / 32 * 32);
    // sources summed in one chain (float32 round-off grows with its length); the parts are added in order
    int part = a.S;
    while (part > 1 && (size_t)a.K * part * (a.N * 8 + 28) > 96 * 1024) part = (part + 1) / 2;
    const dim3 grid(a.Tmax, a.A, groups);
    const size_t smem = predict_smem(a.N, KG, chunk);
    if (small)
        k_predict<PRED_THREADS_SMALL, 3><<<grid, threads, smem, s>>>(a, KG, chunk, part);
    else
        k_predict<PRED_THREADS, 1><<<grid, threads, smem, s>>>(a, KG, chunk, part);
    return cudaGetLastError();
}
cudaError_t launch_gram_weights(const float2* C, const DiagDesc* desc, const int* slot, const int* T, float* gw,
                                int A, int D, int K, int N, cudaStream_t s) {
    const cudaError_t e = cudaMemsetAsync(gw, 0, (size_t)A * K * N * ((N + 3) / 4 * 4) * sizeof(float), s);
    if (e != cudaSuccess) return e;
    k_gram_weights<<<dim3(D, A), 128, 0, s>>>(C, desc, slot, T, gw, D, K, N);
    return cudaGetLastError();
}
// Shared memory of a CTA of the staged statistics pass: the largest V + C block.
size_t ss_stats_smem(int N, int K, int Tmax) { return (size_t)Tmax * ((N + 3) / 4 * 4) * (32 + 8 * K); }

template <int KB>
cudaError_t ss_stats_go(const float2* V, const float2* C, float2* U, float2* S, float* gw, int N, const DiagDesc* desc, const int* slot,
                        const int* T, int A, int D, int K, int NP, size_t smem, int* status, cudaStream_t s) {
    const int threads = std::min(512, ((NP * K + 31) / 32) * 32);
    dim3 grid(D, A);
    const bool staged = smem <= SS_STATS_STAGED_MAX;
    const auto kernel = staged ? (gw ? k_ss_stats<KB, true, true> : k_ss_stats<KB, true, false>)
                               : (gw ? k_ss_stats<KB, false, true> : k_ss_stats<KB, false, false>);
    kernel<<<grid, threads, staged ? smem : 0, s>>>(V, C, U, S, gw, N, desc, slot, T, D, K, NP, status);
    return cudaGetLastError();
}

cudaError_t launch_ss_stats(const float2* V, const float2* C, float2* U, float2* S, float* gw, const DiagDesc* desc,
                            const int* slot, const int* T, int A, int D, int K, int N, int Tmax, int* status,
                            cudaStream_t s) {
    const int NP = (N + 3) / 4 * 4;
    const size_t smem = ss_stats_smem(N, K, Tmax);
    if (K <= 4) return ss_stats_go<4>(V, C, U, S, gw, N, desc, slot, T, A, D, K, NP, smem, status, s);
    if (K <= 8) return ss_stats_go<8>(V, C, U, S, gw, N, desc, slot, T, A, D, K, NP, smem, status, s);
    return ss_stats_go<MAX_K>(V, C, U, S, gw, N, desc, slot, T, A, D, K, NP, smem, status, s);
}

}  // namespace calib
