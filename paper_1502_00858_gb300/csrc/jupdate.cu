// The whole J-update of an agent (Section 3, Eq. M1) in one CTA, for problems small enough that the
// separate kernels of lm.cu, ss.cu and ss_hessvec.cu spend their time on launches and on chains of dependent
// loads: all n_lm Levenberg-Marquardt or trust-region steps, each with its n_cg Hessian passes, its CG
// steps, its trial pass and its accept decision, with the statistics, J, J', the CG direction and the partial
// sums in shared memory and x, r in registers. (A thread's 128 registers do not hold a whole slot's trial pass at
// K = 3: 816 bytes are spilled there by the LM form, 656 by the trust region; 36 and 112 at K = 2, none at K = 1.)
//
// The arithmetic is that of those kernels, operation by operation: a slot's Q_l, S Q and station terms as in
// k_ss_hessvec, W, W' and the decrease as in k_ss_sweep, a station's terms summed over the diagonals in
// order, one (first + second station) sum per diagonal, the CG and accept steps as in lm.cu. The first
// iterations hold the gauge mode by little more than round-off, so another order of operations would move
// the solutions by 1e-5 and more; with one diagonal per piece the separate kernels give the same bits.
//
// Bound by latency: at 8 stations an LM step is about 20 k cycles, of which a slot pass 0.9 k, its sums
// 0.5 k and a PCG step's two reductions and divisions 1.4 k, four times each; float64 operations take about
// 100 cycles each, so the decrease's sum is left to one warp and the damping to one idle thread. A step
// took 30 us as 10 launches and takes 12 us here (8 stations, K = 1), 46 -> 23 us at 47 stations, 47 -> 29 us
// at 30 stations, K = 3 (10 steps x 4 PCG steps, one agent an SM).
//
// Mapping. Slots (diagonal d, position i) go over all threads in chunks of diagonals; a thread writes its
// slot's two station terms to shared memory (each station is first and second of one slot a diagonal), and
// after a barrier each float of the sums is added up by one thread. The CG and LM steps have one thread
// per (direction, station) block.
#include <algorithm>

#include "lm_common.cuh"
#include "ss_common.cuh"

namespace calib {
namespace {

using namespace ss;

constexpr float4 Z4 = {0.f, 0.f, 0.f, 0.f};

__device__ __forceinline__ float2 xy(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 zw(float4 v) { return make_float2(v.z, v.w); }

// Packed statistics entry (k, l) of a slot; conjugated below the diagonal.
template <int K>
__device__ __forceinline__ float2 stat(const float2* S, int k, int l) {
    const int lo = k < l ? k : l, hi = k < l ? l : k;
    float2 v = S[lo * K - lo * (lo - 1) / 2 + (hi - lo)];
    if (k > l) v.y = -v.y;
    return v;
}

// Planes in shared memory: [K][2 rows][N] float4; f and s are the slot's stations.
// H_GN p of one slot: its terms of the first (F) and second (B) station's sums (see k_ss_hessvec).
template <int K>
__device__ __forceinline__ void hessian_slot(const float4* Js, const float4* Es, const float2* S, int N, int f, int s, float4* F, float4* B) {
    float2 X[K][4];
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
        for (int e = 0; e < 4; ++e) X[k][e] = make_float2(0.f, 0.f);
#pragma unroll
    for (int l = 0; l < K; ++l) {
        const float4 js0 = Js[2 * l * N + s], js1 = Js[(2 * l + 1) * N + s], es0 = Es[2 * l * N + s], es1 = Es[(2 * l + 1) * N + s];
        const float4 jf0 = Js[2 * l * N + f], jf1 = Js[(2 * l + 1) * N + f], ef0 = Es[2 * l * N + f], ef1 = Es[(2 * l + 1) * N + f];
        const float2 z2 = make_float2(0.f, 0.f);
        float2 q[4];
        q[0] = cdot2_acc(cdot2_acc(z2, ef0, js0), jf0, es0);
        q[1] = cdot2_acc(cdot2_acc(z2, ef0, js1), jf0, es1);
        q[2] = cdot2_acc(cdot2_acc(z2, ef1, js0), jf1, es0);
        q[3] = cdot2_acc(cdot2_acc(z2, ef1, js1), jf1, es1);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float2 skl = stat<K>(S, k, l);
#pragma unroll
            for (int e = 0; e < 4; ++e) cmac(X[k][e], skl, q[e]);
        }
    }
    const float2 z2 = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const float4 s0 = Js[2 * k * N + s], s1 = Js[(2 * k + 1) * N + s], f0 = Js[2 * k * N + f], f1 = Js[(2 * k + 1) * N + f];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float2 a0 = cmul2_acc(z2, 1.f, X[k][2 * r], xy(s0), X[k][2 * r + 1], xy(s1));
            const float2 a1 = cmul2_acc(z2, 1.f, X[k][2 * r], zw(s0), X[k][2 * r + 1], zw(s1));
            F[(2 * k + r) * N + f] = make_float4(a0.x, a0.y, a1.x, a1.y);
            const float2 b0 = cmul2c_acc(z2, 1.f, X[k][r], xy(f0), X[k][2 + r], xy(f1));
            const float2 b1 = cmul2c_acc(z2, 1.f, X[k][r], zw(f0), X[k][2 + r], zw(f1));
            B[(2 * k + r) * N + s] = make_float4(b0.x, b0.y, b1.x, b1.y);
        }
    }
}

// Trial pass of one slot at J' (Ts): gradient terms of its stations at J', and the decrease of its data cost
// (see k_ss_sweep; the two rows there are two threads). U: the slot's [K][2][2].
template <int K>
__device__ __forceinline__ double trial_slot(const float4* Js, const float4* Ts, const float2* S, const float4* __restrict__ U, int N, int f, int s,
                                             float4* F, float4* B) {
    float2 W[K][4], Y[K][4], dP[K][4];  // entries 2 row + column
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
        for (int e = 0; e < 4; ++e) W[k][e] = Y[k][e] = make_float2(0.f, 0.f);
#pragma unroll
    for (int l = 0; l < K; ++l) {
        const float4 js[2] = {Js[2 * l * N + s], Js[(2 * l + 1) * N + s]}, es[2] = {Ts[2 * l * N + s], Ts[(2 * l + 1) * N + s]};
        const float4 jf[2] = {Js[2 * l * N + f], Js[(2 * l + 1) * N + f]}, ef[2] = {Ts[2 * l * N + f], Ts[(2 * l + 1) * N + f]};
        const float2 z2 = make_float2(0.f, 0.f);
        float2 p[4];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float4 xf = f4sub(ef[r], jf[r]);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                p[2 * r + c] = cdot2_acc(z2, jf[r], js[c]);
                dP[l][2 * r + c] = cdot2_acc(cdot2_acc(z2, xf, es[c]), jf[r], f4sub(es[c], js[c]));
            }
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float2 skl = stat<K>(S, k, l);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                cmac(W[k][e], skl, p[e]);
                cmac(Y[k][e], skl, dP[l][e]);
            }
        }
    }
    float dc[2] = {0.f, 0.f};
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const float4 u0 = __ldg(U + 2 * k), u1 = __ldg(U + 2 * k + 1);
        const float2 u[4] = {xy(u0), zw(u0), xy(u1), zw(u1)};
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int d = 2 * r + r, o = 2 * r + (r ^ 1);  // columns r and 1 - r of row r
            const float2 Wd = f2sub(u[d], W[k][d]), Wo = f2sub(u[o], W[k][o]);
            dc[r] = fmaf(dP[k][d].x, 2.f * Wd.x - Y[k][d].x, fmaf(dP[k][d].y, 2.f * Wd.y - Y[k][d].y, dc[r]));
            dc[r] = fmaf(dP[k][o].x, 2.f * Wo.x - Y[k][o].x, fmaf(dP[k][o].y, 2.f * Wo.y - Y[k][o].y, dc[r]));
            W[k][d] = f2sub(Wd, Y[k][d]);  // W'_k
            W[k][o] = f2sub(Wo, Y[k][o]);
        }
    }
    const float2 z2 = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const float4 sv[2] = {Ts[2 * k * N + s], Ts[(2 * k + 1) * N + s]}, fv[2] = {Ts[2 * k * N + f], Ts[(2 * k + 1) * N + f]};
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int d = 2 * r + r, o = 2 * r + (r ^ 1), c = 2 * (r ^ 1) + r;  // c: row 1 - r, column r
            const float2 a0 = cmul2_acc(z2, -1.f, W[k][d], xy(sv[r]), W[k][o], xy(sv[r ^ 1]));
            const float2 a1 = cmul2_acc(z2, -1.f, W[k][d], zw(sv[r]), W[k][o], zw(sv[r ^ 1]));
            F[(2 * k + r) * N + f] = make_float4(a0.x, a0.y, a1.x, a1.y);
            const float2 b0 = cmul2c_acc(z2, -1.f, W[k][d], xy(fv[r]), W[k][c], xy(fv[r ^ 1]));
            const float2 b1 = cmul2c_acc(z2, -1.f, W[k][d], zw(fv[r]), W[k][c], zw(fv[r ^ 1]));
            B[(2 * k + r) * N + s] = make_float4(b0.x, b0.y, b1.x, b1.y);
        }
    }
    return (double)dc[0] + (double)dc[1];
}

__device__ __forceinline__ Blk ld_plane(const float4* P, int k, int p, int N) {
    const float4 a = P[2 * k * N + p], b = P[(2 * k + 1) * N + p];
    return Blk{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}
__device__ __forceinline__ void st_plane(float4* P, int k, int p, int N, const Blk& v) {
    P[2 * k * N + p] = make_float4(v.v[0], v.v[1], v.v[2], v.v[3]);
    P[(2 * k + 1) * N + p] = make_float4(v.v[4], v.v[5], v.v[6], v.v[7]);
}

// block_sum over the first nw warps, which hold every block; the others' values are zero and left out.
template <int NV>
__device__ __forceinline__ void own_sum(float (&v)[NV], float* red, int nw) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (w < nw) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
            if (lane == 0) red[i * 32 + w] = v[i];
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        float s = 0.f;
        for (int k = 0; k < nw; ++k) s += red[i * 32 + k];
        v[i] = s;
    }
}

// Dynamic shared memory: S and the Jacobi weights of the agent, the planes J, J', p, the sums, Y and B Z,
// then the chunk's station terms ([chunk][first, second] planes), which also serve the gauge terms, J^H J
// and the threads' shares of the decrease.
template <int K, bool RTR, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) k_jupdate(const LMArgs a, const JUpdateArgs q, const int mode) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ float red[6][64];
    __shared__ float4 Asol[K];
    __shared__ AgentState sst;
    __shared__ int accept_s;
    __shared__ float mu_s;
    __shared__ double dL_s;
    const int agent = blockIdx.x, tid = threadIdx.x, T = blockDim.x;
    const int N = a.N, D = a.D, NP = (N + 3) / 4 * 4, KN = K * N;
    constexpr int KK = K * (K + 1) / 2;
    const size_t off = (size_t)agent * KN * 8;
    const size_t sbytes = (size_t)D * NP * KK * 8;
    float2* Ss = reinterpret_cast<float2*>(smem);
    const size_t wbytes = RTR ? 0 : (size_t)KN * NP * 4;
    float* Ws = reinterpret_cast<float*>(smem + (sbytes + 127) / 128 * 128);  // [K][N][NP]
    float4* Js = reinterpret_cast<float4*>(smem + (sbytes + 127) / 128 * 128 + (wbytes + 127) / 128 * 128);
    float4* Ts = Js + 2 * KN;
    float4* Ps = Ts + 2 * KN;
    float4* Hs = Ps + 2 * KN;
    float4* buf = Hs + 6 * KN;
    float* scratch = reinterpret_cast<float*>(buf);
    float4* Ys = buf - 4 * KN;
    float4* Zs = buf - 2 * KN;
    const float2* Sg = q.S + (size_t)agent * D * NP * KK;
    const float4* Ug = reinterpret_cast<const float4*>(q.U + (size_t)agent * D * NP * K * 4);

    if (tid == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
        mbar_expect_tx(&bar, (uint32_t)(sbytes + wbytes));
        bulk_g2s(Ss, Sg, (uint32_t)sbytes, &bar);
        if (!RTR) bulk_g2s(Ws, a.gw + (size_t)agent * KN * NP, (uint32_t)wbytes, &bar);
        sst = a.st[agent];
    }
    const bool own = tid < KN;
    const int k = own ? tid / N : 0, st_p = own ? tid - k * N : 0;
    const int nwo = (KN + 31) / 32;  // the warps that own blocks
    const float rk = a.rho[k];
    Blk j = zero_blk(), gg = zero_blk();
    if (own) {
        j = ld_blk(a.J + off, tid);
        st_plane(Js, k, st_p, N, j);
        st_plane(Ys, k, st_p, N, ld_blk(a.Y + off, tid));
        st_plane(Zs, k, st_p, N, ld_blk(a.BZ + off, tid));
    }
    __syncthreads();
    const bool ok = mbar_wait_bounded(&bar, 0u);
    if (__syncthreads_or(!ok)) {
        if (tid == 0) {
            atomicOr(q.status, STATUS_TIMEOUT);
            mbar_wait_bounded(&bar, 0u);  // the copy in flight still targets this CTA's memory
        }
        return;
    }

    // this thread's first slot of a chunk, and the step to the next one
    const int dd0 = tid / N, i0 = tid - dd0 * N, dd_step = T / N, i_step = T - dd_step * N;
    // Sums over the diagonals, in order, of the slots' station terms: slot(d, i, f, s, F, B) forms those of
    // position i on diagonal d. Into Hs.
    auto sweep = [&](auto&& slot) {
        for (int c0 = 0; c0 < D; c0 += q.chunk) {
            const int nc = min(q.chunk, D - c0);
            int dd = dd0, i = i0;
            for (; dd < nc; dd += dd_step, i += i_step) {
                if (i >= N) {
                    i -= N;
                    if (++dd >= nc) break;
                }
                const int d = c0 + dd + 1;
                const int s = i + d < N ? i + d : i + d - N;
                float4* F = buf + (size_t)dd * 4 * KN;
                float4* B = F + 2 * KN;
                if (i < ((2 * d == N) ? N / 2 : N)) {
                    slot(d, i, s, F, B);
                } else {
#pragma unroll
                    for (int r = 0; r < 2 * K; ++r) F[r * N + i] = B[r * N + s] = Z4;
                }
            }
            __syncthreads();
            float* H = reinterpret_cast<float*>(Hs);
            for (int e = tid; e < 8 * KN; e += T) {
                const float* v = scratch + e;
                float sum = c0 == 0 ? v[0] + v[8 * KN] : H[e];
#pragma unroll 8
                for (int dd = c0 == 0 ? 1 : 0; dd < nc; ++dd) sum += v[dd * 16 * KN] + v[dd * 16 * KN + 8 * KN];
                H[e] = sum;
            }
            __syncthreads();
        }
    };

    // ---- begin (LM_BEGIN_FROM_PARTIALS after a direct residual sweep at J, else LM_BEGIN_REUSE)
    bool fresh = mode == LM_BEGIN_FROM_PARTIALS;
    {
        float v[2] = {0.f, 0.f};
        if (own) {
            gg = fresh ? sum_parts(a, agent, tid, KN) : ld_blk(a.gradg + off, tid);
            v[0] = penalty_blk(j, ld_plane(Ys, k, st_p, N), ld_plane(Zs, k, st_p, N), rk);
            v[1] = dot8(j, j);
        }
        own_sum<2>(v, red[0], nwo);
        if (tid == 0) {
            if (fresh) {
                double g = 0.0;
                for (int ch = 0; ch < n_parts(a, agent); ++ch) g += a.part_cost[(size_t)agent * a.part_stride + ch];
                sst.g = g;
            }
            sst.L = sst.g + (double)v[0];
            if (RTR) {
                sst.delta_bar = sqrt(2.0 * (double)v[1]);
                sst.delta = sst.delta_bar / 8.0;
            }
        }
        __syncthreads();
    }
    float G[1][4] = {{0.f, 0.f, 0.f, 0.f}};
    if (!RTR && !fresh && own) {
        const float4 v = reinterpret_cast<const float4*>(a.Gm + (size_t)agent * KN * 4)[tid];
        G[0][0] = v.x; G[0][1] = v.y; G[0][2] = v.z; G[0][3] = v.w;
    }
    auto bar_owners = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(nwo * 32) : "memory"); };
    // Jacobi block of this thread, G_pk = sum_o s_(p,o)k J_ok^H J_ok (gram_blocks; the weights are symmetric, so
    // that the threads read them along a row)
    auto gram_block = [&](const Blk& b) {
        const float* v = b.v;
        float4* X = buf;
        if (own)
            X[tid] = make_float4(v[0] * v[0] + v[1] * v[1] + v[4] * v[4] + v[5] * v[5], v[2] * v[2] + v[3] * v[3] + v[6] * v[6] + v[7] * v[7],
                                 v[0] * v[2] + v[1] * v[3] + v[4] * v[6] + v[5] * v[7],
                                 v[0] * v[3] - v[1] * v[2] + v[4] * v[7] - v[5] * v[6]);
        bar_owners();
        if (own) {
            const float* W = Ws + (size_t)k * N * NP + st_p;
            float g0 = 0.f, g1 = 0.f, g2 = 0.f, g3 = 0.f;
#pragma unroll 8
            for (int o = 0; o < N; ++o) {
                const float w = W[o * NP];
                const float4 x = X[k * N + o];
                g0 = fmaf(w, x.x, g0);
                g1 = fmaf(w, x.y, g1);
                g2 = fmaf(w, x.z, g2);
                g3 = fmaf(w, x.w, g3);
            }
            G[0][0] = g0; G[0][1] = g1; G[0][2] = g2; G[0][3] = g3;
        }
    };
    // Projected data gradient and, for the PCG, the Jacobi blocks at a new J. The owning warps alone take part
    // (their own barrier) up to the barrier at the end; the gauge sums run over a direction's stations in
    // the order of project_out_gauge.
    auto refresh = [&]() {
        if (tid < nwo * 32) {
            if (own) gauge_terms(j, gg, scratch + (size_t)tid * GT);
            bar_owners();
            const int lane = tid & 31;
            for (int d = tid >> 5; d < K; d += nwo) {
                DF t[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
                float s4[4] = {0.f, 0.f, 0.f, 0.f};
                gauge_sums(scratch + (size_t)d * N * GT, N, lane, t, s4);
                if (lane == 0) {
                    const float tt[GT] = {t[0].hi, t[0].lo, t[1].hi, t[1].lo, t[2].hi, t[2].lo, t[3].hi, t[3].lo,
                                          s4[0], s4[1], s4[2], s4[3]};
                    Asol[d] = gauge_solve(tt);
                }
            }
            bar_owners();
            if (own) {
                remove_gauge(j, Asol[k], gg);
                st_blk(a.gradg + off, tid, gg);
            }
            if constexpr (!RTR) gram_block(j);
        }
        __syncthreads();
    };
    if (fresh) refresh();
    if (!RTR) {  // mu0 = tau * max_{p,k} max diag(G_pk + rho_k/2 I)
        float m = own ? fmaxf(G[0][0], G[0][1]) + 0.5f * rk : 0.f;
        m = block_max(m, red[1]);
        if (tid == 0) {
            sst.mu = a.tau * (double)m;
            sst.nu = 2.0;
            mu_s = (float)sst.mu;
        }
        __syncthreads();
    }

    for (int step = 0; step < q.n_lm; ++step) {
        // ---- gradient, CG start
        const float mu = RTR ? 0.f : mu_s, lam = RTR ? 0.5f * rk : 0.5f * rk + mu;
        Blk x = zero_blk(), r = zero_blk(), gr = zero_blk();
        float4 M = Z4;  // (G + lam I)^-1, the same for the whole step
        float s0[1] = {0.f};
        if (own) {
            const Blk y = ld_plane(Ys, k, st_p, N), bz = ld_plane(Zs, k, st_p, N);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                gr.v[e] = gg.v[e] + 0.5f * y.v[e] + 0.5f * rk * (j.v[e] - bz.v[e]);
                r.v[e] = -gr.v[e];
            }
            if constexpr (!RTR) M = precond_inverse(G[0], lam);
            const Blk z = RTR ? r : precond_apply(r, M);
            st_plane(Ps, k, st_p, N, z);
            s0[0] = dot8(r, z);
        }
        own_sum<1>(s0, red[2], nwo);  // its barrier also publishes p
        double rr = 2.0 * (double)s0[0];
        const double r0sq = rr, delta = RTR ? sst.delta : 0.0;
        double ee = 0.0;
        float rz = (float)rr;
        int stop = RTR ? (rr > 0.0 ? TCG_RUNNING : TCG_RESIDUAL) : (rr > 0.0 ? 0 : 1);

        for (int it = 0; it < q.n_cg && !stop; ++it) {  // stop: the same in every thread
            sweep([&](int d, int i, int s, float4* F, float4* B) {
                hessian_slot<K>(Js, Ps, Ss + ((size_t)(d - 1) * NP + i) * KK, N, i, s, F, B);
            });
            Blk p = zero_blk(), ap = zero_blk();
            if (own) {
                p = ld_plane(Ps, k, st_p, N);
                ap = ld_plane(Hs, k, st_p, N);
#pragma unroll
                for (int e = 0; e < 8; ++e) ap.v[e] = fmaf(lam, p.v[e], ap.v[e]);
            }
            if constexpr (!RTR) {  // PCG (k_cg_step)
                float v[1] = {own ? dot8(p, ap) : 0.f};
                own_sum<1>(v, red[3], nwo);
                const float pAp = 2.f * v[0];
                if (!(pAp > 0.f)) {
                    stop = 1;
                    break;
                }
                const float alpha = rz / pAp;
                float w[1] = {0.f};
                if (own) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        x.v[e] = fmaf(alpha, p.v[e], x.v[e]);
                        r.v[e] = fmaf(-alpha, ap.v[e], r.v[e]);
                    }
                    ap = precond_apply(r, M);  // z
                    w[0] = dot8(r, ap);
                }
                own_sum<1>(w, red[4], nwo);
                const float rzn = 2.f * w[0], beta = rzn / rz;
                if (own) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) p.v[e] = fmaf(beta, p.v[e], ap.v[e]);
                    st_plane(Ps, k, st_p, N, p);
                }
                rz = rzn;
                if (!(rzn > 0.f)) stop = 1;
                __syncthreads();  // p is published
            } else {  // truncated CG (k_tcg_step)
                float v[3] = {0.f, 0.f, 0.f};
                if (own) {
                    v[0] = dot8(p, ap);
                    v[1] = dot8(x, p);
                    v[2] = dot8(p, p);
                }
                own_sum<3>(v, red[3], nwo);  // uses red[3] and red[4]
                const double dHd = 2.0 * v[0], ed = 2.0 * v[1], dd = 2.0 * v[2];
                int why = TCG_RUNNING;
                double len = 0.0, ee_new = ee;
                if (!(dHd > 0.0)) {
                    why = TCG_CURVATURE;
                } else {
                    len = rr / dHd;
                    ee_new = ee + 2.0 * len * ed + len * len * dd;
                    if (ee_new >= delta * delta) why = TCG_BOUNDARY;
                }
                if (why != TCG_RUNNING) {  // to the boundary along d
                    len = (dd > 0.0) ? (-ed + sqrt(fmax(ed * ed + dd * (delta * delta - ee), 0.0))) / dd : 0.0;
                    ee_new = delta * delta;
                }
                const float sf = (float)len;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    x.v[e] = fmaf(sf, p.v[e], x.v[e]);
                    r.v[e] = fmaf(-sf, ap.v[e], r.v[e]);
                }
                double rr_new = rr;
                if (why == TCG_RUNNING) {
                    float w[1] = {own ? dot8(r, r) : 0.f};
                    own_sum<1>(w, red[5], nwo);
                    rr_new = 2.0 * w[0];
                    if (rr_new <= r0sq * fmin(r0sq, TCG_KAPPA * TCG_KAPPA)) {
                        why = TCG_RESIDUAL;
                    } else {
                        const float beta = (float)(rr_new / rr);
                        if (own) {
#pragma unroll
                            for (int e = 0; e < 8; ++e) p.v[e] = fmaf(beta, p.v[e], r.v[e]);
                            st_plane(Ps, k, st_p, N, p);
                        }
                    }
                }
                rr = rr_new;
                ee = ee_new;
                stop = why;
                __syncthreads();
            }
        }

        // ---- trial point, predicted decrease, trial pass
        Blk jt = zero_blk();
        {
            float v[2] = {0.f, 0.f};
            if (own) {
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    jt.v[e] = j.v[e] + x.v[e];
                    v[0] = fmaf(x.v[e], r.v[e] - gr.v[e], v[0]);
                    v[1] = fmaf(x.v[e], x.v[e], v[1]);
                }
                st_plane(Ts, k, st_p, N, jt);
            }
            own_sum<2>(v, red[0], nwo);  // its barrier also publishes J'
            if (tid == T - 1) sst.pred = RTR ? (double)v[0] : (double)v[0] + sst.mu * (double)v[1];
        }
        double dc = 0.0;
        sweep([&](int d, int i, int s, float4* F, float4* B) {
            const size_t pos = (size_t)(d - 1) * NP + i;
            dc += trial_slot<K>(Js, Ts, Ss + pos * KK, Ug + pos * K * 2, N, i, s, F, B);
        });
        // The decrease's shares are float64, whose rate is low: one warp adds them up.
        double* share = reinterpret_cast<double*>(buf);
        share[tid] = dc;
        __syncthreads();
        if (tid < 32) {
            dc = 0.0;
            for (int t = tid; t < T; t += 32) dc += share[t];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) dc += __shfl_xor_sync(0xffffffffu, dc, o);
        }

        // ---- accept or reject (k_lm_eval, k_rtr_eval)
        float v[2] = {0.f, 0.f};
        if (own) {
            const Blk y = ld_plane(Ys, k, st_p, N), bz = ld_plane(Zs, k, st_p, N);
            v[0] = penalty_blk(jt, y, bz, rk);
            v[1] = penalty_decrease_blk(j, jt, y, bz, rk);
        }
        own_sum<2>(v, red[1], nwo);
        if (tid == 0) {
            const double g_t = sst.g - dc, L_t = g_t + (double)v[0], dL = dc + (double)v[1];
            sst.g_t = g_t;
            sst.L_t = L_t;
            dL_s = dL;
            int acc;
            if (RTR) {
                const double ratio = (sst.pred > 0.0 && isfinite(L_t) && isfinite(dL)) ? dL / sst.pred : -INFINITY;
                if (ratio < 0.25)
                    sst.delta *= 0.25;
                else if (ratio > 0.75 && (stop == TCG_BOUNDARY || stop == TCG_CURVATURE))
                    sst.delta = fmin(2.0 * sst.delta, sst.delta_bar);
                acc = ratio > RTR_ACCEPT;
            } else {
                acc = (sst.pred > 0.0) && isfinite(L_t) && isfinite(dL) && (dL > 0.0);
            }
            if (acc) {
                sst.g = g_t;
                sst.L = L_t;
                sst.accepted += 1;
            } else {
                sst.rejected += 1;
            }
            accept_s = acc;
        }
        __syncthreads();
        // The damping update is a chain of float64 operations (about 100 cycles each on this GPU): the last
        // thread runs it while the others refresh the gradient, if they do.
        if (!RTR && tid == T - 1) {
            if (accept_s) {
                const double t = 2.0 * (dL_s / sst.pred) - 1.0;
                sst.mu *= fmax(1.0 / 3.0, 1.0 - t * t * t);
                sst.nu = 2.0;
            } else {
                sst.mu *= sst.nu;
                sst.nu *= 2.0;
            }
            mu_s = (float)sst.mu;
        }
        if (accept_s) {
            if (own) {
                j = jt;
                st_plane(Js, k, st_p, N, j);
                gg = ld_plane(Hs, k, st_p, N);
            }
            refresh();
        } else {
            __syncthreads();
        }
    }
    if (own) {
        st_blk(a.J + off, tid, j);
        if (!RTR) reinterpret_cast<float4*>(a.Gm + (size_t)agent * KN * 4)[tid] = make_float4(G[0][0], G[0][1], G[0][2], G[0][3]);
    }
    if (tid == 0) a.st[agent] = sst;
}

size_t fixed_smem(int N, int K) {
    const size_t NP = (N + 3) / 4 * 4, S = (size_t)(N / 2) * NP * (K * (K + 1) / 2) * 8;
    return (S + 127) / 128 * 128 + (K * N * NP * 4 + 127) / 128 * 128 + (size_t)6 * 2 * K * N * 16;
}
size_t diagonal_smem(int N, int K) { return (size_t)4 * K * N * 16; }
// a chunk's station terms; the gauge terms (48 bytes a block) and a float64 per thread use the same place
size_t scratch_smem(int N, int K, int chunk, int threads) {
    return std::max((size_t)chunk * diagonal_smem(N, K), (size_t)threads * 8);
}

template <int K, bool RTR>
cudaError_t prep() {
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(k_jupdate<K, RTR, 512, 1>, attr, JUPDATE_SMEM_MAX);
    return e == cudaSuccess ? cudaFuncSetAttribute(k_jupdate<K, RTR, 256, 2>, attr, JUPDATE_SMEM_MAX) : e;
}
template <int K, bool RTR>
cudaError_t go(const LMArgs& a, const JUpdateArgs& q, int mode, size_t smem, cudaStream_t s) {
    if (q.threads > 256)
        k_jupdate<K, RTR, 512, 1><<<a.A, q.threads, smem, s>>>(a, q, mode);
    else
        k_jupdate<K, RTR, 256, 2><<<a.A, q.threads, smem, s>>>(a, q, mode);
    return cudaGetLastError();
}
template <bool RTR>
cudaError_t dispatch(const LMArgs& a, const JUpdateArgs& q, int mode, size_t smem, cudaStream_t s) {
    switch (a.K) {
        case 1: return go<1, RTR>(a, q, mode, smem, s);
        case 2: return go<2, RTR>(a, q, mode, smem, s);
        case 3: return go<3, RTR>(a, q, mode, smem, s);
        default: return cudaErrorInvalidConfiguration;
    }
}

}  // namespace

cudaError_t prepare_jupdate_kernels() {
    cudaError_t e = prep<1, false>();
    if (e == cudaSuccess) e = prep<2, false>();
    if (e == cudaSuccess) e = prep<3, false>();
    if (e == cudaSuccess) e = prep<1, true>();
    if (e == cudaSuccess) e = prep<2, true>();
    if (e == cudaSuccess) e = prep<3, true>();
    return e;
}

// Whether one launch is the faster one, by the slots (N / 2) N of an agent and the agents an SM has to take. Both sides
// in us a step of 4 CG steps, separate kernels (autotuned) -> this one, at the edges of the rule (LM unless marked;
// 8 to 128 stations and 4 to 10240 agents were measured). What a row cites beyond a limit is why the limit lies there.
//   at most one agent an SM: this one's time does not depend on their number, the separate kernels' grows with it
//     K = 1: 80 stations, 16 agents 52 -> 44; 96 stations 53 -> 56, but with more than half of the SMs at work every size
//       (128 stations, 80 agents 96 -> 90, 152: 127 -> 90). Trust region: 80 stations 61 -> 55, 96 59 -> 67
//     K = 2: 63 stations, 16 agents 58 -> 56. Trust region: 47 stations 62 -> 53, 63 66 -> 75
//     K = 3: 47 stations, 16 agents 58 -> 53. Trust region: 42 stations 71 -> 65, 44 70 -> 71 (47, 80 agents 80 -> 71)
//   two (both CTAs resident), 160 agents: K = 1, 80 stations 86 -> 71, 84 84 -> 87; trust region 64 stations 71 -> 55, 80
//     87 -> 87. 34 stations, K = 2 64 -> 41, K = 3 77 -> 62, trust region 69 -> 59, 85 -> 76
//   up to eight, or four: K = 1, 80 stations, 320 agents 120 -> 117, 88 139 -> 171; 28 stations, 1200 agents 82 -> 70. 20 stations,
//     1200 agents, K = 2 91 -> 78, K = 3 127 -> 100. Trust region, 640 agents: 16 stations, K = 1 59 -> 44, K = 3 86 -> 80, K = 2
//     66 -> 66 (12 stations 68 -> 34); 20 stations, K = 1 65 -> 74; 16 stations, K = 1, 1280 agents 72 -> 73
//   more: 16 stations, 5120 agents, K = 1 135 -> 127, K = 3 301 -> 246; 20 and 32 stations, K = 1, 2560 agents 112 -> 121 and
//     137 -> 157, but 33 (where the separate kernels' CTAs grow) 214 -> 183 and 80 681 -> 583; 18 stations, K = 2, 5120
//     agents 259 -> 289. Trust region: 10 stations, 9600 agents 235 -> 226, 12, 2560 agents 97 -> 99; 16, K = 3 208 -> 200
static bool one_launch_faster(int slots, int K, int A, int sms, bool rtr) {
    if (A <= sms) {
        if (2 * A > sms && (rtr ? K == 3 && slots <= 1104 : K == 1)) return true;
        return slots <= (K == 1 ? 3200 : rtr ? (K == 2 ? 1104 : 900) : K == 2 ? 2048 : 1104);
    }
    if (A <= 2 * sms) return slots <= (K == 1 ? (rtr ? 2048 : 3200) : 600);
    if (A <= (rtr ? 4 : 8) * sms) return slots <= (rtr ? (K == 2 ? 72 : 128) : K == 1 ? 3200 : 200);
    if (A > 64 * sms) return false;  // not measured
    if (rtr) return slots <= (K == 3 ? 128 : 50);
    return slots <= 128 || (K == 1 && slots > 512 && slots <= 3200);
}

bool jupdate_plan(int N, int K, int A, int sms, bool rtr, JUpdateArgs& q) {
    if (K > 3 || K * N > 512) return false;
    if (!one_launch_faster(N / 2 * N, K, A, sms, rtr)) return false;
    const size_t fixed = fixed_smem(N, K), diag = diagonal_smem(N, K);
    const int D = N / 2;
    const bool one = A <= sms;  // at most one agent an SM: as many threads as have work
    // equal rounds of slots over at most 512 or 256 threads
    const int most = std::max(one ? 512 : 256, K * N), rounds = (D * N + most - 1) / most;
    q.threads = std::max(64, (std::max(K * N, (D * N + rounds - 1) / rounds) + 31) / 32 * 32);
    const size_t budget = q.threads <= 256 && !one ? JUPDATE_SMEM_MAX / 2 - 2048 : JUPDATE_SMEM_MAX;
    if (fixed + scratch_smem(N, K, 1, q.threads) > JUPDATE_SMEM_MAX) return false;
    const size_t room = fixed + scratch_smem(N, K, 1, q.threads) > budget ? JUPDATE_SMEM_MAX : budget;
    q.chunk = std::max(1, (int)std::min<size_t>(D, (room - fixed) / diag));
    return true;
}

cudaError_t launch_jupdate(const LMArgs& a, const JUpdateArgs& q, bool rtr, int mode, cudaStream_t s) {
    const size_t smem = fixed_smem(a.N, a.K) + scratch_smem(a.N, a.K, q.chunk, q.threads);
    return rtr ? dispatch<true>(a, q, mode, smem, s) : dispatch<false>(a, q, mode, smem, s);
}

}  // namespace calib
