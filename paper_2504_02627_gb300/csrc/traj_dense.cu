// traj_dense.cu -- FP32 leapfrog trajectories (Algorithm 1) of the dense Gaussian
// with 32 < D <= 128.
//
// A CTA moves G particles.  A step's gradient -P (theta - mu) is a product with
// a register tile of RT rows x PT particles per thread, P (transposed) and the
// deviations theta - mu coming from shared memory; the row pairs of the tile go
// through packed FP32x2 FMAs.  Each (row, particle) sum runs over the columns
// in order, in one chain, so tile and CTA size change no rounding.  The
// momenta stay in registers, theta and the (double-buffered) deviations in
// shared memory: one barrier a step.
//
// What bounds it is the data return of shared memory, 128 bytes per clock and SM
// whether or not the lanes read the same word, against about 105 packed FMAs
// per clock and SM: a value loaded must feed more than three FMAs.  The 4 x 4 tile before
// this one fed two (10.6 us a step at D = 100, 8192 particles); keeping a row
// of P per thread in registers and loading the deviations as broadcasts feeds one
// (the same 10.6 us); 8 x 8 feeds four but leaves one warp a scheduler with
// nothing to hide its chains behind (12.5 us).  The 8 x 4 tile here: 20 steps of
// 8192 particles at D = 100 in 156 instead of 221 us, with the caller's copies (170 with the
// FP64 sums as trees over a warp per particle and a launch order that gained nothing).
#include <algorithm>
#include <type_traits>
#include <math_constants.h>
#include "tc_ptx.cuh"
#include "traj.cuh"

namespace smc {
namespace {

constexpr int DENSE_MAX_THREADS = 256;   // 16 row groups x 16 particle groups
constexpr int DENSE_SHARES = 8;          // parts of an FP64 sum over the dimensions

// Shared memory, in floats: P^T [D][RP] (RP = rows padded to the tile), deviations
// [2][D][G], theta [RP][G], the final gradients [RP][G].
struct DenseLayout {
    int nrg, rp, dl, th, g, total;
    __host__ __device__ DenseLayout(int D, int RT, int G) {
        nrg = (D + RT - 1) / RT;
        rp = nrg * RT;
        dl = D * rp;
        th = dl + 2 * D * G;
        g = th + rp * G;
        total = g + rp * G;
    }
};

// G / PT particle groups x ceil(D / RT) row groups of threads; particle groups
// run along the lanes.  A thread's rows (and, with PT = 8, particles) come in
// fours, 4 x the number of groups apart: neighbouring lanes read neighbouring
// 16 bytes.
template <int RT, int PT, int G>
__global__ void __launch_bounds__(DENSE_MAX_THREADS) traj_dense_kernel(DevModel m, TrajArgs a) {
    constexpr int NPG = G / PT, PV = PT < 4 ? PT : 4;     // particle groups; particles per vector access
    static_assert(RT % 4 == 0 && (PT == 2 || PT % 4 == 0), "vector accesses");
    extern __shared__ __align__(16) float sm[];
    const int D = m.D, NT = blockDim.x, tid = threadIdx.x;
    const DenseLayout L(D, RT, G);
    const int RP = L.rp, NRG = L.nrg;
    float* const Pt = sm;
    float* const dl_s = sm + L.dl;
    float* const th_s = sm + L.th;
    float* const g_s = sm + L.g;
    __shared__ int64_t j_s[G], src_s[G];
    __shared__ int S_s[G];
    __shared__ float eps_s[G];
    __shared__ uint64_t seed_s[G];
    __shared__ uint32_t k_s[G], jl_s[G];
    __shared__ double part_s[3][DENSE_SHARES][G], e_s[3][G];   // |p_0|^2, (theta - mu)' grad, |p|^2

    for (int e = tid; e < D * RP; e += NT) {
        const int r = e / D, k = e - r * D;               // reads of a row of P
        Pt[k * RP + r] = r < D ? m.P[r * D + k] : 0.0f;
    }
    wait_order(a);
    for (int q = tid; q < G; q += NT) {
        const int64_t t = (int64_t)blockIdx.x * G + q;
        int64_t j = -1, src = -1;
        int S = 0;
        float ef = 0.0f;
        if (t < a.N) {
            j = a.perm ? a.perm[t] : t;
            src = a.src ? a.src[j] : j;
            S = a.eval_only ? 0 : a.steps[j];
            int r;
            double eps;
            uint64_t seed;
            uint32_t kk, jl;
            particle_run(a, j, r, eps, seed, kk, jl);
            ef = (float)eps;
            seed_s[q] = seed;
            k_s[q] = kk;
            jl_s[q] = jl;
        }
        j_s[q] = j;
        src_s[q] = src;
        S_s[q] = S;
        eps_s[q] = ef;
    }
    __syncthreads();
    int smax = 0;
    for (int q = 0; q < G; ++q) smax = max(smax, S_s[q]);

    // ---- state: theta in place, p and the cached gradient staged over the two
    //      deviation buffers; rows past D are zero
    float* const p_st = dl_s;
    float* const g_st = dl_s + D * G;
    for (int e = tid; e < RP * G; e += NT) {
        const int d = e / G, q = e % G;
        const int64_t src = src_s[q];
        float tv = 0.0f, gv = 0.0f, pv = 0.0f;
        if (src >= 0 && d < D) {
            tv = a.theta_in[(int64_t)d * a.ld + src];
            if (!a.eval_only) gv = a.grad_in[(int64_t)d * a.ld + src];
            if (a.p_in && !a.eval_only) pv = a.p_in[(int64_t)d * a.ld + j_s[q]];
        }
        th_s[e] = tv;
        g_s[e] = gv;       // kept when no step is made
        if (d < D) {
            g_st[e] = gv;
            p_st[e] = pv;
        }
    }
    if (!a.p_in && !a.eval_only) {
        __syncthreads();
        for (int e = tid; e < (D + 1) / 2 * G; e += NT) {
            const int i = e / G, q = e % G;
            if (j_s[q] < 0) continue;
            double z0, z1;
            normal_pair(seed_s[q], (uint32_t)i, jl_s[q], k_s[q], TAG_MOM, z0, z1);
            p_st[(2 * i) * G + q] = (float)z0;
            if (2 * i + 1 < D) p_st[(2 * i + 1) * G + q] = (float)z1;
        }
    }
    __syncthreads();
    // FP64 sums over the dimensions, here and at the end: a lane per particle and
    // share of the dimensions, so that no lane idles and no tree is needed (an FP64
    // instruction takes its warp 64 clocks whatever the lanes do); the shares are
    // added in order.  Not unrolled: that cost the step loop 14 registers and 15%
    if (!a.eval_only)
        for (int i = tid; i < DENSE_SHARES * G; i += NT) {
            double kin = 0.0;
#pragma unroll 1
            for (int d = i / G; d < D; d += DENSE_SHARES) {
                const double v = widen(p_st[d * G + i % G]);
                kin += v * v;
            }
            part_s[0][i / G][i % G] = kin;
        }
    const int rg = tid / NPG, pg = tid % NPG;
    const bool on = rg < NRG;
    auto row = [&](int i) { return (i < 4 ? 4 * rg : 4 * NRG + 4 * rg - 4) + i; };
    auto part = [&](int i) { return PT < 4 ? PT * pg + i : (i < 4 ? 4 * pg : 4 * NPG + 4 * pg - 4) + i; };
    float p[RT][PT], mu[RT], ef[PT];
    int S[PT];
#pragma unroll
    for (int i = 0; i < RT; ++i) mu[i] = on && row(i) < D ? m.mu[row(i)] : 0.0f;
#pragma unroll
    for (int c = 0; c < PT; ++c) {
        S[c] = on ? S_s[part(c)] : 0;
        ef[c] = on ? eps_s[part(c)] : 0.0f;
    }
    // ---- first half kick and drift
    if (on) {
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int c = 0; c < PT; ++c) {
                const int r = row(i), q = part(c);
                p[i][c] = 0.0f;
                if (r < D) {
                    p[i][c] = p_st[r * G + q];
                    if (S[c] >= 1) {
                        p[i][c] = fmaf(0.5f * ef[c], g_st[r * G + q], p[i][c]);
                        th_s[r * G + q] = fmaf(ef[c], p[i][c], th_s[r * G + q]);
                    }
                }
            }
    }
    __syncthreads();
    for (int e = tid; e < D * G; e += NT) dl_s[e] = th_s[e] - m.mu[e / G];
    __syncthreads();

    const int nsteps = a.eval_only ? 1 : smax;
    for (int s = 1; s <= nsteps; ++s) {
        const float* dl = dl_s + ((s - 1) & 1) * D * G;
        float* dn = dl_s + (s & 1) * D * G;
        if (on) {
            uint64_t acc[RT / 2][PT];
#pragma unroll
            for (int i = 0; i < RT / 2; ++i)
#pragma unroll
                for (int c = 0; c < PT; ++c) acc[i][c] = 0ull;
            const float* pr = Pt + 4 * rg;
            const float* dr = dl + PV * pg;
            // the next column's operands are loaded before this one's FMAs
            ulonglong2 ra[RT / 4], rn[RT / 4];
            float b[PT], bn[PT];
            auto load = [&](int k, ulonglong2 (&x)[RT / 4], float (&y)[PT]) {
#pragma unroll
                for (int i = 0; i < RT / 4; ++i)
                    x[i] = *reinterpret_cast<const ulonglong2*>(pr + k * RP + i * 4 * NRG);
                if constexpr (PT < 4) {
                    const float2 v = *reinterpret_cast<const float2*>(dr + k * G);
                    y[0] = v.x;
                    y[1] = v.y;
                } else {
#pragma unroll
                    for (int c = 0; c < PT; c += 4) {
                        const float4 v = *reinterpret_cast<const float4*>(dr + k * G + c * NPG);
                        y[c] = v.x;
                        y[c + 1] = v.y;
                        y[c + 2] = v.z;
                        y[c + 3] = v.w;
                    }
                }
            };
            auto mul = [&](const ulonglong2 (&x)[RT / 4], const float (&y)[PT]) {
                uint64_t bb[PT];
#pragma unroll
                for (int c = 0; c < PT; ++c) bb[c] = tc::f32x2_pack(y[c], y[c]);
#pragma unroll
                for (int i = 0; i < RT / 4; ++i)
#pragma unroll
                    for (int c = 0; c < PT; ++c) {
                        acc[2 * i][c] = tc::f32x2_fma(x[i].x, bb[c], acc[2 * i][c]);
                        acc[2 * i + 1][c] = tc::f32x2_fma(x[i].y, bb[c], acc[2 * i + 1][c]);
                    }
            };
            load(0, ra, b);
            int k = 0;
            for (; k + 2 < D; k += 2) {
                load(k + 1, rn, bn);
                mul(ra, b);
                load(k + 2, ra, b);
                mul(rn, bn);
            }
            if (k + 1 < D) load(k + 1, rn, bn);
            mul(ra, b);
            if (k + 1 < D) mul(rn, bn);
            // closing half kick of step s, opening kick and drift of s + 1
#pragma unroll
            for (int i = 0; i < RT; ++i) {
                const int r = row(i);
                if (r >= D) continue;
#pragma unroll
                for (int c0 = 0; c0 < PT; c0 += PV) {
                    const int o = r * G + part(c0);
                    using V = typename std::conditional<PV == 4, float4, float2>::type;
                    V tv = *reinterpret_cast<const V*>(th_s + o), dv;
                    float* const t = &tv.x;
                    float* const dd = &dv.x;
#pragma unroll
                    for (int c = 0; c < PV; ++c) {
                        float lo, hi;
                        tc::f32x2_unpack(acc[i / 2][c0 + c], lo, hi);
                        const float gv = -((i & 1) ? hi : lo);
                        const int Sc = S[c0 + c];
                        const float he = 0.5f * ef[c0 + c];
                        if (a.eval_only || s == Sc) g_s[o + c] = gv;
                        if (!a.eval_only && s <= Sc) {
                            float pv = fmaf(he, gv, p[i][c0 + c]);
                            if (s < Sc) {
                                pv = fmaf(he, gv, pv);
                                t[c] = fmaf(ef[c0 + c], pv, t[c]);
                            }
                            p[i][c0 + c] = pv;
                        }
                    }
#pragma unroll
                    for (int c = 0; c < PV; ++c) dd[c] = t[c] - mu[i];
                    *reinterpret_cast<V*>(th_s + o) = tv;
                    *reinterpret_cast<V*>(dn + o) = dv;
                }
            }
        }
        __syncthreads();   // the step's deviations are read, the next one's written
    }
    // ---- end point: the momenta into the deviations' buffer, then log pi = c -
    //      1/2 (theta - mu)' P (theta - mu) = c + 1/2 (theta - mu)' grad, FP64
    //      accumulation of the FP32 gradient of the final position
    if (on)
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int c = 0; c < PT; ++c)
                if (row(i) < D) p_st[row(i) * G + part(c)] = p[i][c];
    __syncthreads();
    for (int i = tid; i < DENSE_SHARES * G; i += NT) {
        const int q = i % G;
        double q2 = 0.0, kin = 0.0;
#pragma unroll 1
        for (int d = i / G; d < D; d += DENSE_SHARES) {
            q2 += (widen(th_s[d * G + q]) - widen(m.mu[d])) * widen(g_s[d * G + q]);
            if (a.eval_only) continue;
            const double v = widen(p_st[d * G + q]);
            kin += v * v;
        }
        part_s[1][i / G][q] = q2;
        part_s[2][i / G][q] = kin;
    }
    __syncthreads();
    for (int i = tid; i < 3 * G; i += NT) {
        double t = 0.0;
        if (!a.eval_only || i / G == 1)
#pragma unroll 1
            for (int h = 0; h < DENSE_SHARES; ++h) t += part_s[i / G][h][i % G];
        e_s[i / G][i % G] = t;
    }
    __syncthreads();
    for (int q = tid; q < G; q += NT) {
        const int64_t j = j_s[q];
        if (j < 0) continue;
        const double lp1 = m.lconst + 0.5 * e_s[1][q];
        a.logpi_out[j] = lp1;
        if (!a.eval_only) {
            const double H0 = 0.5 * e_s[0][q] - a.logpi_in[src_s[q]];
            double dH = (0.5 * e_s[2][q] - lp1) - H0;
            if (!isfinite(dH)) dH = CUDART_INF;
            if (a.dH) a.dH[j] = dH;
            if (a.alpha) a.alpha[j] = dH <= 0.0 ? 1.0 : exp(-dH);
        }
    }
    for (int e = tid; e < D * G; e += NT) {
        const int64_t j = j_s[e % G];
        if (j < 0) continue;
        const int64_t o = (int64_t)(e / G) * a.ld + j;
        if (!a.eval_only) a.theta_out[o] = th_s[e];
        a.grad_out[o] = g_s[e];
        if (a.p_out && !a.eval_only) a.p_out[o] = p_st[e];
    }
}

template <int RT, int PT, int G>
cudaError_t launch_dense(const DevModel& m, const TrajArgs& a, cudaStream_t s) {
    const DenseLayout L(m.D, RT, G);
    const size_t sm = sizeof(float) * (size_t)L.total;
    auto kern = traj_dense_kernel<RT, PT, G>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    const int64_t grid = (a.N + G - 1) / G;
    if (grid == 0) return cudaSuccess;
    // four warps at least: the product needs fewer for small tiles, what comes
    // before and after it does not
    return launch_ordered(kern, grid, std::max((L.nrg * (G / PT) + 31) / 32 * 32, 128), sm, s, m, a);
}

}  // namespace

// From 96 CTAs of 64 particles on a large tile, where its threads fill the CTA:
// 8 x 4 above 96 dimensions, 4 x 4 between 48 and 64.  Otherwise smaller tiles, which
// load more per FMA but put more threads to work and leave no SM idle.  us for 15
// steps in tiles of 8 x 4 x 64 particles / 4 x 4 x 64 / 4 x 2 x 16 / 4 x 2 x 8:
//   D = 128, 16384 particles 284 / - / 340 / 476   3500 particles 149 / - / 102 / 139
//   D = 100,  8192 particles 116 / - / 124 / 134   1500 particles 121 / - / 46 / 51
//   D = 80,  16384 particles 209 / - / 132 / 170   3500 particles 108 / - / 50 / 49
//   D = 64,  16384 particles 95 / 89 / 107 / 131   3500 particles 76 / 60 / 38 / 37
//   D = 48,  16384 particles 75 / 62 / 58 / 81     3500 particles 62 / 50 / 28 / 27
int64_t dense_tile(const DevModel& m, int64_t N) {
    if (N >= 64 * 96) return m.D > 96 || (m.D > 48 && m.D <= 64) ? 64 : 16;
    return m.D > 64 && N >= 32 * 96 ? 16 : 8;
}

cudaError_t launch_traj_dense(const DevModel& m, const TrajArgs& a, cudaStream_t s) {
    if (m.D > 128) return cudaErrorInvalidValue;
    switch (dense_tile(m, a.N)) {
        case 64: return m.D > 96 ? launch_dense<8, 4, 64>(m, a, s) : launch_dense<4, 4, 64>(m, a, s);
        case 16: return launch_dense<4, 2, 16>(m, a, s);
        default: return launch_dense<4, 2, 8>(m, a, s);
    }
}

}  // namespace smc
