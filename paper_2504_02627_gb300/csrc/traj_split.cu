// traj_split.cu -- leapfrog trajectories (Algorithm 1) with one particle spread
// over several threads, for the cheap targets whose gradient splits without
// changing a single rounding:
//  * the banana: its pairs (theta_2i, theta_2i+1) never meet, so each pair is
//    a trajectory of its own, in one thread's registers;
//  * the dense Gaussian with D <= 32: a lane per row of the precision, the
//    deviations exchanged through shared memory each step.
// A particle per thread (traj_thread.cu) leaves the GPU idle at the particle
// counts of one run: a step is then one thread's chain over all dimensions,
// with a warp or less per scheduler to hide it.
#include <algorithm>
#include <math_constants.h>
#include "traj.cuh"

namespace smc {
namespace {

// What a thread needs of its particle.
struct Slot {
    int64_t j, src;
    int S;
    double eps;
    uint64_t seed;
    uint32_t kk, jl;
};
__device__ __forceinline__ Slot slot_of(const TrajArgs& a, int64_t t) {
    Slot x;
    x.j = a.perm ? a.perm[t] : t;
    x.src = a.src ? a.src[x.j] : x.j;
    int r;
    particle_run(a, x.j, r, x.eps, x.seed, x.kk, x.jl);
    x.S = a.eval_only ? 0 : a.steps[x.j];
    return x;
}

// Energies of the particle in slot order: H_0 from p_0, log pi at the end.
__device__ __forceinline__ void finish(const TrajArgs& a, int64_t j, double lp1, double H0, double kin1) {
    a.logpi_out[j] = lp1;
    if (a.eval_only) return;
    double dH = (0.5 * kin1 - lp1) - H0;
    if (!isfinite(dH)) dH = CUDART_INF;
    if (a.dH) a.dH[j] = dH;
    if (a.alpha) a.alpha[j] = dH <= 0.0 ? 1.0 : exp(-dH);
}

// ============================================================ banana
// Banana pairs (Sec. 4, Rosenbrock): x_o ~ N(0, a), x_e ~ N(b (x_o^2 - a), 1).
// Its constants come from the host: two FP64 divisions, in every warp of a kernel
// that spreads a particle over warps, were half of a gradient evaluation (D = 2:
// 6.2 us a call, D = 32, 100000 particles 37.2).
struct BananaC {
    float a, b, inva, half_inva;
};
__device__ __forceinline__ void banana_grad(float a, float b, float inva, float xo, float xe, float& g0, float& g1) {
    float u = xe - b * (xo * xo - a);
    g0 = -xo * inva + 2.0f * b * u * xo;
    g1 = -u;
}
// A pair's part of log pi.  Which of its two products is rounded on its own is
// written out, so that the value does not vary with what the compiler contracts in
// an instance of the kernel: the second, and for a single pair the first, as a
// thread that holds the whole particle has it.
__device__ __forceinline__ float banana_term(float a, float b, float half_inva, float xo, float xe, bool single) {
    const float u = xe - b * (xo * xo - a);
    const float s = __fmul_rn(-half_inva, xo), t = __fmul_rn(0.5f, u);
    return single ? fmaf(-t, u, __fmul_rn(s, xo)) : fmaf(s, xo, -__fmul_rn(t, u));
}

// A warp holds 32 consecutive slots; the PW warps of a slot group share the
// particles' pairs, warp w taking pairs w, w + PW, ..., NPT of them side by
// side (independent chains that fill each other's latency).  Loads and stores
// are those of 32 consecutive particles of one dimension.  The FP64 sums (p'p
// before and after, log pi) run in the order of the dimensions, a warp each,
// from shared memory, so they have the bits of a thread that holds the whole
// particle.  Bound by the FMA pipe (12 operations a pair and step)
// and, in unsorted launches, by the longest of a warp's 32 trajectories: 50-d,
// 8192 particles, up to 100 steps 59.6 -> 38.9 us with the caller's copies (24
// of them this kernel; a thread per particle filled 64 CTAs).
template <int NPT>
__global__ void __launch_bounds__(256) traj_banana_kernel(DevModel m, TrajArgs a, BananaC c, int pw) {
    extern __shared__ __align__(16) float sm[];
    const int D = m.D, np = D / 2;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int w = wid % pw, grp = wid / pw, ngrp = (blockDim.x >> 5) / pw;
    const int64_t t = ((int64_t)blockIdx.x * ngrp + grp) * 32 + lane;
    const bool on = t < a.N;
    float* sp0 = sm + (size_t)grp * 32 * (2 * D + np + 6); // [D][32] momenta before
    float* sp1 = sp0 + 32 * D;                              // [D][32] momenta after
    float* slp = sp1 + 32 * D;                              // [np][32] log pi terms
    double* se = reinterpret_cast<double*>(slp + 32 * np);   // [3][32] log pi, p'p before and after
    const float fa = c.a, fb = c.b, inva = c.inva, half_inva = c.half_inva;
    Slot x{};
    double lp0 = 0.0;
    // a group of one warp needs no other
    auto sync = [&] {
        if (pw == 1) __syncwarp();
        else __syncthreads();
    };
    if (on) {
        x = slot_of(a, t);
        if (w == 0 && !a.eval_only) lp0 = a.logpi_in[x.src];
        float xo[NPT], xe[NPT], po[NPT], pe[NPT], g0[NPT], g1[NPT];
        const float ef = (float)x.eps, he = (float)(0.5 * x.eps);
#pragma unroll
        for (int k = 0; k < NPT; ++k) {
            const int i = w + k * pw;
            xo[k] = xe[k] = po[k] = pe[k] = g0[k] = g1[k] = 0.0f;
            if (i >= np) continue;
            const int64_t o = (int64_t)(2 * i) * a.ld;
            xo[k] = a.theta_in[o + x.src];
            xe[k] = a.theta_in[o + a.ld + x.src];
            if (a.eval_only) {
                banana_grad(fa, fb, inva, xo[k], xe[k], g0[k], g1[k]);
                continue;
            }
            g0[k] = a.grad_in[o + x.src];
            g1[k] = a.grad_in[o + a.ld + x.src];
            if (a.p_in) {
                po[k] = a.p_in[o + x.j];
                pe[k] = a.p_in[o + a.ld + x.j];
            } else {
                normal_pair_f32(x.seed, (uint32_t)i, x.jl, x.kk, TAG_MOM, po[k], pe[k]);
            }
            sp0[2 * i * 32 + lane] = po[k];
            sp0[(2 * i + 1) * 32 + lane] = pe[k];
        }
        for (int s = 0; s < x.S; ++s) {
#pragma unroll
            for (int k = 0; k < NPT; ++k) {
                po[k] = fmaf(he, g0[k], po[k]);
                pe[k] = fmaf(he, g1[k], pe[k]);
                xo[k] = fmaf(ef, po[k], xo[k]);
                xe[k] = fmaf(ef, pe[k], xe[k]);
                banana_grad(fa, fb, inva, xo[k], xe[k], g0[k], g1[k]);
                po[k] = fmaf(he, g0[k], po[k]);
                pe[k] = fmaf(he, g1[k], pe[k]);
            }
        }
#pragma unroll
        for (int k = 0; k < NPT; ++k) {
            const int i = w + k * pw;
            if (i >= np) continue;
            const int64_t o = (int64_t)(2 * i) * a.ld + x.j;
            slp[i * 32 + lane] = banana_term(fa, fb, half_inva, xo[k], xe[k], np == 1);
            a.grad_out[o] = g0[k];
            a.grad_out[o + a.ld] = g1[k];
            if (a.eval_only) continue;
            sp1[2 * i * 32 + lane] = po[k];
            sp1[(2 * i + 1) * 32 + lane] = pe[k];
            a.theta_out[o] = xo[k];
            a.theta_out[o + a.ld] = xe[k];
            if (a.p_out) {
                a.p_out[o] = po[k];
                a.p_out[o + a.ld] = pe[k];
            }
        }
    }
    sync();
    // three warps (of four schedulers) take a sum each: an FP64 instruction
    // occupies a warp's scheduler for 64 clocks
    if (on)
        for (int e = w; e < (a.eval_only ? 1 : 3); e += pw) {
            double s = 0.0;
            if (e == 0)
                for (int i = 0; i < np; ++i) s += widen(slp[i * 32 + lane]);
            else
                for (int d = 0; d < D; ++d) {
                    const double v = widen((e == 1 ? sp0 : sp1)[d * 32 + lane]);
                    s += v * v;
                }
            se[e * 32 + lane] = s;
        }
    sync();
    if (on && w == 0)
        finish(a, x.j, se[lane] + m.lconst, a.eval_only ? 0.0 : 0.5 * se[32 + lane] - lp0, a.eval_only ? 0.0 : se[64 + lane]);
}

template <int NPT>
cudaError_t launch_banana_n(const DevModel& m, const TrajArgs& a, int pw, int ngrp, cudaStream_t s) {
    const size_t sm = (size_t)ngrp * 32 * (2 * m.D + m.D / 2 + 6) * sizeof(float);
    auto kern = traj_banana_kernel<NPT>;
    if (sm > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
    }
    const int64_t grid = (a.N + 32 * ngrp - 1) / (32 * ngrp);
    const BananaC c{(float)m.h0, (float)m.h1, (float)(1.0 / m.h0), (float)(0.5 / m.h0)};
    kern<<<(unsigned)grid, 32 * pw * ngrp, sm, s>>>(m, a, c, pw);
    return cudaGetLastError();
}

// ============================================================ dense Gaussian, row per lane
// G lanes per particle (G the power of two from D on): lane r keeps row r of P
// and dimension r of theta and p in registers.  A step: the deviations go to
// shared memory, each lane reads them back as 16-byte broadcasts and runs its
// row's sum in the order of the columns (the sum, and so every bit, of a
// thread that holds the whole particle).  Bound by the step's chain (exchange
// and one row's sum): the 10-d Gaussian's move of 256 particles, up to about 100
// steps, takes 9 instead of 30.5 us.
//
// The FP64 sums of the end point (log pi, p'p before and after: FP32 terms, added
// in the order of the dimensions) go to one warp of the CTA, a lane per particle
// and sum: an FP64 instruction takes its warp 64 clocks however few of its lanes
// need it (three lanes per particle in its own warp: D = 32, 8192 particles, 15
// steps 27.6 us instead of 21.7, 256 particles 7.0 instead of 6.8).
template <int G>
__global__ void __launch_bounds__(128) traj_gauss_rows_kernel(DevModel m, TrajArgs a) {
    constexpr int PPC = 128 / G;                       // particles per CTA
    __shared__ __align__(16) float P_s[G][G + 4], dl_s[PPC][G];
    __shared__ float p0_s[PPC][G], p1_s[PPC][G], q_s[PPC][G];
    __shared__ double e_s[3][PPC], lp0_s[PPC];
    __shared__ int64_t j_s[PPC];
    const int D = m.D, tid = threadIdx.x, r = tid % G, pi = tid / G;
    const int64_t t = (int64_t)blockIdx.x * PPC + pi;
    // the lanes of one particle; all of them take every branch together
    const unsigned gmask = G == 32 ? 0xffffffffu : ((1u << (G % 32)) - 1u) << ((tid & 31) / G * G);
    const bool on = t < a.N, in = on && r < D;
    // P once per CTA: a lane's row straight from global memory is a sector per
    // lane and column
    float pv[(G * G + 127) / 128];
#pragma unroll
    for (int k = 0; k < (G * G + 127) / 128; ++k) {
        const int i = tid + 128 * k, row = i / G, c = i % G;
        pv[k] = (row < D && c < D) ? m.P[row * D + c] : 0.0f;
    }
    Slot x{};
    float mu = 0.0f, th = 0.0f, p = 0.0f, g = 0.0f;
    if (on) x = slot_of(a, t);
    const int64_t o = (int64_t)r * a.ld;
    // (kept in a register until the end: a store here would wait for it)
    const double lp0 = on && r == 0 && !a.eval_only ? a.logpi_in[x.src] : 0.0;
    if (in) {
        mu = m.mu[r];
        th = a.theta_in[o + x.src];
        if (!a.eval_only) {
            g = a.grad_in[o + x.src];
            if (a.p_in) {
                p = a.p_in[o + x.j];
            } else {   // both lanes of a pair draw it
                float z0, z1;
                normal_pair_f32(x.seed, (uint32_t)(r >> 1), x.jl, x.kk, TAG_MOM, z0, z1);
                p = (r & 1) ? z1 : z0;
            }
        }
    } else {
        dl_s[pi][r] = 0.0f;   // and stays zero
    }
#pragma unroll
    for (int k = 0; k < (G * G + 127) / 128; ++k) {
        const int i = tid + 128 * k;
        if (G * G >= 128 || i < G * G) P_s[i / G][i % G] = pv[k];
    }
    __syncthreads();
    float P[G];
#pragma unroll
    for (int b = 0; b < G; b += 4) {
        const float4 v = *reinterpret_cast<const float4*>(&P_s[r][b]);
        P[b] = v.x;
        P[b + 1] = v.y;
        P[b + 2] = v.z;
        P[b + 3] = v.w;
    }
    // grad log pi = -P (theta - mu), this lane's row
    auto grad = [&]() {
        if (in) dl_s[pi][r] = th - mu;
        __syncwarp(gmask);
        float acc = 0.0f;
#pragma unroll
        for (int b = 0; b < G; b += 4) {
            if (b < D) {
                const float4 v = *reinterpret_cast<const float4*>(&dl_s[pi][b]);
                acc = fmaf(P[b], v.x, acc);
                acc = fmaf(P[b + 1], v.y, acc);
                acc = fmaf(P[b + 2], v.z, acc);
                acc = fmaf(P[b + 3], v.w, acc);
            }
        }
        __syncwarp(gmask);
        return -acc;
    };
    if (on) {
        if (a.eval_only) {
            g = grad();
        } else {
            p0_s[pi][r] = p;
            const float ef = (float)x.eps, he = (float)(0.5 * x.eps);
            for (int s = 0; s < x.S; ++s) {
                p = fmaf(he, g, p);
                th = fmaf(ef, p, th);
                g = grad();
                p = fmaf(he, g, p);
            }
            p1_s[pi][r] = p;
        }
        q_s[pi][r] = (th - mu) * g;
        if (r == 0) {
            j_s[pi] = x.j;
            lp0_s[pi] = lp0;
        }
        if (in) {
            a.grad_out[o + x.j] = g;
            if (!a.eval_only) {
                a.theta_out[o + x.j] = th;
                if (a.p_out) a.p_out[o + x.j] = p;
            }
        }
    }
    __syncthreads();
    // log pi = c + 1/2 (theta - mu)' g
    const int e = tid / PPC, k = tid % PPC;
    if (e < (a.eval_only ? 1 : 3)) {
        const float* v = e == 0 ? q_s[k] : e == 1 ? p0_s[k] : p1_s[k];
        double sum = 0.0;
        for (int d = 0; d < D; ++d) {
            const double w = widen(v[d]);
            sum = fma(w, e == 0 ? 1.0 : w, sum);
        }
        e_s[e][k] = sum;
    }
    __syncthreads();
    if (tid < PPC && (int64_t)blockIdx.x * PPC + tid < a.N)
        finish(a, j_s[tid], m.lconst + 0.5 * e_s[0][tid], a.eval_only ? 0.0 : 0.5 * e_s[1][tid] - lp0_s[tid],
               a.eval_only ? 0.0 : e_s[2][tid]);
}

template <int G>
cudaError_t launch_rows(const DevModel& m, const TrajArgs& a, cudaStream_t s) {
    traj_gauss_rows_kernel<G><<<(unsigned)((a.N + 128 / G - 1) / (128 / G)), 128, 0, s>>>(m, a);
    return cudaGetLastError();
}

}  // namespace

// All launch plans of the banana are this one launch.
cudaError_t launch_traj_banana(const DevModel& m, const TrajArgs& a, cudaStream_t s) {
    if (m.D > 64) return cudaErrorInvalidValue;
    const int np = m.D / 2;
    int pw = 1;
    while (pw < 8 && pw < np) pw <<= 1;
    // two pairs per thread where one each would put more than four warps on a
    // scheduler (D = 16, 16384 particles, 30 steps: 12.5 us with one)
    if (np <= 2 * (pw / 2) && (a.N + 31) / 32 * pw > 152 * 4 * 4) pw /= 2;
    // CTAs of four warps where a particle's pairs take fewer: an FP64 sum per
    // scheduler (eight warps: D = 2, 1500 particles, 15 steps 3.5 us, so 3.3)
    const int ngrp = std::max(1, 4 / pw);
    switch ((np + pw - 1) / pw) {
        case 1: return launch_banana_n<1>(m, a, pw, ngrp, s);
        case 2: return launch_banana_n<2>(m, a, pw, ngrp, s);
        case 3: return launch_banana_n<3>(m, a, pw, ngrp, s);
        default: return launch_banana_n<4>(m, a, pw, ngrp, s);
    }
}

// A particle per thread needs fewer instructions for each (no exchange, no idle
// lanes), but its chain is long and its launch starts late: where N particles
// leave most of the GPU idle the rows are faster.  us by rows / by particles, 15
// steps: D = 8, 8192 particles 4.8 / 9.3, 32768 9.4 / 10.2, 65536 14.5 / 13.0; D = 16,
// 16384 13.0 / 21.0, 32768 22.0 / 22.7, 65536 39.8 / 29.9; D = 32, 16384 39 / 89, 65536
// 138 / 192 (one step: 27.6 / 17.3 and 92 / 38).  Gradients alone cross at 131072
// lanes: D = 8, 16384 particles 3.0 / 3.0, D = 16, 8192 4.0 / 4.2, D = 32, 8192 10.7 / 7.6.
// Below five dimensions there is nothing to split.
bool gauss_rows_supported(const DevModel& m, const TrajArgs& a) {
    if (m.kind != GAUSS_DENSE || m.D <= 4 || m.D > 32) return false;
    const int64_t lanes = m.D <= 8 ? 8 : m.D <= 16 ? 16 : 32;
    if (a.eval_only) return a.N * lanes <= 131072;
    return m.D <= 16 ? a.N <= 32768 : a.N * m.D <= 1245184;
}

cudaError_t launch_traj_gauss_rows(const DevModel& m, const TrajArgs& a, cudaStream_t s) {
    if (m.D <= 8) return launch_rows<8>(m, a, s);
    if (m.D <= 16) return launch_rows<16>(m, a, s);
    return launch_rows<32>(m, a, s);
}

}  // namespace smc
