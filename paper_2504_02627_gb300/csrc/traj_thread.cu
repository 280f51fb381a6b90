// traj_thread.cu -- thread-per-particle leapfrog trajectories (Algorithm 1)
// for targets whose gradient is cheap per particle: the dense Gaussian with
// D <= 32 and the non-centred hierarchical normal.  One thread carries theta
// and p of its particle in registers for the whole trajectory, draws its
// momentum from the (seed, i, j, k, MOM) Philox stream and returns the
// end-point energy error Delta H and min(1, exp(-Delta H)).
//
// What bounds them is the FMA pipe and, before that, the registers: a
// gradient component is used up as it is formed (it closes its dimension's
// kick, opens the next one and drifts the position at once), so no gradient
// array lives next to theta and p during the steps.  The 52-d hierarchical normal
// then runs four CTAs an SM on 128 registers with 324 bytes of spills (223
// registers, or 168 with 2 KB of spills, before): 64 runs, 278k particles, three
// iterations 8.73 -> 5.87 ms.  Launches of up to two CTAs an SM take 255 registers
// and spill nothing.
#include <algorithm>
#include <cstdio>
#include <math_constants.h>
#include "traj.cuh"

namespace smc {

// ============================================================ thread models
// A model's grad_each forms the gradient component by component and hands
// each to f(d, g_d), which may already move theta_d and p_d: every value that
// other components still need is read before the first call.
template <int DM>
struct GaussDenseM {
    static constexpr bool ENERGY_FROM_GRAD = true;
    static constexpr int CTAS = DM > 16 ? 3 : 4;   // resident CTAs of 128 that the registers are capped for
    static constexpr int FEW = CTAS;               // the same in launches of two CTAs an SM at most
    static constexpr int VW = DM <= 2 ? 2 : 4;     // elements of P per shared load
    static constexpr int LD = (DM + VW - 1) / VW * VW;   // row stride of P in shared memory
    static size_t smem_bytes(const DevModel&) { return (size_t)(DM * LD + LD) * sizeof(float); }
    __device__ static void load(const DevModel& m, float* sm) {
        for (int i = threadIdx.x; i < DM * LD; i += blockDim.x) {
            const int r = i / LD, c = i % LD;
            sm[i] = (r < m.D && c < m.D) ? m.P[r * m.D + c] : 0.0f;
        }
        for (int i = threadIdx.x; i < LD; i += blockDim.x) sm[DM * LD + i] = i < m.D ? m.mu[i] : 0.0f;
    }
    // grad log pi = -P (theta - mu); a row's sum runs over the padded width
    // (zero times zero adds nothing), VW elements of P per shared load.  Up to
    // four dimensions the rows past D run too: a branch per row costs more
    // (D = 2, 300 particles, up to 30 steps 6.8 us with it, 5.7 without)
    template <class F>
    __device__ static void grad_each(const DevModel& m, const float* sm, const float (&th)[DM], F&& f) {
        const float* mu = sm + DM * LD;
        float dl[LD];
#pragma unroll
        for (int d = 0; d < LD; ++d) dl[d] = d < DM ? th[d < DM ? d : 0] - mu[d] : 0.0f;
#pragma unroll
        for (int a = 0; a < DM; ++a) {
            if (DM > 4 && a >= m.D) break;
            float acc = 0.0f;
#pragma unroll
            for (int b = 0; b < LD; b += VW) {
                if constexpr (VW == 2) {
                    const float2 v = *reinterpret_cast<const float2*>(sm + a * LD + b);
                    acc = fmaf(v.x, dl[b], acc);
                    acc = fmaf(v.y, dl[b + 1], acc);
                } else {
                    const float4 v = *reinterpret_cast<const float4*>(sm + a * LD + b);
                    acc = fmaf(v.x, dl[b], acc);
                    acc = fmaf(v.y, dl[b + 1], acc);
                    acc = fmaf(v.z, dl[b + 2], acc);
                    acc = fmaf(v.w, dl[b + 3], acc);
                }
            }
            if (DM > 4 || a < m.D) f(a, -acc);
        }
    }
    // log pi = c - 1/2 (theta - mu)' P (theta - mu) = c + 1/2 (theta - mu)' g
    // with g = -P (theta - mu) the FP32 gradient at theta: FP32 products,
    // FP64 accumulation (the FP64 quadratic form costs D^2 operations at the
    // FP64 rate, a small fraction of the FP32 rate here)
    __device__ static double energy_term(const float* sm, const float (&th)[DM], int d, float g) {
        return widen((th[d] - sm[DM * LD + d]) * g);
    }
    __device__ static double logpi(const DevModel& m, const float*, const float (&)[DM], double q) {
        return m.lconst + 0.5 * q;
    }
};

// Non-centred hierarchical normal with group sufficient statistics:
// theta = (mu, log tau, eta_1..eta_G), b_g = mu + tau eta_g.
template <int DM>
struct HierM {
    static constexpr bool ENERGY_FROM_GRAD = false;
    static constexpr int CTAS = DM > 52 ? 3 : 4;   // resident CTAs of 128 that the registers are capped for
    static constexpr int FEW = 2;                  // the same in launches of two CTAs an SM at most (no spills)
    // shared memory: (ybar_g, n_g / sigma^2) pairs for the gradient (one 8-byte
    // load per group), then n_g and the within-group sums of squares
    static size_t smem_bytes(const DevModel& m) { return (size_t)4 * m.n * sizeof(float); }
    __device__ static void load(const DevModel& m, float* sm) {
        const float inv_s2 = (float)(1.0 / (m.h0 * m.h0));
        for (int i = threadIdx.x; i < m.n; i += blockDim.x) {
            sm[2 * i] = m.gmean[i];
            sm[2 * i + 1] = m.gn[i] * inv_s2;
            sm[2 * m.n + i] = m.gn[i];
            sm[3 * m.n + i] = m.gss[i];
        }
    }
    template <class F>
    __device__ static void grad_each(const DevModel& m, const float* sm, const float (&th)[DM], F&& f) {
        const float2* st = reinterpret_cast<const float2*>(sm);
        const float mu = th[0], logtau = th[1], tau = expf(logtau);
        float dmu = 0.0f, dlt = 0.0f;
        auto group = [&](int d) {
            const float2 yn = st[d - 2];               // ybar_g, n_g / sigma^2
            const float eta = th[d];
            const float r = yn.y * (yn.x - fmaf(tau, eta, mu));
            dmu += r;
            dlt = fmaf(r * tau, eta, dlt);
            f(d, fmaf(r, tau, -eta));
        };
        // groups in fours, one bounds check each, so that the scheduler has
        // four independent groups between branches
#pragma unroll
        for (int d0 = 2; d0 < DM; d0 += 4) {
            if (d0 + 4 <= DM && d0 + 4 <= m.D) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (d0 + u < DM) group(d0 + u);
            } else if (d0 < m.D) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (d0 + u < DM && d0 + u < m.D) group(d0 + u);
            }
        }
        f(0, dmu - mu);
        f(1, dlt - logtau);
    }
    __device__ static double energy_term(const float*, const float (&)[DM], int, float) { return 0.0; }
    // FP32 terms per group, FP64 accumulation (as the GEMM-shaped models'
    // end points): FP64 runs at a small fraction of the FP32 rate here
    __device__ static double logpi(const DevModel& m, const float* sm, const float (&th)[DM], double) {
        const float inv_2s2 = (float)(0.5 / (m.h0 * m.h0));
        const float mu = th[0], logtau = th[1], tau = expf(logtau);
        double s = -0.5 * (double)mu * (double)mu - 0.5 * (double)logtau * (double)logtau;
#pragma unroll
        for (int d = 2; d < DM; ++d) {
            if (d < m.D) {
                const int k = d - 2;
                const float eta = th[d];
                const float dev = sm[2 * k] - fmaf(tau, eta, mu);
                const float term = -fmaf(sm[2 * m.n + k] * dev, dev, sm[3 * m.n + k]) * inv_2s2 - 0.5f * eta * eta;
                s += widen(term);
            }
        }
        return s + m.lconst;
    }
};

// The move of the particle in slot t (Algorithm 1 for its S_j steps, the
// end-point energy and Delta H), the model's data already in shared memory.
// ROOM: the registers hold a gradient beside theta and p.
template <template <int> class MT, int DM, bool ROOM>
__device__ __forceinline__ void particle_move(const DevModel& m, const TrajArgs& a, const float* sm, int64_t t) {
    using M = MT<DM>;
    const int64_t j = a.perm ? a.perm[t] : t;
    const int64_t src = a.src ? a.src[j] : j;
    const int D = m.D;
    int r;
    double eps;
    uint64_t seed;
    uint32_t kk, jl;
    particle_run(a, j, r, eps, seed, kk, jl);

    float th[DM], p[DM];
#pragma unroll
    for (int d = 0; d < DM; ++d) th[d] = d < D ? a.theta_in[(int64_t)d * a.ld + src] : 0.0f;

    if (a.eval_only) {
        double q = 0.0;
        M::grad_each(m, sm, th, [&](int d, float g) {
            if (M::ENERGY_FROM_GRAD) q += M::energy_term(sm, th, d, g);
            a.grad_out[(int64_t)d * a.ld + j] = g;
        });
        a.logpi_out[j] = M::logpi(m, sm, th, q);
        return;   // from the particle's move
    }

    const double lp0 = a.logpi_in[src];
    if (a.p_in) {
#pragma unroll
        for (int d = 0; d < DM; ++d) p[d] = d < D ? a.p_in[(int64_t)d * a.ld + j] : 0.0f;
    } else {
#pragma unroll
        for (int d = 0; d < DM; d += 2) {
            float z0 = 0.0f, z1 = 0.0f;
            if (d < D) normal_pair_f32(seed, (uint32_t)(d >> 1), jl, kk, TAG_MOM, z0, z1);
            p[d] = d < D ? z0 : 0.0f;
            if (d + 1 < DM) p[d + 1] = d + 1 < D ? z1 : 0.0f;
        }
    }
    // the cached gradient, GB loads in flight at a time (zeros past D, where p and
    // theta are zero too); with room in the registers all of it, behind nothing
    constexpr int GB = ROOM ? DM : 16;
    float g[GB];
    auto load_grad = [&](int d0) {
#pragma unroll
        for (int u = 0; u < GB; ++u) g[u] = d0 + u < D ? a.grad_in[(int64_t)(d0 + u) * a.ld + src] : 0.0f;
    };
    if (ROOM) load_grad(0);
    double kin0 = 0.0;
#pragma unroll
    for (int d = 0; d < DM; ++d)
        if (d < D) {
            const double v = widen(p[d]);
            kin0 += v * v;
        }
    const double H0 = 0.5 * kin0 - lp0;

    const int S = a.steps[j];
    const float ef = (float)eps, he = (float)(0.5 * eps);
    double q = 0.0;
    if (S > 0) {
        // the first half kick and drift from the cached gradient
#pragma unroll
        for (int d0 = 0; d0 < DM; d0 += GB) {
            if (!ROOM) load_grad(d0);
#pragma unroll
            for (int u = 0; u < GB; ++u)
                if (d0 + u < DM) {
                    p[d0 + u] = fmaf(he, g[u], p[d0 + u]);
                    th[d0 + u] = fmaf(ef, p[d0 + u], th[d0 + u]);
                }
        }
        // a step's gradient closes its kick, opens the next and drifts
        for (int s = 1; s < S; ++s)
            M::grad_each(m, sm, th, [&](int d, float g) {
                const float pv = fmaf(he, g, fmaf(he, g, p[d]));
                p[d] = pv;
                th[d] = fmaf(ef, pv, th[d]);
            });
        M::grad_each(m, sm, th, [&](int d, float g) {
            if (M::ENERGY_FROM_GRAD) q += M::energy_term(sm, th, d, g);
            p[d] = fmaf(he, g, p[d]);
            a.grad_out[(int64_t)d * a.ld + j] = g;
        });
    } else {
#pragma unroll
        for (int d = 0; d < DM; ++d)
            if (d < D) {
                const float g = a.grad_in[(int64_t)d * a.ld + src];
                if (M::ENERGY_FROM_GRAD) q += M::energy_term(sm, th, d, g);
                a.grad_out[(int64_t)d * a.ld + j] = g;
            }
    }
    const double lp1 = M::logpi(m, sm, th, q);
    double kin1 = 0.0;
#pragma unroll
    for (int d = 0; d < DM; ++d)
        if (d < D) {
            const double v = widen(p[d]);
            kin1 += v * v;
        }
    double dH = (0.5 * kin1 - lp1) - H0;
    if (!isfinite(dH)) dH = CUDART_INF;
#pragma unroll
    for (int d = 0; d < DM; ++d) {
        if (d < D) {
            a.theta_out[(int64_t)d * a.ld + j] = th[d];
            if (a.p_out) a.p_out[(int64_t)d * a.ld + j] = p[d];
        }
    }
    a.logpi_out[j] = lp1;
    if (a.dH) a.dH[j] = dH;
    if (a.alpha) a.alpha[j] = dH <= 0.0 ? 1.0 : exp(-dH);
}

// One particle per thread, one CTA per NT slots.
template <template <int> class MT, int DM, int NT = 128, int MINB = 1>
__global__ void __launch_bounds__(NT, MINB) traj_thread_kernel(DevModel m, TrajArgs a) {
    extern __shared__ __align__(16) float sm[];
    MT<DM>::load(m, sm);
    __syncthreads();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < a.N) particle_move<MT, DM, (NT * MINB <= 256)>(m, a, sm, t);
}

// Persistent form: as many CTAs as fit on the GPU at once, each loading the
// model's data once and then taking tiles of NT slots from a device counter
// (zeroed by the launcher) in slot order, i.e. longest trajectories first.
// Every particle's arithmetic is that of traj_thread_kernel.
template <template <int> class MT, int DM, int NT = 128, int MINB = 1>
__global__ void __launch_bounds__(NT, MINB) traj_thread_persist_kernel(DevModel m, TrajArgs a, int64_t ntiles) {
    extern __shared__ __align__(16) float sm[];
    __shared__ unsigned int tile_s;
    MT<DM>::load(m, sm);
    for (;;) {
        if (threadIdx.x == 0) tile_s = atomicAdd(a.work, 1u);
        __syncthreads();
        const int64_t tile = tile_s;
        __syncthreads();   // every thread has the tile before the next one is taken
        if (tile >= ntiles) break;
        const int64_t t = tile * NT + threadIdx.x;
        if (t < a.N) particle_move<MT, DM, (NT * MINB <= 256)>(m, a, sm, t);
    }
}


int sm_count() {
    static int sms = 0;
    if (sms == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
            sms = 1;
    }
    return sms;
}

namespace {

template <template <int> class MT, int DM, int NT, int MINB>
cudaError_t launch_thread_v(const DevModel& m, const TrajArgs& a, cudaStream_t s) {
    const size_t sm = MT<DM>::smem_bytes(m);
    auto kern = traj_thread_kernel<MT, DM, NT, MINB>;
    if (sm > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
    }
    const int64_t grid = (a.N + NT - 1) / NT;
    if (grid == 0) return cudaSuccess;
    kern<<<(unsigned)grid, NT, sm, s>>>(m, a);
    return cudaGetLastError();
}

template <template <int> class MT, int DM, int NT, int MINB>
cudaError_t launch_thread_persist(const DevModel& m, const TrajArgs& a, cudaStream_t s) {
    const size_t sm = MT<DM>::smem_bytes(m);
    auto kern = traj_thread_persist_kernel<MT, DM, NT, MINB>;
    if (sm > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
    }
    const int64_t ntiles = (a.N + NT - 1) / NT;
    if (ntiles == 0) return cudaSuccess;
    const int sms = sm_count();
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    const int64_t grid = std::min<int64_t>(ntiles, (int64_t)sms * per_sm);
    e = cudaMemsetAsync(a.work, 0, sizeof(unsigned int), s);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)grid, NT, sm, s>>>(m, a, ntiles);
    return cudaGetLastError();
}

// Variants of the thread-per-particle kernel for the autotuner: CTA size
// (the granularity with which length-sorted slots are dealt to the SMs),
// registers capped for three or four resident CTAs of 128, and for each of
// these the persistent form (4-7: tiles from a device counter; they need
// TrajArgs::work, else the launch falls back to the one-shot form).  Same
// code, same arithmetic.  Small particles (DM < 16) have only the default.
constexpr int32_t THREAD_TILES = 8;
template <template <int> class MT, int DM>
cudaError_t launch_thread(const DevModel& m, const TrajArgs& a, cudaStream_t s) {
    if constexpr (DM >= 16) {
        constexpr int C = MT<DM>::CTAS, O = 7 - C;   // the default cap, and the other one
        const int v = (a.tile >= 4 && !a.work) ? a.tile - 4 : a.tile;
        switch (v) {
            case 1: return launch_thread_v<MT, DM, 64, 2 * C>(m, a, s);
            case 2: return launch_thread_v<MT, DM, 256, 2>(m, a, s);
            case 3: return launch_thread_v<MT, DM, 128, O>(m, a, s);
            case 4: return launch_thread_persist<MT, DM, 128, C>(m, a, s);
            case 5: return launch_thread_persist<MT, DM, 64, 2 * C>(m, a, s);
            case 6: return launch_thread_persist<MT, DM, 256, 2>(m, a, s);
            case 7: return launch_thread_persist<MT, DM, 128, O>(m, a, s);
            default: break;
        }
        // while two CTAs an SM hold all particles, more registers for each beat more
        // CTAs: 52-d hierarchical normal, 300 or 8192 particles, 15 steps 46 -> 41 us,
        // one step 29 -> 25
        return a.N <= 2 * 128 * (int64_t)sm_count() ? launch_thread_v<MT, DM, 128, MT<DM>::FEW>(m, a, s)
                                                    : launch_thread_v<MT, DM, 128, C>(m, a, s);
    } else {
        return launch_thread_v<MT, DM, 128, 1>(m, a, s);
    }
}

template <template <int> class MT>
cudaError_t dispatch_thread(const DevModel& m, const TrajArgs& a, cudaStream_t s) {
    const int D = m.D;
    if (D <= 2) return launch_thread<MT, 2>(m, a, s);
    if (D <= 4) return launch_thread<MT, 4>(m, a, s);
    if (D <= 8) return launch_thread<MT, 8>(m, a, s);
    if (D <= 12) return launch_thread<MT, 12>(m, a, s);
    if (D <= 16) return launch_thread<MT, 16>(m, a, s);
    if (D <= 32) return launch_thread<MT, 32>(m, a, s);
    return cudaErrorInvalidValue;
}

template <template <int> class MT>
cudaError_t dispatch_thread_wide(const DevModel& m, const TrajArgs& a, cudaStream_t s) {
    const int D = m.D;
    if (D <= 32) return dispatch_thread<MT>(m, a, s);
    if (D <= 52) return launch_thread<MT, 52>(m, a, s);
    if (D <= 64) return launch_thread<MT, 64>(m, a, s);
    return cudaErrorInvalidValue;
}

}  // namespace

int32_t traj_thread_tiles(const DevModel& m) { return m.D > 12 ? THREAD_TILES : 1; }

cudaError_t launch_traj_thread(const DevModel& m, const TrajArgs& a, cudaStream_t s) {
    switch (m.kind) {
        case GAUSS_DENSE:
            if (m.D > 32) return cudaErrorInvalidValue;
            return a.tile == 0 && gauss_rows_supported(m, a) ? launch_traj_gauss_rows(m, a, s)
                                                               : dispatch_thread<GaussDenseM>(m, a, s);
        case BANANA: return launch_traj_banana(m, a, s);
        case HIER_NORMAL: return dispatch_thread_wide<HierM>(m, a, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace smc
