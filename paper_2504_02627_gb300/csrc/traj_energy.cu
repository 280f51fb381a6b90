// traj_energy.cu -- end-point energies of the regressions for trajectory kernels
// that leave them out: log pi at every particle's final position from the FP32
// data, and with it Delta H and the acceptance probability.
//
// The energy costs every particle the same whatever its trajectory's length, so
// a launch of its own spreads it evenly over the GPU; inside the trajectory
// kernel it ran on that kernel's terms (one CTA an SM, registers and shared
// memory of the tensor-core pipeline, at the end of the longest tile).
//
// eta = X theta is an FP32 product: a CTA takes 128 particles (theta^T in shared
// memory for the whole launch) and streams X in chunks of 128 observations; a
// thread's tile is 8 observations x 8 particles, particle pairs through packed
// FP32x2 FMAs.  Each eta is one chain over the dimensions, a thread's eight
// terms of a particle are summed in FP32, everything else in FP64.  Bound by
// the FMA pipe (its throttle is the first stall, 1.7 of 4.2 warps; a value
// loaded feeds four FMAs); one chunk buffer, so that two CTAs share an SM (up to
// 104 padded dimensions) and one computes while the other's copy is in flight.
// Logistic regression, n = 1e5, D = 100, 16384 particles: 9.1 ms, of which the
// 1.6e11 FMAs are 5.4; the move with it 18.2 -> 15.2 ms.  With log1pf(expf(.))
// written for either sign of eta apart this kernel took 12.4 ms.
#include <algorithm>
#include <math_constants.h>
#include "tc_ptx.cuh"
#include "traj.cuh"

namespace smc {
namespace {

constexpr int EP = 128;                   // particles per CTA
constexpr int EC = CENTRED_CHUNK;         // observations per chunk (128)
constexpr int ET = 256;                   // threads: 16 observation groups x 16 particle groups

constexpr int SEGS = 8;                   // segments of the chunks, summed on their own: the same for every split

// theta^T and a chunk of X, which the reductions' scratch shares
size_t energy_smem(int Dp) {
    const size_t x = sizeof(float) * (size_t)Dp * EC, scratch = sizeof(double) * (ET / 32 + 4) * EP;
    return sizeof(float) * (size_t)Dp * EP + std::max(x, scratch);
}

template <bool LOGIT>
__global__ void __launch_bounds__(ET, 2) k_regression_energy(DevModel m, TrajArgs a) {
    extern __shared__ __align__(16) float sm[];
    const int Dp = m.Dp, D = m.D, n = m.n;
    float* const th_s = sm;                // [Dp][EP]
    float* const x_s = sm + Dp * EP;       // [EC][Dp]
    double* const red = reinterpret_cast<double*>(x_s);          // [8 warps][EP]
    double* const e_s = red + ET / 32 * EP;                       // [4][EP]
    __shared__ double ll_s[SEGS][EP];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int kc = (int)a.c_split, rank = (int)tc::cluster_rank();
    const int64_t j0 = (int64_t)(blockIdx.x / kc) * EP;
    const bool evalm = a.eval_only != 0;
    // theta^T; rows past D and columns past N are zero
    for (int e = tid; e < Dp * EP; e += ET) {
        const int d = e / EP;
        const int64_t j = j0 + e % EP;
        float v = 0.0f;
        if (d < D && j < a.N)
            v = evalm ? a.theta_in[(int64_t)d * a.ld + (a.src ? a.src[j] : j)] : a.theta_out[(int64_t)d * a.ld + j];
        th_s[e] = v;
    }
    const int og = tid >> 4, pg = tid & 15;      // observations 8 og .., particles 4 pg .. and 64 + 4 pg ..
    const float inv_s = LOGIT ? 0.0f : (float)(1.0 / m.h0);
    const int nch = (n + EC - 1) / EC;
    const int per = SEGS / kc;                   // this CTA's segments: rank * per ..
    for (int seg = rank * per; seg < (rank + 1) * per; ++seg) {
        const int c_lo = (int)((int64_t)seg * nch / SEGS), c_hi = (int)((int64_t)(seg + 1) * nch / SEGS);
        double ll[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) ll[k] = 0.0;
        for (int c = c_lo; c < c_hi; ++c) {
            const int64_t row0 = (int64_t)c * EC;
            const int rows = (int)(n - row0 < EC ? n - row0 : EC);
            __syncthreads();                         // the previous chunk is used up
            const float* src = m.X + row0 * Dp;
            for (int v = tid; v < rows * Dp / 4; v += ET) tc::cp_async16(x_s + 4 * v, src + 4 * v);
            tc::cp_async_commit();
            tc::cp_async_wait<0>();
            __syncthreads();
            uint64_t acc[8][4];
#pragma unroll
            for (int o = 0; o < 8; ++o)
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[o][k] = 0ull;
            const float* xr = x_s + 8 * og * Dp;
            const float* tr = th_s + 4 * pg;
#pragma unroll 2
            for (int d = 0; d < Dp; d += 2) {
                float2 x[8];
#pragma unroll
                for (int o = 0; o < 8; ++o) x[o] = *reinterpret_cast<const float2*>(xr + o * Dp + d);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const ulonglong2 t0 = *reinterpret_cast<const ulonglong2*>(tr + (d + u) * EP);
                    const ulonglong2 t1 = *reinterpret_cast<const ulonglong2*>(tr + (d + u) * EP + 64);
#pragma unroll
                    for (int o = 0; o < 8; ++o) {
                        const float xv = u ? x[o].y : x[o].x;
                        const uint64_t xx = tc::f32x2_pack(xv, xv);
                        acc[o][0] = tc::f32x2_fma(xx, t0.x, acc[o][0]);
                        acc[o][1] = tc::f32x2_fma(xx, t0.y, acc[o][1]);
                        acc[o][2] = tc::f32x2_fma(xx, t1.x, acc[o][2]);
                        acc[o][3] = tc::f32x2_fma(xx, t1.y, acc[o][3]);
                    }
                }
            }
            float part[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) part[k] = 0.0f;
#pragma unroll
            for (int o = 0; o < 8; ++o) {
                const int64_t i = row0 + 8 * og + o;
                if (i >= n) continue;                // rows past the data hold what was there before
                const float yv = __ldg(m.y + i);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    float lo, hi;
                    tc::f32x2_unpack(acc[o][k / 2], lo, hi);
                    const float eta = (k & 1) ? hi : lo;
                    float term;
                    if (LOGIT) {
                        const float sp = softplus(eta);
                        term = yv * eta - sp;
                    } else {
                        const float z = (yv - eta) * inv_s;
                        term = -0.5f * z * z;
                    }
                    part[k] += term;
                }
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) ll[k] += widen(part[k]);
        }
        // the segment's sums: lane pairs, then warps, in order
        __syncthreads();                             // the last chunk is used up
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            ll[k] += __shfl_xor_sync(0xffffffffu, ll[k], 16);
            if (lane < 16) red[wid * EP + (k < 4 ? 4 * pg : 60 + 4 * pg) + k] = ll[k];
        }
        __syncthreads();
        if (tid < EP) {
            double s = 0.0;
            for (int w = 0; w < ET / 32; ++w) s += red[w * EP + tid];
            ll_s[seg][tid] = s;
        }
    }
    // |theta|^2 and |p|^2, half of the dimensions a thread (rank 0's are used)
    if (rank == 0) {
        const int p = tid & (EP - 1), h = tid / EP;
        const int64_t j = j0 + p;
        double sq = 0.0, kin = 0.0;
        for (int d = h; d < D; d += 2) {
            const double t = widen(th_s[d * EP + p]);
            sq += t * t;
            if (!evalm && a.dH && j < a.N) {
                const double v = widen(a.p_out[(int64_t)d * a.ld + j]);
                kin += v * v;
            }
        }
        e_s[h * EP + p] = sq;
        e_s[(2 + h) * EP + p] = kin;
    }
    __syncthreads();
    tc::cluster_sync();                          // every CTA's sums are in its shared memory
    const int64_t j = j0 + tid;
    if (rank == 0 && tid < EP && j < a.N) {
        double s = 0.0;
        for (int g = 0; g < SEGS; ++g)
            s += tc::ld_cluster_f64(tc::map_to_rank(tc::smem_u32(&ll_s[g][tid]), (uint32_t)(g / per)));
        const double inv_tau2 = LOGIT ? 1.0 / (m.h0 * m.h0) : 1.0 / (m.h1 * m.h1);
        const double lp1 = s - 0.5 * (e_s[tid] + e_s[EP + tid]) * inv_tau2 + m.lconst;
        a.logpi_out[j] = lp1;
        if (!evalm && a.dH) {
            double dH = (0.5 * (e_s[2 * EP + tid] + e_s[3 * EP + tid]) - lp1) - a.dH[j];   // H_0, left there by the trajectories
            if (!isfinite(dH)) dH = CUDART_INF;
            a.dH[j] = dH;
            if (a.alpha) a.alpha[j] = dH <= 0.0 ? 1.0 : exp(-dH);
        }
    }
    tc::cluster_sync();                          // nobody leaves while its sums may be read
}

template <bool LOGIT>
cudaError_t launch_energy(const DevModel& m, const TrajArgs& a, cudaStream_t s) {
    static int sms = 0;
    if (sms == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
            sms = 1;
    }
    const size_t smem = energy_smem(m.Dp);
    auto kern = k_regression_energy<LOGIT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // CTAs per particle tile (a cluster, each with a share of the chunks): the
    // split that leaves the fullest SM the least, a CTA's start counted as two
    // chunks (128 tiles on 152 SMs: split by 8, not one CTA on each of 128)
    const int64_t tiles = (a.N + EP - 1) / EP, nch = (m.n + EC - 1) / EC;
    int64_t best = 0;
    int split = 1;
    for (int k = 1; k <= 8 && k <= nch; k *= 2) {
        const int64_t cost = (tiles * k + sms - 1) / sms * ((nch + k - 1) / k + 2);
        if (k == 1 || cost < best) {
            best = cost;
            split = k;
        }
    }
    TrajArgs a2 = a;
    a2.c_split = split;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * split));
    cfg.blockDim = dim3(ET);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)split;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, m, a2);
}

}  // namespace

// log pi of the N positions in theta_out (eval_only: theta_in) into logpi_out;
// with dH, which holds H_0 and whose momenta are in p_out, also Delta H and alpha.
// D <= 128.
cudaError_t launch_regression_energy(const DevModel& m, const TrajArgs& a, cudaStream_t s) {
    if ((m.kind != LOGISTIC && m.kind != LINEAR_GAUSS) || m.D > 128 || (a.dH && !a.eval_only && !a.p_out) ||
        (a.alpha && !a.dH))
        return cudaErrorInvalidValue;
    return m.kind == LOGISTIC ? launch_energy<true>(m, a, s) : launch_energy<false>(m, a, s);
}

}  // namespace smc
