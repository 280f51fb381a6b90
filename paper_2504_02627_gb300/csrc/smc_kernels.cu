// smc_kernels.cu -- the SMC stages around the trajectories (Algorithm 3 of
// arXiv 2504.02627): initial draw and weights, weight normalisation and ESS,
// fixed-point systematic resampling with a decoupled look-back scan, Halton
// jitter and step counts with a counting sort by step count, and the
// reweighting / evidence / ChEES-adaptation epilogue.
#include <algorithm>
#include <cmath>
#include <math_constants.h>
#include "smc_kernels.cuh"

namespace smc {

constexpr int RUN_THREADS = 1024;
constexpr double LOG_2PI = 1.8378770664093454835606594728112;

// ============================================================ initial draw
// theta_0 ~ q_init = N(0, s^2 I) (Eq. for theta_0), or N(m, L L') when the
// run has a general Gaussian initial distribution, and log q_init(theta_0)
// parked in logw until the target has been evaluated.  Bound by FP64 (a pair of
// normals is some 90 instructions, 64 clocks each in a warp), so a particle's
// pairs are spread over the INIT_SPLIT warps of a CTA of 32 particles (a thread
// per particle had 256 particles of 10 dimensions on one SM: the whole run of ten
// iterations 786 -> 752 us with the split; ten runs of 4096 x 25 155 -> 89 us here).
constexpr int INIT_SPLIT = 4;
__global__ void __launch_bounds__(32 * INIT_SPLIT) k_init_draw(StepBufs b, float* theta) {
    __shared__ double zz_s[INIT_SPLIT][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t j = (int64_t)blockIdx.x * 32 + lane;
    const bool on = j < b.N;
    const RunParams rp = b.runs[on ? b.run_of[j] : 0];
    const uint32_t jl = (uint32_t)(j - rp.off);
    if (on && rp.init_general && w == 0) {
        // theta_d = m_d + L_d0 z_0 + ... + L_dd z_d in FP64, added column by
        // column (the same order for every d), every product and sum rounded
        // on its own (no contraction), so the result is that of the plain
        // sum written in this order
        double acc[MAX_CHEES_DIM];
        const int64_t D = b.D;
        for (int64_t d = 0; d < D; ++d) acc[d] = rp.init_mean ? rp.init_mean[d] : 0.0;
        double zz = 0.0;
        for (int64_t e = 0; e < D; e += 2) {
            double z[2];
            normal_pair(rp.seed, (uint32_t)(e >> 1), jl, 0u, TAG_INIT, z[0], z[1]);
            for (int u = 0; u < 2 && e + u < D; ++u) {
                const int64_t c = e + u;
                zz = __dadd_rn(zz, __dmul_rn(z[u], z[u]));
                if (rp.init_chol) {
                    for (int64_t d = c; d < D; ++d) acc[d] = __dadd_rn(acc[d], __dmul_rn(rp.init_chol[d * D + c], z[u]));
                } else {
                    acc[c] = __dadd_rn(acc[c], __dmul_rn(rp.init_scale, z[u]));
                }
            }
        }
        for (int64_t d = 0; d < D; ++d) theta[d * b.ld + j] = (float)acc[d];
        b.logw[j] = __dsub_rn(-0.5 * zz, __dadd_rn(__dmul_rn(0.5 * (double)D, LOG_2PI), rp.init_logdet));
    }
    // a particle of a general run is done (its run's other lanes too: every lane
    // still reaches the barrier)
    const bool iso = on && !rp.init_general;
    double zz = 0.0;
    if (iso)
        for (int64_t d = 2 * w; d < b.D; d += 2 * INIT_SPLIT) {
            double z0, z1;
            normal_pair(rp.seed, (uint32_t)(d >> 1), jl, 0u, TAG_INIT, z0, z1);
            theta[d * b.ld + j] = (float)(rp.init_scale * z0);
            zz += z0 * z0;
            if (d + 1 < b.D) {
                theta[(d + 1) * b.ld + j] = (float)(rp.init_scale * z1);
                zz += z1 * z1;
            }
        }
    zz_s[w][lane] = zz;
    __syncthreads();
    if (!iso || w != 0) return;
    for (int u = 1; u < INIT_SPLIT; ++u) zz += zz_s[u][lane];
    b.logw[j] = -0.5 * zz - 0.5 * (double)b.D * (LOG_2PI + 2.0 * log(rp.init_scale));
}

// Resampling uniform of iteration k: Philox block (0, 0, k, RESAMPLE).
__device__ __forceinline__ unsigned long long resample_r64(uint64_t seed, int64_t k) {
    const Philox4 w = philox4x32_10(Philox4{0u, 0u, (uint32_t)k, TAG_RESAMPLE}, seed);
    return ((unsigned long long)w.x << 32) | w.y;
}

// Decision for the next iteration from the current log-weights: LSE, ESS
// (Eqs. for W and J_eff) and the resampling test J_eff < frac J (Sec. 3).
__device__ __forceinline__ void set_decision(RunState& st, const RunParams& rp, double m, double lse, double ess,
                                             double L) {
    if (!(m > -CUDART_INF)) {
        st.status = -4;
        st.resample = 0;
        return;
    }
    st.lse = lse;
    st.ess_pre = ess;
    st.resample = ess < rp.ess_frac * (double)rp.n;
    st.L_used = L;
    st.T = 0ull;
    st.r64 = resample_r64(rp.seed, st.k);
}

// w_1 = pi(theta_0) / q_init(theta_0) (Eq. for w_1); log Z_0 = LSE(log w) - log J;
// and the weight decision of iteration 1.
__global__ void __launch_bounds__(RUN_THREADS) k_init_finish(StepBufs b, const double* logpi) {
    __shared__ double buf[2 * 32], tot_s[2];
    __shared__ long long lbuf[32];
    const int r = blockIdx.x;
    const RunParams rp = b.runs[r];
    long long mk = order_key(-CUDART_INF);
    for (int64_t i = threadIdx.x; i < rp.n; i += blockDim.x) {
        const int64_t j = rp.off + i;
        const double lp = logpi[j];
        // independent chains (Algorithm 2) carry no importance weight
        const double lw = rp.mcmc ? 0.0 : (isfinite(lp) ? lp - b.logw[j] : -CUDART_INF);
        b.logw[j] = lw;
        mk = max(mk, order_key(lw));
    }
    const double m = from_order_key(block_reduce(mk, lbuf, OpMax()));
    double s = 0.0, s2 = 0.0;
    if (m > -CUDART_INF)
        for (int64_t i = threadIdx.x; i < rp.n; i += blockDim.x) {
            const double e = exp(b.logw[rp.off + i] - m);
            s += e;
            s2 += e * e;
        }
    const double sums[2] = {s, s2};
    const double tot = block_sums(sums, buf);
    if (threadIdx.x < 2) tot_s[threadIdx.x] = tot;
    __syncthreads();
    if (threadIdx.x == 0) {
        s = tot_s[0];
        s2 = tot_s[1];
        RunState& st = b.rstate[r];
        const double lse = (m > -CUDART_INF) ? m + log(s) : -CUDART_INF;
        st.log_z = (m > -CUDART_INF) ? lse - rp.log_n : -CUDART_INF;
        st.status = 0;
        set_decision(st, rp, m, lse, s * s / s2, exp(st.log_L));
        b.done[r] = 0u;
    }
}

// atomicAdd(&counter[key], number of active lanes with this key) once per
// distinct key in the warp; returns this lane's old-value-plus-rank (the
// warp-aggregated form: particles of a warp often share a step count)
__device__ __forceinline__ int warp_agg_inc(int* counter, int key) {
    const unsigned peers = __match_any_sync(__activemask(), key);
    const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(counter + key, __popc(peers));
    base = __shfl_sync(peers, base, leader);
    return base + __popc(peers & ((1u << lane) - 1u));
}

// ============================================================ weights + steps
// Per particle slice: normalised weight W_j = exp(log w_j - LSE), the
// fixed-point weight q_j = floor(W_j 2^S) with S = 62 - ceil(log2 N) when the
// run resamples (its slice total is added to T with an exact integer atomic),
// the 1-d Halton jitter h_j of n = j K + k (Sec. 3.2), the step count
// S_j = ceil(h_j L / eps) clipped to [1, max] (Algorithm 2), and the
// histogram of S_j for the counting sort.
__global__ void __launch_bounds__(SLICE) k_weights_steps(StepBufs b) {
    __shared__ unsigned long long ubuf[32];
    const int c = blockIdx.x;
    const int r = b.slice_run[c];
    const RunParams& rp = b.runs[r];
    RunState& st = b.rstate[r];
    if (c == 0 && threadIdx.x == 0) {
        b.counter[0] = 0u;      // dynamic scan-tile counter of the next launch
        b.counter[1] += 1u;     // look-back epoch: never repeats within a handle
    }
    const int64_t i = b.slice_start[c] + threadIdx.x;
    const bool valid = i < rp.n;
    const int64_t j = rp.off + i;
    const bool ok = st.status == 0;
    unsigned long long qi = 0ull;
    if (valid) {
        int32_t S = 0;
        if (ok) {
            const double w = exp(b.logw[j] - st.lse);
            b.W[j] = w;
            if (st.resample) {
                int sh = 0;
                while (((int64_t)1 << sh) < rp.n) ++sh;
                const double v = w * ldexp(1.0, 62 - sh);
                qi = v > 0.0 ? __double2ull_rz(v) : 0ull;
                b.q[j] = qi;
            }
            const double h = jitter_h(rp.jitter, rp.seed, i, st.k, rp.n, rp.n_iters, b.primes);
            S = step_count(h, st.L_used, st.eps, rp.max_steps);
        }
        b.steps[j] = S;
        warp_agg_inc(b.hist, b.max_steps_all - S);
    }
    if (ok && st.resample) {
        qi = block_reduce(qi, ubuf, OpSum());
        if (threadIdx.x == 0 && qi) atomicAdd(&st.T, qi);
    }
}

// ============================================================ resampling scan
// Inclusive prefix C of q within each run by a single-pass decoupled
// look-back scan (tiles of SCAN_TILE elements; a tile id is taken from an
// atomic counter, so every predecessor tile has already started).  Each
// particle j then owns the output slots i with N C_{j-1} <= i T + U < N C_j,
// i.e. [cnt(C_{j-1}), cnt(C_j)) with cnt(C) = ceil((N C - U) / T) clipped to
// [0, N], and writes its own index there (systematic resampling).  Runs that
// do not resample write the identity source index.
constexpr long long LOOKBACK_SPIN_LIMIT = 1ll << 22;

// floor(X / T) with rT = 1 / (float)T: the FP32 quotient is off by at most
// about 2^-22 of itself, so two of them (the second on the remainder) leave
// the exact quotient within one unit, which the two loops settle.  About 25
// instructions instead of the roughly 100 of the 64-bit division; T up to
// 2^62 (every normalised weight vector) keeps the remainders in an int64,
// larger totals divide.
__host__ __device__ __forceinline__ unsigned long long quotient_u64(unsigned long long X, unsigned long long T, float rT) {
    if (T >> 62) return X / T;
    unsigned long long c = (unsigned long long)((float)X * rT);
    long long rem = (long long)(X - c * T);
    const long long d = (long long)((float)rem * rT);
    c += (unsigned long long)d;
    rem -= d * (long long)T;
    while (rem < 0) {
        --c;
        rem += (long long)T;
    }
    while (rem >= (long long)T) {
        ++c;
        rem -= (long long)T;
    }
    return c;
}

__device__ __forceinline__ unsigned long long systematic_count(unsigned long long C, unsigned long long N,
                                                               unsigned long long T, unsigned long long U, float rT) {
    const unsigned long long NC = N * C;
    if (NC <= U) return 0ull;
    const unsigned long long c = quotient_u64(NC - U + T - 1ull, T, rT);
    return c < N ? c : N;
}

// Decoupled look-back of tile g, by the 32 lanes of one warp: publishes the
// tile's aggregate, walks back over the predecessors of its run (tiles first ..
// g-1), 32 descriptors at a time, summing aggregates until an inclusive prefix,
// and publishes its own inclusive prefix.  (One thread walking tile by tile
// pays an L2 round trip per predecessor.)  Every wait on
// a predecessor is bounded: after `limit` polls without progress it gives up,
// sets *failed (*status is set to -5 before the publication) and returns the
// partial sum; the tile still publishes, so no successor waits forever.
// Returns the exclusive prefix of the tile to every lane.
__device__ unsigned long long lookback_prefix(TileDesc* tiles, int64_t g, int64_t first, unsigned int epoch,
                                              unsigned long long tile_agg, long long limit, int* status,
                                              bool& failed) {
    TileDesc* me = tiles + g;
    const int lane = threadIdx.x & 31;
    unsigned long long excl = 0ull;
    failed = false;
    if (g == first) {
        if (lane == 0) {
            me->incl = tile_agg;
            __threadfence();
            atomicExch(&me->flag, (epoch << 2) | 2u);
        }
        return 0ull;
    }
    if (lane == 0) {
        me->agg = tile_agg;
        __threadfence();
        atomicExch(&me->flag, (epoch << 2) | 1u);
    }
    int64_t pred = g - 1;
    long long spins = 0;
    while (true) {
        // lane l reads predecessor pred - l; lanes before the run's first tile
        // count as ready and empty (the first tile publishes its prefix, so
        // the walk ends there)
        const int64_t t = pred - lane;
        const bool in = t >= first;
        const volatile TileDesc* pd = tiles + (in ? t : first);
        const unsigned int f = in ? pd->flag : 0u;
        const bool ready = !in || ((f >> 2) == epoch && (f & 3u) != 0u);
        const unsigned rmask = __ballot_sync(0xffffffffu, ready);
        const unsigned imask = __ballot_sync(0xffffffffu, in && ready && (f & 3u) == 2u);
        const int n_ready = rmask == 0xffffffffu ? 32 : __ffs(~rmask) - 1;   // ready lanes without a gap
        const int n_incl = imask ? __ffs(imask) - 1 : 32;                     // nearest inclusive prefix
        if (n_ready > 0) {
            __threadfence();
            const bool done = n_incl < n_ready;
            const int n = done ? n_incl + 1 : n_ready;
            unsigned long long v = 0ull;
            if (in && lane < n) v = lane == n_incl ? pd->incl : pd->agg;
            excl += warp_sum(v);
            if (done) break;
            pred -= n;
            spins = 0;
            continue;
        }
        if (++spins > limit) {   // bounded wait: report, never hang
            if (lane == 0) {
                *(volatile int*)status = -5;
                __threadfence();
            }
            failed = true;
            break;
        }
        __nanosleep(64);
    }
    if (lane == 0) {
        me->incl = excl + tile_agg;
        __threadfence();
        atomicExch(&me->flag, (epoch << 2) | 2u);
    }
    return excl;
}

// Output ranges longer than EMIT_SHORT slots are written by a warp (by the
// whole CTA from EMIT_BLOCK on) instead of their particle's thread: where a few
// particles hold the mass (the first weighting of a run), one thread writing
// its range slot by slot is the whole launch.
constexpr unsigned int EMIT_SHORT = 8, EMIT_BLOCK = 2048;

struct EmitList {
    unsigned int lo[SCAN_TILE], hi[SCAN_TILE];   // a tile's long output ranges
    int i[SCAN_TILE];
    int n;
};

// Inclusive prefixes of this thread's SCAN_ITEMS consecutive values (zero past
// n); returns the exclusive prefix of the thread within the tile and, in
// tile_agg, the tile's total.
__device__ __forceinline__ unsigned long long tile_scan(const unsigned long long* q, int64_t base, int64_t n,
                                                        unsigned long long (&v)[SCAN_ITEMS], unsigned long long* wsum,
                                                        unsigned long long& tile_agg) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    unsigned long long acc = 0ull;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        const int64_t i = base + (int64_t)tid * SCAN_ITEMS + k;
        acc += i < n ? q[i] : 0ull;
        v[k] = acc;
    }
    unsigned long long x = acc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    unsigned long long before = 0ull;
    tile_agg = 0ull;
#pragma unroll
    for (int w = 0; w < SCAN_THREADS / 32; ++w) {
        before += w < wid ? wsum[w] : 0ull;
        tile_agg += wsum[w];
    }
    return before + (x - acc);
}

// Systematic resampling of a tile: particle i (run-local) owns the output slots
// [cnt(C_{i-1}), cnt(C_i)), C its inclusive prefix off + v.  list.n is zero
// and all threads are past a barrier since then.
__device__ __forceinline__ void emit_systematic(const unsigned long long (&v)[SCAN_ITEMS], unsigned long long off,
                                                int64_t base, int64_t n, unsigned long long T, unsigned long long U,
                                                int32_t* anc, int32_t* src, int32_t src0, EmitList& list) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned long long N = (unsigned long long)n;
    const float rT = 1.0f / (float)T;
    // a particle's range ends where the next one's begins: one count per particle
    unsigned int lo = (unsigned int)systematic_count(off, N, T, U, rT);
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        const int64_t i = base + (int64_t)tid * SCAN_ITEMS + k;
        if (i >= n) break;
        const unsigned int hi = (unsigned int)systematic_count(off + v[k], N, T, U, rT);
        if (hi - lo > EMIT_SHORT && hi > lo) {
            const int e = atomicAdd(&list.n, 1);   // the list's order does not matter: disjoint ranges
            list.lo[e] = lo;
            list.hi[e] = hi;
            list.i[e] = (int)i;
        } else {
            for (unsigned int o = lo; o < hi; ++o) {
                anc[o] = (int32_t)i;
                if (src) src[o] = src0 + (int32_t)i;
            }
        }
        lo = hi;
    }
    __syncthreads();
    const int nl = list.n;
    for (int e = 0; e < nl; ++e) {
        const unsigned int l = list.lo[e], h = list.hi[e];
        const int32_t i = list.i[e];
        const bool by_block = h - l >= EMIT_BLOCK;
        if (!by_block && (e % (SCAN_THREADS / 32)) != wid) continue;
        const unsigned int step = by_block ? SCAN_THREADS : 32u;
        for (unsigned int o = l + (by_block ? (unsigned)tid : (unsigned)lane); o < h; o += step) {
            anc[o] = i;
            if (src) src[o] = src0 + i;
        }
    }
}

__global__ void __launch_bounds__(SCAN_THREADS) k_resample_scan(StepBufs b) {
    __shared__ unsigned int tile_s;
    __shared__ unsigned long long wsum[SCAN_THREADS / 32];
    __shared__ unsigned long long excl_s;
    __shared__ int failed_s;
    __shared__ EmitList list;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid == 0) {
        tile_s = atomicAdd(b.counter, 1u);
        list.n = 0;
    }
    __syncthreads();
    const int64_t g = tile_s;
    if (g >= b.n_tiles) return;
    const int r = b.tile_run ? b.tile_run[g] : 0;
    const RunParams rp = b.runs[r];
    RunState& st = b.rstate[r];
    const int64_t t_in_run = g - rp.tile0;
    const int64_t base = t_in_run * SCAN_TILE;
    if (!st.resample || st.status != 0) {
        if (b.src)
            for (int k = 0; k < SCAN_ITEMS; ++k) {
                const int64_t i = base + (int64_t)k * SCAN_THREADS + tid;
                if (i < rp.n) b.src[rp.off + i] = (int32_t)(rp.off + i);
            }
        return;
    }
    const unsigned int epoch = b.counter[1] & 0x3fffffffu;
    const unsigned long long T = st.T;
    if (T == 0ull) {                 // no mass at all: degenerate
        if (tid == 0) st.status = -4;
        return;
    }
    const unsigned long long U = __umul64hi(st.r64, T);

    unsigned long long v[SCAN_ITEMS], tile_agg;
    const unsigned long long thread_excl = tile_scan(b.q + rp.off, base, rp.n, v, wsum, tile_agg);

    // look-back over predecessor tiles of the same run
    if (wid == 0) {
        bool failed;
        const unsigned long long excl =
            lookback_prefix(b.tiles, g, rp.tile0, epoch, tile_agg, LOOKBACK_SPIN_LIMIT, &st.status, failed);
        // a run whose look-back gave up anywhere (here or in a predecessor,
        // whose status store precedes its publication) gets no resampling from
        // this tile on: identity source indices for the tile's own slots
        if (lane == 0) {
            excl_s = excl;
            failed_s = failed || *(volatile int*)&st.status != 0;
        }
    }
    __syncthreads();
    if (failed_s) {
        for (int k = 0; k < SCAN_ITEMS; ++k) {
            const int64_t i = base + (int64_t)k * SCAN_THREADS + tid;
            if (i < rp.n) {
                b.anc[rp.off + i] = (int32_t)i;
                if (b.src) b.src[rp.off + i] = (int32_t)(rp.off + i);
            }
        }
        return;
    }
    const unsigned long long off = excl_s + thread_excl;
    // multinomial: the prefix is kept for k_multinomial_search; systematic:
    // particle i of the run owns output slots [cnt(C_{i-1}), cnt(C_i))
    if (rp.resample_scheme == 1) {
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; ++k) {
            const int64_t i = base + (int64_t)tid * SCAN_ITEMS + k;
            if (i < rp.n) b.cprefix[rp.off + i] = off + v[k];
        }
        return;
    }
    emit_systematic(v, off, base, rp.n, T, U, b.anc + rp.off, b.src ? b.src + rp.off : nullptr, (int32_t)rp.off, list);
}

// Multinomial resampling (the paper's scheme, Sec. 3) after the scan: output
// i of a resampling run takes the first particle j whose inclusive prefix C_j
// exceeds P_i = floor(u_i T / 2^64), u_i the 64-bit word pair of Philox block
// (1, i, k, RESAMPLE): a binary search over the run's prefix (C_{n-1} = T > P_i).
__global__ void k_multinomial_search(StepBufs b) {
    const int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= b.N) return;
    const int r = b.run_of ? b.run_of[o] : 0;
    const RunParams& rp = b.runs[r];
    const RunState& st = b.rstate[r];
    if (rp.resample_scheme != 1 || !st.resample || st.status != 0) return;
    const int64_t i = o - rp.off;
    const Philox4 w = philox4x32_10(Philox4{1u, (uint32_t)i, (uint32_t)st.k, TAG_RESAMPLE}, rp.seed);
    const unsigned long long u = ((unsigned long long)w.x << 32) | w.y;
    const unsigned long long P = __umul64hi(u, st.T);
    const unsigned long long* C = b.cprefix + rp.off;
    int64_t lo = 0, hi = rp.n - 1;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (C[mid] > P) hi = mid;
        else lo = mid + 1;
    }
    b.anc[o] = (int32_t)lo;
    if (b.src) b.src[o] = (int32_t)(rp.off + lo);
}

// ============================================================ sort by steps
// Exclusive scan of the step histogram (one CTA), in place.
__global__ void __launch_bounds__(1024) k_hist_scan(StepBufs b) {
    __shared__ int wsum[32];
    const int nb = b.max_steps_all + 1;
    int carry = 0;
    for (int base = 0; base < nb; base += blockDim.x) {
        const int i = base + threadIdx.x;
        const int v = i < nb ? b.hist[i] : 0;
        int x = v;
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[wid] = x;
        __syncthreads();
        if (wid == 0) {
            int w = lane < (int)(blockDim.x >> 5) ? wsum[lane] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                int y = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += y;
            }
            wsum[lane] = w;
        }
        __syncthreads();
        const int excl = carry + (x - v) + (wid > 0 ? wsum[wid - 1] : 0);
        const int total = wsum[(blockDim.x >> 5) - 1];
        __syncthreads();
        if (i < nb) b.hist[i] = excl;
        carry += total;
    }
}

// Slot of each particle in descending-step order, so that particles with
// similar trajectory lengths share a CTA / warp in the trajectory kernels.
__global__ void k_sort_scatter(StepBufs b) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= b.N) return;
    const int slot = warp_agg_inc(b.hist, b.max_steps_all - b.steps[j]);
    b.perm[slot] = (int32_t)j;
}

// Resampling and order of one run that fits a scan tile, in one CTA instead of
// three kernels of one CTA each (11 us one after the other, now 5): the
// tile's prefix needs no look-back, and the step histogram is scanned and its
// slots taken in shared memory.
constexpr int SMALL_BINS = 4096;
static bool small_order(const StepBufs& b) { return b.n_runs == 1 && b.n_tiles == 1 && b.max_steps_all < SMALL_BINS; }
__global__ void __launch_bounds__(SCAN_THREADS) k_resample_order_small(StepBufs b) {
    __shared__ unsigned long long wsum[SCAN_THREADS / 32];
    __shared__ EmitList list;
    __shared__ int slot[SMALL_BINS], wcnt[SCAN_THREADS / 32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid == 0) list.n = 0;
    // the first slot of each step count, longest first
    const int nb = b.max_steps_all + 1, per = (nb + SCAN_THREADS - 1) / SCAN_THREADS;
    int cnt = 0;
    for (int i = tid; i < nb; i += SCAN_THREADS) slot[i] = b.hist[i];
    __syncthreads();
    for (int i = tid * per; i < min(nb, (tid + 1) * per); ++i) cnt += slot[i];
    int x = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wcnt[wid] = x;
    __syncthreads();
    int first = x - cnt;
    for (int w = 0; w < wid; ++w) first += wcnt[w];
    for (int i = tid * per; i < min(nb, (tid + 1) * per); ++i) {
        const int c = slot[i];
        slot[i] = first;
        first += c;
    }
    __syncthreads();
    const int n = (int)b.N;
    for (int j = tid; j < n; j += SCAN_THREADS) b.perm[warp_agg_inc(slot, b.max_steps_all - b.steps[j])] = j;

    RunState& st = b.rstate[0];
    const RunParams& rp = b.runs[0];
    if (!st.resample || st.status != 0) {
        for (int j = tid; j < n; j += SCAN_THREADS) b.src[j] = j;
        return;
    }
    const unsigned long long T = st.T;
    __syncthreads();                 // everyone has read the status
    if (T == 0ull) {                 // no mass at all: degenerate
        if (tid == 0) st.status = -4;
        return;
    }
    unsigned long long v[SCAN_ITEMS], tile_agg;
    const unsigned long long off = tile_scan(b.q, 0, n, v, wsum, tile_agg);
    if (rp.resample_scheme == 1) {
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; ++k)
            if (tid * SCAN_ITEMS + k < n) b.cprefix[tid * SCAN_ITEMS + k] = off + v[k];
        return;
    }
    emit_systematic(v, off, 0, n, T, __umul64hi(st.r64, T), b.anc, b.src, 0, list);
}

// ============================================================ move statistics
// Per particle slice (first pass): with the momentum change-of-variable
// L-kernel the Jacobians cancel and log w += -Delta H (Sec. 3.1); pieces of
// log sum_j W_j exp(-Delta H_j) (evidence factor), of the new ESS, sum alpha,
// sum S_j, and the ChEES column sums of the pre-move and proposed states.
struct SliceIdx {
    int r;
    int64_t i, j;
    bool valid;
};
__device__ __forceinline__ SliceIdx slice_idx(const StepBufs& b) {
    SliceIdx x;
    const int c = blockIdx.x;
    x.r = b.slice_run[c];
    x.i = b.slice_start[c] + threadIdx.x;
    x.valid = x.i < b.runs[x.r].n;
    x.j = b.runs[x.r].off + x.i;
    return x;
}

__global__ void __launch_bounds__(SLICE) k_move_stats(StepBufs b) {
    __shared__ double buf[5 * 32];
    __shared__ long long lbuf[2 * 32];
    __shared__ int ibuf[2 * 32];
    const SliceIdx x = slice_idx(b);
    const RunParams& rp = b.runs[x.r];
    const RunState& st = b.rstate[x.r];
    const int c = blockIdx.x;
    // the step histogram of the next iteration starts empty (this one's order
    // has been made)
    for (int i = c * SLICE + threadIdx.x; i <= b.max_steps_all; i += gridDim.x * SLICE) b.hist[i] = 0;
    if (st.status != 0) return;
    double za = -CUDART_INF, lw = -CUDART_INF, al = 0.0;
    long long S = 0;
    int smin = 0x7fffffff, smax = 0;
    if (x.valid) {
        // with the Metropolis select the incremental weight is one
        const double dH = rp.accept_reject ? 0.0 : b.dH[x.j];
        const double old = b.logw[x.j];
        za = (st.resample ? -rp.log_n : old - st.lse) - dH;
        lw = (st.resample ? -rp.log_n : old) - dH;
        b.logw[x.j] = lw;
        al = b.alpha[x.j];
        S = b.steps[x.j];
        smin = smax = (int)S;
    }
    // the slice's reductions, each with block_reduce's tree, in three passes:
    // the two maxima (by their bits), then the sums that need them; the
    // integer parts.  After resampling the two log-weights are the same value.
    SlicePart& part = b.parts[c];
    double* const pd = reinterpret_cast<double*>(&part);   // za_m, za_s, w_m, w_e1, w_e2, alpha_sum, inv_alpha_sum
    long long mx[2] = {order_key(za), order_key(lw)};
    block_reduce_n(mx, lbuf, OpMax());
    const double za_m = from_order_key(mx[0]), w_m = from_order_key(mx[1]);
    const double e = (x.valid && w_m > -CUDART_INF) ? exp(lw - w_m) : 0.0;
    const double ez = st.resample ? e : (za_m > -CUDART_INF ? exp(za - za_m) : 0.0);
    const bool step_rule = rp.step_rate > 0.0 && st.k < rp.n_warmup;
    if (step_rule) {
        const double sm[5] = {ez, e, e * e, al, x.valid ? 1.0 / al : 0.0};
        const double r = block_sums(sm, buf);
        if (threadIdx.x < 5) pd[threadIdx.x == 0 ? 1 : threadIdx.x + 2] = r;
    } else {
        const double sm[4] = {ez, e, e * e, al};
        const double r = block_sums(sm, buf);
        if (threadIdx.x < 4) pd[threadIdx.x == 0 ? 1 : threadIdx.x + 2] = r;
        if (threadIdx.x == 4) part.inv_alpha_sum = 0.0;
    }
    long long ls[1] = {S};
    block_reduce_n(ls, lbuf, OpSum());
    int mm[2] = {-smin, smax};   // min S as -max(-S)
    block_reduce_n(mm, ibuf, OpMax());
    if (threadIdx.x == 0) {
        part.za_m = za_m;
        part.w_m = w_m;
        part.steps_sum = ls[0];
        part.smin = -mm[0];
        part.smax = mm[1];
        part.g_num = 0.0;
        part.g_den = 0.0;
    }
    if (rp.adapt && st.k < rp.n_warmup) {
        // ChEES column sums of the pre-move states (after resampling) and the
        // proposals: warp w takes dimensions w, w + SLICE / 32, ...; a lane
        // sums its particles lane, lane + 32, ... of the slice in order, then
        // the warp adds its lanes (fixed order)
        constexpr int PL = SLICE / 32;   // particles per lane
        const int D = (int)b.D, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        const int64_t i0 = b.slice_start[c];
        int64_t jj[PL], ss[PL];
#pragma unroll
        for (int u = 0; u < PL; ++u) {
            const int64_t i = i0 + lane + 32 * u;
            jj[u] = i < rp.n ? rp.off + i : -1;
            ss[u] = (jj[u] >= 0 && !b.chees0) ? b.src[jj[u]] : 0;
        }
        // two dimensions per pass, their loads issued together
        const float* t0 = b.chees0 ? b.chees0 : b.theta_prev;
        const float* t1 = b.chees1 ? b.chees1 : b.theta_new;
        for (int d = wid; d < D; d += 2 * (SLICE / 32)) {
            const int d2 = d + SLICE / 32;
            float a0[2][PL], a1[2][PL];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int dd = h ? d2 : d;
                const int64_t o = (int64_t)dd * b.ld;
#pragma unroll
                for (int u = 0; u < PL; ++u) {
                    const bool in = jj[u] >= 0 && dd < D;
                    a0[h][u] = in ? t0[o + (b.chees0 ? jj[u] : ss[u])] : 0.0f;
                    a1[h][u] = in ? t1[o + jj[u]] : 0.0f;
                }
            }
            f2sum v[4];                                  // FP32 pairs (about 48 bits): d before, after, d2 before, after
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                f2sum v0{0.0f, 0.0f}, v1{0.0f, 0.0f};
#pragma unroll
                for (int u = 0; u < PL; ++u) {
                    if (jj[u] < 0) continue;
                    v0 = f2_add_f(v0, a0[h][u]);
                    v1 = f2_add_f(v1, a1[h][u]);
                }
                v[2 * h] = v0;
                v[2 * h + 1] = v1;
            }
            const f2sum t = warp_sum4_f2(v, lane);
            const int w = lane >> 3, dd = (w & 2) ? d2 : d;
            if ((lane & 7) == 0 && dd < D) b.colsum[(int64_t)c * 2 * D + ((w & 1) ? D : 0) + dd] = f2_to_double(t);
        }
    }
}

// Bound by FP64 (an exponential is some 25 instructions) and by the pair sums
// over the dimensions: 64 hierarchical runs, 278k particles, 129 -> 60 us; one
// run of 256 particles 13 -> 8 us.
//
// Second pass: ChEES gradient estimates g_j = l_j (|t1_j - mean t1|^2 -
// |t0_j - mean t0|^2) (t1_j - mean t1)' p_j weighted by alpha_j (Algorithm 2),
// then the last slice of each run combines every slice in a fixed order:
// evidence, log-weights' ESS, Adam ascent on log L, Lbar, the freeze at
// M_warmup, statistics, and the weight decision of the next iteration.  One run of
// 256 particles: 34 -> 20 us alone and cold, the FP64 latency of the last slice's
// chain and the fetch of the unrolled sums; 64 hierarchical runs: 115 -> 103 us,
// the pair arithmetic.
__global__ void __launch_bounds__(SLICE) k_chees_finish(StepBufs b) {
    __shared__ double buf[7 * 32], tot_s[7], res_s[4];
    __shared__ long long lbuf[2 * 32];
    __shared__ int ibuf[2 * 32];
    __shared__ float mean_s[4 * MAX_CHEES_DIM];   // negated means as FP32 pairs: hi [2D], lo [2D]
    __shared__ bool last_s;
    const SliceIdx x = slice_idx(b);
    const RunParams& rp = b.runs[x.r];
    RunState& st = b.rstate[x.r];
    if (st.status != 0) return;
    const int c = blockIdx.x;
    const int D = (int)b.D;
    const bool adapting = rp.adapt && st.k < rp.n_warmup;
    if (adapting) {
        // loads are issued in batches ahead of the sums (the sums keep their
        // order): a serial load-then-add loop waits one L2 round trip per term
        constexpr int BQ = 8;
        for (int t = threadIdx.x; t < 2 * D; t += blockDim.x) {
            double s = 0.0;
            const double* cs = b.colsum + (int64_t)rp.slice0 * 2 * D + t;
            int q = 0;
            for (; q + BQ <= rp.n_slices; q += BQ) {
                double v[BQ];
#pragma unroll
                for (int u = 0; u < BQ; ++u) v[u] = cs[(int64_t)(q + u) * 2 * D];
#pragma unroll
                for (int u = 0; u < BQ; ++u) s += v[u];
            }
            for (; q < rp.n_slices; ++q) s += cs[(int64_t)q * 2 * D];
            // the mean as a negated FP32 pair, ready to add to each value
            const f2sum m = f2_from_double(s / (double)rp.n);
            mean_s[t] = -m.hi;
            mean_s[2 * D + t] = -m.lo;
        }
        __syncthreads();
        double num = 0.0, den = 0.0;
        if (x.valid) {
            const int64_t src = b.src[x.j];
            const int64_t j0 = b.chees0 ? x.j : src;
            const float* t0 = b.chees0 ? b.chees0 : b.theta_prev;
            const float* t1 = b.chees1 ? b.chees1 : b.theta_new;
            // |t - mean|^2 and the projection, sums of products of FP32 pairs
            f2dot sq0{0.0f, 0.0f, 0.0f}, sq1{0.0f, 0.0f, 0.0f}, proj{0.0f, 0.0f, 0.0f};
            constexpr int BD = 8;
            for (int d0 = 0; d0 < D; d0 += BD) {
                float v0[BD], v1[BD], vp[BD];
#pragma unroll
                for (int u = 0; u < BD; ++u) {
                    const int64_t o = (int64_t)(d0 + u) * b.ld;
                    const bool in = d0 + u < D;
                    v0[u] = in ? t0[o + j0] : 0.0f;
                    v1[u] = in ? t1[o + x.j] : 0.0f;
                    vp[u] = in ? b.p_final[o + x.j] : 0.0f;
                }
#pragma unroll
                for (int u = 0; u < BD; ++u) {
                    const int d = d0 + u;
                    if (d >= D) break;
                    const f2sum e0 = f2_add_f(f2sum{mean_s[d], mean_s[2 * D + d]}, v0[u]);
                    const f2sum e1 = f2_add_f(f2sum{mean_s[D + d], mean_s[3 * D + d]}, v1[u]);
                    f2_dot(sq0, e0, e0);
                    f2_dot(sq1, e1, e1);
                    f2_dot(proj, e1, f2sum{vp[u], 0.0f});
                }
            }
            const double h = jitter_h(rp.jitter, rp.seed, x.i, st.k, rp.n, rp.n_iters, b.primes);
            const double a = b.alpha[x.j];
            num = a * ((h * st.L_used) * (f2_to_double(sq1) - f2_to_double(sq0)) * f2_to_double(proj));
            den = a;
        }
        const double nd[2] = {num, den};
        const double r = block_sums(nd, buf);
        if (threadIdx.x < 2) (threadIdx.x == 0 ? b.parts[c].g_num : b.parts[c].g_den) = r;
    }
    // Metropolis variant (Eqs. for alpha and the select rule): keep the
    // proposal when u < alpha, otherwise restore the start state; the ChEES
    // statistics above used the proposals, as in Algorithm 2.
    if (rp.accept_reject && x.valid) {
        const Philox4 w = philox4x32_10(Philox4{0u, (uint32_t)x.i, (uint32_t)st.k, TAG_MH}, rp.seed);
        if (!(u01_52(w.x, w.y) < b.alpha[x.j])) {
            const int64_t src = b.src[x.j];
            for (int d = 0; d < D; ++d) {
                b.theta_new[(int64_t)d * b.ld + x.j] = b.theta_prev[(int64_t)d * b.ld + src];
                b.grad_new[(int64_t)d * b.ld + x.j] = b.grad_prev[(int64_t)d * b.ld + src];
            }
            b.logpi_new[x.j] = b.logpi_prev[src];
        }
    }
    // ticket: the last slice of the run to get here finishes the iteration
    if (threadIdx.x < 2) __threadfence();   // the threads that wrote this slice's sums
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned int t = atomicAdd(&b.done[x.r], 1u);
        last_s = (t == (unsigned int)rp.n_slices - 1u);
    }
    __syncthreads();
    if (!last_s) return;
    __threadfence();
    // fixed-order combination of the run's slices: thread t takes slices
    // t, t + SLICE, ... and the block reduces in a fixed tree
    // (the other slices' parts are read from L2 with cache-global loads, after
    // the fence that followed the ticket, so no stale L1 copy is seen)
    long long mx[2] = {order_key(-CUDART_INF), order_key(-CUDART_INF)};
    for (int q = threadIdx.x; q < rp.n_slices; q += blockDim.x) {
        const SlicePart* p = b.parts + rp.slice0 + q;
        mx[0] = max(mx[0], order_key(__ldcg(&p->za_m)));
        mx[1] = max(mx[1], order_key(__ldcg(&p->w_m)));
    }
    block_reduce_n(mx, lbuf, OpMax());
    const double za_m = from_order_key(mx[0]), w_m = from_order_key(mx[1]);
    double za_s = 0.0, w_e1 = 0.0, w_e2 = 0.0, asum = 0.0, gnum = 0.0, gden = 0.0, iasum = 0.0;
    long long ssum = 0;
    int smin = 0x7fffffff, smax = 0;
    for (int q = threadIdx.x; q < rp.n_slices; q += blockDim.x) {
        const SlicePart* pp = b.parts + rp.slice0 + q;
        SlicePart p;
        p.za_m = __ldcg(&pp->za_m);
        p.za_s = __ldcg(&pp->za_s);
        p.w_m = __ldcg(&pp->w_m);
        p.w_e1 = __ldcg(&pp->w_e1);
        p.w_e2 = __ldcg(&pp->w_e2);
        p.alpha_sum = __ldcg(&pp->alpha_sum);
        p.inv_alpha_sum = __ldcg(&pp->inv_alpha_sum);
        p.g_num = __ldcg(&pp->g_num);
        p.g_den = __ldcg(&pp->g_den);
        p.steps_sum = __ldcg(&pp->steps_sum);
        p.smin = __ldcg(&pp->smin);
        p.smax = __ldcg(&pp->smax);
        if (p.za_m > -CUDART_INF) za_s += p.za_s * exp(p.za_m - za_m);
        if (p.w_m > -CUDART_INF) {
            const double f = exp(p.w_m - w_m);
            w_e1 += p.w_e1 * f;
            w_e2 += p.w_e2 * f * f;
        }
        asum += p.alpha_sum;
        iasum += p.inv_alpha_sum;
        gnum += p.g_num;
        gden += p.g_den;
        ssum += p.steps_sum;
        smin = min(smin, p.smin);
        smax = max(smax, p.smax);
    }
    // the run's sums, each with block_reduce's tree, in one pass per type
    {
        const double sm[7] = {za_s, w_e1, w_e2, asum, iasum, gnum, gden};
        const double r = block_sums(sm, buf);
        if (threadIdx.x < 7) tot_s[threadIdx.x] = r;
    }
    long long ls[1] = {ssum};
    block_reduce_n(ls, lbuf, OpSum());
    ssum = ls[0];
    int mm[2] = {-smin, smax};   // min S as -max(-S)
    block_reduce_n(mm, ibuf, OpMax());
    smin = -mm[0];
    smax = mm[1];
    // (the barriers above order tot_s)
    // The run's update is a chain of FP64 logarithms, exponentials and
    // divisions, a microsecond each in one thread: its independent parts run in
    // one warp each.  Warp 1: the evidence factor; warp 2: the new LSE; warp 3:
    // the ESS and the mean acceptance; warp 0: Adam on log L.
    const int wid = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0 && wid > 0) {
        if (wid == 1) res_s[0] = za_m > -CUDART_INF ? za_m + log(tot_s[0]) : -CUDART_INF;
        if (wid == 2) res_s[1] = w_m > -CUDART_INF ? w_m + log(tot_s[1]) : -CUDART_INF;
        if (wid == 3) {
            res_s[2] = w_m > -CUDART_INF ? tot_s[1] * tot_s[1] / tot_s[2] : 0.0;
            res_s[3] = tot_s[3] / (double)rp.n;
        }
    }
    const int64_t k = st.k;
    double L_next = 0.0;      // exp(log L) of the next iteration
    if (threadIdx.x == 0) {
        bool have = false;
        double log_L = st.log_L;
        if (adapting) {
            gnum = tot_s[5];
            gden = tot_s[6];
            if (gden > 0.0 && isfinite(gnum / gden)) {
                const double gh = gnum / gden;
                st.adam_t += 1.0;
                st.adam_m = rp.adam_b1 * st.adam_m + (1.0 - rp.adam_b1) * gh;
                st.adam_v = rp.adam_b2 * st.adam_v + (1.0 - rp.adam_b2) * gh * gh;
                st.adam_b1t *= rp.adam_b1;     // b1^t, b2^t by running products (no FP64 pow)
                st.adam_b2t *= rp.adam_b2;
                const double mh = st.adam_m / (1.0 - st.adam_b1t);
                const double vh = st.adam_v / (1.0 - st.adam_b2t);
                log_L += rp.adam_lr * mh / (sqrt(vh) + rp.adam_eps);
                // clamp L to [eps, max_steps eps] of this iteration's step size
                const double lo = rp.step_rate > 0.0 ? log(st.eps) : rp.log_L_lo;
                const double hi = rp.step_rate > 0.0 ? log((double)rp.max_steps * st.eps) : rp.log_L_hi;
                log_L = fmin(fmax(log_L, lo), hi);
            }
            L_next = exp(log_L);
            have = true;
            st.Lbar = 0.9 * st.Lbar + 0.1 * L_next;
        }
        if (rp.adapt && k == rp.n_warmup && st.Lbar > 0.0) {
            log_L = log(st.Lbar);
            have = false;
        }
        st.log_L = log_L;
        if (!have) L_next = exp(log_L);
        // optional warm-up step-size rule (not in the paper), after the ChEES
        // update: log eps += rate (a_h - target), a_h = n / sum 1/alpha_j the
        // harmonic mean (0 when some alpha_j = 0: the sum is +inf)
        if (rp.step_rate > 0.0 && k < rp.n_warmup)
            st.eps = exp(log(st.eps) + rp.step_rate * ((double)rp.n / tot_s[4] - rp.step_target));
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    const double inc = res_s[0];
    st.log_z += inc;
    st.log_z_inc = inc;
    st.mean_alpha = res_s[3];
    st.ess = res_s[2];
    st.stat_ess_pre = st.ess_pre;
    st.stat_resampled = st.resample;
    st.L_last = st.L_used;
    st.grad_evals = ssum;
    st.steps_min = smin;
    st.steps_max = smax;
    st.iters_total += 1;
    st.grad_evals_total += ssum;
    st.resamples_total += st.resample;
    st.ess_sum += st.ess;
    if (k > rp.n_warmup) st.ess_sum_post += st.ess;
    st.k = k + 1;
    set_decision(st, rp, w_m, res_s[1], res_s[2], L_next);
    b.done[x.r] = 0u;
}

// ============================================================ launchers
cudaError_t launch_init_draw(const StepBufs& b, float* theta, cudaStream_t s) {
    k_init_draw<<<(unsigned)((b.N + 31) / 32), 32 * INIT_SPLIT, 0, s>>>(b, theta);
    return cudaGetLastError();
}
cudaError_t launch_init_finish(const StepBufs& b, const double* logpi, cudaStream_t s) {
    k_init_finish<<<(unsigned)b.n_runs, RUN_THREADS, 0, s>>>(b, logpi);
    return cudaGetLastError();
}
cudaError_t launch_weights_steps(const StepBufs& b, cudaStream_t s) {
    k_weights_steps<<<(unsigned)b.n_slices, SLICE, 0, s>>>(b);
    return cudaGetLastError();
}
cudaError_t launch_resample_scan(const StepBufs& b, cudaStream_t s) {
    if (small_order(b)) k_resample_order_small<<<1, SCAN_THREADS, 0, s>>>(b);
    else k_resample_scan<<<(unsigned)b.n_tiles, SCAN_THREADS, 0, s>>>(b);
    if (b.any_multinomial && b.N > 0) k_multinomial_search<<<(unsigned)((b.N + 255) / 256), 256, 0, s>>>(b);
    return cudaGetLastError();
}
int kernels_per_iteration(const StepBufs& b) { return small_order(b) ? 5 : 7; }
cudaError_t launch_sort(const StepBufs& b, cudaStream_t s) {
    if (small_order(b)) return cudaSuccess;   // with the resampling
    const int bs = 256;
    k_hist_scan<<<1, 1024, 0, s>>>(b);
    k_sort_scatter<<<(unsigned)((b.N + bs - 1) / bs), bs, 0, s>>>(b);
    return cudaGetLastError();
}
cudaError_t launch_move_stats(const StepBufs& b, cudaStream_t s) {
    if (b.D > MAX_CHEES_DIM) return cudaErrorInvalidValue;
    k_move_stats<<<(unsigned)b.n_slices, SLICE, 0, s>>>(b);
    k_chees_finish<<<(unsigned)b.n_slices, SLICE, 0, s>>>(b);
    return cudaGetLastError();
}

// ============================================================ stand-alone stages
__global__ void k_philox(uint64_t seed, const uint32_t* ctr, uint32_t* out, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Philox4 w = philox4x32_10(Philox4{ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]}, seed);
    out[4 * i] = w.x;
    out[4 * i + 1] = w.y;
    out[4 * i + 2] = w.z;
    out[4 * i + 3] = w.w;
}
cudaError_t launch_philox(uint64_t seed, const uint32_t* ctr, uint32_t* out, int64_t n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_philox<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(seed, ctr, out, n);
    return cudaGetLastError();
}

__global__ void k_normals(uint64_t seed, uint32_t tag, uint32_t k, int64_t N, int64_t D, double* out,
                          int64_t ld) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    for (int64_t d = 0; d < D; d += 2) {
        double z0, z1;
        normal_pair(seed, (uint32_t)(d >> 1), (uint32_t)j, k, tag, z0, z1);
        out[d * ld + j] = z0;
        if (d + 1 < D) out[(d + 1) * ld + j] = z1;
    }
}
cudaError_t launch_normals(uint64_t seed, uint32_t tag, uint32_t k, int64_t N, int64_t D, double* out,
                           int64_t ld, cudaStream_t s) {
    if (N <= 0) return cudaSuccess;
    k_normals<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(seed, tag, k, N, D, out, ld);
    return cudaGetLastError();
}

__global__ void k_jitter_only(int32_t scheme, uint64_t seed, int64_t J, int64_t K, int64_t k,
                              const int32_t* primes, double* out_h) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= J) return;
    out_h[i] = jitter_h(scheme, seed, i, k, J, K, primes);
}
cudaError_t launch_jitter_only(int32_t scheme, uint64_t seed, int64_t J, int64_t K, int64_t k,
                               const int32_t* primes, double* out_h, cudaStream_t s) {
    if (J <= 0) return cudaSuccess;
    k_jitter_only<<<(unsigned)((J + 255) / 256), 256, 0, s>>>(scheme, seed, J, K, k, primes, out_h);
    return cudaGetLastError();
}
__global__ void k_steps_only(int64_t N, int64_t K, int64_t k, double L, double eps, int32_t max_steps,
                             int32_t jitter, double* out_h, int32_t* out_steps) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    const double h = jitter ? halton2((uint32_t)(j * K + k)) : 1.0;
    if (out_h) out_h[j] = h;
    out_steps[j] = step_count(h, L, eps, max_steps);
}
cudaError_t launch_steps_only(int64_t N, int64_t K, int64_t k, double L, double eps, int32_t max_steps,
                              int32_t jitter, double* out_h, int32_t* out_steps, cudaStream_t s) {
    if (N <= 0) return cudaSuccess;
    k_steps_only<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(N, K, k, L, eps, max_steps, jitter, out_h,
                                                             out_steps);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(RUN_THREADS) k_normalise_flat(const double* logw, int64_t N, double* W,
                                                                double* lse_out, double* ess_out) {
    __shared__ double buf[32];
    double m = -CUDART_INF;
    for (int64_t i = threadIdx.x; i < N; i += blockDim.x) m = fmax(m, logw[i]);
    m = block_reduce(m, buf, OpMax());
    if (!(m > -CUDART_INF)) {
        for (int64_t i = threadIdx.x; i < N; i += blockDim.x) W[i] = 0.0;
        if (threadIdx.x == 0) {
            *lse_out = -CUDART_INF;
            *ess_out = 0.0;
        }
        return;
    }
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < N; i += blockDim.x) s += exp(logw[i] - m);
    s = block_reduce(s, buf, OpSum());
    const double lse = m + log(s);
    double s2 = 0.0;
    for (int64_t i = threadIdx.x; i < N; i += blockDim.x) {
        const double w = exp(logw[i] - lse);
        W[i] = w;
        s2 += w * w;
    }
    s2 = block_reduce(s2, buf, OpSum());
    if (threadIdx.x == 0) {
        *lse_out = lse;
        *ess_out = 1.0 / s2;
    }
}
// The same over the whole GPU, for more than one CTA's worth of weights.  FP64
// exponentials bound it (an SM retires about two FP64 operations per clock),
// so each is taken once, relative to the largest of its CTA's share, and
// scaled when the total is known; one CTA took 962 us at 100003 weights,
// separate exponentials for the sum and the weights over the whole GPU 32,
// this 27.  The partials (max, sum exp, sum exp^2 of each CTA's contiguous
// share) wait in the first 3 gridDim.x entries of W, whose exponentials a last
// small kernel takes again, so nothing is allocated.
constexpr int NORM_THREADS = 512, NORM_MAX_PARTS = 152;   // a share per SM
__device__ __forceinline__ int64_t norm_share(int64_t N, int64_t parts, int64_t b) { return N * b / parts; }
__global__ void __launch_bounds__(NORM_THREADS) k_norm_part(const double* logw, int64_t N, double* W) {
    __shared__ double buf[2 * 32], tot_s[2];
    __shared__ long long lbuf[32];
    const int64_t lo = norm_share(N, gridDim.x, blockIdx.x), hi = norm_share(N, gridDim.x, blockIdx.x + 1);
    long long mk = order_key(-CUDART_INF);
    int nan = 0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += NORM_THREADS) {
        const double x = logw[i];
        if (isnan(x)) nan = 1;
        else mk = max(mk, order_key(x));
    }
    const double m = from_order_key(block_reduce(mk, lbuf, OpMax()));
    const bool mass = m > -CUDART_INF;
    double s[2] = {0.0, 0.0};
    for (int64_t i = lo + threadIdx.x; i < hi; i += NORM_THREADS) {
        const double x = logw[i];
        // without mass the share is -inf and NaN
        const double e = mass ? exp(x - m) : (nan && isnan(x) ? x : 0.0);
        s[0] += e;
        s[1] += e * e;
        if (i >= 3 * (int64_t)gridDim.x) W[i] = e;
    }
    const double r = block_sums(s, buf);
    if (threadIdx.x < 2) tot_s[threadIdx.x] = r;
    __syncthreads();
    if (threadIdx.x < 3) W[3 * (int64_t)blockIdx.x + threadIdx.x] = threadIdx.x == 0 ? m : tot_s[threadIdx.x - 1];
}
// Every CTA combines the partials and scales its share; CTA 0 also writes the
// scalars.
__global__ void __launch_bounds__(NORM_THREADS) k_norm_scale(double* W, int64_t N, int n_parts, double* lse_out,
                                                             double* ess_out) {
    __shared__ double buf[2 * 32], tot_s[2], f_s;
    __shared__ long long lbuf[32];
    const int p = threadIdx.x;
    const bool in = p < n_parts;
    const double m = in ? W[3 * p] : -CUDART_INF;
    const double M = from_order_key(block_reduce(order_key(m), lbuf, OpMax()));
    double s[2] = {0.0, 0.0};
    if (in) {
        const double f = m > -CUDART_INF ? exp(m - M) : 1.0;   // without mass the sums are 0, or NaN
        s[0] = W[3 * p + 1] * f;
        s[1] = W[3 * p + 2] * f * f;
    }
    const double r = block_sums(s, buf);
    if (threadIdx.x < 2) tot_s[threadIdx.x] = r;
    __syncthreads();
    const bool any = M > -CUDART_INF;
    if (threadIdx.x == 0) {
        const double lse = any ? M + log(tot_s[0]) : -CUDART_INF;
        if (blockIdx.x == 0) {
            *lse_out = lse;
            *ess_out = any ? tot_s[0] * tot_s[0] / tot_s[1] : 0.0;
        }
        // W_i = exp(x_i - m_b) exp(m_b - lse), m_b this share's largest
        f_s = any ? exp(W[3 * (int64_t)blockIdx.x] - lse) : 0.0;
    }
    __syncthreads();
    const double f = f_s;
    const int64_t first = 3 * (int64_t)n_parts;
    const int64_t lo = norm_share(N, n_parts, blockIdx.x), hi = norm_share(N, n_parts, blockIdx.x + 1);
    for (int64_t i = max(lo, first) + threadIdx.x; i < hi; i += NORM_THREADS) W[i] = any ? W[i] * f : 0.0;
}
// The entries that held the partials.
constexpr int FIRST_THREADS = 64;   // a few warps of exponentials per SM (1e5 weights: 26.6 -> 24.6 us a call; 512: one SM)
__global__ void __launch_bounds__(FIRST_THREADS) k_norm_first(const double* logw, int64_t n, const double* lse, double* W) {
    const int64_t i = (int64_t)blockIdx.x * FIRST_THREADS + threadIdx.x;
    if (i >= n) return;
    const double l = *lse;
    W[i] = l == -CUDART_INF ? 0.0 : exp(logw[i] - l);
}

cudaError_t launch_normalise_flat(const double* logw, int64_t N, double* W, double* lse, double* ess,
                                  cudaStream_t s) {
    if (N <= 0) return cudaErrorInvalidValue;
    const int64_t nb = std::min<int64_t>((N + NORM_THREADS - 1) / NORM_THREADS, NORM_MAX_PARTS);
    // one CTA: a single share, or weights written over the log-weights (W holds
    // the partials while the log-weights are still read)
    const bool overlap = W < logw + N && logw < W + N;
    if (nb == 1 || overlap) {
        k_normalise_flat<<<1, RUN_THREADS, 0, s>>>(logw, N, W, lse, ess);
        return cudaGetLastError();
    }
    k_norm_part<<<(unsigned)nb, NORM_THREADS, 0, s>>>(logw, N, W);
    k_norm_scale<<<(unsigned)nb, NORM_THREADS, 0, s>>>(W, N, (int)nb, lse, ess);
    k_norm_first<<<(unsigned)((3 * nb + FIRST_THREADS - 1) / FIRST_THREADS), FIRST_THREADS, 0, s>>>(logw, 3 * nb, lse, W);
    return cudaGetLastError();
}

// Stand-alone systematic resampling of given normalised weights W.
struct FlatScratch {
    RunParams rp;
    RunState st;
    unsigned int counter[4];
};
static int64_t flat_tiles(int64_t N) { return (N + SCAN_TILE - 1) / SCAN_TILE; }
int64_t resample_scratch_bytes(int64_t N) {
    return (int64_t)(((sizeof(FlatScratch) + 255) / 256) * 256 + sizeof(TileDesc) * (size_t)flat_tiles(N));
}

// q_j = floor(W_j 2^S), with the total of every scan tile.  Bound by memory: 16
// bytes per weight (one CTA over all of them took most of the 942 us of a
// 1M-particle resampling).
__global__ void __launch_bounds__(SCAN_THREADS) k_quantise_flat(const double* W, int64_t N, unsigned long long* q,
                                                                unsigned long long* agg, double scale) {
    __shared__ unsigned long long ubuf[32];
    unsigned long long T = 0ull;
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + threadIdx.x;
    double w[SCAN_ITEMS];
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        const int64_t i = base + (int64_t)k * SCAN_THREADS;
        w[k] = i < N ? W[i] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        const int64_t i = base + (int64_t)k * SCAN_THREADS;
        const double v = w[k] * scale;
        const unsigned long long qi = v > 0.0 ? __double2ull_rz(v) : 0ull;
        if (i < N) q[i] = qi;
        T += qi;
    }
    T = block_reduce(T, ubuf, OpSum());
    if (threadIdx.x == 0) agg[blockIdx.x] = T;
}

// The ancestors where the tiles' totals are at hand: every CTA adds up those
// before its tile, and all of them, itself (two round trips to L2, where the
// look-back's walk takes one per 32 tiles): 1048576 weights 46 -> 30 us in all.
constexpr int64_t FLAT_DIRECT_TILES = 2048;   // 4194304 particles: 16 KB of totals per CTA
__global__ void __launch_bounds__(SCAN_THREADS) k_resample_flat(const unsigned long long* q, int64_t N, uint64_t r64,
                                                                const unsigned long long* agg, int32_t* anc,
                                                                int32_t* status) {
    __shared__ unsigned long long wsum[SCAN_THREADS / 32], ubuf[2 * 32];
    __shared__ EmitList list;
    if (threadIdx.x == 0) list.n = 0;
    unsigned long long t[2] = {0ull, 0ull};   // before this tile, all
    for (int64_t g = threadIdx.x; g < gridDim.x; g += SCAN_THREADS) {
        const unsigned long long x = agg[g];
        t[0] += g < blockIdx.x ? x : 0ull;
        t[1] += x;
    }
    block_reduce_n(t, ubuf, OpSum());
    const unsigned long long T = t[1];
    if (blockIdx.x == 0 && threadIdx.x == 0) *status = T == 0ull ? -4 : 0;   // no mass at all: degenerate
    if (T == 0ull) return;
    unsigned long long v[SCAN_ITEMS], tile_agg;
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    const unsigned long long off = t[0] + tile_scan(q, base, N, v, wsum, tile_agg);
    emit_systematic(v, off, base, N, T, __umul64hi((unsigned long long)r64, T), anc, nullptr, 0, list);
}

// With more tiles the scan looks back; its header from the tiles' totals, which
// lie where its descriptors will (they are zeroed in between).
__global__ void __launch_bounds__(RUN_THREADS) k_flat_header(FlatScratch* fs, const unsigned long long* agg, int64_t N,
                                                             uint64_t r64, int64_t n_tiles) {
    __shared__ unsigned long long ubuf[32];
    unsigned long long T = 0ull;
    for (int64_t g = threadIdx.x; g < n_tiles; g += RUN_THREADS) T += agg[g];
    T = block_reduce(T, ubuf, OpSum());
    if (threadIdx.x == 0) {
        RunParams rp = {};
        rp.n = N;
        rp.n_tiles = (int32_t)n_tiles;
        fs->rp = rp;
        RunState st = {};
        st.k = 1;
        st.T = T;
        st.r64 = (unsigned long long)r64;
        st.resample = 1;            // T == 0 is found (status -4) by the scan
        fs->st = st;
        fs->counter[0] = 0u;
        fs->counter[1] = 1u;        // the descriptors' epoch
    }
}
__global__ void k_copy_status(const FlatScratch* fs, int32_t* status) { *status = fs->st.status; }

// The look-back wait of the resampling scan against a predecessor that never
// publishes: tile 1 of a two-tile run whose tile 0 descriptor holds no flag
// of the current epoch, with the caller's poll limit; the wait must give up
// and report -5 in *status (device), never hang.
__global__ void k_lookback_wait_check(TileDesc* tiles, long long limit, int* status) {
    if (threadIdx.x == 0) {
        tiles[0].flag = 0u;   // epoch 0, not ready: nothing will ever publish it
        tiles[0].agg = tiles[0].incl = 0ull;
        *status = 0;
        __threadfence();
    }
    __syncwarp();
    bool failed;
    (void)lookback_prefix(tiles, 1, 0, 1u, 1ull, limit, status, failed);
    if (!failed && threadIdx.x == 0) *status = 1;   // cannot happen: the predecessor never publishes
}
cudaError_t launch_lookback_wait_check(long long limit, TileDesc* tiles, int* status, cudaStream_t s) {
    k_lookback_wait_check<<<1, 32, 0, s>>>(tiles, limit, status);
    return cudaGetLastError();
}

cudaError_t launch_resample_flat(const double* W, int64_t N, uint64_t r64, unsigned long long* q,
                                 int32_t* anc, int32_t* status, void* scratch, cudaStream_t s) {
    if (N <= 0 || N > (1ll << 30)) return cudaErrorInvalidValue;
    const int64_t nt = flat_tiles(N);
    FlatScratch* fs = reinterpret_cast<FlatScratch*>(scratch);
    TileDesc* tiles = reinterpret_cast<TileDesc*>(reinterpret_cast<char*>(scratch) +
                                                  ((sizeof(FlatScratch) + 255) / 256) * 256);
    int c = 0;
    while (((int64_t)1 << c) < N) ++c;
    unsigned long long* agg = reinterpret_cast<unsigned long long*>(tiles);
    k_quantise_flat<<<(unsigned)nt, SCAN_THREADS, 0, s>>>(W, N, q, agg, std::ldexp(1.0, 62 - c));
    if (nt <= FLAT_DIRECT_TILES) {
        k_resample_flat<<<(unsigned)nt, SCAN_THREADS, 0, s>>>(q, N, r64, agg, anc, status);
        return cudaGetLastError();
    }
    k_flat_header<<<1, RUN_THREADS, 0, s>>>(fs, agg, N, r64, nt);
    cudaError_t e = cudaMemsetAsync(tiles, 0, sizeof(TileDesc) * (size_t)nt, s);
    if (e != cudaSuccess) return e;
    StepBufs b = {};
    b.runs = &fs->rp;
    b.rstate = &fs->st;
    b.tile_run = nullptr;
    b.n_runs = 1;
    b.N = N;
    b.q = q;
    b.anc = anc;
    b.counter = fs->counter;
    b.tiles = tiles;
    b.n_tiles = nt;
    k_resample_scan<<<(unsigned)nt, SCAN_THREADS, 0, s>>>(b);
    k_copy_status<<<1, 1, 0, s>>>(fs, status);
    return cudaGetLastError();
}

}  // namespace smc
