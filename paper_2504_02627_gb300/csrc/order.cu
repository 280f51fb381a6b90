// order.cu -- launch order of a stage-level move: particles by descending step
// count, so that the particles of a tile, which run in lockstep, end together.
#include <cooperative_groups.h>
#include "traj.cuh"

namespace smc {
namespace {

namespace cg = cooperative_groups;
constexpr int ORDER_CTAS = 8, ORDER_THREADS = 1024, ORDER_BINS = 512;

// One cluster: every CTA takes a contiguous share of the particles; the range of
// the counts, then per-bin counts, then each share's slots per bin go through
// distributed shared memory.  Counts that span more than ORDER_BINS values
// share bins (an order within a five-hundredth of the range is enough), and
// equal counts come in any order: no result depends on it.  The kernel that
// reads the order may start at once (programmatic launch): it waits for this
// one's end before it reads it, and by then has loaded the model's data.
// 7 to 9 us at 8192 particles, all of it latency (an atomic's, a cluster barrier's).
__global__ void __cluster_dims__(ORDER_CTAS, 1, 1) __launch_bounds__(ORDER_THREADS)
    k_order_steps(const int32_t* steps, int64_t N, int32_t* perm) {
    __shared__ int range_s[2];              // this share's largest and smallest count
    __shared__ int hist[ORDER_BINS], offs[ORDER_BINS], wsum[32];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    cg::cluster_group cl = cg::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int rank = (int)cl.block_rank();
    const int64_t lo = N * rank / ORDER_CTAS, hi = N * (rank + 1) / ORDER_CTAS;
    if (tid == 0) {
        range_s[0] = INT32_MIN;
        range_s[1] = INT32_MAX;
    }
    for (int b = tid; b < ORDER_BINS; b += ORDER_THREADS) hist[b] = 0;
    __syncthreads();
    int mx = INT32_MIN, mn = INT32_MAX;
    for (int64_t i = lo + tid; i < hi; i += ORDER_THREADS) {
        const int s = steps[i];
        mx = max(mx, s);
        mn = min(mn, s);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    mn = __reduce_min_sync(0xffffffffu, mn);
    if (lane == 0) {
        atomicMax(&range_s[0], mx);
        atomicMin(&range_s[1], mn);
    }
    cl.sync();
    for (int r = 0; r < ORDER_CTAS; ++r) {
        const int* p = cl.map_shared_rank(range_s, r);
        mx = max(mx, p[0]);
        mn = min(mn, p[1]);
    }
    if (mx <= mn) {                          // equal counts: the particles as they are
        for (int64_t i = lo + tid; i < hi; i += ORDER_THREADS) perm[i] = (int32_t)i;
        cl.sync();                           // nobody leaves while its range may be read
        return;
    }
    const float scale = (float)ORDER_BINS / ((float)mx - (float)mn + 1.0f);
    auto bin = [&](int s) { return min(ORDER_BINS - 1, (int)(((float)mx - (float)s) * scale)); };
    for (int64_t i = lo + tid; i < hi; i += ORDER_THREADS) atomicAdd(&hist[bin(steps[i])], 1);
    cl.sync();
    // bin b starts after every share's earlier bins, and this share's part of it
    // after the lower ranks' parts
    int total = 0, before = 0;
    if (tid < ORDER_BINS)
        for (int r = 0; r < ORDER_CTAS; ++r) {
            const int h = cl.map_shared_rank(hist, r)[tid];
            if (r < rank) before += h;
            total += h;
        }
    int x = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    if (tid < ORDER_BINS) {
        int base = 0;
        for (int w = 0; w < wid; ++w) base += wsum[w];
        offs[tid] = base + x - total + before;
    }
    __syncthreads();
    for (int64_t i = lo + tid; i < hi; i += ORDER_THREADS) perm[atomicAdd(&offs[bin(steps[i])], 1)] = (int32_t)i;
    cl.sync();   // nobody leaves while its counts may be read
}

}  // namespace

cudaError_t launch_order_steps(const int32_t* steps, int64_t N, int32_t* perm, cudaStream_t s) {
    k_order_steps<<<ORDER_CTAS, ORDER_THREADS, 0, s>>>(steps, N, perm);
    return cudaGetLastError();
}

// Ordering pays where the particles of a tile share the longest trajectory, a step
// of the launch takes about a microsecond or more (some 5e7 operations, 1e8 on
// the matrix units; the move is over in the time that ordering takes below that)
// and there are more tiles than SMs: otherwise the longest tile is the launch,
// ordered or not, and only slower when all of its particles run on.  us in order
// / in the particles' own order, counts uniform on 0 .. 30, then all 15:
//   regression, n = 1000, D = 25, 16 particles a tile: 4096 particles 228 / 442, 242 / 237;
//     1000 particles 228 / 222
//   regression, n = 300, D = 64, 64 a tile: 12000 2620 / 3261; 4096 2366 / 2207
//   Gaussian in FP32, D = 100: 5000 123 / 163, 97 / 93; 10000 199 / 360; 8192, 128 tiles of
//     64, 199 / 183; D = 40, 20011 76 / 108, 68 / 63
// On tensor cores a tile's 16 lanes gather their particles, which short moves
// hardly repay: D = 80, 16384 particles in BF16x3, to 30 steps 84 / 84, to 100 158 / 228; in
// BF16 70 / 62 and 111 / 135; D = 64 to 30 69 / 65, D = 40 as much as it costs.
// The centred and the other tcgen05 kernels keep state at the particles' indices
// and read it every step, coalesced only in the particles' own order.
bool order_pays(const DevModel& m, int32_t precision, int64_t N) {
    const double n = (double)N;
    if (m.kind == GAUSS_DENSE && (precision == 1 || precision == 2)) return m.D > 64 && 2.0 * m.D * m.D * n >= 1e8;
    if (precision != 0) return false;
    int64_t tile;
    if (m.kind == GAUSS_DENSE && m.D > 32) {
        if (2.0 * m.D * m.D * n < 5e7) return false;
        tile = dense_tile(m, N);
    } else if (m.kind == LOGISTIC || m.kind == LINEAR_GAUSS) {
        if (4.0 * m.n * m.D * n < 5e7) return false;
        tile = glm_tile(m);
    } else {
        return false;
    }
    return (N + tile - 1) / tile > sm_count();
}

}  // namespace smc
