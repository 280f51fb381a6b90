// flow_mma.cu -- the BF16 forms of the learned preconditioner (flow.cu): HMC in
// the latent space of the coupling flow, and the gradient of its training loss,
// with every conditioner product on m16n8k16 warp MMAs (BF16 operands, FP32
// accumulation).
//
// A CTA holds 32 particles.  A product's operands are the weights, as
// fragments from L2, and the activations as BF16 particle-major rows in shared
// memory; its accumulators become the next product's operand without a detour:
// bias, tanh or tanh' are applied in registers and a transposing matrix store
// writes them back as particle-major rows (the hidden activations of the
// backward products stay in registers, since every product with H rows has
// the same fragment layout).  One barrier per product, and the next product's
// weights are requested before it.
//
// What bounds it is latency: a product is 32 MMAs a warp behind an L2 round
// trip and a barrier.  So the shared memory is cut until two CTAs share an SM
// (at D = 100, H = 128, L = 4: 103 and 111 KB; each layer keeps the half it
// changes, the other half being the half of its neighbour).  At that shape and
// 8192 particles (one wave of CTAs, two before): a move of four steps 921 ->
// 518 us, the training gradient 313 -> 199 us, of which this kernel 274 -> 153.
#include <cuda_bf16.h>
#include <math_constants.h>
#include "flow.cuh"
#include "tc_ptx.cuh"

namespace smc {
namespace {

constexpr int FG = 32;           // particles per CTA
constexpr int FT = 256;          // threads per CTA
constexpr int NW = FT / 32;
constexpr int LDB = 136;         // BF16 row stride of the particle-major operands: 17 16-byte units, conflict-free
constexpr int WLD = FG + 8;      // BF16 row stride of the weight-gradient operands

__device__ __forceinline__ void stsm4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b),
                 "r"(c), "r"(d)
                 : "memory");
}
__device__ __forceinline__ void stsm4_t(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b),
                 "r"(c), "r"(d)
                 : "memory");
}
__device__ __forceinline__ uint32_t pk(float x, float y) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// A warp's share of a product with MT 16-row tiles over 32 particles (four
// 8-column tiles): two pieces of one row tile and two neighbouring column
// tiles each.  With eight or more row tiles, both halves of row tile `wid`,
// else pieces wid and wid + 8 of the 2 MT.  Accumulators acc[2 h + u]: column
// tile nt(h) + u.
struct Piece {
    int MT, wid;
    __device__ bool both() const { return MT >= NW; }
    __device__ bool on(int h) const { return both() || wid + NW * h < 2 * MT; }
    __device__ int mt(int h) const { return both() ? wid : (wid + NW * h) >> 1; }
    __device__ int nt(int h) const { return both() ? 2 * h : 2 * ((wid + NW * h) & 1); }
};

struct Frag {
    uint4 a[8];
    // the row tile's K / 16 <= 8 fragments, all requested at once
    __device__ __forceinline__ void load(const uint4* __restrict__ Af, const Piece& pc, int h, int KS, int lane) {
        if (!pc.on(h)) return;
        const uint4* p = Af + (int64_t)pc.mt(h) * KS * 32 + lane;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
            if (ks < KS) a[ks] = __ldg(p + ks * 32);
    }
};

// acc = A . B for the warp's pieces; fr holds piece 0's fragments
__device__ __forceinline__ void product(Frag& fr, const uint4* __restrict__ Af, const Piece& pc, int KS, uint32_t pm,
                                        float (&acc)[4][4], int lane) {
    const int mi = lane >> 3, mr = lane & 7;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = 0.0f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (!pc.on(h)) continue;
        if (h == 1 && !pc.both()) fr.load(Af, pc, 1, KS, lane);
        const uint32_t b0 = pm + (uint32_t)(((8 * (pc.nt(h) + (mi >> 1)) + mr) * LDB + 8 * (mi & 1)) * 2);
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            if (ks >= KS) break;
            uint32_t b[4];
            tc::ldsm4(b, b0 + 32 * ks);
            const uint32_t av[4] = {fr.a[ks].x, fr.a[ks].y, fr.a[ks].z, fr.a[ks].w};
            tc::mma_bf16_16816(acc[2 * h], av, b[0], b[1]);
            tc::mma_bf16_16816(acc[2 * h + 1], av, b[2], b[3]);
        }
    }
}

// acc += bias of the row (rows below Mvalid), then tanh
template <bool TANH>
__device__ __forceinline__ void bias_act(float (&acc)[4][4], const Piece& pc, const float* __restrict__ bias, int Mvalid,
                                         int lane) {
    const int g = lane >> 2;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (!pc.on(h)) continue;
        const int r0 = 16 * pc.mt(h) + g, r1 = r0 + 8;
        const float b0 = r0 < Mvalid ? __ldg(bias + r0) : 0.0f, b1 = r1 < Mvalid ? __ldg(bias + r1) : 0.0f;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            float(&c)[4] = acc[2 * h + u];
            c[0] += b0;
            c[1] += b0;
            c[2] += b1;
            c[3] += b1;
            if (TANH) {
#pragma unroll
                for (int v = 0; v < 4; ++v) c[v] = tanhf(c[v]);
            }
        }
    }
}
// acc *= 1 - h^2
__device__ __forceinline__ void times_dtanh(float (&acc)[4][4], const float (&hv)[4][4]) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = acc[u][v] * (1.0f - hv[u][v] * hv[u][v]);
}

// accumulators as BF16: particle-major rows (the next product's operand) ...
__device__ __forceinline__ void store_pm(const float (&acc)[4][4], const Piece& pc, uint32_t pm, int lane) {
    const int mi = lane >> 3, mr = lane & 7;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (!pc.on(h)) continue;
        const float(&c0)[4] = acc[2 * h];
        const float(&c1)[4] = acc[2 * h + 1];
        stsm4_t(pm + (uint32_t)(((8 * (pc.nt(h) + (mi >> 1)) + mr) * LDB + 16 * pc.mt(h) + 8 * (mi & 1)) * 2),
                pk(c0[0], c0[1]), pk(c0[2], c0[3]), pk(c1[0], c1[1]), pk(c1[2], c1[3]));
    }
}
// ... and rows of particles (an operand of the weight-gradient products)
__device__ __forceinline__ void store_rows(const float (&acc)[4][4], const Piece& pc, uint32_t rows, int lane) {
    const int mi = lane >> 3, mr = lane & 7;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (!pc.on(h)) continue;
        const float(&c0)[4] = acc[2 * h];
        const float(&c1)[4] = acc[2 * h + 1];
        stsm4(rows + (uint32_t)(((16 * pc.mt(h) + 8 * (mi & 1) + mr) * WLD + 8 * (pc.nt(h) + (mi >> 1))) * 2),
              pk(c0[0], c0[1]), pk(c0[2], c0[3]), pk(c1[0], c1[1]), pk(c1[2], c1[3]));
    }
}
// accumulators into FP32 rows of particles (rows below Mvalid); ADD: added to
// what is there (each element belongs to one thread)
template <bool ADD>
__device__ __forceinline__ void store_f32(const float (&acc)[4][4], const Piece& pc, float* Y, int Mvalid, int lane) {
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (!pc.on(h)) continue;
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int r = 16 * pc.mt(h) + g + 8 * e;
                if (r >= Mvalid) continue;
                float2* y = reinterpret_cast<float2*>(Y + r * FG + 8 * (pc.nt(h) + u) + 2 * t);
                float2 v = make_float2(acc[2 * h + u][2 * e], acc[2 * h + u][2 * e + 1]);
                if (ADD) {
                    const float2 o = *y;
                    v.x = o.x + v.x;
                    v.y = o.y + v.y;
                }
                *y = v;
            }
    }
}

// Elementwise passes over [rows x 32]: a thread takes its lane's particle and
// blocks of eight rows, so FP32 row accesses are conflict-free and eight BF16
// values of a particle go out as 16 bytes.
__device__ __forceinline__ void put_pm8(__nv_bfloat16* pm, int q, int k0, const float (&v)[8]) {
    *reinterpret_cast<uint4*>(pm + q * LDB + k0) = make_uint4(pk(v[0], v[1]), pk(v[2], v[3]), pk(v[4], v[5]), pk(v[6], v[7]));
}
__device__ __forceinline__ void to_pm(const float* X, int R, int Kpad, __nv_bfloat16* pm) {
    const int q = threadIdx.x & 31;
    for (int b = threadIdx.x >> 5; b < Kpad / 8; b += NW) {
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = 8 * b + i < R ? X[(8 * b + i) * FG + q] : 0.0f;
        put_pm8(pm, q, 8 * b, v);
    }
}

// The weights of a layer: fragments, biases.
struct Layer {
    const uint4 *W1, *W2, *W3, *W1t, *W2t, *W3t;
    const float *b1, *b2, *b3;
};
__device__ __forceinline__ Layer layer_of(const DevFlow& f, int l) {
    const FlowFragOff fo = flow_frag_off(f.H, f.kp1, f.o4p);
    const FlowLayerOff o = flow_layer_off(f.H, f.Dh, f.Dh4, f.O4);
    const uint4* fr = f.frag + (int64_t)l * f.layer_frag;
    const float* w = f.work + (int64_t)l * f.layer_work;
    return {fr + fo.W1, fr + fo.W2, fr + fo.W3, fr + fo.W1t, fr + fo.W2t, fr + fo.W3t, w + o.b1, w + o.b2, w + o.b3};
}

// FP64 sums over a CTA's rows, per particle: a thread's part (lane = particle)
// into [8][32], added warp by warp by the particle's thread of warp 0
__device__ __forceinline__ double row_total(double* ldp, double v) {
    __syncthreads();
    ldp[threadIdx.x] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < FG)
        for (int w = 0; w < NW; ++w) s += ldp[w * FG + threadIdx.x];
    return s;
}

// Shared memory of the trajectories, in order (floats, FG per row): z, p, x (which
// also holds the cotangent), the changed half of every layer, the last
// layer's kept half, the conditioner's output; two BF16 operands; FP64 parts.
struct MoveSmem {
    float *z, *p, *x, *zb, *za, *o;
    __nv_bfloat16* pm[2];
    double* ldp;
    int scratch;                   // floats from o on that P may be staged in
};
__host__ __device__ inline size_t move_floats(int D, int L, int O4) { return (size_t)FG * (3 * D + (L + 1) * (D / 2) + O4); }
__host__ __device__ inline size_t move_bytes(int D, int L, int O4) {
    return 4 * move_floats(D, L, O4) + 2 * sizeof(uint16_t) * FG * LDB + 8 * FT;
}
__device__ __forceinline__ MoveSmem move_smem(unsigned char* base, int D, int L, int O4) {
    MoveSmem s;
    s.z = reinterpret_cast<float*>(base);
    s.p = s.z + D * FG;
    s.x = s.p + D * FG;
    s.zb = s.x + D * FG;
    s.za = s.zb + L * (D / 2) * FG;
    s.o = s.za + (D / 2) * FG;
    s.pm[0] = reinterpret_cast<__nv_bfloat16*>(s.o + O4 * FG);
    s.pm[1] = s.pm[0] + FG * LDB;
    s.ldp = reinterpret_cast<double*>(s.pm[1] + FG * LDB);
    s.scratch = O4 * FG + FG * LDB;            // o and both operands (2 x FG x LDB BF16)
    return s;
}

// Conditioner of a layer on the particle-major half in pm[0] (kp1 columns): o in
// FP32; with KEEP the hidden activations stay in h1, h2.  pm[1] and pm[0] are
// overwritten.  Begins and ends with every thread past a barrier.
__device__ __forceinline__ void conditioner(const DevFlow& f, const Layer& w, __nv_bfloat16* const (&pm)[2], float* o,
                                            float (&h1)[4][4], float (&h2)[4][4], Frag& fr, const Piece& ph,
                                            const Piece& po, int lane) {
    const uint32_t a0 = tc::smem_u32(pm[0]), a1 = tc::smem_u32(pm[1]);
    fr.load(w.W1, ph, 0, f.kp1 / 16, lane);
    product(fr, w.W1, ph, f.kp1 / 16, a0, h1, lane);
    fr.load(w.W2, ph, 0, f.H / 16, lane);
    bias_act<true>(h1, ph, w.b1, f.H, lane);
    store_pm(h1, ph, a1, lane);
    __syncthreads();
    product(fr, w.W2, ph, f.H / 16, a1, h2, lane);
    fr.load(w.W3, po, 0, f.H / 16, lane);
    bias_act<true>(h2, ph, w.b2, f.H, lane);
    store_pm(h2, ph, a0, lane);
    __syncthreads();
    float acc[4][4];
    product(fr, w.W3, po, f.H / 16, a0, acc, lane);
    bias_act<false>(acc, po, w.b3, f.O4, lane);
    store_f32<false>(acc, po, o, f.O4, lane);
    __syncthreads();
}

// x <- T(x) (INV: T^-1(x)), recording every layer's changed half as the
// forward layer finds it; returns this thread's part of log|det| (lane =
// particle).  x in place, all threads synchronised before and after.
template <bool INV>
__device__ __forceinline__ double flow_pass(const DevFlow& f, const MoveSmem& s, const Piece& ph, const Piece& po,
                                            int lane) {
    const int Dh = f.Dh, q = lane, wid = threadIdx.x >> 5;
    double part = 0.0;
    const int first = INV ? f.L - 1 : 0;
    to_pm(s.x + ((first & 1) ? Dh : 0) * FG, Dh, f.kp1, s.pm[0]);
    __syncthreads();
    for (int i = 0; i < f.L; ++i) {
        const int l = INV ? f.L - 1 - i : i;
        float h1[4][4], h2[4][4];
        Frag fr;
        conditioner(f, layer_of(f, l), s.pm, s.o, h1, h2, fr, ph, po, lane);
        const int boff = (l & 1) ? 0 : Dh, aoff = (l & 1) ? Dh : 0;
        float* xb = s.x + boff * FG;
        float* zb = s.zb + l * Dh * FG;
        if (l == f.L - 1)
            for (int k = wid; k < Dh; k += NW) s.za[k * FG + q] = s.x[(aoff + k) * FG + q];
        // the changed half, which is also the next layer's kept half
        for (int b = wid; b < f.kp1 / 8; b += NW) {
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int k = 8 * b + e;
                v[e] = 0.0f;
                if (k >= Dh) continue;
                const float sv = 2.0f * tanhf(s.o[k * FG + q]);
                const float tv = s.o[(f.Dh4 + k) * FG + q];
                const float x0 = xb[k * FG + q];
                if (INV) {
                    v[e] = (x0 - tv) * expf(-sv);
                    part -= (double)sv;
                    zb[k * FG + q] = v[e];
                } else {
                    v[e] = fmaf(x0, expf(sv), tv);
                    part += (double)sv;
                    zb[k * FG + q] = x0;
                }
                xb[k * FG + q] = v[e];
            }
            put_pm8(s.pm[0], q, 8 * b, v);
        }
        __syncthreads();
    }
    return part;
}

// c (in s.x) <- J_T(z)^T c + grad_z log|det dT/dz| with the recorded halves.
__device__ __forceinline__ void flow_back(const DevFlow& f, const MoveSmem& s, const Piece& ph, const Piece& po,
                                          int lane) {
    const int Dh = f.Dh, H = f.H, q = lane, wid = threadIdx.x >> 5;
    const Piece pa{f.kp1 / 16, wid};
    const uint32_t a0 = tc::smem_u32(s.pm[0]), a1 = tc::smem_u32(s.pm[1]);
    float* c = s.x;
    to_pm(s.za, Dh, f.kp1, s.pm[0]);
    __syncthreads();
    for (int l = f.L - 1; l >= 0; --l) {
        const Layer w = layer_of(f, l);
        float h1[4][4], h2[4][4], acc[4][4];
        Frag fr;
        conditioner(f, w, s.pm, s.o, h1, h2, fr, ph, po, lane);
        fr.load(w.W3t, ph, 0, f.o4p / 16, lane);
        const int boff = (l & 1) ? 0 : Dh, aoff = (l & 1) ? Dh : 0;
        const float* in = s.zb + l * Dh * FG;
        for (int b = wid; b < (f.Dh4 + 7) / 8; b += NW) {
            float vs[8], vt[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int k = 8 * b + e;
                vs[e] = vt[e] = 0.0f;
                if (k >= Dh) continue;
                const float th = tanhf(s.o[k * FG + q]);
                const float es = expf(2.0f * th);
                const float cbp = c[(boff + k) * FG + q];
                const float cs = fmaf(cbp * in[k * FG + q], es, 1.0f);   // + d logdet / ds
                vs[e] = cs * 2.0f * (1.0f - th * th);
                vt[e] = cbp;
                c[(boff + k) * FG + q] = cbp * es;
            }
            // rows [0, Dh4) and [Dh4, 2 Dh4); Dh4 is a multiple of four only
            __nv_bfloat16* r = s.pm[1] + q * LDB;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int k = 8 * b + 4 * u;
                if (k < f.Dh4) {
                    *reinterpret_cast<uint2*>(r + k) = make_uint2(pk(vs[4 * u], vs[4 * u + 1]), pk(vs[4 * u + 2], vs[4 * u + 3]));
                    *reinterpret_cast<uint2*>(r + f.Dh4 + k) = make_uint2(pk(vt[4 * u], vt[4 * u + 1]), pk(vt[4 * u + 2], vt[4 * u + 3]));
                }
            }
        }
        for (int k = f.O4 + 4 * wid; k < f.o4p; k += 4 * NW)
            *reinterpret_cast<uint2*>(s.pm[1] + q * LDB + k) = make_uint2(0u, 0u);
        __syncthreads();
        product(fr, w.W3t, ph, f.o4p / 16, a1, acc, lane);
        fr.load(w.W2t, ph, 0, H / 16, lane);
        times_dtanh(acc, h2);
        store_pm(acc, ph, a0, lane);
        __syncthreads();
        product(fr, w.W2t, ph, H / 16, a0, acc, lane);
        fr.load(w.W1t, pa, 0, H / 16, lane);
        times_dtanh(acc, h1);
        store_pm(acc, ph, a1, lane);
        __syncthreads();
        product(fr, w.W1t, pa, H / 16, a1, acc, lane);
        store_f32<true>(acc, pa, c + aoff * FG, Dh, lane);
        if (l > 0) to_pm(s.zb + l * Dh * FG, Dh, f.kp1, s.pm[0]);   // layer l - 1 keeps the half that layer l changes
        __syncthreads();
    }
}

// grad log pi at x, over x; with LAST, x and the gradient go out to theta_out,
// grad_out, and the return value is this thread's part (lane = particle) of
// the FP64 sum of log pi without its constant.
template <int TARGET>
__device__ __forceinline__ double target_grad(const DevModel& m, const MoveSmem& s, const TrajArgs& a,
                                              const int64_t* j_s, bool last) {
    const int t = threadIdx.x, D = m.D, lane = t & 31, wid = t >> 5;
    float* x = s.x;
    double part = 0.0;
    if (last)
        for (int e = t; e < D * FG; e += FT)
            if (j_s[e % FG] >= 0) a.theta_out[(int64_t)(e / FG) * a.ld + j_s[e % FG]] = x[e];
    if constexpr (TARGET == 0) {
        // -P (x - mu): 4 rows x 4 particles a thread, the columns of P staged in
        // chunks (transposed, rows padded to four) in the idle operand buffers
        const int D4 = (D + 3) & ~3, KC = min(D, s.scratch / D4);
        const int db = t >> 3, pb = t & 7;
        float acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[i][u] = 0.0f;
        for (int k0 = 0; k0 < D; k0 += KC) {
            const int kc = min(KC, D - k0);
            __syncthreads();
            for (int e = t; e < D4 * kc; e += FT) {
                const int d = e / kc, k = e - d * kc;
                s.o[k * D4 + d] = d < D ? __ldg(m.P + (int64_t)d * D + k0 + k) : 0.0f;
            }
            __syncthreads();
            if (4 * db < D)
                for (int k = 0; k < kc; ++k) {
                    const float mk = __ldg(m.mu + k0 + k);
                    const float4 x4 = *reinterpret_cast<const float4*>(x + (k0 + k) * FG + 4 * pb);
                    const float4 p4 = *reinterpret_cast<const float4*>(s.o + k * D4 + 4 * db);
                    const float b0 = x4.x - mk, b1 = x4.y - mk, b2 = x4.z - mk, b3 = x4.w - mk;
                    const float av[4] = {p4.x, p4.y, p4.z, p4.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        acc[i][0] = fmaf(av[i], b0, acc[i][0]);
                        acc[i][1] = fmaf(av[i], b1, acc[i][1]);
                        acc[i][2] = fmaf(av[i], b2, acc[i][2]);
                        acc[i][3] = fmaf(av[i], b3, acc[i][3]);
                    }
                }
        }
        __syncthreads();
        float* g = s.o;                      // the gradient, then over x
        if (last) {
            if (4 * db < D)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (4 * db + i < D)
                        *reinterpret_cast<float4*>(g + (4 * db + i) * FG + 4 * pb) =
                            make_float4(-acc[i][0], -acc[i][1], -acc[i][2], -acc[i][3]);
            __syncthreads();
            // log pi = c + 1/2 (x - mu)' g: FP64 sums of the FP32 gradient
            for (int d = wid; d < D; d += NW) {
                part += ((double)x[d * FG + lane] - (double)m.mu[d]) * (double)g[d * FG + lane];
                if (j_s[lane] >= 0) a.grad_out[(int64_t)d * a.ld + j_s[lane]] = g[d * FG + lane];
            }
            __syncthreads();
        }
        if (4 * db < D)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (4 * db + i < D)
                    *reinterpret_cast<float4*>(x + (4 * db + i) * FG + 4 * pb) =
                        make_float4(-acc[i][0], -acc[i][1], -acc[i][2], -acc[i][3]);
        __syncthreads();
        return 0.5 * part;
    } else {
        const float fa = (float)m.h0, fb = (float)m.h1, inva = (float)(1.0 / m.h0);
        __syncthreads();                     // theta_out has been read from x
        for (int i = wid; i < D / 2; i += NW) {
            const float xo = x[(2 * i) * FG + lane], xe = x[(2 * i + 1) * FG + lane];
            const float u = xe - fb * (xo * xo - fa);
            const float g0 = -xo * inva + 2.0f * fb * u * xo, g1 = -u;
            x[(2 * i) * FG + lane] = g0;
            x[(2 * i + 1) * FG + lane] = g1;
            if (last) {
                const double dxo = xo, dxe = xe;
                const double du = dxe - m.h1 * (dxo * dxo - m.h0);
                part += -0.5 * dxo * dxo / m.h0 - 0.5 * du * du;
                if (j_s[lane] >= 0) {
                    a.grad_out[(int64_t)(2 * i) * a.ld + j_s[lane]] = g0;
                    a.grad_out[(int64_t)(2 * i + 1) * a.ld + j_s[lane]] = g1;
                }
            }
        }
        __syncthreads();
        return part;
    }
}

template <int TARGET>
__global__ void __launch_bounds__(FT, 2) traj_flow_mma_kernel(DevModel m, DevFlow f, TrajArgs a, float* z0out,
                                                              float* z1out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const MoveSmem s = move_smem(smem_raw, f.D, f.L, f.O4);
    __shared__ int64_t j_s[FG], src_s[FG];
    __shared__ int S_s[FG];
    __shared__ float eps_s[FG];
    __shared__ uint64_t seed_s[FG];
    __shared__ uint32_t k_s[FG], jl_s[FG];
    const int t = threadIdx.x, D = f.D, lane = t & 31, wid = t >> 5;
    const Piece ph{f.H / 16, wid}, po{f.o4p / 16, wid};
    if (t < FG) {
        const int64_t sl = (int64_t)blockIdx.x * FG + t;
        int64_t j = -1, src = -1;
        int S = 0;
        float ef = 0.0f;
        if (sl < a.N) {
            j = a.perm ? a.perm[sl] : sl;
            src = a.src ? a.src[j] : j;
            S = a.steps[j];
            int r;
            double eps;
            uint64_t seed;
            uint32_t kk, jl;
            particle_run(a, j, r, eps, seed, kk, jl);
            ef = (float)eps;
            seed_s[t] = seed;
            k_s[t] = kk;
            jl_s[t] = jl;
        }
        j_s[t] = j;
        src_s[t] = src;
        S_s[t] = S;
        eps_s[t] = ef;
    }
    __syncthreads();
    int smax = 0;
    for (int q = 0; q < FG; ++q) smax = max(smax, S_s[q]);
    // lane = particle in every pass below that goes row by row
    const int64_t j = j_s[lane], src = src_s[lane];
    for (int d = wid; d < D; d += NW) s.x[d * FG + lane] = src >= 0 ? a.theta_in[(int64_t)d * a.ld + src] : 0.0f;
    __syncthreads();
    // latent start z0 = T^-1(theta), its log pi_z and gradient
    const double ld0 = flow_pass<true>(f, s, ph, po, lane);
    for (int d = wid; d < D; d += NW) {
        const int e = d * FG + lane;
        const float z = s.x[e];
        s.z[e] = z;
        if (z0out && j >= 0) z0out[(int64_t)d * a.ld + j] = z;
        s.x[e] = src >= 0 ? a.grad_in[(int64_t)d * a.ld + src] : 0.0f;
        if (a.p_in) s.p[e] = src >= 0 ? a.p_in[(int64_t)d * a.ld + j] : 0.0f;
    }
    if (!a.p_in)
        for (int i = wid; i < D / 2; i += NW) {
            double z0 = 0.0, z1 = 0.0;
            if (j >= 0) normal_pair(seed_s[lane], (uint32_t)i, jl_s[lane], k_s[lane], TAG_MOM, z0, z1);
            s.p[(2 * i) * FG + lane] = (float)z0;
            s.p[(2 * i + 1) * FG + lane] = (float)z1;
        }
    double H0 = row_total(s.ldp, ld0);              // of particle t, threads t < 32
    const double logpi0 = t < FG && src >= 0 ? a.logpi_in[src] : 0.0;
    H0 = -(logpi0 - H0);                            // - log pi_z(z0) = -(log pi - log|det dT^-1|)
    const double ldT0 = -(H0 + logpi0);             // log|det dT| at z0, for a CTA without steps
    double kin = 0.0;
    for (int d = wid; d < D; d += NW) kin += (double)s.p[d * FG + lane] * (double)s.p[d * FG + lane];
    H0 += 0.5 * row_total(s.ldp, kin);
    flow_back(f, s, ph, po, lane);                  // s.x = grad_z log pi_z(z0)
    for (int d = wid; d < D; d += NW) {
        const int e = d * FG + lane;
        float z = s.z[e];
        if (S_s[lane] >= 1) {
            const float he = 0.5f * eps_s[lane];
            const float pv = fmaf(he, s.x[e], s.p[e]);
            s.p[e] = pv;
            z = fmaf(eps_s[lane], pv, z);
            s.z[e] = z;
        }
        s.x[e] = z;
    }
    __syncthreads();
    double ldT = ldT0, lpx = 0.0;
    for (int st = 1; st <= smax; ++st) {
        const double ldp = flow_pass<false>(f, s, ph, po, lane);        // s.x = T(z)
        const double lp = target_grad<TARGET>(m, s, a, j_s, st == smax);   // s.x = grad_x log pi
        if (st == smax) {
            ldT = row_total(s.ldp, ldp);
            lpx = row_total(s.ldp, lp);
        }
        flow_back(f, s, ph, po, lane);              // s.x = grad_z log pi_z
        for (int d = wid; d < D; d += NW) {
            const int e = d * FG + lane;
            float z = s.z[e];
            if (st <= S_s[lane]) {
                const float he = 0.5f * eps_s[lane];
                const float g = s.x[e];
                float pv = fmaf(he, g, s.p[e]);
                if (st + 1 <= S_s[lane]) {
                    pv = fmaf(he, g, pv);
                    z = fmaf(eps_s[lane], pv, z);
                    s.z[e] = z;
                }
                s.p[e] = pv;
            }
            s.x[e] = z;
        }
        __syncthreads();
    }
    if (smax == 0) {   // nothing moved: theta and its gradient as they were
        double lp = 0.0;
        for (int d = wid; d < D; d += NW) {
            const int64_t o = (int64_t)d * a.ld;
            const float tv = src >= 0 ? a.theta_in[o + src] : 0.0f, gv = src >= 0 ? a.grad_in[o + src] : 0.0f;
            if (TARGET == 0) lp += 0.5 * (((double)tv - (double)m.mu[d]) * (double)gv);
            if (TARGET == 1) s.x[d * FG + lane] = tv;
            if (j >= 0) {
                a.theta_out[o + j] = tv;
                a.grad_out[o + j] = gv;
            }
        }
        __syncthreads();
        if (TARGET == 1)
            for (int i = wid; i < D / 2; i += NW) {
                const double xo = s.x[(2 * i) * FG + lane], xe = s.x[(2 * i + 1) * FG + lane];
                const double u = xe - m.h1 * (xo * xo - m.h0);
                lp += -0.5 * xo * xo / m.h0 - 0.5 * u * u;
            }
        lpx = row_total(s.ldp, lp);
    }
    // end point: theta' = T(z') went out with its gradient; exact energy in FP64
    kin = 0.0;
    for (int d = wid; d < D; d += NW) {
        const int e = d * FG + lane;
        kin += (double)s.p[e] * (double)s.p[e];
        if (j >= 0) {
            if (a.p_out) a.p_out[(int64_t)d * a.ld + j] = s.p[e];
            if (z1out) z1out[(int64_t)d * a.ld + j] = s.z[e];
        }
    }
    kin = row_total(s.ldp, kin);
    if (t < FG && j >= 0) {
        lpx += m.lconst;
        double dH = (0.5 * kin - (lpx + ldT)) - H0;
        if (!isfinite(dH)) dH = CUDART_INF;
        a.logpi_out[j] = lpx;
        if (a.dH) a.dH[j] = dH;
        if (a.alpha) a.alpha[j] = dH <= 0.0 ? 1.0 : exp(-dH);
    }
}

// ============================================================ training
// out[row(m) * ldo + n] = sum over the CTA's 32 particles p of A[m][p] B[n][p]
// for m < 16 MT, n < min(16 NP, Nvalid); A, B BF16 rows [.][WLD] in shared
// memory (K = the particles: two k-steps of m16n8k16).  A warp takes one
// m-tile and four n-tiles.  CMAP: A's rows are the conditioner's padded
// output rows (s rows from 0, t rows from Dh4), stored at the canonical rows
// of W3 (s then t, Dh each); otherwise rows m < Mvalid are stored as they are.
template <bool CMAP>
__device__ __forceinline__ void cta_wgrad(const __nv_bfloat16* A, int MT, const __nv_bfloat16* B, int NP, float* out,
                                          int ldo, int Mvalid, int Nvalid, int Dh, int Dh4) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int mi = lane >> 3, mr = lane & 7;
    const int NQ = (NP + 1) >> 1;
    const uint32_t abase = tc::smem_u32(A), bbase = tc::smem_u32(B);
    auto row_of = [&](int m) -> int {
        if (!CMAP) return m < Mvalid ? m : -1;
        return m < Dh ? m : (m >= Dh4 && m < Dh4 + Dh ? Dh + (m - Dh4) : -1);
    };
    for (int it = wid; it < MT * NQ; it += NW) {
        const int mt = it / NQ, q = it % NQ;
        float acc[4][4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[u][v] = 0.0f;
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
            uint32_t a[4];
            tc::ldsm4(a, abase + (uint32_t)(((16 * mt + (lane & 15)) * WLD + 16 * ks + 8 * (lane >> 4)) * 2));
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int np = 2 * q + h;     // n-tiles 2 np and 2 np + 1
                if (np < NP) {
                    uint32_t b[4];
                    tc::ldsm4(b, bbase + (uint32_t)(((16 * np + 8 * (mi >> 1) + mr) * WLD + 16 * ks + 8 * (mi & 1)) * 2));
                    tc::mma_bf16_16816(acc[2 * h], a, b[0], b[1]);
                    tc::mma_bf16_16816(acc[2 * h + 1], a, b[2], b[3]);
                }
            }
        }
        const int r0 = row_of(16 * mt + g), r1 = row_of(16 * mt + g + 8);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (2 * q + (u >> 1) < NP) {
                const int c0 = 8 * (4 * q + u) + 2 * t;
                if (r0 >= 0) {
                    if (c0 < Nvalid) out[(int64_t)r0 * ldo + c0] = acc[u][0];
                    if (c0 + 1 < Nvalid) out[(int64_t)r0 * ldo + c0 + 1] = acc[u][1];
                }
                if (r1 >= 0) {
                    if (c0 < Nvalid) out[(int64_t)r1 * ldo + c0] = acc[u][2];
                    if (c0 + 1 < Nvalid) out[(int64_t)r1 * ldo + c0 + 1] = acc[u][3];
                }
            }
        }
    }
}

// FP32 sums over the 32 particles of the accumulators' rows (the bias
// gradients): a row's columns over its quad of lanes, then, where two warps
// share a row tile, the two halves at rs[half][row] are added by the reader.
__device__ __forceinline__ void row_sums(const float (&acc)[4][4], const Piece& pc, float* rs, int lane) {
    const int g = lane >> 2, t = lane & 3;
    auto quad = [](float v) {
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        return v + __shfl_xor_sync(0xffffffffu, v, 2);
    };
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        float v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h)
            v[h] = quad((acc[2 * h][2 * e] + acc[2 * h][2 * e + 1]) + (acc[2 * h + 1][2 * e] + acc[2 * h + 1][2 * e + 1]));
        if (t != 0) continue;
        if (pc.both()) {
            rs[16 * pc.mt(0) + g + 8 * e] = v[0];
            rs[128 + 16 * pc.mt(0) + g + 8 * e] = v[1];
        } else {
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (pc.on(h)) rs[64 * pc.nt(h) + 16 * pc.mt(h) + g + 8 * e] = v[h];
        }
    }
}

// Shared memory of the training gradient: x, which becomes the cotangent c, the
// first layer's kept half, every layer's changed half, the conditioner's
// output (later the BF16 rows of c_h2); the two particle-major operands; BF16
// rows of c_o / c_h1, h1, h2 and the kept half; the bias sums.
struct TrainSmem {
    float *x, *za, *zb, *o;
    __nv_bfloat16 *pm[2], *A, *A2, *h1, *h2, *ar;
    float* rs;
};
__host__ __device__ inline size_t train_bytes(int D, int H, int L, int O4, int kp1, int o4p) {
    const size_t o = 4 * FG * (size_t)O4 > 2 * WLD * (size_t)H ? 4 * FG * (size_t)O4 : 2 * WLD * (size_t)H;
    return 4 * (size_t)FG * (D + (L + 1) * (D / 2)) + o + 2 * 2 * (size_t)FG * LDB +
           2 * (size_t)WLD * ((o4p > H ? o4p : H) + 2 * H + kp1) + 4 * 256;
}
__device__ __forceinline__ TrainSmem train_smem(unsigned char* base, int D, int H, int L, int O4, int kp1, int o4p) {
    TrainSmem s;
    s.x = reinterpret_cast<float*>(base);
    s.za = s.x + D * FG;
    s.zb = s.za + (D / 2) * FG;
    s.o = s.zb + L * (D / 2) * FG;
    s.A2 = reinterpret_cast<__nv_bfloat16*>(s.o);
    const int ob = 4 * FG * O4 > 2 * WLD * H ? 4 * FG * O4 : 2 * WLD * H;
    s.pm[0] = reinterpret_cast<__nv_bfloat16*>(reinterpret_cast<unsigned char*>(s.o) + ob);
    s.pm[1] = s.pm[0] + FG * LDB;
    s.A = s.pm[1] + FG * LDB;
    s.h1 = s.A + (o4p > H ? o4p : H) * WLD;
    s.h2 = s.h1 + H * WLD;
    s.ar = s.h2 + H * WLD;
    s.rs = reinterpret_cast<float*>(s.ar + kp1 * WLD);
    return s;
}

// FP32 rows X [R x 32] -> BF16 rows [Rpad][WLD], zero for R <= r < Rpad
__device__ __forceinline__ void to_rows(const float* X, int R, int Rpad, __nv_bfloat16* Y) {
    for (int e = threadIdx.x; e < Rpad * 4; e += FT) {
        const int r = e >> 2, p0 = 8 * (e & 3);
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (r < R) {
            const float4 a = *reinterpret_cast<const float4*>(X + r * FG + p0);
            const float4 b = *reinterpret_cast<const float4*>(X + r * FG + p0 + 4);
            w = make_uint4(pk(a.x, a.y), pk(a.z, a.w), pk(b.x, b.y), pk(b.z, b.w));
        }
        *reinterpret_cast<uint4*>(Y + r * WLD + p0) = w;
    }
}

// The weighted-NLL gradient of k_flow_train (flow.cu) with BF16 products; the
// same partials layout (canonical parameter order, one row per CTA).
__global__ void __launch_bounds__(FT, 2) k_flow_train_mma(DevFlow f, const float* theta, int64_t ld, const int32_t* src,
                                                          const double* W, FlowGate gate, int64_t N, float* partials) {
    if (!gate.open()) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int D = f.D, H = f.H, Dh = f.Dh, Dh4 = f.Dh4;
    const TrainSmem s = train_smem(smem_raw, D, H, f.L, f.O4, f.kp1, f.o4p);
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5, q = lane;
    const Piece ph{H / 16, wid}, po{f.o4p / 16, wid}, pa{f.kp1 / 16, wid};
    const uint32_t a0 = tc::smem_u32(s.pm[0]), a1 = tc::smem_u32(s.pm[1]);
    const int64_t j = (int64_t)blockIdx.x * FG + q;
    float wq = 0.0f;                         // the lane's particle's weight
    if (j < N) wq = (gate.rs && gate.rs->resample) ? (float)(1.0 / (double)gate.rp->n) : (float)W[j];
    // a particle of zero weight adds nothing; its position may be non-finite
    // (the end of a divergent trajectory), so it enters as zeros
    const int64_t sj = (j < N && wq != 0.0f) ? (src ? (int64_t)src[j] : j) : -1;
    for (int d = wid; d < D; d += NW) s.x[d * FG + q] = sj >= 0 ? theta[(int64_t)d * ld + sj] : 0.0f;
    __syncthreads();
    to_pm(s.x + (((f.L - 1) & 1) ? Dh : 0) * FG, Dh, f.kp1, s.pm[0]);
    __syncthreads();
    // inverse pass, recording every layer's changed half before it changes
    for (int l = f.L - 1; l >= 0; --l) {
        float h1[4][4], h2[4][4];
        Frag fr;
        conditioner(f, layer_of(f, l), s.pm, s.o, h1, h2, fr, ph, po, lane);
        float* xb = s.x + ((l & 1) ? 0 : Dh) * FG;
        float* zb = s.zb + l * Dh * FG;
        for (int b = wid; b < f.kp1 / 8; b += NW) {
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int k = 8 * b + e;
                v[e] = 0.0f;
                if (k >= Dh) continue;
                const float sv = 2.0f * tanhf(s.o[k * FG + q]);
                const float tv = s.o[(Dh4 + k) * FG + q];
                const float x0 = xb[k * FG + q];
                zb[k * FG + q] = x0;
                v[e] = (x0 - tv) * expf(-sv);
                xb[k * FG + q] = v[e];
            }
            put_pm8(s.pm[0], q, 8 * b, v);
        }
        __syncthreads();
    }
    // layer 0 keeps dimensions 0 .. Dh - 1 of z; c = d(1/2 |z|^2) weighted
    for (int d = wid; d < D; d += NW) {
        const float z = s.x[d * FG + q];
        if (d < Dh) s.za[d * FG + q] = z;
        s.x[d * FG + q] = wq * z;
    }
    __syncthreads();
    to_pm(s.za, Dh, f.kp1, s.pm[0]);
    __syncthreads();
    float* c = s.x;
    const int64_t lsz = (int64_t)H * Dh + H + (int64_t)H * H + H + (int64_t)D * H + D;
    float* part = partials + (int64_t)blockIdx.x * f.n_params;
    for (int l = 0; l < f.L; ++l) {
        const Layer w = layer_of(f, l);
        float* gl = part + l * lsz;
        float *gW1 = gl, *gb1 = gW1 + (int64_t)H * Dh, *gW2 = gb1 + H, *gb2 = gW2 + (int64_t)H * H, *gW3 = gb2 + H,
              *gb3 = gW3 + (int64_t)D * H;
        const int boff = (l & 1) ? 0 : Dh, aoff = (l & 1) ? Dh : 0;
        const float* kept = l == 0 ? s.za : s.zb + (l - 1) * Dh * FG;
        const float* in = s.zb + l * Dh * FG;
        float h1[4][4], h2[4][4], acc[4][4];
        Frag fr;
        to_rows(kept, Dh, f.kp1, s.ar);
        conditioner(f, w, s.pm, s.o, h1, h2, fr, ph, po, lane);
        fr.load(w.W3t, ph, 0, f.o4p / 16, lane);
        store_rows(h1, ph, tc::smem_u32(s.h1), lane);
        store_rows(h2, ph, tc::smem_u32(s.h2), lane);
        // c_o, as both operands, and its row sums db3 (s rows, then t rows)
        for (int b = wid; b < (Dh4 + 7) / 8; b += NW) {
            float vs[8], vt[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int k = 8 * b + e;
                vs[e] = vt[e] = 0.0f;
                if (k < Dh) {
                    const float th = tanhf(s.o[k * FG + q]);
                    const float ems = expf(-2.0f * th);
                    const float bb = (in[k * FG + q] - s.o[(Dh4 + k) * FG + q]) * ems;
                    const float cb = c[(boff + k) * FG + q];
                    const float cs = fmaf(-cb, bb, wq);            // + W_j from sum s
                    vs[e] = cs * 2.0f * (1.0f - th * th);
                    vt[e] = -cb * ems;
                    c[(boff + k) * FG + q] = cb * ems;
                }
                if (k < Dh4) {
                    s.A[k * WLD + q] = __float2bfloat16_rn(vs[e]);
                    s.A[(Dh4 + k) * WLD + q] = __float2bfloat16_rn(vt[e]);
                }
                const float ss = warp_sum(vs[e]), ts = warp_sum(vt[e]);
                if (lane == 0 && k < Dh) {
                    gb3[k] = ss;
                    gb3[Dh + k] = ts;
                }
            }
            __nv_bfloat16* r = s.pm[1] + q * LDB;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int k = 8 * b + 4 * u;
                if (k < Dh4) {
                    *reinterpret_cast<uint2*>(r + k) = make_uint2(pk(vs[4 * u], vs[4 * u + 1]), pk(vs[4 * u + 2], vs[4 * u + 3]));
                    *reinterpret_cast<uint2*>(r + Dh4 + k) = make_uint2(pk(vt[4 * u], vt[4 * u + 1]), pk(vt[4 * u + 2], vt[4 * u + 3]));
                }
            }
        }
        for (int k = f.O4 + 4 * wid; k < f.o4p; k += 4 * NW) {
            *reinterpret_cast<uint2*>(s.pm[1] + q * LDB + k) = make_uint2(0u, 0u);
#pragma unroll
            for (int u = 0; u < 4; ++u) s.A[(k + u) * WLD + q] = __float2bfloat16_rn(0.0f);
        }
        __syncthreads();
        // dW3 = c_o h2^T; c_h2 = (W3^T c_o) (1 - h2^2)
        product(fr, w.W3t, ph, f.o4p / 16, a1, acc, lane);
        fr.load(w.W2t, ph, 0, H / 16, lane);
        times_dtanh(acc, h2);
        store_pm(acc, ph, a0, lane);
        store_rows(acc, ph, tc::smem_u32(s.A2), lane);
        row_sums(acc, ph, s.rs, lane);
        cta_wgrad<true>(s.A, f.o4p / 16, s.h2, H / 16, gW3, H, 0, H, Dh, Dh4);
        __syncthreads();
        // dW2 = c_h2 h1^T; c_h1 = (W2^T c_h2) (1 - h1^2)
        if (t < H) gb2[t] = s.rs[t] + s.rs[128 + t];
        product(fr, w.W2t, ph, H / 16, a0, acc, lane);
        fr.load(w.W1t, pa, 0, H / 16, lane);
        times_dtanh(acc, h1);
        store_pm(acc, ph, a1, lane);
        store_rows(acc, ph, tc::smem_u32(s.A), lane);
        cta_wgrad<false>(s.A2, H / 16, s.h1, H / 16, gW2, H, H, H, Dh, Dh4);
        __syncthreads();
        // dW1 = c_h1 a^T; c_a += W1^T c_h1
        row_sums(acc, ph, s.rs, lane);
        cta_wgrad<false>(s.A, H / 16, s.ar, f.kp1 / 16, gW1, Dh, H, Dh, Dh, Dh4);
        product(fr, w.W1t, pa, H / 16, a1, acc, lane);
        store_f32<true>(acc, pa, c + aoff * FG, Dh, lane);
        if (l + 1 < f.L) to_pm(in, Dh, f.kp1, s.pm[0]);   // layer l + 1 keeps the half that layer l changes
        __syncthreads();
        if (t < H) gb1[t] = s.rs[t] + s.rs[128 + t];
    }
}

}  // namespace

cudaError_t launch_traj_flow_mma(const DevModel& m, const DevFlow& f, const TrajArgs& a, float* z0, float* z1,
                                 cudaStream_t s) {
    const int64_t grid = (a.N + FG - 1) / FG;
    const size_t sm = move_bytes(f.D, f.L, f.O4);
    auto kern = m.kind == GAUSS_DENSE ? traj_flow_mma_kernel<0> : traj_flow_mma_kernel<1>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)grid, FT, sm, s>>>(m, f, a, z0, z1);
    return cudaGetLastError();
}

cudaError_t launch_flow_train_mma(const DevFlow& f, const float* theta, int64_t ld, const int32_t* src, const double* W,
                                  FlowGate gate, int64_t N, float* partials, cudaStream_t s) {
    const int64_t grid = (N + FG - 1) / FG;
    const size_t sm = train_bytes(f.D, f.H, f.L, f.O4, f.kp1, f.o4p);
    cudaError_t e = cudaFuncSetAttribute(k_flow_train_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k_flow_train_mma<<<(unsigned)grid, FT, sm, s>>>(f, theta, ld, src, W, gate, N, partials);
    return cudaGetLastError();
}

}  // namespace smc
