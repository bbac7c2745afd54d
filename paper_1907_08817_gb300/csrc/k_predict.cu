// k_predict.cu -- the translate, map and rounding steps of Fig. "Algorithm NN-sort":
// w <- translate(A), w_pos <- w.map(f), pos <- round(w_pos * m), for every key, in binary32.
//
// One pass over the keys, the position written as a global position gs = gs_base + pos. A block
// takes a contiguous range of tiles, so it looks its first array up once and stages a model's
// parameters only when the range enters another array.
//   k_predict1 -- one hidden layer: eight keys per thread as four pairs of packed binary32 lanes.
//   k_predict2 -- two hidden layers: the second layer as a register-tiled block product.
// Every output is the fixed sequence of IEEE operations of mlp_fwd_f32, whatever the kernel.
#include "common.cuh"
#include "internal.h"

namespace nns {
static inline cudaError_t nns_launched(cudaError_t e, int k = 1) {
    if (e == cudaSuccess) note_launch(k);
    return e;
}
}  // namespace nns

namespace nns {

__device__ __forceinline__ int seg_of_tile(const Seg *segs, int nseg, uint32_t tile) {
    int lo = 0, hi = nseg - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (segs[mid].tbase <= tile) lo = mid; else hi = mid - 1;
    }
    return lo;
}

namespace {
// what a key's outputs need of its array (copied to registers: the outputs' stores could alias the
// table in memory)
struct Out {
    uint64_t n, ebase, L;
    uint32_t gs_base;
    float nm_hi, nm_lo;
    const int32_t *payload;
    __device__ __forceinline__ explicit Out(const Seg &s)
        : n(s.n), ebase(s.ebase), L(s.L), gs_base((uint32_t)s.gs_base), nm_hi(s.nm_hi), nm_lo(s.nm_lo),
          payload(s.payload) {}
};

// a worker's contiguous share of the work units
__device__ __forceinline__ void work_range(uint32_t total, uint32_t worker, uint32_t workers, uint32_t &t0,
                                           uint32_t &t1) {
    const uint32_t per = (total + workers - 1) / workers;
    t0 = min(total, worker * per);
    t1 = min(total, t0 + per);
}

// one key's outputs
template <typename W>
__device__ __forceinline__ void put(const PredictArgs &a, const Out &o, uint64_t i, W w, uint32_t slot, float y) {
    const uint64_t e = o.ebase + i;
    if (a.gs) a.gs[e] = o.gs_base + slot;
    if (a.key_copy) reinterpret_cast<W *>(a.key_copy)[e] = w;
    if (a.pay_copy && o.payload) a.pay_copy[e] = (uint32_t)o.payload[i];
    if (a.row_init) a.row_init[e] = (uint32_t)i;
    if (a.slots_out) a.slots_out[e] = slot;
    if (a.y_out) a.y_out[e] = y;
}

// `count` keys of injected positions instead of a model's
template <typename W>
__device__ __forceinline__ void put_injected(const PredictArgs &a, const Seg &sg, uint64_t start, int count,
                                             int threads, uint32_t &err) {
    const Out o(sg);
    const W *keys = reinterpret_cast<const W *>(sg.keys);
    const uint32_t *slots = sg.slots;
    for (int k = threadIdx.x; k < count; k += threads) {
        const uint64_t i = start + k;
        if (i >= o.n) break;
        const W w = keys[i];
        if (key_is_nan(word64(w), a.dtype)) err |= ERR_NAN;
        uint32_t slot = slots[i];
        if ((uint64_t)slot >= o.L) { err |= ERR_SLOT; slot = 0; }
        put<W>(a, o, i, w, slot, 0.0f);
    }
}
}  // namespace

// One hidden layer. Bound by the FMA and ALU pipes (two packed FMAs and two maxima per unit and key
// pair); a unit's parameters are staged as lane pairs, so one 128-bit and one 64-bit shared-memory
// read serve the eight keys of a thread. Four blocks of 256 threads per SM (64 registers). 26.2M
// binary32 keys of 1-32-1: 0.157 ms (0.385 ms with one key at a time and 64-bit conversions); 147M
// keys in 1,024 arrays of 1-16-1 with their key copies: 0.63 ms (1.86 ms).
template <int H, typename W>
__global__ void __launch_bounds__(PRED_THREADS, 4) k_predict1(PredictArgs a) {
    __shared__ ulonglong2 wb[H];           // (W1, W1), (b1, b1)
    __shared__ unsigned long long w3[H];   // (W3, W3)
    __shared__ float sb3;
    const int tid = threadIdx.x;
    uint32_t t0, t1, err = 0;
    work_range(a.total_tiles, blockIdx.x, gridDim.x, t0, t1);
    int si = t0 < t1 ? seg_of_tile(a.segs, a.nseg, t0) : 0, loaded = -1;
    for (uint32_t tile = t0; tile < t1; ++tile) {
        while (si + 1 < a.nseg && a.segs[si + 1].tbase <= tile) ++si;
        const Seg &sg = a.segs[si];
        const uint64_t start = (uint64_t)(tile - sg.tbase) * PRED_TILE;
        if (sg.slots) {
            put_injected<W>(a, sg, start, PRED_TILE, PRED_THREADS, err);
            continue;
        }
        if (si != loaded) {
            __syncthreads();
            for (int j = tid; j < H; j += PRED_THREADS) {
                const float *P = sg.params;
                wb[j] = make_ulonglong2(pk2(P[j], P[j]), pk2(P[H + j], P[H + j]));
                w3[j] = pk2(P[2 * H + j], P[2 * H + j]);
            }
            if (tid == 0) sb3 = sg.params[3 * H];
            loaded = si;
            __syncthreads();
        }
        const Norm nm = sg.norm;
        const Out o(sg);
        const uint64_t n = o.n;
        const W *keys = reinterpret_cast<const W *>(sg.keys);
        W w[PRED_ITEMS];
#pragma unroll
        for (int k = 0; k < PRED_ITEMS; ++k) {
            const uint64_t i = start + (uint64_t)k * PRED_THREADS + tid;
            w[k] = i < n ? keys[i] : (W)0;
        }
        constexpr int NP = PRED_ITEMS / 2;
        unsigned long long x[NP], y[NP];
        const float b3 = sb3;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            x[p] = pk2(translate_key<W>(w[2 * p], nm), translate_key<W>(w[2 * p + 1], nm));
            y[p] = pk2(b3, b3);
        }
#pragma unroll 4
        for (int j = 0; j < H; ++j) {
            const ulonglong2 c = wb[j];
            const unsigned long long c3 = w3[j];
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                float h0, h1;
                upk2(fma2_rn(c.x, x[p], c.y), h0, h1);
                y[p] = fma2_rn(c3, pk2(relu_f(h0), relu_f(h1)), y[p]);
            }
        }
#pragma unroll
        for (int k = 0; k < PRED_ITEMS; ++k) {
            const uint64_t i = start + (uint64_t)k * PRED_THREADS + tid;
            if (i >= n) break;
            float y0, y1;
            upk2(y[k / 2], y0, y1);
            const float yk = (k & 1) ? y1 : y0;
            if (key_is_nan(word64(w[k]), a.dtype)) err |= ERR_NAN;
            put<W>(a, o, i, w[k], slot_of(yk, o.nm_hi, o.nm_lo, o.L), yk);
        }
    }
    if (err) atomicOr(a.err, err);
}

// Two hidden layers of padded width H. A block of 128 threads stages the first layer's activations of
// M keys transposed in shared memory; each thread then accumulates an 8-key by 8-unit tile of
// z = b2 + H1 W2^T over the units j in order (64 FMAs, as 32 packed ones over key pairs, per four
// 128-bit shared-memory reads), writes relu(z) back transposed, and each key's owner sums the output
// layer in unit order. M = 8,192 / H keys keep the buffer at 34 KB for every width.
// Thread (tm, tn) holds units tn + NT i and keys 4 tm + {0..3}, M / 2 + 4 tm + {0..3}; the row stride
// M + 32 / NT spreads a quarter warp's 16-byte stores over all banks.
// A thread that kept one key's activations in registers read 16 bytes of weights per four FMAs and was
// bound by those reads: 16.8M keys of 1-64-64-1 took 4.39 ms, 2.68 ms now (53 TFLOP/s; the FMA pipe
// is busy 77% of the time). 256-thread blocks of the same tile measured 2.79 ms, scalar FMAs the
// same, and 16 x 8 tiles (12 warps per SM) 3.56 ms.
constexpr int F2_THREADS = 128;
template <int H> struct Fwd2 {
    static constexpr int NT = H / 8;                    // threads along the units
    static constexpr int M = 8 * F2_THREADS / NT;       // keys per step
    static constexpr int S = M + 32 / NT;               // row stride (floats)
    static constexpr int KPT = M / F2_THREADS;          // keys a thread owns in the first and last layer
    static constexpr int OFF_W2 = H * S;                // W2 transposed, units permuted to the threads' order
    static constexpr int OFF_B2 = OFF_W2 + H * H;       // b2 in the same order
    static constexpr int OFF_P = OFF_B2 + H;            // W1 | b1 | W3 | b3
    static constexpr int FLOATS = OFF_P + 3 * H + 4;
    static constexpr uint32_t STEPS = PRED_TILE / M;    // work units per tile
    static_assert(M <= PRED_TILE && PRED_TILE % M == 0, "whole steps per tile");
};

template <int H, typename W>
__global__ void __launch_bounds__(F2_THREADS, 4) k_predict2(PredictArgs a) {
    using F = Fwd2<H>;
    constexpr int NT = F::NT, M = F::M, S = F::S;
    extern __shared__ __align__(16) float sm[];
    float *buf = sm, *w2 = sm + F::OFF_W2, *b2 = sm + F::OFF_B2, *par = sm + F::OFF_P;
    const int tid = threadIdx.x, tn = tid % NT, tm = tid / NT;
    uint32_t t0, t1, err = 0;
    work_range(a.total_tiles * F::STEPS, blockIdx.x, gridDim.x, t0, t1);
    int si = t0 < t1 ? seg_of_tile(a.segs, a.nseg, t0 / F::STEPS) : 0, loaded = -1;
    for (uint32_t step = t0; step < t1; ++step) {
        while (si + 1 < a.nseg && a.segs[si + 1].tbase <= step / F::STEPS) ++si;
        const Seg &sg = a.segs[si];
        const uint64_t start = (uint64_t)(step - sg.tbase * F::STEPS) * M;
        if (start >= sg.n) continue;  // uniform over the block
        if (sg.slots) {
            put_injected<W>(a, sg, start, M, F2_THREADS, err);
            continue;
        }
        if (si != loaded) {
            __syncthreads();
            const float *P = sg.params;  // W1 b1 W2 b2 W3 b3
            // unit k = tn + NT (4 q + r) at column q (H / 2) + 4 tn + r
            for (int e = tid; e < H * H; e += F2_THREADS) {
                const int k = e / H, j = e % H, i = k / NT;
                w2[j * H + (i / 4) * (H / 2) + 4 * (k % NT) + i % 4] = P[2 * H + e];
            }
            for (int k = tid; k < H; k += F2_THREADS) {
                const int i = k / NT;
                b2[(i / 4) * (H / 2) + 4 * (k % NT) + i % 4] = P[2 * H + H * H + k];
                par[k] = P[k];
                par[H + k] = P[H + k];
                par[2 * H + k] = P[3 * H + H * H + k];
            }
            if (tid == 0) par[3 * H] = P[4 * H + H * H];
            loaded = si;
            __syncthreads();
        }
        const Norm nm = sg.norm;
        const Out o(sg);
        const uint64_t n = o.n;
        const W *keys = reinterpret_cast<const W *>(sg.keys);
#pragma unroll 4
        for (int q = 0; q < F::KPT; ++q) {
            const uint64_t i = start + (uint64_t)q * F2_THREADS + tid;
            const W w = i < n ? keys[i] : (W)0;
            if (key_is_nan(word64(w), a.dtype)) err |= ERR_NAN;
            const float x = translate_key<W>(w, nm);
            float *col = buf + q * F2_THREADS + tid;
#pragma unroll
            for (int j = 0; j < H; j += 4) {
                const float4 c = *reinterpret_cast<const float4 *>(par + j);
                const float4 d = *reinterpret_cast<const float4 *>(par + H + j);
                col[(j + 0) * S] = relu_f(__fmaf_rn(c.x, x, d.x));
                col[(j + 1) * S] = relu_f(__fmaf_rn(c.y, x, d.y));
                col[(j + 2) * S] = relu_f(__fmaf_rn(c.z, x, d.z));
                col[(j + 3) * S] = relu_f(__fmaf_rn(c.w, x, d.w));
            }
        }
        __syncthreads();
        unsigned long long z[8][4];  // [unit][key pair]
        {
            const float4 u = *reinterpret_cast<const float4 *>(b2 + 4 * tn);
            const float4 v = *reinterpret_cast<const float4 *>(b2 + H / 2 + 4 * tn);
            const float bb[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c) z[i][c] = pk2(bb[i], bb[i]);
        }
        const float *hp = buf + 4 * tm, *wp = w2 + 4 * tn;
#pragma unroll 4
        for (int j = 0; j < H; ++j) {
            const ulonglong2 h0 = *reinterpret_cast<const ulonglong2 *>(hp + j * S);
            const ulonglong2 h1 = *reinterpret_cast<const ulonglong2 *>(hp + j * S + M / 2);
            const float4 u = *reinterpret_cast<const float4 *>(wp + j * H);
            const float4 v = *reinterpret_cast<const float4 *>(wp + j * H + H / 2);
            const unsigned long long hh[4] = {h0.x, h0.y, h1.x, h1.y};
            const float ww[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const unsigned long long w2v = pk2(ww[i], ww[i]);
#pragma unroll
                for (int c = 0; c < 4; ++c) z[i][c] = fma2_rn(w2v, hh[c], z[i][c]);
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float *row = buf + (tn + NT * i) * S + 4 * tm;
            float r[8];
#pragma unroll
            for (int c = 0; c < 4; ++c) upk2(z[i][c], r[2 * c], r[2 * c + 1]);
            *reinterpret_cast<float4 *>(row) = make_float4(relu_f(r[0]), relu_f(r[1]), relu_f(r[2]), relu_f(r[3]));
            *reinterpret_cast<float4 *>(row + M / 2) =
                make_float4(relu_f(r[4]), relu_f(r[5]), relu_f(r[6]), relu_f(r[7]));
        }
        __syncthreads();
#pragma unroll 4
        for (int q = 0; q < F::KPT; ++q) {
            const uint64_t i = start + (uint64_t)q * F2_THREADS + tid;
            if (i >= n) break;
            const float *col = buf + q * F2_THREADS + tid;
            float y = par[3 * H];
#pragma unroll 16
            for (int k = 0; k < H; ++k) y = __fmaf_rn(par[2 * H + k], col[k * S], y);
            put<W>(a, o, i, a.key_copy ? keys[i] : (W)0, slot_of(y, o.nm_hi, o.nm_lo, o.L), y);
        }
        __syncthreads();
    }
    if (err) atomicOr(a.err, err);
}

// blocks for `units` work units: enough to fill the GPU, and no more than `most` units in a block. A
// block that took its full share of a long run (units / resident blocks) would leave its SM's later
// blocks behind, since the schedulers favour the older warps: the SM then ends with few warps.
static int work_blocks(uint64_t units, uint64_t resident, uint64_t most) {
    return (int)std::max<uint64_t>(std::min(units, resident), (units + most - 1) / most);
}

template <int H>
static cudaError_t go1(const PredictArgs &p, int sms, cudaStream_t s) {
    const int grid = work_blocks(p.total_tiles, (uint64_t)sms * 4, 8);
    if (grid == 0) return cudaSuccess;
    if (p.key_bytes == 4)
        k_predict1<H, uint32_t><<<grid, PRED_THREADS, 0, s>>>(p);
    else
        k_predict1<H, uint64_t><<<grid, PRED_THREADS, 0, s>>>(p);
    return nns_launched(cudaGetLastError());
}

template <int H>
static cudaError_t go2(const PredictArgs &p, int sms, cudaStream_t s) {
    const size_t smem = sizeof(float) * Fwd2<H>::FLOATS;
    const int grid = work_blocks((uint64_t)p.total_tiles * Fwd2<H>::STEPS, (uint64_t)sms * 4, 16);
    if (grid == 0) return cudaSuccess;
    auto kfn = p.key_bytes == 4 ? k_predict2<H, uint32_t> : k_predict2<H, uint64_t>;
    cudaError_t e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kfn<<<grid, F2_THREADS, smem, s>>>(p);
    return nns_launched(cudaGetLastError());
}

cudaError_t launch_predict_bf16(const PadArch &a, const PredictArgs &p, bool split, int sms, cudaStream_t s);

cudaError_t launch_predict(const PadArch &a, int precision, const PredictArgs &p, int sms,
                           cudaStream_t s) {
    if (precision == NNSORT_PREC_PWL) return launch_predict_pwl(p, sms, s);
    if ((precision == NNSORT_PREC_BF16 || precision == NNSORT_PREC_BF16X2) && a.layers == 2)
        return launch_predict_bf16(a, p, precision == NNSORT_PREC_BF16X2, sms, s);
    if (a.layers == 1) {
        switch (a.h1) {
        case 8: return go1<8>(p, sms, s);
        case 16: return go1<16>(p, sms, s);
        case 32: return go1<32>(p, sms, s);
        case 64: return go1<64>(p, sms, s);
        }
    } else {
        switch (a.h1) {
        case 8: return go2<8>(p, sms, s);
        case 16: return go2<16>(p, sms, s);
        case 32: return go2<32>(p, sms, s);
        case 64: return go2<64>(p, sms, s);
        }
    }
    return cudaErrorInvalidValue;
}

}  // namespace nns
