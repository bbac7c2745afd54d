// k_train_block.cu -- training many small models at once (Sec. "Training"), one thread block per
// model, entirely on chip: the block draws its array's sample, sorts it, labels it, initialises the
// network and runs every Adam step without leaving the kernel.
//
// For a model with one hidden layer of at most 32 units and a sample of at most TB_MAX_S keys the
// whole training set fits in shared memory and the gradient is a few hundred numbers, so launching
// two kernels per step over the whole GPU (the path of nnsort_train for large models) would spend
// its time on launches. Here:
//   * sample: S draws with replacement from the SplitMix64 stream (seed, 1), as nnsort_train;
//   * sort: a bitonic sort of the sample's order images in shared memory (equal keys give equal
//     inputs and consecutive labels, so the order among them does not change the training data);
//   * normaliser, inputs and labels: the sample's extremes, x_j = translate(key_j), label_j = j / S;
//   * initial weights: stream (seed, 2) in the same order and binary64 arithmetic as nnsort_train;
//   * each step: forward and backward over the full batch, or the minibatch drawn from stream
//     (seed, 3), every sum in a fixed order, then Adam in binary32.
#include <cstdint>

#include "common.cuh"
#include "internal.h"
#include "train_math.cuh"

namespace nns {
static inline cudaError_t nns_launched(cudaError_t e, int k = 1) {
    if (e == cudaSuccess) note_launch(k);
    return e;
}

namespace {
__device__ __forceinline__ double tb_unit53(uint64_t u) {
    return __dmul_rn((double)(u >> 11), 1.0 / 9007199254740992.0);
}

// the key word whose order image is u (the inverse of ordbits)
__device__ __forceinline__ uint64_t key_of_image(uint64_t u, int dtype) {
    if (dtype == NNSORT_F32) {
        const uint32_t b = (uint32_t)u;
        return (b & 0x80000000u) ? (uint64_t)(b & 0x7FFFFFFFu) : (uint64_t)(uint32_t)~b;
    }
    if (dtype == NNSORT_F64) return (u >> 63) ? (u & 0x7FFFFFFFFFFFFFFFull) : ~u;
    return u;
}
__device__ __forceinline__ double value_of_key(uint64_t w, int dtype) {
    if (dtype == NNSORT_F32) return (double)__uint_as_float((uint32_t)w);
    if (dtype == NNSORT_F64) return __longlong_as_double((long long)w);
    if (dtype == NNSORT_U32) return (double)(uint32_t)w;
    return __ull2double_rn(w);
}

template <int N> __device__ __forceinline__ float pairwise_sum(const float *v) {
    if constexpr (N == 1) return v[0];
    else return __fadd_rn(pairwise_sum<N / 2>(v), pairwise_sum<N / 2>(v + N / 2));
}

// fixed-order sum of v over the 32 lanes (the result in lane 0)
__device__ __forceinline__ float tb_warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = __fadd_rn(v, __shfl_down_sync(0xFFFFFFFFu, v, o));
    return v;
}
}  // namespace

// Samples a model's arrays hold: the sort's images, then inputs and labels in their place, and the
// upstream gradients beside them. A step walks its batch in chunks of at most tb_chunk samples (one chunk
// when the whole sample is the batch; a mini-batch stages its inputs too, in the gradients' array).
constexpr uint32_t TB_ROWS = 64;  // rows of a chunk at most
__host__ __device__ constexpr uint32_t tb_chunk(uint32_t cap, bool minibatch) { return minibatch ? cap / 2 : cap; }
template <int H> __host__ __device__ constexpr size_t tb_smem(uint32_t cap) {
    return (size_t)cap * 12 + (size_t)TB_ROWS * (3 * H) * 4;
}

// A step in three phases: (1) four samples per thread: forward pass, loss term and upstream gradient gy;
// (2) a (row, unit) per thread: over the row's samples with a positive activation, the sums of gy, gy x and
// gy h (two samples per packed instruction; the gradients of W1 and b1 are W3 times the first two); (3)
// a parameter per thread: its row sums pairwise, then Adam. Every sum has a fixed order. The first form
// kept all 3 H + 1 sums per thread and reduced each over the block by shuffles; 1,024 models of
// 1-16-1 on 1% samples of 1K..1M keys, 100 full-batch steps: 4.42 ms, now 2.59 ms. Rows of consecutive
// samples, added one after another, took the sums' rms error from 4.6e-8 to 8.3e-8 of their terms'
// magnitudes (and 2.70 ms); dealt out and added pairwise it is 4.6e-8 again.
template <typename W, int H, int T>
__global__ void __launch_bounds__(T) k_train_block(TrainBlockArgs a) {
    constexpr int P = 3 * H + 1;  // W1[H] b1[H] W3[H] b3 (padded layout of one hidden layer)
    constexpr int NW = T / 32;
    extern __shared__ __align__(16) unsigned char tb_raw[];
    unsigned long long *img = reinterpret_cast<unsigned long long *>(tb_raw);  // [cap] order images
    float *sx = reinterpret_cast<float *>(tb_raw);                             // then [cap] inputs
    float *slab = sx + a.cap;                                                  //      [cap] labels
    float *sgy = slab + a.cap;                                                 // [cap]
    float *part = sgy + a.cap;                                                 // [TB_ROWS][3 H]
    __shared__ __align__(16) float dp[4 * H];  // (W1, W1, b1, b1) per unit
    __shared__ __align__(8) float d3[2 * H];   // (W3, W3)
    __shared__ float sp[P], sm_[P], sv[P];
    __shared__ float red[NW][2];
    __shared__ Norm nm;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t m = a.ids[blockIdx.x];
    const uint64_t n = a.n[m];
    const uint32_t S = (uint32_t)a.S[m];
    const W *keys = reinterpret_cast<const W *>(a.keys[m]);
    const uint64_t seed = a.seed0 + m;
    uint32_t err = 0;

    // sample and its order images, up to the next power of two; the rest sorts last
    uint32_t cap = 2;
    while (cap < S) cap <<= 1;
    const uint64_t ss = rng_draw(seed, 1);
    for (uint32_t i = tid; i < cap; i += T) {
        unsigned long long u = ~0ull;
        if (i < S) {
            const uint64_t r = __umul64hi(rng_draw(ss, i), n);
            const uint64_t w = word64(keys[r]);
            if (key_is_nan(w, a.dtype)) err |= ERR_NAN;
            u = ordbits(w, a.dtype);
        }
        img[i] = u;
    }
    __syncthreads();
    // bitonic sort of the images, ascending
    for (uint32_t k = 2; k <= cap; k <<= 1) {
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            for (uint32_t q = tid; q < cap / 2; q += T) {
                const uint32_t i = 2 * q - (q & (j - 1)), p = i + j;  // i has bit j clear
                const unsigned long long x = img[i], y = img[p];
                if ((x > y) == ((i & k) == 0)) { img[i] = y; img[p] = x; }
            }
            __syncthreads();
        }
    }
    // normaliser from the sample's extremes (as nnsort_sample_labels computes it)
    if (tid == 0) {
        const uint64_t lo = img[0], hi = img[S - 1];
        Norm q;
        q.dtype = a.dtype;
        q.translate = a.translate;
        q.lo_bits = lo;
        q.lo_val = value_of_key(key_of_image(lo, a.dtype), a.dtype);
        const bool ob = a.translate == NNSORT_TRANSLATE_ORDBITS || a.dtype == NNSORT_U32 || a.dtype == NNSORT_U64;
        if (ob) {
            q.scale = (hi > lo) ? __ddiv_rn(1.0, __ull2double_rn(hi - lo)) : 1.0;
        } else {
            const double hv = value_of_key(key_of_image(hi, a.dtype), a.dtype);
            q.scale = (hv > q.lo_val) ? __ddiv_rn(1.0, __dsub_rn(hv, q.lo_val)) : 1.0;
        }
        q.lo_f = __double2float_rn(q.lo_val);
        q.scale_f = __double2float_rn(q.scale);
        nm = q;
        a.norm_out[m] = q;
    }
    // initial weights: W1_j in (-sqrt 6, sqrt 6), kink c_j in [0, 1) (b1_j = -W1_j c_j), output weights
    // in (-sqrt(6/h1), sqrt(6/h1)), b3 = 0; padding units stay 0
    for (int u = tid; u < P; u += T) { sp[u] = 0.0f; sm_[u] = 0.0f; sv[u] = 0.0f; }
    __syncthreads();
    if (tid < a.h1) {
        const uint64_t si = rng_draw(seed, 2);
        const double r1 = __dsqrt_rn(6.0), r3 = __dsqrt_rn(__ddiv_rn(6.0, (double)a.h1));
        const int j = tid, h1 = a.h1;
        const float w1 = __double2float_rn(__dmul_rn(__dsub_rn(__dmul_rn(2.0, tb_unit53(rng_draw(si, j))), 1.0), r1));
        sp[j] = w1;
        sp[H + j] = __double2float_rn(__dmul_rn(-(double)w1, tb_unit53(rng_draw(si, h1 + j))));
        sp[2 * H + j] = __double2float_rn(
            __dmul_rn(__dsub_rn(__dmul_rn(2.0, tb_unit53(rng_draw(si, 2 * h1 + j))), 1.0), r3));
    }
    // inputs and labels in place of the sorted images (each thread keeps its images over the barrier)
    {
        constexpr uint32_t MAXI = TB_MAX_S / 1024;  // images per thread: every class has cap <= MAXI * T
        unsigned long long mine[MAXI];
#pragma unroll
        for (uint32_t q = 0; q < MAXI; ++q) mine[q] = tid + q * T < S ? img[tid + q * T] : 0ull;
        __syncthreads();
#pragma unroll
        for (uint32_t q = 0; q < MAXI; ++q) {
            const uint32_t j = tid + q * T;
            if (j < a.cap) {
                sx[j] = j < S ? translate_x(key_of_image(mine[q], a.dtype), nm) : 0.0f;
                slab[j] = j < S ? __double2float_rn(__ddiv_rn((double)j, (double)S)) : 0.0f;
            }
        }
    }
    auto spread = [&]() {  // the parameters as lane pairs
        for (int j = tid; j < H; j += T) {
            dp[4 * j] = dp[4 * j + 1] = sp[j];
            dp[4 * j + 2] = dp[4 * j + 3] = sp[H + j];
            d3[2 * j] = d3[2 * j + 1] = sp[2 * H + j];
        }
    };
    spread();
    __syncthreads();

    const uint64_t B = a.batch ? a.batch : S;
    const float inv_n = 1.0f / (float)B;
    const uint64_t bseed = rng_draw(seed, 3);
    const uint32_t CH = tb_chunk(a.cap, a.batch != 0);
    float *cx = a.batch ? sgy + CH : sx;  // the chunk's inputs
    for (int step = 0; step < a.steps; ++step) {
        float gsum = 0.0f, lsum = 0.0f;
        uint32_t rows = 0;
        for (uint64_t c0 = 0; c0 < B; c0 += CH) {
            const uint32_t cn = (uint32_t)min((uint64_t)CH, B - c0), cn4 = (cn + 3) & ~3u;
            if (c0) __syncthreads();  // the last chunk's readers are done
            const float b3 = sp[3 * H];
            for (uint32_t i = 4 * tid; i < cn4; i += 4 * T) {
                float x[4], lab[4], gy[4];
                if (a.batch) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        x[q] = lab[q] = 0.0f;
                        if (i + q < cn) {
                            const uint64_t src = __umul64hi(rng_draw(bseed, (uint64_t)step * B + c0 + i + q), S);
                            x[q] = sx[src];
                            lab[q] = slab[src];
                        }
                    }
                    *reinterpret_cast<float4 *>(cx + i) = make_float4(x[0], x[1], x[2], x[3]);
                } else {
                    const float4 xv = *reinterpret_cast<const float4 *>(sx + i);
                    const float4 lv = *reinterpret_cast<const float4 *>(slab + i);
                    x[0] = xv.x; x[1] = xv.y; x[2] = xv.z; x[3] = xv.w;
                    lab[0] = lv.x; lab[1] = lv.y; lab[2] = lv.z; lab[3] = lv.w;
                }
                const unsigned long long x01 = pk2(x[0], x[1]), x23 = pk2(x[2], x[3]);
                unsigned long long y01 = pk2(b3, b3), y23 = y01;
#pragma unroll 4
                for (int j = 0; j < H; ++j) {
                    const ulonglong2 c = *reinterpret_cast<const ulonglong2 *>(dp + 4 * j);
                    const unsigned long long w3 = *reinterpret_cast<const unsigned long long *>(d3 + 2 * j);
                    float h0, h1, h2, h3;
                    upk2(fma2_rn(c.x, x01, c.y), h0, h1);
                    upk2(fma2_rn(c.x, x23, c.y), h2, h3);
                    y01 = fma2_rn(w3, pk2(relu_f(h0), relu_f(h1)), y01);
                    y23 = fma2_rn(w3, pk2(relu_f(h2), relu_f(h3)), y23);
                }
                float y[4];
                upk2(y01, y[0], y[1]);
                upk2(y23, y[2], y[3]);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float lv;
                    loss_term(__fsub_rn(y[q], lab[q]), a.loss, a.delta, inv_n, gy[q], lv);
                    if (i + q >= cn) { gy[q] = 0.0f; lv = 0.0f; }
                    gsum = __fadd_rn(gsum, gy[q]);
                    lsum = __fadd_rn(lsum, lv);
                }
                *reinterpret_cast<float4 *>(sgy + i) = make_float4(gy[0], gy[1], gy[2], gy[3]);
            }
            __syncthreads();
            // rows of groups of four samples, enough of them to spread the chunk over the threads. Row k takes
            // groups k, k + nrow, ...: neighbours in the sorted sample share their residual's sign, and a sum
            // that runs through neighbours grows, and rounds, far beyond the whole sum
            uint32_t nrow = (cn + 15) / 16;
            nrow = nrow < TB_ROWS ? nrow : TB_ROWS;
            const uint32_t stride = 4 * nrow;
            for (uint32_t t = tid; t < nrow * H; t += T) {
                const uint32_t k = t / H, j = t % H;
                const unsigned long long w1 = pk2(sp[j], sp[j]), b1 = pk2(sp[H + j], sp[H + j]);
                unsigned long long sa1 = 0, sa2 = 0, sa3 = 0, sb1 = 0, sb2 = 0, sb3 = 0;
#pragma unroll 2
                for (uint32_t i = 4 * k; i < cn4; i += stride) {
                    const ulonglong2 xv = *reinterpret_cast<const ulonglong2 *>(cx + i);
                    const float4 gv = *reinterpret_cast<const float4 *>(sgy + i);
                    const unsigned long long ha = fma2_rn(w1, xv.x, b1), hb = fma2_rn(w1, xv.y, b1);
                    float h0, h1, h2, h3;
                    upk2(ha, h0, h1);
                    upk2(hb, h2, h3);
                    const unsigned long long ga = pk2(h0 > 0.0f ? gv.x : 0.0f, h1 > 0.0f ? gv.y : 0.0f);
                    const unsigned long long gb = pk2(h2 > 0.0f ? gv.z : 0.0f, h3 > 0.0f ? gv.w : 0.0f);
                    sa1 = fma2_rn(ga, xv.x, sa1);
                    sa2 = add2_rn(sa2, ga);
                    sa3 = fma2_rn(ga, ha, sa3);
                    sb1 = fma2_rn(gb, xv.y, sb1);
                    sb2 = add2_rn(sb2, gb);
                    sb3 = fma2_rn(gb, hb, sb3);
                }
                float *o = part + k * (3 * H);
                const bool add = c0 && k < rows;  // a row of an earlier chunk
                auto put = [&](float *q, unsigned long long u, unsigned long long v) {
                    float e, f;
                    upk2(add2_rn(u, v), e, f);
                    e = __fadd_rn(e, f);
                    *q = add ? __fadd_rn(*q, e) : e;
                };
                put(o + j, sa1, sb1);
                put(o + H + j, sa2, sb2);
                put(o + 2 * H + j, sa3, sb3);
            }
            rows = rows > nrow ? rows : nrow;
        }
        // db3 and the loss: shuffle tree inside each warp, then the warps in order
        gsum = tb_warp_sum(gsum);
        lsum = tb_warp_sum(lsum);
        if (lane == 0) { red[warp][0] = gsum; red[warp][1] = lsum; }
        __syncthreads();
        float np = 0.0f;
        if (tid < P) {
            float gs = 0.0f;
            if (tid < 3 * H) {
                // the rows pairwise, eight at a time
                float blk[TB_ROWS / 8];
#pragma unroll
                for (uint32_t q = 0; q < TB_ROWS / 8; ++q) {
                    float v[8];
#pragma unroll
                    for (uint32_t r = 0; r < 8; ++r)
                        v[r] = 8 * q + r < rows ? part[(8 * q + r) * (3 * H) + tid] : 0.0f;
                    blk[q] = pairwise_sum<8>(v);
                }
                gs = pairwise_sum<TB_ROWS / 8>(blk);
                if (tid < 2 * H) gs = __fmul_rn(gs, sp[2 * H + tid % H]);
            } else {
#pragma unroll
                for (int w = 0; w < NW; ++w) gs = __fadd_rn(gs, red[w][0]);
            }
            np = adam_step(sp[tid], gs, sm_[tid], sv[tid], a.lr, a.b1, a.b2, a.eps, a.c1[step], a.c2[step], 0.0f);
        } else if (tid == P && a.loss_out) {
            float l = 0.0f;
#pragma unroll
            for (int w = 0; w < NW; ++w) l = __fadd_rn(l, red[w][1]);
            a.loss_out[(size_t)m * a.steps + step] = l * inv_n;
        }
        __syncthreads();  // W3 has been read
        if (tid < P) {
            sp[tid] = np;
            if (tid < H) dp[4 * tid] = dp[4 * tid + 1] = np;
            else if (tid < 2 * H) dp[4 * (tid - H) + 2] = dp[4 * (tid - H) + 3] = np;
            else if (tid < 3 * H) d3[2 * (tid - 2 * H)] = d3[2 * (tid - 2 * H) + 1] = np;
        }
        __syncthreads();
    }
    for (int u = tid; u < P; u += T) a.params_out[(size_t)m * P + u] = sp[u];
    if (err) atomicOr(a.err, err);
}

template <typename W, int T>
static cudaError_t tb_go(const TrainBlockArgs &a, int H, uint32_t blocks, cudaStream_t s) {
    constexpr uint32_t most = T == 128 ? 1024 : T == 512 ? 4096 : TB_MAX_S;  // the class's largest sample
    auto go = [&](auto kfn, size_t smem, size_t top) -> cudaError_t {
        cudaError_t e = allow_smem(kfn, top);
        if (e != cudaSuccess) return e;
        kfn<<<blocks, T, smem, s>>>(a);
        return nns_launched(cudaGetLastError());
    };
    switch (H) {
    case 8: return go(k_train_block<W, 8, T>, tb_smem<8>(a.cap), tb_smem<8>(most));
    case 16: return go(k_train_block<W, 16, T>, tb_smem<16>(a.cap), tb_smem<16>(most));
    case 32: return go(k_train_block<W, 32, T>, tb_smem<32>(a.cap), tb_smem<32>(most));
    }
    return cudaErrorInvalidValue;
}

// threads per model by the class's sample size: what a step of its samples keeps busy (and at most 16
// images per thread)
template <typename W>
static cudaError_t tb_class(const TrainBlockArgs &a, int H, uint32_t blocks, cudaStream_t s) {
    if (a.cap <= 1024) return tb_go<W, 128>(a, H, blocks, s);
    if (a.cap <= 4096) return tb_go<W, 512>(a, H, blocks, s);
    return tb_go<W, 1024>(a, H, blocks, s);
}

cudaError_t launch_train_block(const TrainBlockArgs &a, int key_bytes, int padded_h, uint32_t blocks,
                               cudaStream_t s) {
    if (blocks == 0) return cudaSuccess;
    if (a.cap < 8 || a.cap > TB_MAX_S || (a.cap & (a.cap - 1))) return cudaErrorInvalidValue;
    return key_bytes == 4 ? tb_class<uint32_t>(a, padded_h, blocks, s) : tb_class<uint64_t>(a, padded_h, blocks, s);
}

}  // namespace nns
