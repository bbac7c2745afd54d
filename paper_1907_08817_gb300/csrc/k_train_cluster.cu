// k_train_cluster.cu -- every Adam step of one-hidden-layer models in one launch (Sec. "Training"):
// one cluster of 16 blocks per model.
//
// A step's batch is cut into the same rows of at most 64 samples as the per-step gradient kernel
// (k_grad), and block c of the cluster takes rows c, c + 16, ...: the rows that warp c of the per-step
// reduction (k_reduce) adds up, in the same order. So the block's sums are that warp's sums, the
// sixteen of them meet through distributed shared memory in the reduction's final order, and every
// parameter is bit for bit what the two-kernel steps give. Within a row a thread owns one unit and walks
// the row's samples in order, recomputing the activation from the sample's input (three sums in
// registers, nothing staged but the input and upstream gradient of each sample). Every block applies
// Adam to its own copy of the parameters, so a step needs one cluster barrier.
//
// What bounds a step is that chain: a sample's forward pass, a row's 64 samples, the barrier and the
// remote reads. Two launches a step took 15 us for 10,000 samples of 1-32-1 (8 us of kernels, the rest
// between them): with one launch, training and sorting 1,000,000 keys takes 1.20 ms instead of 2.23 ms.
#include <algorithm>
#include <cooperative_groups.h>

#include "common.cuh"
#include "internal.h"
#include "train_math.cuh"

namespace nns {
namespace {
namespace cg = cooperative_groups;

constexpr int TC1_CTAS = 16;      // = the warps of k_reduce
constexpr int TC1_THREADS = 512;
constexpr int TC1_ROW = 64;       // samples per row at most
constexpr uint64_t TC1_MAX_BATCH = 65536;  // 1,024 rows: beyond, rows hold several chunks

template <int H>
__global__ void __launch_bounds__(TC1_THREADS) k_train_cluster(const TrainJob *jobs, TrainHyper hp, uint32_t cap,
                                                               uint32_t rcap) {
    constexpr int P = 3 * H + 1;
    extern __shared__ __align__(16) float dyn[];
    float2 *xg = reinterpret_cast<float2 *>(dyn);            // [cap] input, upstream gradient
    float2 *xl = xg + cap;                                   // [cap] input, label (kept across steps: full batch)
    float *slv = reinterpret_cast<float *>(xl + cap);        // [cap] loss terms
    float *part = slv + cap;                                 // [rcap][P + 1] row sums, the loss last
    __shared__ float sp[P], sums[2][P + 1];
    cg::cluster_group cl = cg::this_cluster();
    const uint32_t c = cl.block_rank();
    const int tid = threadIdx.x;
    const TrainJob J = jobs[blockIdx.y];
    if (J.blocks == 0) return;  // refused (every block of the cluster)
    // the rows of the per-step kernel: `nrow` rows of `per` samples
    const uint32_t B = (uint32_t)J.B, nrow = J.blocks, per = (B + nrow - 1) / nrow;
    const uint32_t rows = c < nrow ? (nrow - c + TC1_CTAS - 1) / TC1_CTAS : 0u;
    const uint32_t nloc = rows * per;
    auto global_of = [&](uint32_t i) -> uint32_t { return (c + TC1_CTAS * (i / per)) * per + i % per; };
    for (int p = tid; p < P; p += TC1_THREADS) sp[p] = J.params[p];
    if (!hp.batch)
        for (uint32_t i = tid; i < nloc; i += TC1_THREADS) {
            const uint32_t g = global_of(i);
            xl[i] = g < B ? make_float2(J.x[g], J.label[g]) : make_float2(0.0f, 0.0f);
        }
    float am = 0.0f, av = 0.0f;  // Adam moments of parameter `tid`
    const float mask = (J.mask && tid < P) ? J.mask[tid] : 0.0f;
    __syncthreads();
    for (int step = 0; step < hp.steps; ++step) {
        // a sample per thread: forward pass, loss term, upstream gradient
        for (uint32_t i = tid; i < nloc; i += TC1_THREADS) {
            const uint32_t g = global_of(i);
            float2 v = make_float2(0.0f, 0.0f);
            if (hp.batch) {
                if (g < B) {
                    const uint64_t src = __umul64hi(rng_draw(J.bseed, (uint64_t)step * B + g), J.S);
                    v = make_float2(J.x[src], J.label[src]);
                }
            } else {
                v = xl[i];
            }
            float y = sp[3 * H];
#pragma unroll
            for (int j = 0; j < H; ++j) y = __fmaf_rn(sp[2 * H + j], relu_f(__fmaf_rn(sp[j], v.x, sp[H + j])), y);
            float gy, lv;
            loss_term(y - v.y, hp.loss, hp.delta, J.inv_n, gy, lv);
            xg[i] = make_float2(v.x, gy);
            slv[i] = lv;
        }
        __syncthreads();
        // a (row, unit) per thread: the row's samples in order; then b3 and the loss, a row per thread
        const uint32_t tasks = rows * H;
        for (uint32_t t = tid; t < tasks; t += TC1_THREADS) {
            const uint32_t k = t / H, j = t % H;
            const uint32_t r0 = (c + TC1_CTAS * k) * per;
            const uint32_t cn = r0 < B ? min(per, B - r0) : 0u;
            const float w1 = sp[j], b1 = sp[H + j], w3 = sp[2 * H + j];
            const float2 *row = xg + k * per;
            float s1 = 0.0f, s2 = 0.0f, s3 = 0.0f;
#pragma unroll 8
            for (uint32_t q = 0; q < cn; ++q) {
                const float2 v = row[q];
                const float h = relu_f(__fmaf_rn(w1, v.x, b1));
                const float d1 = (h > 0.0f) ? __fmul_rn(v.y, w3) : 0.0f;
                s1 = __fmaf_rn(d1, v.x, s1);
                s2 = __fadd_rn(s2, d1);
                s3 = __fmaf_rn(v.y, h, s3);
            }
            float *o = part + k * (P + 1);
            o[j] = __fadd_rn(0.0f, s1);  // the row's accumulator starts at +0
            o[H + j] = __fadd_rn(0.0f, s2);
            o[2 * H + j] = __fadd_rn(0.0f, s3);
        }
        // the last threads take the two remaining sums, so that they run beside the units' tasks
        for (uint32_t t = TC1_THREADS - 1 - tid; t < 2 * rows; t += TC1_THREADS) {
            const uint32_t k = t >> 1;
            const uint32_t r0 = (c + TC1_CTAS * k) * per;
            const uint32_t cn = r0 < B ? min(per, B - r0) : 0u;
            float s = 0.0f;
            if (t & 1) {
#pragma unroll 8
                for (uint32_t q = 0; q < cn; ++q) s = __fadd_rn(s, slv[k * per + q]);
                part[k * (P + 1) + P] = s;
            } else {
#pragma unroll 8
                for (uint32_t q = 0; q < cn; ++q) s = __fadd_rn(s, xg[k * per + q].y);
                part[k * (P + 1) + P - 1] = __fadd_rn(0.0f, s);
            }
        }
        __syncthreads();
        float *mine = sums[step & 1];
        for (int p = tid; p <= P; p += TC1_THREADS) {
            float s = 0.0f;
#pragma unroll 4
            for (uint32_t k = 0; k < rows; ++k) s = __fadd_rn(s, part[k * (P + 1) + p]);
            mine[p] = s;
        }
        // one barrier a step: the sums alternate between two buffers, so that the next step's writes
        // cannot meet this step's remote reads (a block that writes a buffer again has passed the
        // barrier that every reader of it reached after reading)
        cl.sync();
        if (tid <= P) {
            float q[TC1_CTAS];
#pragma unroll
            for (int r = 0; r < TC1_CTAS; ++r) q[r] = cl.map_shared_rank(mine, r)[tid];
            float g = 0.0f;
#pragma unroll
            for (int r = 0; r < TC1_CTAS; ++r) g = __fadd_rn(g, q[r]);
            if (tid < P)
                sp[tid] = adam_step(sp[tid], g, am, av, hp.lr, hp.b1, hp.b2, hp.eps, hp.c12[step],
                                    hp.c12[hp.steps + step], mask);
            else if (c == 0)
                J.loss_out[step] = g * J.inv_n;
        }
        __syncthreads();
    }
    if (c == 0)
        for (int p = tid; p < P; p += TC1_THREADS) J.params[p] = sp[p];
    cl.sync();  // no block's shared memory goes away while another may still read it
}

template <int H>
cudaError_t go(const TrainJob *jobs, uint32_t models, const TrainHyper &hp, uint64_t max_batch, bool probe,
               cudaStream_t s) {
    static_assert(3 * H + 2 <= TC1_THREADS, "a thread per sum");
    auto rows_of = [](uint64_t batch) {  // of a block
        return (uint32_t)(((batch + TC1_ROW - 1) / TC1_ROW + TC1_CTAS - 1) / TC1_CTAS);
    };
    auto smem_of = [](uint32_t rows) { return (size_t)rows * TC1_ROW * 20 + (size_t)rows * (3 * H + 2) * 4; };
    const uint32_t rcap = rows_of(max_batch), cap = rcap * TC1_ROW;
    const size_t smem = smem_of(rcap);
    auto kfn = k_train_cluster<H>;
    cudaError_t e = allow_smem(kfn, smem_of(rows_of(TC1_MAX_BATCH)));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kfn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(TC1_CTAS, std::max<uint32_t>(1, models));
    cfg.blockDim = dim3(TC1_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = TC1_CTAS;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (probe) {
        int n = 0;
        e = cudaOccupancyMaxActiveClusters(&n, kfn, &cfg);
        return e != cudaSuccess ? e : (n >= 1 ? cudaSuccess : cudaErrorNotSupported);
    }
    e = cudaLaunchKernelEx(&cfg, kfn, jobs, hp, cap, rcap);
    if (e == cudaSuccess) note_launch(1);
    return e;
}

cudaError_t dispatch(int h, const TrainJob *jobs, uint32_t models, const TrainHyper &hp, uint64_t max_batch,
                     bool probe, cudaStream_t s) {
    switch (h) {
    case 8: return go<8>(jobs, models, hp, max_batch, probe, s);
    case 16: return go<16>(jobs, models, hp, max_batch, probe, s);
    case 32: return go<32>(jobs, models, hp, max_batch, probe, s);
    case 64: return go<64>(jobs, models, hp, max_batch, probe, s);
    }
    return cudaErrorInvalidValue;
}
}  // namespace

// One hidden layer and batches of at most 65,536 samples. At that size a step takes as long as the
// chain of one block's 4,096 samples; beyond it the per-step kernels' 1,024 blocks are as fast.
bool train_cluster_ok(const PadArch &a, uint64_t max_batch) {
    if (a.layers != 1 || max_batch == 0 || max_batch > TC1_MAX_BATCH) return false;
    if (dispatch(a.h1, nullptr, 1, TrainHyper{}, max_batch, true, nullptr) == cudaSuccess) return true;
    cudaGetLastError();  // a device partition without room for a 16-block cluster: the per-step kernels
    return false;
}

cudaError_t launch_train_cluster(const PadArch &a, const TrainJob *jobs, uint32_t models, const TrainHyper &hp,
                                 uint64_t max_batch, cudaStream_t s) {
    if (hp.steps == 0) return cudaSuccess;
    return dispatch(a.h1, jobs, models, hp, max_batch, false, s);
}

}  // namespace nns
