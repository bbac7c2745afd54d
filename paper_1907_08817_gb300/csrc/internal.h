// internal.h -- host-side declarations shared by the library's translation units.
#pragma once
#include <cstddef>
#include <cstdint>
#include <memory>
#include <vector>
#include <cuda_runtime.h>

#include "nnsort.h"

namespace nns {

// counts kernels launched by the library (nnsort_launch_count)
void note_launch(int kernels);

// Allows a kernel `most` bytes of dynamic shared memory: the most that any launch of it takes, not this
// launch's own share. The attribute is the function's, so a call that set what it needs itself could lower
// it between another thread's setting and launch, which then fails.
template <typename K> inline cudaError_t allow_smem(K kfn, size_t most) {
    return cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}
constexpr size_t BLOCK_SMEM = 227 * 1024;  // of one block

struct Seg;
struct Norm;
struct SegStats;
struct OKey;

constexpr int RADIX_MAX_BITS = 9;
constexpr int RADIX_BINS = 1 << RADIX_MAX_BITS;  // 512
constexpr int PRED_THREADS = 256;
constexpr int PRED_ITEMS = 8;
constexpr int PRED_TILE = PRED_THREADS * PRED_ITEMS;  // 2048
constexpr int MAX_PASSES = 4;

struct PassPlan {
    int npass;
    int wlog;                 // log2 of the bucket width in positions
    int shift[MAX_PASSES];    // digit shift applied to the global position
    int bits[MAX_PASSES];
};

// padded architecture actually instantiated on the device
struct PadArch {
    int layers, h1, h2;  // padded widths (8, 16, 32 or 64; h2 = 0 for one hidden layer)
};
PadArch pad_arch(int layers, int h1, int h2);
size_t padded_param_count(const PadArch &a);

// ---- predict (k_predict.cu)
// Fills gs (global position per element) and optional key / payload / row copies into the element
// space. Also serves nnsort_predict through slots_out / y_out (element space of a single array).
// one segment of the compiled piecewise-linear model in the keys' order-image domain (pwl.cu)
struct PwlEntry {
    unsigned long long thr;  // smallest order image in the segment (0 for the first)
    float Ah, Al, Ch, Cl;    // position = floor(A d + C), d = translate offset of the key, with
                             // A = Ah + Al and C = Ch + Cl (pairs of binary32: ~48 significant bits)
};
struct PwlDev {
    const PwlEntry *tab;     // device table, null when the compiled form is not used
    uint32_t S;              // segments
};

struct PredictArgs {
    const Seg *segs;
    int nseg;
    uint32_t total_tiles;
    uint32_t *gs;            // nullable
    void *key_copy;          // nullable
    uint32_t *pay_copy;      // nullable
    uint32_t *row_init;      // nullable
    uint32_t *slots_out;     // nullable
    float *y_out;            // nullable
    uint32_t *err;
    int key_bytes;
    int dtype;
    PwlDev pwl;              // NNSORT_PREC_PWL (single array)
    int single_model;        // 1: one array whose positions come from its model (no injected slots)
    const Seg *host_seg;     // single_model: the array's segment in host memory
    const float *host_pad;   // single_model: that model's padded parameters in host memory
};
cudaError_t launch_predict(const PadArch &a, int precision, const PredictArgs &p, int sms,
                           cudaStream_t s);
cudaError_t launch_predict_pwl(const PredictArgs &p, int sms, cudaStream_t s);
// host side of the compiled form (pwl.cu)
void pwl_segments(int layers, int h1, int h2, const float *params, std::vector<double> &brk,
                  std::vector<double> &slope, std::vector<double> &icept);
uint32_t pwl_max_segments(int layers, int h1, int h2);
void pwl_key_table(const nnsort_model_desc &d, const std::vector<double> &brk, const std::vector<double> &slope,
                   const std::vector<double> &icept, double nm, PwlEntry *out);

// ---- partition (k_partition.cu)
// One pass of the stable digit partition without inter-block waits (reduce, then scan, then
// scatter): per tile of SC_TILE elements a digit histogram, per chunk of SC_CHUNK tiles the
// in-chunk exclusive prefixes and chunk totals (and the digit totals), the chunk bases over all
// chunks and digits, then the scatter of every tile to its chunk's base + its in-chunk prefix.
// The pass finds its own digit offsets, so no histogram is needed beforehand; tile_hist, chunk and
// bin_total are scratch.
constexpr int SC_TILE = 4096;
constexpr int SC_CHUNK = 65536 / SC_TILE;  // tiles per chunk (in-chunk prefix < 2^16)
struct PartitionArgs {
    uint64_t N;
    const uint32_t *gs_in;  uint32_t *gs_out;   // null when sorting by key bits
    const void *key_in;     void *key_out;
    const uint32_t *pay_in; uint32_t *pay_out;  // nullable
    const uint32_t *row_in; uint32_t *row_out;  // nullable
    int key_digits;         // 1: digit from the key's order image, 0: from gs
    int shift, bits;
    uint16_t *tile_hist;    // [tiles * RADIX_BINS] scratch
    uint32_t *chunk;        // [chunks * RADIX_BINS] scratch
    uint32_t *bin_total;    // [RADIX_BINS] scratch: elements per digit
    int key_bytes, dtype;
};
inline uint64_t partition_tiles(uint64_t N) { return (N + SC_TILE - 1) / SC_TILE; }
inline uint64_t partition_chunks(uint64_t N) { return (partition_tiles(N) + SC_CHUNK - 1) / SC_CHUNK; }
cudaError_t launch_partition(const PartitionArgs &a, cudaStream_t s);
// bucket starts by binary search over the partitioned global positions
cudaError_t launch_bucket_bounds(const uint32_t *gs, uint64_t N, uint32_t nb, int wlog,
                                 uint32_t *bstart, cudaStream_t s);

// ---- rounds / finalize / polish / seam / repair (k_solve.cu)
// an output range [lo, hi) of array `seg` (positions relative to the array) to be re-sorted
struct SeamRange {
    unsigned long long lo, hi;
    uint32_t seg, pad;
};

// a bucket too large for one block's polish: partitioned elements [lo, hi) of array `seg`, bucket b,
// offset `off` in the packed buffer
struct BigRange {
    unsigned long long lo, hi;
    uint32_t seg, off, b, pad;
};
constexpr uint32_t POLISH_BIG = 1u << 16;  // two-kernel form: larger buckets sort multi-block
constexpr uint32_t GIANT_LEAST = 8192;     // no listed bucket is smaller (sizes the lists)

struct SolveArgs {
    const Seg *segs;
    int nseg;
    uint32_t NB;
    int wlog;
    const uint32_t *bstart;   // [NB + 1]
    const uint32_t *gs;       // partitioned
    const void *keys;         // partitioned
    const uint32_t *pay;      // partitioned, nullable
    const uint32_t *rows;     // partitioned, nullable
    uint8_t *rank;            // [N]
    SegStats *stats;          // [nseg]
    OKey *bmax;               // [NB * MAXR]
    OKey *carry;              // [NB * MAXR]
    OKey *blo, *bhi;          // [NB]
    // global scratch for buckets beyond on-chip capacity
    uint8_t *g_flag;          // [N]
    uint32_t *g_x, *g_y;  // [N] each
    uint64_t N;               // elements (the sizes of the [N] scratch arrays)
    int8_t *fate;             // nullable, per row (single array only)
    uint32_t *out_rows;       // [N] rows of the output order (when rows are carried)
    void *key_scratch;        // [N] free partition buffer reused by the seam repair
    uint32_t *pay_scratch, *row_scratch;
    uint32_t *err;
    int key_bytes, dtype;
    int polish_cap;           // elements that a bucket of the two-kernel form may hold on chip
    size_t polish_smem;
    int allow_defer;          // 1: seam repairs above seam_max are left to the host's
                              //    multi-block sort (never when rows are carried)
    uint32_t seam_max;        // elements of the largest repair that one block performs
    SeamRange *ranges;        // [max_ranges]: block-sized repairs from the front, large from the back
    uint32_t max_ranges;      // >= NB + nseg
    uint32_t *seam_cnt;       // [4], zero before the seam: block-sized ranges, large ranges, next range to repair
    OKey *seam_suf;           // [NB] scratch: smallest element of the later buckets
    OKey *seam_pre;           // [NB] scratch: largest element of the earlier buckets
    unsigned long long *seam_cut;  // [2 NB] scratch: first and last sorted-boundary cut per bucket
    // one-pass buckets (launch_buckets; null rk: not used): the in-order runs that await their carries,
    // as order images and tie-breaks in partitioned element order, and where each round's run ends
    void *rk;                 // [N] keys' width
    uint32_t *rt;             // [N]
    uint32_t *rend;           // [NB * MAXR]
    int bucket_cap[3];        // elements that a one-pass block holds: of the width's own size, with two
                              //   512-thread blocks per SM, with one
    int bucket_threads;       // threads of the first of these
    int seam_cap;             // elements that a block of the on-chip seam repair holds
    const uint32_t *heavy_cnt;  // with rk: the order's first *heavy_cnt buckets exceed bucket_cap[0]
    uint32_t giant_min;       // buckets above this many elements are listed in giant
    int list_refused;         // 1: also after an error (their rounds only; nothing is written back)
    const uint32_t *order;    // [NB] nullable: block i of k_bucket / k_rounds / k_polish takes bucket order[i]
    BigRange *giant;          // nullable: k_bucket_order lists buckets above giant_min here, in any order;
    uint32_t *giant_cnt;      //   [2] their count and their elements. k_bucket and k_rounds leave them to
                              //   launch_giant_buckets and launch_giant_rounds
    BigRange *big;            // nullable: k_polish lists buckets above POLISH_BIG here (and only
    uint32_t *big_cnt;        //   splits their runs); their sort is left to the host's multi-block sort
};
// largest seam repair one block performs (less where its on-chip form holds less, at least SEAM_CTA_LEAST):
// blocks that took up to 65,536 elements, with their lists in global memory, held the whole sort up (1,024
// arrays, 147M keys: 0.65 ms of repairs; 0.18 with 16,384, 0.07 with 8,192)
constexpr uint64_t SEAM_CTA_MAX = 1u << 13, SEAM_CTA_LEAST = 1u << 12;
constexpr uint64_t SEAM_SMALL = 1u << 16;  // arrays of at most this many elements: what one block can hold
// order[]: buckets holding more than `heavy` elements first (they run longest), the rest after
cudaError_t launch_bucket_order(const SolveArgs &a, uint32_t heavy, uint32_t *order,
                                uint32_t *cnt /*[2], zero, as giant_cnt*/, cudaStream_t s);
// buckets above giant_min elements run their rounds on the whole GPU (global claim tables); the
// list, its count and the per-(bucket, round) statistics live in GiantRounds
struct GiantRounds {
    BigRange *list;               // [N / giant_min + 1]
    uint32_t *count;              // [2] entries, their elements
    unsigned long long *table;    // [list entries x W] round-tagged claims
    unsigned int *cnt;            // [entries x MAXR] elements stored per round
    unsigned long long *kmax;     // [entries x MAXR] largest order image stored per round
    unsigned int *tbmax;          // [entries x MAXR] its largest tie-break
    uint32_t cap;                 // list entries
};
// the same for buckets that no one-pass block holds, their runs split round by round from the claim
// table (cnt: elements stored and run elements so far, two words per entry); the list receives their packed
// offsets
cudaError_t launch_giant_buckets(const SolveArgs &a, const GiantRounds &g, int eps, int sms, cudaStream_t s);
cudaError_t launch_giant_rounds(const SolveArgs &a, const GiantRounds &g, int eps, int sms, cudaStream_t s);
cudaError_t launch_rounds(const SolveArgs &a, cudaStream_t s);
// every bucket of at most bucket_cap[0] elements in one pass (rounds, runs and sorted output), then the
// heavy ones of at most bucket_cap[2] (if the array can hold any), and their out-of-order counts once the
// carries are known; larger ones are left to launch_giant_buckets and the host's multi-block sort
bool buckets_ok(int wlog, bool rows);
void bucket_capacities(SolveArgs &a, bool payload);
cudaError_t launch_buckets(const SolveArgs &a, cudaStream_t s);
cudaError_t launch_heavy_buckets(const SolveArgs &a, int sms, cudaStream_t s);
cudaError_t launch_carried(const SolveArgs &a, cudaStream_t s);
// one array of few buckets: bounds and order, finalize and carried counts, in one launch each
bool small_solve(const SolveArgs &a);
cudaError_t launch_bounds_order_small(const SolveArgs &a, uint32_t *bstart, uint32_t heavy, uint32_t *order,
                                      uint32_t *cnt, cudaStream_t s);
cudaError_t launch_finalize_small(const SolveArgs &a, cudaStream_t s);
cudaError_t launch_finalize(const SolveArgs &a, cudaStream_t s);
cudaError_t launch_polish(const SolveArgs &a, cudaStream_t s);
cudaError_t launch_seam_repair(const SolveArgs &a, int sms, cudaStream_t s);
cudaError_t launch_big_pack(const BigRange *br, uint32_t nr, const Seg *segs, uint64_t total, int key_bytes,
                            const void *src_k, const uint32_t *src_p, void *pk, uint32_t *pp, uint32_t *pj,
                            int unpack, int sms, cudaStream_t s);
cudaError_t launch_big_bounds(const BigRange *br, uint32_t nr, const Seg *segs, int key_bytes, int dtype,
                              OKey *blo, OKey *bhi, cudaStream_t s);
cudaError_t launch_seam_pack(const SeamRange *rg, uint32_t nr, const Seg *segs, uint64_t total,
                             int key_bytes, void *pk, uint32_t *pp, uint32_t *ps, int unpack, int sms,
                             cudaStream_t s);
int polish_capacity(int key_bytes, bool payload, bool rows, int wlog, int blocks_per_sm,
                    size_t *smem_bytes);

// ---- training (k_train.cu)
cudaError_t launch_sample(const void *keys, uint64_t n, int key_bytes, int dtype, uint64_t S,
                          uint64_t stream_seed, void *sample_keys, uint32_t *sample_rows,
                          uint32_t *err, cudaStream_t s);
cudaError_t launch_make_xy(const void *sorted_keys, uint64_t S, int key_bytes, const Norm *nm_dev,
                           float *x, float *label, cudaStream_t s);
// a training run of the two-layer model of width 64 (k_train_tc.cu)
struct TrainStepArgs {
    float *params;        // padded layout, updated in place
    float *m, *v;         // Adam moments (padded layout)
    float *partials;      // [blocks * P]
    float *loss_partials; // [blocks]
    float *loss_out;      // [steps]
    const float *x, *label;
    uint64_t S;
    uint32_t batch;       // 0 = full
    uint64_t batch_seed;
    int loss; float delta;
    float lr, b1, b2, eps;
    const float *mask;    // nullable: +1/-1 sign a parameter must keep, 0 free
    const uint32_t *refused;  // device word: not zero when the model's sample was refused
};
// One model of a training call (models of one architecture trained side by side): its sample, its
// batch and its parameters. Sample arrays of all models are packed; `off` is the model's first entry.
struct TrainJob {
    const void *keys;        // device keys to sample
    uint64_t n, S, off;      // keys, sample size, offset in the packed sample arrays
    uint64_t sseed, bseed;   // sample and mini-batch streams
    uint64_t B;              // samples per step
    float inv_n;             // 1 / B
    uint32_t blocks;         // partial gradient rows of a step (0 on the device: the model is refused)
    float *params, *m, *v;   // padded layout
    const float *mask;       // nullable: signs to keep
    const float *x, *label;  // [S]
    float *partials, *loss_partials;  // [blocks * P], [blocks] (null where no kernel uses them)
    float *loss_out;         // [steps]
};
struct TrainHyper {
    int steps;
    uint32_t batch;          // 0: full batch
    int loss;
    float delta, lr, b1, b2, eps;
    const float *c12;        // device [2 * steps]: 1 - beta1^(t+1), then 1 - beta2^(t+1)
};
// sample keys of every job (packed; `group` nullable: the job index of each), their inputs, labels and
// normalisers once sorted
cudaError_t launch_sample_jobs(const TrainJob *jobs, uint32_t models, uint64_t max_S, int key_bytes, int dtype,
                               void *sample_keys, uint32_t *group, uint32_t *err, cudaStream_t s);
cudaError_t launch_norm_xy(TrainJob *jobs, uint32_t models, uint64_t max_S, int key_bytes, int dtype, int translate,
                           const void *sorted_keys, Norm *norms, const uint32_t *err, cudaStream_t s);
// one Adam step of every job (per-step kernels), all steps of one-hidden-layer jobs in one launch
// (k_train_cluster.cu)
cudaError_t launch_train_step(const PadArch &a, const TrainJob *jobs, uint32_t models, uint32_t max_blocks,
                              const TrainHyper &hp, size_t P, int step, float c1, float c2, cudaStream_t s);
bool train_cluster_ok(const PadArch &a, uint64_t max_batch);
cudaError_t launch_train_cluster(const PadArch &a, const TrainJob *jobs, uint32_t models, const TrainHyper &hp,
                                 uint64_t max_batch, cudaStream_t s);
// many small models at once, one block per model (k_train_block.cu): one hidden layer of padded
// width 8, 16 or 32, samples of at most TB_MAX_S keys; the sort buffer holds `cap` keys (a power of
// two >= every S of the launch)
constexpr uint32_t TB_MAX_S = 16384;
struct TrainBlockArgs {
    const void *const *keys;   // [models] device key arrays
    const uint64_t *n, *S;     // [models] keys, sample size
    const uint32_t *ids;       // [blocks] model index of each block
    uint32_t cap;
    int dtype, translate, h1;  // h1: real hidden width (<= padded width)
    uint64_t seed0;            // model m uses seed seed0 + m
    int steps;
    uint64_t batch;            // 0: full batch
    int loss;
    float delta, lr, b1, b2, eps;
    const float *c1, *c2;      // [steps] Adam bias corrections 1 - beta^(t+1)
    float *params_out;         // [models][3 H + 1] padded layout
    Norm *norm_out;            // [models]
    float *loss_out;           // nullable [models][steps]
    uint32_t *err;
};
cudaError_t launch_train_block(const TrainBlockArgs &a, int key_bytes, int padded_h, uint32_t blocks,
                               cudaStream_t s);
// gradient of a sum over samples (k_train.cu, k_train_tc.cu). mode 0: s = sum_i gy_i * y_i (explicit
// upstream gradient); mode 1: mean loss over the batch with labels; mode 2: as mode 1 with batch
// indices drawn from the batch stream. Each block (or block group) writes one partial gradient row.
struct GradArgs {
    const float *params;
    const float *x, *gy, *label;
    uint64_t n;          // samples in the batch
    uint64_t S;          // labelled set size (mode 2)
    uint64_t bseed;      // batch stream (mode 2)
    uint64_t bofs;       // first draw of this step (mode 2)
    int mode, loss;
    float delta;
    float inv_n;
    float *partials;     // [rows * P]
    float *loss_partials;  // [rows], nullable
    float *gx;           // nullable (mode 0)
    const TrainJob *jobs;  // nullable: block row y computes the step of job y (mode 1 or 2)
    int step;              // with jobs: the step
};
int train_grad_blocks(const PadArch &a, uint64_t nsamples);
// two hidden layers of width 64 on the tensor cores (k_train_tc.cu): blocks of the launch (each
// writes one partial row), and the launch; a bounded wait that expired sets ERR_TIMEOUT in the
// library's training error word (train_err_word)
int grad_tc64_blocks(uint64_t nsamples);
cudaError_t launch_grad_tc64(const GradArgs &g, cudaStream_t s);
// every Adam step of a training run of that model in one cooperative launch: c12 = device
// [2 * steps] bias corrections (1 - beta1^(t+1), then 1 - beta2^(t+1)), count = a device word zeroed
// before the launch
cudaError_t launch_train_tc64(const TrainStepArgs &t, uint32_t steps, const float *c12, unsigned int *count,
                              cudaStream_t s);
uint32_t *train_err_word();
// forward / backward / loss-grad for explicit arrays (nnsort_mlp_* entry points)
cudaError_t launch_mlp_forward(const PadArch &a, const float *params, const float *x, uint64_t n,
                               float *y, cudaStream_t s);
cudaError_t launch_mlp_backward(const PadArch &a, const float *params, const float *x,
                                const float *gy, const float *label, uint64_t n, int mode,
                                int loss, float delta, float *partials, float *loss_partials,
                                float *gx, cudaStream_t s, int *blocks_out);
cudaError_t launch_reduce_partials(const float *partials, int blocks, size_t P, float *out,
                                   const float *loss_partials, float *loss_out, float scale,
                                   cudaStream_t s);

// Device memory from the library's own pool (api.cu), ordered on the stream like cudaMallocAsync. The
// device's default pool gives its memory back at every synchronisation, so that each call after one
// maps its buffers again; this one keeps up to POOL_KEEP bytes until nnsort_release.
constexpr size_t POOL_KEEP = (size_t)256 << 20;
cudaError_t pool_alloc(void **p, size_t bytes, cudaStream_t s);

}  // namespace nns

// Trains `count` models of one architecture side by side (the recipe of nnsort_train; api.cu): model j
// on d_keys[j] with sample size S[j] and seed seeds[j]. rc[j] receives each model's status and out[j]
// its model (null unless NNSORT_OK); h_loss (nullable): count x steps. Synchronous. Returns an error
// that concerns the whole call.
int nnsort_train_models(const void *const *d_keys, const uint64_t *ns, uint32_t count, int32_t dtype,
                        const nnsort_train_opts &o, const uint64_t *S, const uint64_t *seeds,
                        struct nnsort_model **out, int *rc, float *h_loss, cudaStream_t s);

// Device bytes of one of its models beside the sample: parameters, moments, partial gradients, losses.
size_t nnsort_train_model_bytes(const nnsort_train_opts &o);

// The model handle behind the opaque nnsort_model of the C ABI: one definition for every
// translation unit that reads it.
struct nnsort_model {
    nnsort_model_desc desc;
    std::vector<float> params;  // caller layout
    std::vector<float> hpad;    // padded layout in host memory (the tensor-core predict passes its
                                // vectors as launch constants)
    nns::PadArch pad;
    size_t P = 0, Ppad = 0;
    float *d_params = nullptr;  // padded layout
    int device = 0;
    std::shared_ptr<void> owner;  // set when d_params lies in a device block shared by several
                                  // models (freed with the last of them), else d_params is its own
};
