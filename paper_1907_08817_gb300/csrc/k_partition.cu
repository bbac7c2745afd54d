// k_partition.cu -- stable digit partition of the element space (one pass per digit, LSD order),
// used two ways:
//   * by the bucket index of each element's predicted position, so that every on-chip bucket of
//     positions ends up contiguous and in input order (which keeps the paper's first-arrival rule
//     and the conflict arrays' arrival order intact inside a bucket), and
//   * by the key's order image, as the radix sort behind the training sample (Sec. "Training"),
//     the multi-block sorts of oversized buckets and long repairs, and the "no model" reference.
//
// One pass reads and writes each element once, in tiles of 4,096. Its offsets come from a scan
// over per-tile digit histograms (reduce, then scan, then scatter), so no block ever waits on
// another and several blocks share each SM. A tile ranks its elements per digit stably (a warp finds
// the lanes holding the same digit through shared-memory match words); writes go out through a
// shared-memory reorder buffer in digit order, so each digit's run leaves as coalesced stores.
#include <algorithm>
#include <cstddef>
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace nns {
static inline cudaError_t nns_launched(cudaError_t e, int k = 1) {
    if (e == cudaSuccess) note_launch(k);
    return e;
}
}  // namespace nns

namespace nns {

// ---------------------------------------------------------------------------------------------
// The partition pass without look-back. The tiles' global offsets come from a scan over tile
// histograms instead of from waits on earlier tiles, so every block is independent: several run
// on each SM and one block's loads overlap the others' ranking and stores.
namespace {
constexpr int TH_THREADS = 256, TH_ITEMS = SC_TILE / TH_THREADS, TH_NW = TH_THREADS / 32;  // histogram blocks
constexpr int SC_THREADS = 256, SC_ITEMS = SC_TILE / SC_THREADS, SC_NW = SC_THREADS / 32;  // scatter blocks

template <typename W, bool KEYDIG>
__device__ __forceinline__ uint32_t sc_digit(const PartitionArgs &a, W key, uint32_t gs, uint32_t mask) {
    if constexpr (KEYDIG) return (uint32_t)(ordbits(word64(key), a.dtype) >> a.shift) & mask;
    else return (gs >> a.shift) & mask;
}
}  // namespace

// per tile: the digit histogram (per-warp counters, so that equal digits contend within a warp only;
// sixteen elements per thread keep the counters to clear and to add up few against the elements)
template <typename W, bool KEYDIG>
__global__ void __launch_bounds__(TH_THREADS) k_tile_hist(PartitionArgs a) {
    __shared__ uint32_t h[TH_NW][RADIX_BINS];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t bins = max(32u, 1u << a.bits), mask = (1u << a.bits) - 1u;
    const uint64_t base = (uint64_t)blockIdx.x * SC_TILE;
    const uint32_t cnt = (uint32_t)min((uint64_t)SC_TILE, a.N - base);
    const W *kin = reinterpret_cast<const W *>(a.key_in) + base;
    const uint32_t *gin = KEYDIG ? nullptr : a.gs_in + base;
    const uint32_t loc0 = (uint32_t)w * (32 * TH_ITEMS) + lane;
    uint32_t d[TH_ITEMS];
#pragma unroll
    for (int r = 0; r < TH_ITEMS; ++r) {
        const uint32_t loc = loc0 + r * 32;
        d[r] = 0xFFFFFFFFu;
        if (loc < cnt) {
            if constexpr (KEYDIG) d[r] = sc_digit<W, true>(a, kin[loc], 0u, mask);
            else d[r] = sc_digit<W, false>(a, W(0), gin[loc], mask);
        }
    }
    for (uint32_t i = lane; i < bins; i += 32) h[w][i] = 0;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < TH_ITEMS; ++r)
        if (d[r] != 0xFFFFFFFFu) atomicAdd(&h[w][d[r]], 1u);
    __syncthreads();
    for (uint32_t i = tid; i < bins; i += TH_THREADS) {
        uint32_t t = 0;
#pragma unroll
        for (int ww = 0; ww < TH_NW; ++ww) t += h[ww][i];
        a.tile_hist[(size_t)blockIdx.x * RADIX_BINS + i] = (uint16_t)t;
    }
    if (blockIdx.x == 0)  // summed by k_chunk_prefix, which runs after; k_chunk_base scans all of them
        for (int i = tid; i < RADIX_BINS; i += TH_THREADS) a.bin_total[i] = 0;
}

// per chunk of SC_CHUNK tiles: each tile's histogram becomes its exclusive prefix inside the chunk,
// the chunk's totals go to chunk[c] and are added to the digit totals
__global__ void __launch_bounds__(RADIX_BINS) k_chunk_prefix(PartitionArgs a, uint32_t tiles) {
    const uint32_t c = blockIdx.x, d = threadIdx.x;  // a thread per digit
    const uint32_t t0 = c * SC_CHUNK;
    uint16_t v[SC_CHUNK];
#pragma unroll
    for (int j = 0; j < SC_CHUNK; ++j)
        v[j] = (t0 + j < tiles) ? a.tile_hist[(size_t)(t0 + j) * RADIX_BINS + d] : (uint16_t)0;
    uint32_t run = 0;
#pragma unroll
    for (int j = 0; j < SC_CHUNK; ++j) {
        if (t0 + j < tiles) a.tile_hist[(size_t)(t0 + j) * RADIX_BINS + d] = (uint16_t)run;
        run += v[j];
    }
    a.chunk[(size_t)c * RADIX_BINS + d] = run;
    if (run) atomicAdd(&a.bin_total[d], run);
}

// one chunk (at most SC_CHUNK tiles): the tiles' prefixes and the digit bases in one block, a digit per
// thread
__global__ void __launch_bounds__(RADIX_BINS) k_chunk_one(PartitionArgs a, uint32_t tiles) {
    __shared__ uint32_t scratch[33];
    const uint32_t d = threadIdx.x;
    uint16_t v[SC_CHUNK];
#pragma unroll
    for (int j = 0; j < SC_CHUNK; ++j) v[j] = (uint32_t)j < tiles ? a.tile_hist[(size_t)j * RADIX_BINS + d] : (uint16_t)0;
    uint32_t run = 0;
#pragma unroll
    for (int j = 0; j < SC_CHUNK; ++j) {
        if ((uint32_t)j < tiles) a.tile_hist[(size_t)j * RADIX_BINS + d] = (uint16_t)run;
        run += v[j];
    }
    a.chunk[d] = block_excl_sum(run, scratch, nullptr);
}

// chunk totals -> chunk bases, the digit's base (elements of all smaller digits) plus the sum over
// earlier chunks, in place. Block b takes digits [32 b, 32 b + 32); its 32 warps take consecutive
// groups of chunks (lane = digit, so every load and store of a warp is one 128-byte line)
__global__ void __launch_bounds__(1024) k_chunk_base(PartitionArgs a, uint32_t chunks) {
    __shared__ uint32_t part[32][33];
    __shared__ uint32_t dbase[RADIX_BINS];
    __shared__ uint32_t scratch[33];
    {   // digit bases: exclusive scan of the digit totals (every block scans all of them)
        const uint32_t v = threadIdx.x < RADIX_BINS ? a.bin_total[threadIdx.x] : 0u;
        const uint32_t ex = block_excl_sum(v, scratch, nullptr);
        if (threadIdx.x < RADIX_BINS) dbase[threadIdx.x] = ex;
        __syncthreads();
    }
    const int i = threadIdx.x & 31, j = threadIdx.x >> 5;
    const uint32_t d = blockIdx.x * 32 + i;
    const uint32_t G = (chunks + 31) / 32;
    const uint32_t c0 = min(chunks, (uint32_t)j * G), c1 = min(chunks, c0 + G);
    uint32_t sum = 0;
    for (uint32_t c = c0; c < c1; ++c) sum += a.chunk[(size_t)c * RADIX_BINS + d];
    part[j][i] = sum;
    __syncthreads();
    if (j == 0) {
        uint32_t run = dbase[d];
        for (int q = 0; q < 32; ++q) {
            const uint32_t x = part[q][i];
            part[q][i] = run;
            run += x;
        }
    }
    __syncthreads();
    uint32_t run = part[j][i];
    for (uint32_t c = c0; c < c1; ++c) {
        const uint32_t x = a.chunk[(size_t)c * RADIX_BINS + d];
        a.chunk[(size_t)c * RADIX_BINS + d] = run;
        run += x;
    }
}

namespace {
// Shared memory of a scatter block: per-warp digit counters, then the reorder buffer that holds every
// carried array; while the tile is ranked, the same bytes hold the warps' two sets of match words.
constexpr size_t SC_MATCH = (size_t)2 * SC_NW * RADIX_BINS * 4;
template <typename W, bool KEYDIG, bool PAY, bool ROW> constexpr size_t sc_buf_bytes() {
    const size_t carried = (size_t)SC_TILE * (sizeof(W) + (KEYDIG ? 0 : 4) + (PAY ? 4 : 0) + (ROW ? 4 : 0));
    return carried > SC_MATCH ? carried : SC_MATCH;
}
}  // namespace

// Per tile: stable rank of every element by digit, then the scatter to its global position through a
// shared-memory reorder buffer that holds every carried array, so each digit's run leaves as coalesced
// stores.
//
// Ranking: each of the warp's 32 elements sets its lane's bit in its digit's match word (one
// shared-memory atomic), reads the word back and counts the bits below its own. One ballot per digit
// bit found the same peers in about three instructions a bit: 123 instructions per element in all,
// against 58 now. The match words alternate between two sets, so that clearing a word and the next
// element's atomics need no barrier between them. Sixteen elements per thread: half the warps, so half
// the counters to clear and to scan per tile. Bound by shared-memory wavefronts (77% of the peak; a warp's
// 32 random digits or places meet in about 3.5 of them) and, for 9-bit digits, by the 32-byte runs a
// tile leaves per digit. A pass over 67M u64 keys with payload: 0.53 ms (0.73 ms with ballots), 50M u64
// keys 0.31 (0.48), 2^28 f32 keys 1.26 and 1.73 ms by 8 and 9 bits (1.60 and 1.82). Measured and slower:
// 16-lane words that hold mask and count together (1.46 and 1.87 ms).
template <typename W, bool KEYDIG, bool PAY, bool ROW, int BITS, bool FULL>
__device__ __forceinline__ void sc_tile(const PartitionArgs &a, uint16_t (*cnt)[RADIX_BINS], unsigned char *buf,
                                        uint32_t *gofs, uint32_t *scratch, uint32_t tile, uint32_t cnt_tile) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int bits = BITS > 0 ? BITS : a.bits;
    const uint32_t bins = 1u << bits, mask = bins - 1u;
    const uint64_t base = (uint64_t)tile * SC_TILE;
    uint32_t gsv[SC_ITEMS], pay[SC_ITEMS], row[SC_ITEMS];
    W key[SC_ITEMS];
    uint32_t rk[SC_ITEMS];  // digit * 2^16 + rank among the warp's earlier elements of that digit
    const W *kin = reinterpret_cast<const W *>(a.key_in) + base;
    const uint32_t *gin = KEYDIG ? nullptr : a.gs_in + base;
    const uint32_t *pin = PAY ? a.pay_in + base : nullptr, *rin = ROW ? a.row_in + base : nullptr;
    const uint32_t loc0 = (uint32_t)w * (32 * SC_ITEMS) + lane;
#pragma unroll
    for (int r = 0; r < SC_ITEMS; ++r) {
        const uint32_t loc = loc0 + r * 32;
        if (FULL || loc < cnt_tile) {
            key[r] = kin[loc];
            if constexpr (!KEYDIG) gsv[r] = gin[loc];
            if constexpr (PAY) pay[r] = pin[loc];
            if constexpr (ROW) row[r] = rin[loc];
        }
    }
    auto digit = [&](int r) -> uint32_t { return sc_digit<W, KEYDIG>(a, key[r], KEYDIG ? 0u : gsv[r], mask); };
    uint32_t *match = reinterpret_cast<uint32_t *>(buf) + (size_t)w * 2 * RADIX_BINS;
    for (uint32_t i = lane; i < bins; i += 32) {
        cnt[w][i] = 0;
        match[i] = 0;
        match[RADIX_BINS + i] = 0;
    }
    __syncwarp();
    const unsigned mine = 1u << lane, below = mine - 1u;
#pragma unroll
    for (int r = 0; r < SC_ITEMS; ++r) {
        const bool valid = FULL || loc0 + r * 32 < cnt_tile;
        const uint32_t d = valid ? digit(r) : 0u;
        uint32_t *m = match + (r & 1) * RADIX_BINS + d;
        if (valid) atomicOr(m, mine);
        __syncwarp();
        const unsigned peers = valid ? *m : 0u;
        const uint32_t c = cnt[w][d];
        __syncwarp();
        const uint32_t before = __popc(peers & below);
        rk[r] = (d << 16) | (c + before);
        if (valid && before == 0) {
            cnt[w][d] = (uint16_t)(c + __popc(peers));
            *m = 0;
        }
    }
    __syncthreads();
    // digit starts inside the tile: thread t takes digits BPT t .. BPT t + BPT - 1
    constexpr int BPT = RADIX_BINS / SC_THREADS;
    uint32_t tot[BPT], sum = 0;
#pragma unroll
    for (int q = 0; q < BPT; ++q) {
        const uint32_t d = tid * BPT + q;
        tot[q] = 0;
        if (d < bins) {
#pragma unroll
            for (int ww = 0; ww < SC_NW; ++ww) tot[q] += cnt[ww][d];
        }
        sum += tot[q];
    }
    uint32_t ls = block_excl_sum(sum, scratch, nullptr);
#pragma unroll
    for (int q = 0; q < BPT; ++q) {
        const uint32_t d = tid * BPT + q;
        if (d < bins) {
            // this tile's global digit offset: chunk base + in-chunk prefix
            gofs[d] = a.chunk[(size_t)(tile / SC_CHUNK) * RADIX_BINS + d] +
                      (uint32_t)a.tile_hist[(size_t)tile * RADIX_BINS + d] - ls;
            uint32_t run = ls;
#pragma unroll
            for (int ww = 0; ww < SC_NW; ++ww) {
                const uint32_t c = cnt[ww][d];
                cnt[ww][d] = (uint16_t)run;
                run += c;
            }
        }
        ls += tot[q];
    }
    __syncthreads();
    W *bk = reinterpret_cast<W *>(buf);
    uint32_t *bg = reinterpret_cast<uint32_t *>(bk + SC_TILE);
    uint32_t *bp = bg + (KEYDIG ? 0 : SC_TILE);
    uint32_t *br = bp + (PAY ? SC_TILE : 0);
#pragma unroll
    for (int r = 0; r < SC_ITEMS; ++r) {
        if (FULL || loc0 + r * 32 < cnt_tile) {
            const uint32_t lp = cnt[w][rk[r] >> 16] + (rk[r] & 0xFFFFu);
            bk[lp] = key[r];
            if constexpr (!KEYDIG) bg[lp] = gsv[r];
            if constexpr (PAY) bp[lp] = pay[r];
            if constexpr (ROW) br[lp] = row[r];
        }
    }
    __syncthreads();
    W *ko = reinterpret_cast<W *>(a.key_out);
#pragma unroll 8
    for (uint32_t k = 0; k < SC_ITEMS; ++k) {
        const uint32_t i = tid + k * SC_THREADS;
        if (FULL || i < cnt_tile) {
            const W kv = bk[i];
            const uint32_t gv = KEYDIG ? 0u : bg[i];
            const uint32_t o = gofs[sc_digit<W, KEYDIG>(a, kv, gv, mask)] + i;
            ko[o] = kv;
            if constexpr (!KEYDIG) a.gs_out[o] = gv;
            if constexpr (PAY) a.pay_out[o] = bp[i];
            if constexpr (ROW) a.row_out[o] = br[i];
        }
    }
}

template <typename W, bool KEYDIG, bool PAY, bool ROW, int BITS, int MINB>
__global__ void __launch_bounds__(SC_THREADS, MINB) k_scatter(PartitionArgs a) {
    extern __shared__ __align__(16) unsigned char buf[];
    __shared__ uint16_t cnt[SC_NW][RADIX_BINS];
    __shared__ uint32_t gofs[RADIX_BINS];
    __shared__ uint32_t scratch[33];
    const uint32_t tile = blockIdx.x;
    const uint32_t cnt_tile = (uint32_t)min((uint64_t)SC_TILE, a.N - (uint64_t)tile * SC_TILE);
    if (cnt_tile == SC_TILE)
        sc_tile<W, KEYDIG, PAY, ROW, BITS, true>(a, cnt, buf, gofs, scratch, tile, cnt_tile);
    else
        sc_tile<W, KEYDIG, PAY, ROW, BITS, false>(a, cnt, buf, gofs, scratch, tile, cnt_tile);
}

template <typename W, bool KD, bool P, bool R, int MB>
static cudaError_t sc_launch(const PartitionArgs &a, uint64_t tiles, cudaStream_t s) {
    constexpr size_t smem = sc_buf_bytes<W, KD, P, R>();
    auto go = [&](auto kfn) -> cudaError_t {
        cudaError_t e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kfn<<<(unsigned)tiles, SC_THREADS, smem, s>>>(a);
        return nns_launched(cudaGetLastError());
    };
    // the digit widths the passes use most as compile-time constants; others at run time
    if (a.bits == 9) return go(k_scatter<W, KD, P, R, 9, MB>);
    if (a.bits == 8) return go(k_scatter<W, KD, P, R, 8, MB>);
    return go(k_scatter<W, KD, P, R, 0, MB>);
}

template <typename W, bool KD>
static cudaError_t sc_go(const PartitionArgs &a, cudaStream_t s) {
    const uint64_t tiles = partition_tiles(a.N), chunks = partition_chunks(a.N);
    k_tile_hist<W, KD><<<(unsigned)tiles, TH_THREADS, 0, s>>>(a);
    cudaError_t e = nns_launched(cudaGetLastError());
    if (e != cudaSuccess) return e;
    const unsigned bins = (unsigned)std::max(32, 1 << a.bits);
    if (chunks == 1) {
        k_chunk_one<<<1, bins, 0, s>>>(a, (uint32_t)tiles);
        if ((e = nns_launched(cudaGetLastError())) != cudaSuccess) return e;
    } else {
        k_chunk_prefix<<<(unsigned)chunks, bins, 0, s>>>(a, (uint32_t)tiles);
        if ((e = nns_launched(cudaGetLastError())) != cudaSuccess) return e;
        k_chunk_base<<<bins / 32, 1024, 0, s>>>(a, (uint32_t)chunks);
        if ((e = nns_launched(cudaGetLastError())) != cudaSuccess) return e;
    }
    const bool pay = a.pay_in != nullptr, row = a.row_in != nullptr;
    // resident blocks per SM: with four-byte keys three (four without positions to carry) pay although
    // a few of the sixteen elements' registers spill (2^28 keys, 8-bit pass: 1.44, 1.26 and 1.29 ms at
    // two, three and four blocks; 33.6M key-value pairs by key digits: 0.187, 0.178 and 0.170 ms a pass)
    constexpr int MB = sizeof(W) == 8 ? 2 : (KD ? 4 : 3);
    if (pay && row) return sc_launch<W, KD, true, true, 2>(a, tiles, s);
    if (pay) return sc_launch<W, KD, true, false, MB>(a, tiles, s);
    if (row) return sc_launch<W, KD, false, true, MB>(a, tiles, s);
    return sc_launch<W, KD, false, false, MB>(a, tiles, s);
}

cudaError_t launch_partition(const PartitionArgs &a, cudaStream_t s) {
    if (a.N == 0) return cudaSuccess;
    if (a.key_bytes == 4)
        return a.key_digits ? sc_go<uint32_t, true>(a, s) : sc_go<uint32_t, false>(a, s);
    return a.key_digits ? sc_go<uint64_t, true>(a, s) : sc_go<uint64_t, false>(a, s);
}

// bstart[b] = first element whose global position is >= b * W (binary search; gs is sorted by
// bucket after the partition)
__global__ void k_bucket_bounds(const uint32_t *gs, uint64_t N, uint32_t nb, int wlog, uint32_t *bstart) {
    const uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b > nb) return;
    uint64_t lo = 0, hi = N;
    while (lo < hi) {
        const uint64_t mid = (lo + hi) >> 1;
        if (((uint64_t)gs[mid] >> wlog) < b) lo = mid + 1; else hi = mid;
    }
    bstart[b] = (uint32_t)lo;
}

cudaError_t launch_bucket_bounds(const uint32_t *gs, uint64_t N, uint32_t nb, int wlog,
                                 uint32_t *bstart, cudaStream_t s) {
    const uint32_t th = 256, grid = (nb + 1 + th - 1) / th;
    k_bucket_bounds<<<grid, th, 0, s>>>(gs, N, nb, wlog, bstart);
    return nns_launched(cudaGetLastError());
}

}  // namespace nns
