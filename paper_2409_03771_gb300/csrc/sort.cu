// Onesweep LSD radix sorts: the vertex order of many packed instances at
// once (Simulation of Simplicity, section "Preprocessing": sort by value,
// ties by global id, per instance), 64-bit keys with or without an int32
// payload (region adjacency), and the ranks of the distinct Morse-Smale pairs.
//
// Keys of a float field: float32 bits mapped to an order-preserving uint32
// (-0.0 first folded onto +0.0 so that the two tie, as IEEE '<' says).
// 8-bit digit passes, least significant first; every pass is stable, and
// the first pass reads the vertices in id order, so equal keys stay in id
// order: the final position of v is its rank under (f[v], v).
//
// One pass = one kernel (the pair ranks make all of theirs in one).  A block
// takes tiles of 4096 keys (64-bit ones: 6144) from a global
// atomic counter (so every predecessor tile is owned by a running block),
// ranks its keys per digit stably within each warp (the lanes of a digit meet
// in a word of shared memory), publishes its per-digit counts to a decoupled
// look-back array, sums its predecessors' counts and scatters through
// shared memory.  The last pass of an order files (vertex id, position)
// pairs into buckets of consecutive ids; the order field is their inverse
// permutation (k_pair_permute).
#include <cuda_runtime.h>

#include <algorithm>
#include <utility>

#include "coop.cuh"
#include "radix.cuh"
#include "sort.cuh"
#include "tma.cuh"

namespace msc {
#ifdef MSC_DEBUG_BOUNDS
__device__ uint32_t g_sort_dbg[16];
#endif
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / kWarp;      // 8
constexpr int kBins = 256;
constexpr unsigned long long kFlagAgg = 1ull << 62;
constexpr unsigned long long kFlagInc = 2ull << 62;
constexpr uint32_t kSpinLimit = 1u << 22;
// The last pass of the vertex order files (id, position) pairs into
// buckets of 2^shift consecutive ids; bucket b holds exactly the ids
// [b << shift, (b + 1) << shift) and so occupies pair slots of the same
// range.  At most kMaxBuckets buckets (see bucket_shift).
constexpr int kMaxBuckets = kOrderMaxBuckets;
constexpr int kFillStride = kOrderFillStride;  // one 128-byte line per bucket counter: the
                                 // tiles' reservations spread over L2 slices
constexpr int kCounterWords = 8 + kMaxBuckets * kFillStride;  // tile counters, bucket fills

// Digit histograms for `npass` passes over the 64-bit keys (16-byte aligned)
// into warp-private shared histograms; blocks then add theirs to the global
// ones.  Lane-consecutive 16-byte loads; a digit that the whole warp shares
// (the high digits of keys from neighbouring grid tiles) is one update.
// Bound: the shared-memory atomics.  52M keys of six digits: 0.36 ms with
// sixteen consecutive keys per thread (128-byte lane stride), 0.16 now.
constexpr int kHistPairs = 8;  // 16-byte loads in flight per thread

// sh: [kWarps][npass][256].  (Loads past the L1: in the pair ranks' kernel the
// keys were written by other blocks.)
__device__ __forceinline__ void add_digit_counts(const unsigned long long* keys, int64_t n, int npass, uint32_t* hist,
                                                 uint32_t* sh) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < kWarps * npass * kBins; i += blockDim.x) sh[i] = 0;
    __syncthreads();
    uint32_t* wsh = sh + warp * npass * kBins;
    constexpr int64_t kStep = 2 * 256 * kHistPairs;
    for (int64_t b = (int64_t)blockIdx.x * kStep; b < n; b += (int64_t)gridDim.x * kStep) {
        if (b + kStep <= n) {
            ulonglong2 k[kHistPairs];
#pragma unroll
            for (int q = 0; q < kHistPairs; ++q)
                k[q] = __ldcg(reinterpret_cast<const ulonglong2*>(keys + b) + q * 256 + tid);
            for (int p = 0; p < npass; ++p) {
                uint32_t* h = wsh + p * kBins;
#pragma unroll
                for (int q = 0; q < 2 * kHistPairs; ++q) {
                    const uint32_t d = (uint32_t)((q & 1 ? k[q / 2].y : k[q / 2].x) >> (8 * p)) & 255u;
                    if (__all_sync(0xffffffffu, d == __shfl_sync(0xffffffffu, d, 0))) {
                        if (lane == 0) atomicAdd(&h[d], 32u);
                    } else {
                        atomicAdd(&h[d], 1u);
                    }
                }
            }
        } else {
            for (int64_t i = b + tid; i < n; i += 256)
                for (int p = 0; p < npass; ++p) atomicAdd(&wsh[p * kBins + ((uint32_t)(keys[i] >> (8 * p)) & 255u)], 1u);
        }
    }
    __syncthreads();
    for (int i = tid; i < npass * kBins; i += blockDim.x) {
        uint32_t c = 0;
        for (int w = 0; w < kWarps; ++w) c += sh[w * npass * kBins + i];
        if (c) atomicAdd(&hist[i], c);
    }
}

__global__ void __launch_bounds__(256) k_hist(const unsigned long long* __restrict__ keys, int64_t n_host,
                                              const int32_t* __restrict__ d_n, int npass, uint32_t* __restrict__ hist) {
    extern __shared__ uint32_t sh[];
    add_digit_counts(keys, d_n ? min((int64_t)*d_n, n_host) : n_host, npass, hist, sh);
}

// Per-segment histograms of the float keys for the 4 passes of a
// segmented sort: hist[seg][pass][256].  Block b takes a contiguous run of
// tiles (one tile = 256 threads x 16 keys, inside one segment) and adds
// its warp-private shared counts to the segment's global histogram each
// time the segment changes and at the end.
constexpr int kSegPasses = 4;

__global__ void __launch_bounds__(256) k_hist_seg(const float* __restrict__ f,
                                                  const int32_t* __restrict__ tile_seg,
                                                  const int32_t* __restrict__ seg_off,
                                                  const int32_t* __restrict__ seg_tile0, int64_t tiles,
                                                  uint32_t* __restrict__ hist, int32_t* status) {
    extern __shared__ uint32_t sh[];  // [kWarps][4][256]
    constexpr int kSeg = kSegPasses * kBins;
    const int tid = threadIdx.x, warp = tid >> 5;
    for (int i = tid; i < kWarps * kSeg; i += blockDim.x) sh[i] = 0;
    __syncthreads();
    uint32_t* wsh = sh + warp * kSeg;
    const int64_t t0 = tiles * blockIdx.x / gridDim.x, t1 = tiles * (blockIdx.x + 1) / gridDim.x;
    bool saw_nan = false;
    auto flush = [&](int seg) {
        __syncthreads();
        for (int i = tid; i < kSeg; i += blockDim.x) {
            uint32_t c = 0;
            for (int w = 0; w < kWarps; ++w) {
                c += sh[w * kSeg + i];
                sh[w * kSeg + i] = 0;
            }
            if (c) atomicAdd(&hist[(int64_t)seg * kSeg + i], c);
        }
        __syncthreads();
    };
    int cur = t0 < t1 ? tile_seg[t0] : 0;
    for (int64_t t = t0; t < t1; ++t) {
        const int seg = tile_seg[t];  // uniform over the block
        if (seg != cur) {
            flush(cur);
            cur = seg;
        }
        const int64_t off = seg_off[seg], n = seg_off[seg + 1] - off;
        const int64_t i0 = (t - seg_tile0[seg]) * kSortTile + (int64_t)tid * kHistRun;
        if (i0 < n) {
            uint32_t k[kHistRun];
            const int cnt = (int)min((int64_t)kHistRun, n - i0);
            load_float_keys16(f + off, i0, cnt, k, saw_nan);
            count_runs(k, cnt, kSegPasses, wsh);
        }
    }
    if (t0 < t1) flush(cur);
    if (saw_nan) record_error(status, MSC_ERR_NAN);
}

// hist[seg][pass][.] -> exclusive bin starts, one block per (seg, pass).
__global__ void __launch_bounds__(256) k_seg_bstart(uint32_t* hist) {
    __shared__ uint32_t s_w[kWarps];
    uint32_t* h = hist + (int64_t)blockIdx.x * kBins;
    const uint32_t c = h[threadIdx.x];
    h[threadIdx.x] = block_scan_256(c, s_w) - c;
}

template <typename KeyT>
struct PassArgs {
    const KeyT* keys_in;
    const float* f_in;
    const int32_t* vals_in;
    KeyT* keys_out;
    int32_t* vals_out;
    int64_t n;
    const int32_t* d_n;
    const uint32_t* hist;  // this pass's 256 counts
    uint32_t* pair_pos;    // BUCKET pass: position of the id in vals_out[slot]
    uint32_t* bucket_fill; // BUCKET pass: slots taken per bucket (stride kFillStride)
    int bucket_shift;      // BUCKET pass: log2 of the ids per bucket
    int shift;
    unsigned long long* lookback;
    uint32_t* tile_counter;
    uint32_t epoch;
    int32_t* status;
    // segmented sort (packed instances): segment of each tile, key offset
    // of each segment, first tile of each segment; `hist` then holds the
    // per-segment exclusive bin starts with a stride of seg_stride words
    const int32_t* tile_seg;
    const int32_t* seg_off;
    const int32_t* seg_tile0;
    int64_t seg_tiles;
    int seg_stride;
    uint32_t* rank_of;  // RANK pass: rank_of[payload] = position; keys_out may be null
};

// Keys per thread: 64-bit sorts take 24 at two blocks per SM (six passes over
// 52M keys and six over 14M with a payload: 2.69 ms, 2.84 with 16 at three);
// segmented ones take the sort tile that their histograms are made by.
template <typename KeyT>
constexpr int kPassItems = sizeof(KeyT) == 8 ? 24 : kSortTile / kThreads;

template <typename KeyT, bool VALS>
constexpr size_t pass_smem_bytes() {
    return (size_t)(2 * kWarps * kBins + 4 * kBins + 32 + 2 * kMaxBuckets) * 4 +
           (size_t)kThreads * kPassItems<KeyT> * (sizeof(KeyT) + (VALS ? 4 : 0));
}

// One onesweep digit pass (64-bit keys alone, 52M of them: 0.40 -> 0.34 ms with
// ranks by shared words instead of ballots and no registers for an absent
// payload).  FROM_F: keys come from the float field and
// the payload is the vertex id.  BUCKET (last pass of the vertex order):
// instead of the sorted (key, payload) arrays, file every (payload,
// position) pair into the bucket of its payload's top bits (a tile
// reserves its share of each bucket with one atomic per bucket).
//
// SEG: the keys are packed segments sorted independently (batched
// instances).  Tiles never straddle two segments, the look-back stops at
// the segment's first tile, bin starts come per segment, and positions are
// segment-local (keys land at seg_off + position; order gets the position).
//
// VALS: with a payload; without, keys alone are moved.  RANK: the payload's
// position goes to rank_of instead.
template <typename KeyT, bool FROM_F, bool BUCKET, bool SEG, bool VALS, bool RANK>
__device__ __forceinline__ void onesweep_tiles(const PassArgs<KeyT>& a, uint8_t* smem) {
    constexpr int kItems = kPassItems<KeyT>, kTile = kThreads * kItems;
    static_assert(kTile >= kSortTile, "the look-back words are sized for tiles of kSortTile keys");
    static_assert(!SEG || kTile == kSortTile, "a segment's tiles and histograms are those of its table");
    uint32_t* s_whist = reinterpret_cast<uint32_t*>(smem);  // [kWarps][256]
    uint32_t* s_match = s_whist + kWarps * kBins;          // [kWarps][256] lanes per digit, 0 between keys
    uint32_t* s_total = s_match + kWarps * kBins;          // [256]
    uint32_t* s_excl = s_total + kBins;                    // [256] tile-local bin starts
    uint32_t* s_gbase = s_excl + kBins;                    // [256] global base of the bin
    uint32_t* s_bstart = s_gbase + kBins;                  // [256] global bin starts
    uint32_t* s_misc = s_bstart + kBins;                   // [0] tile id, [1..8] scan
    uint32_t* s_bucket = s_misc + 32;                      // [2][kMaxBuckets] counts, bases
    KeyT* s_keys = reinterpret_cast<KeyT*>(s_bucket + 2 * kMaxBuckets);
    int32_t* s_vals = reinterpret_cast<int32_t*>(s_keys + kTile);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t n_all = a.d_n ? min((int64_t)*a.d_n, a.n) : a.n;  // a device count never exceeds the buffers
    const int64_t ntiles = SEG ? a.seg_tiles : (n_all + kTile - 1) / kTile;
    if constexpr (!SEG) {
        const uint32_t c = a.hist[tid];
        s_bstart[tid] = block_scan_256(c, s_misc + 1) - c;
    }
    for (int i = tid; i < kWarps * kBins; i += kThreads) s_match[i] = 0;
    for (;;) {
        if (tid == 0) {  // no tiles left once a pass before this one gave up: its payloads are indices
            const bool unfinished = stage_gave_up(a.status);
            const uint32_t next = atomicAdd(a.tile_counter, 1u);
            s_misc[0] = unfinished ? ~0u : next;
        }
        for (int i = tid; i < kWarps * kBins; i += kThreads) s_whist[i] = 0;
        __syncthreads();
        const int64_t tile = s_misc[0];
        if (tile >= ntiles) break;
        // this tile's segment: key offset, key count, tile index within it
        int64_t seg_base = 0, n = n_all, ltile = tile;
        if constexpr (SEG) {
            const int seg = a.tile_seg[tile];
            seg_base = a.seg_off[seg];
            n = a.seg_off[seg + 1] - seg_base;
            ltile = tile - a.seg_tile0[seg];
            s_bstart[tid] = a.hist[(int64_t)seg * a.seg_stride + tid];  // read by this thread only
        }
        // tile-local 32-bit indices from here on: the tile's keys are
        // [tbase, tbase + cnt) of the packed arrays
        const int64_t tbase = seg_base + ltile * kTile;
        const int cnt = (int)min((int64_t)kTile, n - ltile * kTile);
        const int wbase = warp * (kItems * 32) + lane;

        KeyT key[kItems];
        int32_t val[kItems];
        uint32_t rk[kItems];  // (digit << 16) | rank among the warp's equal digits
        {
            const KeyT* kin = FROM_F ? nullptr : a.keys_in + tbase;
            const int32_t* vin = FROM_F || !VALS ? nullptr : a.vals_in + tbase;
            const float* fin = FROM_F ? a.f_in + tbase : nullptr;
#pragma unroll
            for (int k = 0; k < kItems; ++k) {
                const int li = wbase + k * 32;
                if (li < cnt) {
                    if constexpr (FROM_F) {
                        key[k] = (KeyT)float_key(fin[li]);
                        val[k] = (int32_t)tbase + li;
                    } else {
                        key[k] = kin[li];
                        val[k] = VALS ? vin[li] : 0;
                    }
                } else {
                    key[k] = 0;
                    val[k] = -1;
                }
            }
        }
        uint32_t* wh = s_whist + warp * kBins;
        const uint32_t lt = lanemask_lt();
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            // stable rank among the warp's equal digits: earlier iterations
            // (warp counter) + lower lanes of this iteration
            const bool valid = wbase + k * 32 < cnt;
            const uint32_t d = (uint32_t)(key[k] >> a.shift) & 255u;
            rk[k] = ((valid ? d : 256u) << 16) | rank_in_warp(d, valid, 1u << lane, lt, s_match + warp * kBins, wh);
        }
        __syncthreads();
#ifdef MSC_DEBUG_BOUNDS
        {   // each warp's histogram must hold exactly its valid items
            uint32_t sum = 0;
            for (int i = lane; i < kBins; i += 32) sum += wh[i];
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            const int64_t wv = min(kItems * 32, max(0, cnt - warp * kItems * 32));
            if (lane == 0 && sum != (uint32_t)wv && atomicCAS(&g_sort_dbg[14], 0u, 1u) == 0u) {
                g_sort_dbg[15] = (uint32_t)((tile & 0xffffu) << 16 | (warp << 12) | (sum & 0xfffu));
            }
        }
        __syncthreads();
#endif
        // per-digit tile totals; warp counts become warp-exclusive prefixes
        uint32_t run = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t c = s_whist[w * kBins + tid];
            s_whist[w * kBins + tid] = run;
            run += c;
        }
        s_total[tid] = run;
        {
            unsigned long long* lb = a.lookback + (size_t)tile * kBins + tid;
            const unsigned long long ep = (unsigned long long)a.epoch << 32;
            st_volatile_u64(lb, (ltile == 0 ? kFlagInc : kFlagAgg) | ep | run);
            uint32_t excl = 0;
            if (ltile > 0) {  // the segment's first tile publishes inclusive: the walk ends there
                int64_t j = tile - 1;
                uint32_t spins = 0;
                while (j >= 0) {
                    const unsigned long long w = ld_volatile_u64(a.lookback + (size_t)j * kBins + tid);
                    const uint32_t wep = (uint32_t)(w >> 32) & 0x3fffffffu;
                    const unsigned long long flag = w & (3ull << 62);
                    if (wep != a.epoch || flag == 0) {
                        if (++spins > kSpinLimit) {
                            record_give_up(a.status);
                            break;
                        }
                        __nanosleep(32);
                        continue;
                    }
                    excl += (uint32_t)w;
                    if (flag == kFlagInc) break;
                    --j;
                }
                st_volatile_u64(lb, kFlagInc | ep | (unsigned long long)(excl + run));
            }
            s_gbase[tid] = s_bstart[tid] + excl;
        }
        s_excl[tid] = block_scan_256(run, s_misc + 1) - run;
        __syncthreads();  // s_excl is read across threads below
        {
#pragma unroll
            for (int k = 0; k < kItems; ++k) {
                const uint32_t d = rk[k] >> 16;
                if (d < 256u) {
                    const uint32_t lpos = s_excl[d] + s_whist[warp * kBins + d] + (rk[k] & 0xffffu);
#ifdef MSC_DEBUG_BOUNDS
                    if (lpos >= (uint32_t)kTile && atomicCAS(&g_sort_dbg[0], 0u, 1u) == 0u) {
                        g_sort_dbg[1] = (uint32_t)tile; g_sort_dbg[2] = warp; g_sort_dbg[3] = lane;
                        g_sort_dbg[4] = k; g_sort_dbg[5] = d; g_sort_dbg[6] = s_excl[d];
                        g_sort_dbg[7] = s_whist[warp * kBins + d]; g_sort_dbg[8] = rk[k] & 0xffffu;
                        g_sort_dbg[9] = a.shift; g_sort_dbg[10] = s_total[d]; g_sort_dbg[11] = blockIdx.x;
                        g_sort_dbg[12] = (uint32_t)ntiles; g_sort_dbg[13] = gridDim.x;
                    }
#endif
                    MSC_GUARD(lpos < (uint32_t)kTile, a.status, -103) {
                        s_keys[lpos] = key[k];
                        if constexpr (VALS) s_vals[lpos] = val[k];
                    }
                }
            }
            __syncthreads();
            if constexpr (BUCKET) {
                // (id, position) pairs regrouped by bucket in shared memory, then
                // each bucket's run written with consecutive lanes on consecutive slots
                static_assert(kMaxBuckets == kThreads, "one bucket per thread");
                uint32_t* s_bstart2 = s_bucket;              // counts, then tile-local bucket starts
                uint32_t* s_bbase = s_bucket + kMaxBuckets;  // first global slot of the tile's run
                s_bstart2[tid] = 0;
                __syncthreads();
                uint32_t pid[kItems], ppos[kItems], prank[kItems / 2];  // two 16-bit ranks per word
#pragma unroll
                for (int k = 0; k < kItems; ++k) {
                    const int i = tid + k * kThreads;
                    if (k % 2 == 0) prank[k / 2] = 0;
                    if (i < cnt) {
                        pid[k] = (uint32_t)s_vals[i];
                        const uint32_t d = (uint32_t)(s_keys[i] >> a.shift) & 255u;
                        ppos[k] = s_gbase[d] + (uint32_t)i - s_excl[d];
                        prank[k / 2] |= atomicAdd(&s_bstart2[pid[k] >> a.bucket_shift], 1u) << (16 * (k % 2));
                    }
                }
                __syncthreads();
                {
                    const uint32_t c = s_bstart2[tid];
                    const uint32_t start = block_scan_256(c, s_misc + 1) - c;
                    s_bbase[tid] = c ? ((uint32_t)tid << a.bucket_shift) +
                                           atomicAdd(&a.bucket_fill[tid * kFillStride], c)
                                     : 0u;
                    s_bstart2[tid] = start;
                }
                __syncthreads();
#pragma unroll
                for (int k = 0; k < kItems; ++k) {
                    const int i = tid + k * kThreads;
                    if (i < cnt) {
                        const uint32_t j = s_bstart2[pid[k] >> a.bucket_shift] + ((prank[k / 2] >> (16 * (k % 2))) & 0xffffu);
                        s_keys[j] = (KeyT)ppos[k];
                        s_vals[j] = (int32_t)pid[k];
                    }
                }
                __syncthreads();
                for (int i = tid; i < cnt; i += kThreads) {
                    const uint32_t id = (uint32_t)s_vals[i];
                    const uint32_t b = id >> a.bucket_shift;
                    const uint32_t slot = s_bbase[b] + ((uint32_t)i - s_bstart2[b]);
                    const uint32_t pos = (uint32_t)s_keys[i];
                    MSC_GUARD(slot < (uint64_t)a.n && pos < (uint64_t)n, a.status, -102) {
                        a.vals_out[slot] = (int32_t)id;
                        a.pair_pos[slot] = pos;
                    }
                }
            } else {
                KeyT* kout = a.keys_out + seg_base;
                int32_t* vout = VALS && !RANK ? a.vals_out + seg_base : nullptr;
                for (int i = tid; i < cnt; i += kThreads) {
                    const KeyT kk = s_keys[i];
                    const uint32_t d = (uint32_t)(kk >> a.shift) & 255u;
                    const uint32_t pos = s_gbase[d] + (uint32_t)i - s_excl[d];
                    MSC_GUARD(pos < (uint64_t)n, a.status, -102) {
                        if constexpr (RANK) {
                            if (a.keys_out) kout[pos] = kk;
                            a.rank_of[s_vals[i]] = pos;
                        } else {
                            kout[pos] = kk;
                            if constexpr (VALS) vout[pos] = s_vals[i];
                        }
                    }
                }
            }
        }
        __syncthreads();
    }
}

template <typename KeyT, bool FROM_F, bool BUCKET, bool SEG, bool VALS>
__global__ void __launch_bounds__(kThreads, sizeof(KeyT) == 8 ? 2 : 3) k_onesweep(const PassArgs<KeyT> a) {
    extern __shared__ __align__(16) uint8_t smem[];
    onesweep_tiles<KeyT, FROM_F, BUCKET, SEG, VALS, false>(a, smem);
}

// Width of the id buckets the last pass files pairs into: 2^19 ids at
// least (2 MiB of the order array), and at most kMaxBuckets buckets.
int bucket_shift(int64_t n) {
    return std::max(19, ceil_log2(ceil_div(std::max<int64_t>(n, 1), kMaxBuckets)));
}

__global__ void __launch_bounds__(kPermuteThreads) k_pair_permute(const int32_t* __restrict__ ids,
                                                                  const uint32_t* __restrict__ pos, int64_t n, int vec,
                                                                  int32_t* __restrict__ order, int32_t* status) {
    permute_pairs(ids, pos, n, vec, order, status);
}

int launch_pair_permute(const int32_t* ids, const uint32_t* pos, int64_t n, int32_t* order, int32_t* status,
                        cudaStream_t s) {
    const int vec = (((uintptr_t)ids | (uintptr_t)pos) & 15) == 0;
    TraceScope ts_("order.permute", s);
    k_pair_permute<<<(unsigned)ceil_div(n, kPermuteChunk), kPermuteThreads, 0, s>>>(ids, pos, n, vec, order, status);
    MSC_LAUNCHED();
    return MSC_OK;
}

template <typename KeyT, bool FROM_F, bool BUCKET, bool SEG = false, bool VALS = true>
int launch_pass(const PassArgs<KeyT>& a, int64_t max_n, cudaStream_t s, const char* label) {
    constexpr size_t smem = pass_smem_bytes<KeyT, VALS>();
    auto kern = k_onesweep<KeyT, FROM_F, BUCKET, SEG, VALS>;
    static int configured_dev = -1;  // the attribute is set once per device
    if (configured_dev != current_device().id) {
        MSC_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        configured_dev = current_device().id;
    }
    int occ = 0;
    MSC_TRY(max_blocks_per_sm(&occ, kern, kThreads, smem));
    const int64_t ntiles = SEG ? a.seg_tiles : ceil_div(max_n, kThreads * kPassItems<KeyT>);
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(ntiles, (int64_t)current_device().sms * std::max(occ, 1)));
    {
        TraceScope ts_(label, s);
        kern<<<(unsigned)grid, kThreads, smem, s>>>(a);
    }
    MSC_LAUNCHED();
    return MSC_OK;
}

// Ranks of a hash table's keys in one cooperative launch: compact the occupied
// slots into (key, slot) pairs (each thread scans 8 consecutive slots with
// 16-byte loads, one atomic append per block and chunk), radix-sort the pairs
// by key and write vals[slot] = rank of the slot's key.  As separate launches
// the five to seven passes over the few thousand to few million pairs of a
// usual field took some 20 us each, nearly all of it launch and look-back
// latency (64^3 field with noise: 93 us as nine launches, 45 as one).
//
// Up to kPairsCoopMax pairs the digit passes are those of coop.cuh, by only as
// many of the at most two blocks per SM as there are tiles of pairs; a single
// tile needs no barrier at all.  More pairs go through onesweep passes in the
// same launch, whose tiles are read once per pass and three times as large.
// us with the passes of coop.cuh / onesweep passes (the launches of before):
//   490 000 pairs 88 / 122, 810 000 146 / 137, 1.2M 160 / 157, 2.6M 305 / 258,
//   9.1M 834 / 677, 23.4M 2921 / 2121 (2010), 46.5M 5685 / 4030 (3670).
// Per pass the first read and write 32 bytes per pair (24 with one tile per
// block), the others 24.
constexpr int kCompactPer = 8;
constexpr int kPairItems = 8;
using PairSmem = CoopSmem<unsigned long long, kPairItems>;
constexpr int kPairTile = kThreads * kPassItems<unsigned long long>;
constexpr uint32_t kPairsCoopMax = 1u << 20;
// The kernel that holds both ways takes 96 KB of shared memory per block, and 5 us
// more where there are few pairs (43 against 49 for 3600): up to this many
// vertices, where a field has at most kPairsCoopMax pairs (white noise: a
// third of its vertices), the one with the passes of coop.cuh alone.
constexpr int64_t kPairsCoopVertices = 3 << 20;
static_assert(kCoopThreads == kThreads, "one block shape for both sorts");

struct PairArgs {
    PairRanks p;
    uint32_t* scratch;             // kCoopScratchWords
    uint32_t* hist;                // [npass][256] ONESWEEP
    uint32_t* tile_counters;       // [npass] ONESWEEP
    unsigned long long* lookback;  // ONESWEEP
    int32_t* status;
};

template <bool ONESWEEP>
__global__ void __launch_bounds__(kCoopThreads, 2) k_pair_ranks(const PairArgs args) {
    extern __shared__ __align__(16) uint8_t pair_smem[];
    PairSmem& S = *reinterpret_cast<PairSmem*>(pair_smem);
    const PairRanks& a = args.p;
    int32_t* status = args.status;
    __shared__ uint32_t s_warp[kCoopWarps];
    __shared__ uint32_t s_base;
    if (a.ctl[kPairCtlRoute] == 0u) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    {
        const int64_t slots = (int64_t)a.ctl[2] + kPairPad;
        constexpr int64_t kChunkSlots = (int64_t)kCoopThreads * kCompactPer;
        const int64_t nchunks = (slots + kChunkSlots - 1) / kChunkSlots;
        for (int64_t c = blockIdx.x; c < nchunks; c += gridDim.x) {
            const int64_t i0 = c * kChunkSlots + (int64_t)tid * kCompactPer;
            unsigned long long k[kCompactPer];
            if (i0 + kCompactPer <= slots) {  // capacity and pad are multiples of 8: whole groups
#pragma unroll
                for (int q = 0; q < kCompactPer / 2; ++q) {
                    const ulonglong2 v = reinterpret_cast<const ulonglong2*>(a.table + i0)[q];
                    k[2 * q] = v.x;
                    k[2 * q + 1] = v.y;
                }
            } else {
#pragma unroll
                for (int j = 0; j < kCompactPer; ++j) k[j] = i0 + j < slots ? a.table[i0 + j] : kPairEmpty;
            }
            uint32_t cnt = 0;
#pragma unroll
            for (int j = 0; j < kCompactPer; ++j) cnt += k[j] != kPairEmpty;
            uint32_t incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            if (lane == 31) s_warp[warp] = incl;
            __syncthreads();
            if (tid == 0) {
                uint32_t run = 0;
                for (int w = 0; w < kCoopWarps; ++w) {
                    const uint32_t t = s_warp[w];
                    s_warp[w] = run;
                    run += t;
                }
                s_base = run ? atomicAdd(&a.ctl[kPairCtlCount], run) : 0u;
            }
            __syncthreads();
            uint32_t pos = s_base + s_warp[warp] + incl - cnt;
#pragma unroll
            for (int j = 0; j < kCompactPer; ++j) {
                if (k[j] != kPairEmpty) {
                    MSC_GUARD(pos < (uint32_t)slots, status, -131) {
                        a.keys[0][pos] = k[j];
                        a.slots[0][pos] = (int32_t)(i0 + j);
                    }
                    ++pos;
                }
            }
            __syncthreads();
        }
    }
    GridBarrier all{a.ctl + kPairCtlBarrier, gridDim.x, 0};
    if (!grid_barrier(all, status)) return;
    const uint32_t K = __ldcg(a.ctl + kPairCtlCount);
    if (ONESWEEP && K > kPairsCoopMax) {
        const int64_t words = ((int64_t)K + kPairTile - 1) / kPairTile * kBins;
        for (int64_t i = (int64_t)blockIdx.x * kCoopThreads + tid; i < words; i += (int64_t)gridDim.x * kCoopThreads)
            args.lookback[i] = 0;
        for (int i = blockIdx.x * kCoopThreads + tid; i < a.npass * kBins; i += gridDim.x * kCoopThreads) args.hist[i] = 0;
        if (blockIdx.x == 0 && tid < a.npass) args.tile_counters[tid] = 0;
        if (!grid_barrier(all, status)) return;
        add_digit_counts(a.keys[0], K, a.npass, args.hist, reinterpret_cast<uint32_t*>(pair_smem));
        if (!grid_barrier(all, status)) return;
        PassArgs<unsigned long long> w{};
        w.n = K;
        w.lookback = args.lookback;
        w.status = status;
        w.rank_of = a.vals;
#pragma unroll 1
        for (int p = 0; p < a.npass; ++p) {
            const int in = p & 1;
            w.keys_in = in ? a.keys[1] : a.keys[0];
            w.vals_in = in ? a.slots[1] : a.slots[0];
            w.keys_out = in ? a.keys[0] : a.keys[1];
            w.vals_out = in ? a.slots[0] : a.slots[1];
            w.hist = args.hist + p * kBins;
            w.shift = 8 * p;
            w.tile_counter = args.tile_counters + p;
            w.epoch = (uint32_t)(p + 1);
            if (p + 1 < a.npass) {
                onesweep_tiles<unsigned long long, false, false, false, true, false>(w, pair_smem);
                if (!grid_barrier(all, status)) return;
            } else {
                if (!a.keep_keys) w.keys_out = nullptr;
                onesweep_tiles<unsigned long long, false, false, false, true, true>(w, pair_smem);
            }
        }
        return;
    }
    const uint32_t active = min(gridDim.x, (K + PairSmem::kTile - 1) / PairSmem::kTile);
    if (blockIdx.x >= active) return;
    GridBarrier bar{a.ctl + kPairCtlBarrier + 1, active, 0};
#pragma unroll 1
    for (int p = 0; p < a.npass; ++p) {
        const bool last = p + 1 == a.npass;
        const unsigned long long* kin = a.keys[p & 1];
        const int32_t* vin = a.slots[p & 1];
        unsigned long long* kout = a.keys[(p & 1) ^ 1];
        int32_t* vout = a.slots[(p & 1) ^ 1];
        const CoopPass r = coop_radix_pass<unsigned long long, kPairItems>(
            S, K, 8 * p, false, [&](uint32_t i) { return kin[i]; }, [&](uint32_t i) { return (uint32_t)vin[i]; },
            [&](uint32_t pos, unsigned long long k, uint32_t slot) {
                if (!last || a.keep_keys) kout[pos] = k;
                if (!last) vout[pos] = (int32_t)slot;
                else a.vals[slot] = pos;
            },
            args.scratch, bar, status);
        if (r == kPassFailed) return;
    }
}

}  // namespace

int order_bucket_shift(int64_t n) { return bucket_shift(n); }

void size_sort_scratch(Sizer& s, int64_t n) {
    s.take<uint32_t>(kOrderCntWords);
    s.take<uint32_t>(8 * kBins + kCounterWords);
    s.take<unsigned long long>((size_t)std::max<int64_t>(1, ceil_div(n, kSortTile)) * kBins);
}

SortScratch carve_sort_scratch(Carver& c, int64_t n) {
    SortScratch sc;
    sc.ord_cnt = c.take<uint32_t>(kOrderCntWords);
    sc.hist = c.take<uint32_t>(8 * kBins + kCounterWords);
    sc.tile_counters = sc.hist + 8 * kBins;
    sc.max_tiles = std::max<int64_t>(1, ceil_div(n, kSortTile));
    sc.lookback = c.take<unsigned long long>((size_t)sc.max_tiles * kBins);
    return sc;
}

// Clears the look-back words of the tiles that *d_n keys occupy (a sort
// whose count is known only on the device touches no other tile).
__global__ void k_clear_lookback(unsigned long long* lookback, const int32_t* __restrict__ d_n,
                                 int64_t max_n) {
    const int64_t words = ((min((int64_t)*d_n, max_n) + kSortTile - 1) / kSortTile) * kBins;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words;
         i += (int64_t)gridDim.x * blockDim.x)
        lookback[i] = 0ull;
}

static size_t hist_smem(int npass) { return (size_t)kWarps * npass * kBins * sizeof(uint32_t); }

// Allow the histogram kernel the shared memory of 8 passes (64 KiB).
static int configure_hist() {
    static int configured_dev = -1;
    if (configured_dev != current_device().id) {
        MSC_TRY(cudaFuncSetAttribute(k_hist, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hist_smem(8)));
        configured_dev = current_device().id;
    }
    return MSC_OK;
}

static int hist_grid(int64_t n) {
    const int64_t want = ceil_div(std::max<int64_t>(n, 1), 256 * kHistRun);
    return (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)current_device().sms * 8));
}

void size_seg_sort_scratch(Sizer& s, int count, int64_t tiles) {
    s.take<uint32_t>((size_t)count * kSegPasses * kBins + kCounterWords);
    s.take<unsigned long long>((size_t)std::max<int64_t>(1, tiles) * kBins);
}

SortScratch carve_seg_sort_scratch(Carver& c, int count, int64_t tiles) {
    SortScratch sc;
    sc.ord_cnt = nullptr;
    const size_t hist_words = (size_t)count * kSegPasses * kBins;
    sc.hist = c.take<uint32_t>(hist_words + kCounterWords);
    sc.tile_counters = sc.hist + hist_words;
    sc.max_tiles = std::max<int64_t>(1, tiles);
    sc.lookback = c.take<unsigned long long>((size_t)sc.max_tiles * kBins);
    return sc;
}

int run_order_seg(const float* f, const SegTable& t, int32_t* order, uint32_t* key_a, int32_t* id_a,
                  uint32_t* key_b, int32_t* id_b, const SortScratch& sc, int32_t* status,
                  cudaStream_t s) {
    if (t.tiles <= 0) return MSC_OK;
    const size_t hist_words = (size_t)t.count * kSegPasses * kBins;
    MSC_TRY(cudaMemsetAsync(sc.hist, 0, (hist_words + kCounterWords) * sizeof(uint32_t), s));
    MSC_TRY(cudaMemsetAsync(sc.lookback, 0, (size_t)t.tiles * kBins * sizeof(unsigned long long), s));
    int r;
    {
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(t.tiles, (int64_t)current_device().sms * 4));
        TraceScope ts_("order.hist", s);
        k_hist_seg<<<grid, 256, hist_smem(kSegPasses), s>>>(f, t.tile_seg, t.off, t.tile0, t.tiles, sc.hist, status);
    }
    MSC_LAUNCHED();
    {
        TraceScope ts_("order.bstart", s);
        k_seg_bstart<<<(unsigned)(t.count * kSegPasses), 256, 0, s>>>(sc.hist);
    }
    MSC_LAUNCHED();
    PassArgs<uint32_t> a{};
    a.n = t.total;
    a.status = status;
    a.lookback = sc.lookback;
    a.tile_seg = t.tile_seg;
    a.seg_off = t.off;
    a.seg_tile0 = t.tile0;
    a.seg_tiles = t.tiles;
    a.seg_stride = kSegPasses * kBins;
    a.f_in = f;
    a.keys_out = key_a;
    a.vals_out = id_a;
    a.hist = sc.hist;
    a.shift = 0;
    a.tile_counter = sc.tile_counters + 0;
    a.epoch = 1;
    if ((r = launch_pass<uint32_t, true, false, true>(a, t.total, s, "order.pass_first"))) return r;
    uint32_t* kin = key_a;
    int32_t* iin = id_a;
    uint32_t* kout = key_b;
    int32_t* iout = id_b;
    for (int p = 1; p <= 2; ++p) {
        a.f_in = nullptr;
        a.keys_in = kin;
        a.vals_in = iin;
        a.keys_out = kout;
        a.vals_out = iout;
        a.hist = sc.hist + p * kBins;
        a.shift = 8 * p;
        a.tile_counter = sc.tile_counters + p;
        a.epoch = (uint32_t)(p + 1);
        if ((r = launch_pass<uint32_t, false, false, true>(a, t.total, s, "order.pass"))) return r;
        std::swap(kin, kout);
        std::swap(iin, iout);
    }
    a.keys_in = kin;
    a.vals_in = iin;
    a.keys_out = nullptr;
    a.vals_out = iout;
    a.pair_pos = kout;
    a.bucket_fill = sc.tile_counters + 8;
    a.bucket_shift = bucket_shift(t.total);
    a.hist = sc.hist + 3 * kBins;
    a.shift = 24;
    a.tile_counter = sc.tile_counters + 3;
    a.epoch = 4;
    if ((r = launch_pass<uint32_t, false, true, true>(a, t.total, s, "order.pass_last"))) return r;
    return launch_pair_permute(iout, kout, t.total, order, status, s);
}

int run_sort_u64(unsigned long long* keys, int32_t* vals, unsigned long long* keys_alt,
                 int32_t* vals_alt, const int32_t* d_count, int64_t max_count, int key_bits,
                 const SortScratch& sc, int32_t* status, cudaStream_t s, bool* result_in_alt,
                 const char* hist_label, const char* pass_label) {
    *result_in_alt = false;
    if (max_count <= 0 || key_bits <= 0) return MSC_OK;
    const int npass = std::min(8, (key_bits + 7) / 8);
    MSC_TRY(cudaMemsetAsync(sc.hist, 0, (8 * kBins + kCounterWords) * sizeof(uint32_t), s));
    {
        TraceScope ts_("sort.clear_lookback", s);
        k_clear_lookback<<<(unsigned)std::min<int64_t>(ceil_div(ceil_div(max_count, kSortTile) * kBins, 256),
                                                       (int64_t)current_device().sms * 8),
                           256, 0, s>>>(sc.lookback, d_count, max_count);
    }
    MSC_LAUNCHED();
    int r = configure_hist();
    if (r) return r;
    {
        TraceScope ts_(hist_label, s);
        k_hist<<<hist_grid(max_count), 256, hist_smem(npass), s>>>(keys, max_count, d_count, npass, sc.hist);
    }
    MSC_LAUNCHED();
    PassArgs<unsigned long long> a{};
    a.n = max_count;
    a.d_n = d_count;
    a.status = status;
    a.lookback = sc.lookback;
    unsigned long long* kin = keys;
    int32_t* vin = vals;
    unsigned long long* kout = keys_alt;
    int32_t* vout = vals_alt;
    for (int p = 0; p < npass; ++p) {
        a.keys_in = kin;
        a.vals_in = vin;
        a.keys_out = kout;
        a.vals_out = vout;
        a.hist = sc.hist + p * kBins;
        a.shift = 8 * p;
        a.tile_counter = sc.tile_counters + p;
        a.epoch = (uint32_t)(p + 1);
        r = vals ? launch_pass<unsigned long long, false, false>(a, max_count, s, pass_label)
                 : launch_pass<unsigned long long, false, false, false, false>(a, max_count, s, pass_label);
        if (r) return r;
        std::swap(kin, kout);
        std::swap(vin, vout);
    }
    *result_in_alt = (npass & 1) != 0;
    return MSC_OK;
}

template <bool ONESWEEP>
static int launch_pair_ranks(const PairArgs& a, int64_t n, cudaStream_t s) {
    constexpr size_t smem = ONESWEEP ? std::max(sizeof(PairSmem), pass_smem_bytes<unsigned long long, true>()) : sizeof(PairSmem);
    static_assert(!ONESWEEP || smem >= (size_t)kWarps * 8 * kBins * sizeof(uint32_t), "the digit counts fit too");
    auto kern = k_pair_ranks<ONESWEEP>;
    static int configured_dev = -1;
    if (configured_dev != current_device().id) {
        MSC_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        configured_dev = current_device().id;
    }
    int blocks = 0;
    const int r = coop_blocks(kern, kCoopThreads, smem, std::min<int64_t>(ceil_div(n, PairSmem::kTile), kCoopMaxBlocks), s,
                              &blocks);
    if (r) return r;
    TraceScope ts_("msid.pairs", s);
    return coop_launch(kern, blocks, kCoopThreads, smem, s, a);
}

int run_pair_ranks(const PairRanks& p, int64_t n, const SortScratch& sc, int32_t* status, cudaStream_t s) {
    const PairArgs a{p, sc.ord_cnt, sc.hist, sc.tile_counters, sc.lookback, status};
    return n > kPairsCoopVertices ? launch_pair_ranks<true>(a, n, s) : launch_pair_ranks<false>(a, n, s);
}

}  // namespace msc

#ifdef MSC_DEBUG_BOUNDS
extern "C" MSC_API int msc_debug_sort(uint32_t* out16) {
    return cudaMemcpyFromSymbol(out16, msc::g_sort_dbg, sizeof(uint32_t) * 16) == cudaSuccess ? 0 : -3;
}
#endif
