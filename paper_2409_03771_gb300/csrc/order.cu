// Vertex order (Simulation of Simplicity, section "Preprocessing": the
// vertices sorted by scalar value with ties broken by global id; order[v]
// is the position of v).
//
// LSD radix sort of (key, id) pairs, four 8-bit digit passes.  Keys are
// the float bits mapped to an order-preserving uint32 (-0.0 folded onto
// +0.0); every pass is stable and the first reads the vertices in id
// order, so equal keys stay in id order and the final position of v is its
// rank under (f[v], v).
//
// Each pass is an upsweep / scan / downsweep over super-tiles (runs of S
// consecutive 6144-key tiles), so no block ever waits for another:
//   k_ord_up    counts the pass digit of every super-tile (run-length
//               counted into warp-private shared histograms);
//   k_ord_scan  one block per digit turns the super-tile counts into each
//               super-tile's first output position for that digit;
//   k_ord_down  each block takes super-tiles s, s + G, s + 2G, ... (G
//               blocks), walks their tiles in order, ranks each tile's keys
//               stably (the lanes of a digit meet in a word of shared memory,
//               or by match where few digits occur), keeps running per-digit offsets and
//               writes through shared memory in coalesced runs.  The next
//               tile is fetched by a 1D TMA bulk copy into the other half
//               of a shared-memory double buffer while the current one is
//               ranked; the consumed half then serves as the staging area.
//               Interleaved super-tiles keep the blocks' write fronts of a
//               digit next to each other, so partly written lines are
//               completed in L2 before they are written back.
// The last pass files (vertex id, position) pairs into buckets of
// consecutive ids instead of writing sorted keys, and the order field is
// their inverse permutation (k_ord_permute); while the
// order array fits the L2 it scatters the positions itself.  Small fields go
// through all four passes in one cooperative launch (k_ord_coop).
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "coop.cuh"
#include "radix.cuh"
#include "sort.cuh"
#include "tma.cuh"

namespace msc {
namespace {

#ifndef MSC_ORD_ITEMS
#define MSC_ORD_ITEMS 24
#endif
#ifndef MSC_ORD_MIN_BLOCKS
#define MSC_ORD_MIN_BLOCKS 2
#endif
#ifndef MSC_ORD_MATCH_MAX
#define MSC_ORD_MATCH_MAX 64
#endif
constexpr int kT = 256;                // threads per block
constexpr int kI = MSC_ORD_ITEMS;      // keys per thread and tile
constexpr int kTile = kT * kI;  // keys per tile (6144)
static_assert(kI % 4 == 0, "digits are packed four to a word");
constexpr int kW = kT / kWarp;  // 8 warps
constexpr int kB = kRadixBins;  // 256 digits
constexpr uint32_t kWaitLimit = 1u << 22;  // mbarrier polls before giving up (~0.3 s)

static_assert(kRadixScanWarps == kW, "block_scan_256 expects 8 warps");
static_assert(kOrderMaxBuckets == kT, "one id bucket per thread");

// Super-tile s holds tiles [s * per_super, min(tiles, (s + 1) * per_super)).
struct Range {
    int64_t n;
    int64_t tiles;
    int64_t per_super;
    int supers;
};

// The buffers of a sort and what its keys have in common.  varies[0] is the
// OR of all keys and varies[1] the OR of their complements (written by the
// first pass's upsweep): a byte that is the same in every key is zero in
// their AND, and its pass moves nothing (the low mantissa bytes of small
// whole numbers: an 8-bit scan takes two passes instead of four).  The
// passes that do move alternate between the buffers, starting from the field.
struct Buffers {
    const float* f;
    uint32_t* key[2];
    int32_t* id[2];
    const uint32_t* varies;
    int aligned[3];  // 16-byte aligned: buffer 0, buffer 1, the field
};

__device__ __forceinline__ bool pass_moves(const Buffers& b, int p) {
    return p == 3 || ((b.varies[0] & b.varies[1]) >> (8 * p) & 255u) != 0u;  // the last pass writes the result
}

__device__ __forceinline__ uint32_t* key_of(const Buffers& b, int i) { return i ? b.key[1] : b.key[0]; }
__device__ __forceinline__ int32_t* id_of(const Buffers& b, int i) { return i ? b.id[1] : b.id[0]; }

// Buffer holding the keys before pass p (-1: the field); the pass writes the
// other one (0 after the field).
__device__ __forceinline__ int source_of(const Buffers& b, int p) {
    const uint32_t v = b.varies[0] & b.varies[1];
    const int moved = (p > 0 && (v & 0xffu)) + (p > 1 && (v & 0xff00u)) + (p > 2 && (v & 0xff0000u));
    return moved == 0 ? -1 : (moved - 1) & 1;
}

// The 8-bit digit of a key at a compile-time bit offset (one byte permute).
template <int SHIFT>
__device__ __forceinline__ uint32_t digit_of(uint32_t k) {
    if constexpr (SHIFT == 0) return k & 255u;
    else if constexpr (SHIFT == 24) return k >> 24;
    else return __byte_perm(k, 0u, 0x4440u + SHIFT / 8);
}

// Upsweep: per-super-tile counts of the digit at SHIFT, stored digit-major
// (cnt[d * kOrderMaxSuper + s]), plus the pass totals (one atomic per block
// and digit).  The first pass also reports NaNs and gathers `varies`.
// Bound: the shared-memory atomics of the counts (LSU 69 %); 512^3: 0.12 ms
// per pass, reading the keys alone takes 0.08.
template <int SHIFT>
__global__ void __launch_bounds__(kT, 4) k_ord_up(const Buffers bufs, const Range r, uint32_t* __restrict__ cnt,
                                               uint32_t* __restrict__ total, uint32_t* varies, int32_t* status) {
    __shared__ uint32_t sh[kW * kB];
    if (SHIFT > 0 && !pass_moves(bufs, SHIFT / 8)) return;
    const int from = SHIFT == 0 ? -1 : source_of(bufs, SHIFT / 8);
    const bool ff = from < 0;  // keys are made from the float field
    uint32_t any1 = 0, all1 = ~0u, lo = ~0u, hi = 0;  // the first pass's keys
    const int tid = threadIdx.x, warp = tid >> 5;
    uint32_t* wh = sh + warp * kB;
    uint32_t mine = 0;  // this block's total of digit tid
    const uint32_t* src = ff ? reinterpret_cast<const uint32_t*>(bufs.f) : key_of(bufs, from);
    const bool vec = ((uintptr_t)src & 15) == 0;
    for (int s = blockIdx.x; s < r.supers; s += gridDim.x) {
        for (int i = tid; i < kW * kB; i += kT) sh[i] = 0;
        __syncthreads();
        const int64_t k0 = (int64_t)s * r.per_super * kTile;
        const int64_t k1 = min(r.n, k0 + r.per_super * kTile);
        // sixteen keys per thread and step in four lane-consecutive groups of
        // four, the next step's loads in flight while one is counted
        constexpr int kStep4 = kT * 16;
        auto load = [&](int64_t base, uint32_t (&k)[16]) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int64_t i = base + (int64_t)(q * kT + tid) * 4;
                if (vec && i + 4 <= k1) {
                    const uint4 v = __ldcs(reinterpret_cast<const uint4*>(src + i));
                    k[4 * q] = v.x;
                    k[4 * q + 1] = v.y;
                    k[4 * q + 2] = v.z;
                    k[4 * q + 3] = v.w;
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) k[4 * q + j] = i + j < k1 ? src[i + j] : 0u;
                }
            }
        };
        uint32_t a[16];
        if (k0 < k1) load(k0, a);
        for (int64_t b = k0; b < k1; b += kStep4) {
            uint32_t nx[16];
            if (b + kStep4 < k1) load(b + kStep4, nx);
            if (SHIFT == 0 || ff) {
#pragma unroll
                for (int j = 0; j < 16; ++j) a[j] = float_key(__uint_as_float(a[j]));
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int64_t i = b + (int64_t)(q * kT + tid) * 4;
                const int cnt = (int)max((int64_t)0, min((int64_t)4, k1 - i));
                uint32_t cur = 0, run = 0;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (j >= cnt) break;
                    const uint32_t w = a[4 * q + j];
                    if constexpr (SHIFT == 0) {
                        any1 |= w;
                        all1 &= w;
                        lo = min(lo, w);
                        hi = max(hi, w);
                    }
                    const uint32_t d = digit_of<SHIFT>(w);
                    if (j > 0 && d != cur) {
                        atomicAdd(&wh[cur], run);
                        run = 0;
                    }
                    cur = d;
                    ++run;
                }
                if (cnt > 0) atomicAdd(&wh[cur], run);
            }
#pragma unroll
            for (int j = 0; j < 16; ++j) a[j] = nx[j];
        }
        __syncthreads();
        uint32_t c = 0;
#pragma unroll
        for (int w = 0; w < kW; ++w) c += sh[w * kB + tid];
        cnt[(size_t)tid * kOrderMaxSuper + s] = c;
        mine += c;
        __syncthreads();
    }
    if (mine) atomicAdd(&total[tid], mine);
    if (SHIFT == 0) {
        // a NaN's key lies above that of +Inf or below that of -Inf
        if (hi > 0xff800000u || lo < 0x007fffffu) record_error(status, MSC_ERR_NAN);
        any1 = __reduce_or_sync(0xffffffffu, any1);
        all1 = __reduce_and_sync(0xffffffffu, all1);
        if ((tid & 31) == 0) {
            atomicOr(&varies[0], any1);
            atomicOr(&varies[1], ~all1);
        }
    }
}

// Scan: block d takes digit d.  Its super-tiles' counts become exclusive
// output positions starting at the digit's global start (the sum of the
// totals of the smaller digits); warp w scans the w-th eighth of the row.
__global__ void __launch_bounds__(kT) k_ord_scan(const Buffers bufs, int pass, uint32_t* __restrict__ cnt,
                                                 const uint32_t* __restrict__ total, int supers) {
    if (!pass_moves(bufs, pass)) return;
    __shared__ uint32_t s_w[kW];
    __shared__ uint32_t s_g;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int d = blockIdx.x;
    if (warp == 0) {
        uint32_t g = 0;
        for (int j = lane; j < d; j += 32) g += total[j];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
        if (lane == 0) s_g = g;
    }
    uint32_t* row = cnt + (size_t)d * kOrderMaxSuper;
    constexpr int kPer = kOrderMaxSuper / kW / 32;  // entries per lane
    const int per_warp = (supers + kW - 1) / kW;
    const int b0 = warp * per_warp;
    uint32_t x[kPer], wsum = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int i = j * 32 + lane;
        const int b = b0 + i;
        x[j] = (i < per_warp && b < supers) ? row[b] : 0u;
        wsum += x[j];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
    if (lane == 0) s_w[warp] = wsum;
    __syncthreads();
    uint32_t run = s_g;
    for (int w = 0; w < warp; ++w) run += s_w[w];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        if (j * 32 >= per_warp) break;
        uint32_t incl = x[j];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const int i = j * 32 + lane;
        const int b = b0 + i;
        if (i < per_warp && b < supers) row[b] = run + incl - x[j];
        run += __shfl_sync(0xffffffffu, incl, 31);
    }
}

// What a downsweep writes: the sorted (key, id) arrays, (id, position) pairs
// filed by id bucket, or order[id] = position.  Scattering the order
// straight from the last pass is best while the order array stays in L2:
// 2^24 vertices of white noise 684 -> 632 us, of 256 levels 668 -> 545; 2^25
// vertices 1266 against 1527.
enum { kOutSorted, kOutBuckets, kOutOrder };
constexpr int64_t kOrderDirectMax = 1 << 24;

struct DownArgs {
    Buffers bufs;
    int32_t* order;            // kOutOrder
    uint32_t* bucket_fill;     // kOutBuckets: slots taken per id bucket (stride kOrderFillStride)
    int bucket_shift;          // kOutBuckets: log2 of the ids per bucket
    Range r;
    const uint32_t* base;      // [256][kOrderMaxSuper] first output position per digit and super-tile
    const uint32_t* total;     // [256] keys per digit in this pass
    int32_t* status;
};

// Shared memory of k_ord_down: two tile buffers of (key, value) words,
// warp histograms (16-bit; after the count, each warp's tile-local start),
// per-digit words, scan scratch, bucket words, two mbarriers.
constexpr size_t kBufWords = 2 * kTile;
constexpr size_t kDownSmem = 2 * kBufWords * 4 + kW * kB * 2 + 2 * kB * 4 + 32 * 4 + 2 * kB * 4 + 2 * 8 + kW * kB * 4;

// The downsweep.  A key's rank among the warp's lanes with its digit comes
// from one match instruction, whose cost grows with the number of distinct
// digits in the warp, or from a word of shared memory per digit
// (rank_in_warp), which a few digits would crowd.  The middle passes of a 512^3
// field took 1.62 ms with eight ballots per key (issue-bound) and take 1.39 this
// way (LSU 79 %, DRAM half busy); shares of the keys by ballots were no faster
// (1.41 to 1.5).
template <int OUT, int SHIFT>
__global__ void __launch_bounds__(kT, MSC_ORD_MIN_BLOCKS) k_ord_down(const DownArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    uint32_t* buf = reinterpret_cast<uint32_t*>(smem);                     // [2][kTile words | kTile words]
    uint16_t* s_wh = reinterpret_cast<uint16_t*>(buf + 2 * kBufWords);     // [kW][kB]
    uint32_t* s_run = reinterpret_cast<uint32_t*>(s_wh + kW * kB);         // [kB] next output position
    uint32_t* s_delta = s_run + kB;                                        // [kB] output pos - staged pos
    uint32_t* s_misc = s_delta + kB;                                       // [32] scan scratch
    uint32_t* s_bcnt = s_misc + 32;                                        // [kB] BUCKET
    uint32_t* s_bbase = s_bcnt + kB;                                       // [kB] BUCKET
    uint64_t* mbar = reinterpret_cast<uint64_t*>(s_bbase + kB);            // [2]
    uint32_t* s_match = reinterpret_cast<uint32_t*>(mbar + 2);             // [kW][kB]

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const Range r = a.r;
    if ((int)blockIdx.x >= r.supers || !pass_moves(a.bufs, SHIFT / 8)) return;  // block-uniform
    const int from = SHIFT == 0 ? -1 : source_of(a.bufs, SHIFT / 8), to = from == 0;
    const bool ff = from < 0;  // keys from the float field, ids implicit
    constexpr bool FF = SHIFT == 0;
    uint32_t* keys_out = key_of(a.bufs, to);  // kOutBuckets: the positions of the filed pairs
    int32_t* vals_out = id_of(a.bufs, to);    // ... and their ids
    // few populated digits in this pass (a float field's top byte): rank
    // with match
    const bool use_match = __syncthreads_count(a.total[tid] != 0u) <= MSC_ORD_MATCH_MAX;
    const int64_t G = gridDim.x;
    // the tiles of this block in processing order: super-tiles
    // blockIdx.x, blockIdx.x + G, ..., each from its first tile to its last
    auto next_tile = [&](int64_t t) -> int64_t {
        if ((t + 1) % r.per_super != 0 && t + 1 < r.tiles) return t + 1;
        const int64_t s = t / r.per_super + G;
        return s < r.supers ? s * r.per_super : -1;
    };
    for (int i = tid; i < kW * kB / 2; i += kT) reinterpret_cast<uint32_t*>(s_wh)[i] = 0u;
    for (int i = tid; i < kW * kB; i += kT) s_match[i] = 0u;
    if (tid == 0) {
        s_misc[31] = SHIFT > 0 && stage_gave_up(a.status);
        mbar_init(&mbar[0], 1);
        mbar_init(&mbar[1], 1);
        fence_mbar_init();
    }
    __syncthreads();

    if (s_misc[31]) return;  // the ids of an unfinished pass
    const uint32_t* src_k = ff ? reinterpret_cast<const uint32_t*>(a.bufs.f) : key_of(a.bufs, from);
    const int32_t* src_v = ff ? nullptr : id_of(a.bufs, from);
    const bool use_tma = ff ? a.bufs.aligned[2] : from ? a.bufs.aligned[1] : a.bufs.aligned[0];
    // full, aligned tiles come by bulk copy; the ragged last tile by plain loads
    auto by_tma = [&](int64_t t) { return use_tma && (t + 1) * kTile <= r.n; };
    auto issue = [&](int64_t t, int slot) {  // one thread
        if (t < 0 || !by_tma(t)) return;
        uint32_t* dst = buf + slot * kBufWords;
        mbar_expect_tx(&mbar[slot], ff ? kTile * 4 : kTile * 8);
        bulk_load(dst, src_k + t * kTile, kTile * 4, &mbar[slot]);
        if (!ff) bulk_load(dst + kTile, src_v + t * kTile, kTile * 4, &mbar[slot]);
    };
    int64_t t = (int64_t)blockIdx.x * r.per_super;
    if (tid == 0) issue(t, 0);

    const int wb = warp * (kI * 32) + lane;  // tile-local index of this thread's key k: wb + 32 k
    const uint32_t lt = lanemask_lt();
    uint16_t* wh = s_wh + warp * kB;
    for (int it = 0; t >= 0; ++it) {
        const int slot = it & 1;
        const int64_t tn = next_tile(t);
        // input: keys (or the field's words) in bk, values in bv; the keys are
        // staged into bv and the values into bk once each half has been read
        uint32_t* bk = buf + slot * kBufWords;
        uint32_t* bv = bk + kTile;
        if (tid == 0) issue(tn, slot ^ 1);
        // a super-tile starts: its output positions per digit (word tid is
        // read and written by thread tid only)
        if (t % r.per_super == 0) s_run[tid] = a.base[(size_t)tid * kOrderMaxSuper + t / r.per_super];
        const int cnt = (int)min((int64_t)kTile, r.n - t * kTile);
        const int64_t tb = t * kTile;
        if (by_tma(t)) {
            const bool ok = mbar_wait(&mbar[slot], (uint32_t)(it >> 1) & 1u, kWaitLimit);
            if (__syncthreads_or(!ok)) {
                // a copy never landed: report, let the prefetch in flight finish, stop
                if (tid == 0) {
                    record_give_up(a.status);
                    if (tn >= 0 && by_tma(tn)) mbar_wait(&mbar[slot ^ 1], (uint32_t)((it + 1) >> 1) & 1u, kWaitLimit);
                }
                return;
            }
        } else {
            for (int i = tid; i < cnt; i += kT) {
                bk[i] = src_k[tb + i];
                if (!ff) bv[i] = (uint32_t)src_v[tb + i];
            }
            __syncthreads();
        }
        if (!FF && ff) {  // the field after passes that moved nothing: make the pairs in place
            for (int i = tid; i < cnt; i += kT) {
                bk[i] = float_key(__uint_as_float(bk[i]));
                bv[i] = (uint32_t)(tb + i);
            }
            __syncthreads();
        }
        auto key_at = [&](int li) -> uint32_t {
            const uint32_t w = bk[li];
            return FF ? float_key(__uint_as_float(w)) : w;
        };
        // stable rank among the warp's equal digits: earlier keys of the warp
        // (its 16-bit counter) + lower lanes of this step
        uint32_t rk[kI / 2];
        uint32_t dg[kI / 4];  // the digits of the thread's keys, four to a word
        // FULL: every key of the tile is valid (all but a ragged last tile)
        auto rank_tile = [&](auto match_tag, auto full_tag) {
            constexpr bool MATCH = decltype(match_tag)::value;
            constexpr bool FULL = decltype(full_tag)::value;
#pragma unroll
            for (int k = 0; k < kI; ++k) {
                const int li = wb + 32 * k;
                const bool valid = FULL || li < cnt;
                const uint32_t d = valid ? digit_of<SHIFT>(key_at(li)) : 0u;
                dg[k / 4] = (k & 3) ? (dg[k / 4] | d << (8 * (k & 3))) : d;
                uint32_t rank;
                if constexpr (MATCH) {
                    const uint32_t peers = __match_any_sync(0xffffffffu, valid ? d : 0x100u | lane);
                    const uint32_t lower = __popc(peers & lt), before = wh[d];
                    if (valid && lower == 0) wh[d] = (uint16_t)(before + __popc(peers));
                    rank = before + lower;
                    __syncwarp();
                } else {
                    rank = rank_in_warp(d, valid, 1u << lane, lt, s_match + warp * kB, wh);
                }
                rk[k / 2] = (k & 1) ? (rk[k / 2] | rank << 16) : rank;
            }
        };
        if (cnt == kTile) {
            if (use_match) rank_tile(std::true_type{}, std::true_type{});
            else rank_tile(std::false_type{}, std::true_type{});
        } else {
            if (use_match) rank_tile(std::true_type{}, std::false_type{});
            else rank_tile(std::false_type{}, std::false_type{});
        }
        if constexpr (OUT == kOutBuckets) s_bcnt[tid] = 0u;
        __syncthreads();
        {   // digit tid: warp counts -> tile-local start of each warp's run of
            // the digit (16-bit: at most kTile); output start of the tile's run
            uint32_t pre[kW], run = 0;
#pragma unroll
            for (int w = 0; w < kW; ++w) {
                pre[w] = run;
                run += s_wh[w * kB + tid];
            }
            const uint32_t excl = block_scan_256(run, s_misc) - run;
#pragma unroll
            for (int w = 0; w < kW; ++w) s_wh[w * kB + tid] = (uint16_t)(excl + pre[w]);
            const uint32_t g = s_run[tid];
            s_delta[tid] = g - excl;
            s_run[tid] = g + run;
        }
        __syncthreads();
        if constexpr (OUT == kOutSorted) {
            // values into registers first (the field pass makes them from the
            // index), so that bv is free for the staged keys
            uint32_t val[kI];
            if constexpr (!FF) {
#pragma unroll
                for (int k = 0; k < kI; ++k) val[k] = bv[wb + 32 * k];
                __syncthreads();
            }
            // each key to its tile-local sorted position; rk keeps the position
#pragma unroll
            for (int k = 0; k < kI; ++k) {
                const int li = wb + 32 * k;
                uint32_t lpos = 0;
                if (li < cnt) {
                    const uint32_t kk = key_at(li);
                    const uint32_t d = (dg[k / 4] >> (8 * (k & 3))) & 255u;
                    lpos = wh[d] + ((rk[k / 2] >> (16 * (k & 1))) & 0xffffu);
                    MSC_GUARD(lpos < (uint32_t)kTile, a.status, -141) bv[lpos] = kk;
                }
                rk[k / 2] = (k & 1) ? ((rk[k / 2] & 0xffffu) | lpos << 16) : ((rk[k / 2] & 0xffff0000u) | lpos);
            }
            __syncwarp();
            for (int j = lane; j < kB / 2; j += 32) reinterpret_cast<uint32_t*>(wh)[j] = 0u;
            __syncthreads();  // every key read: bk is free
#pragma unroll
            for (int k = 0; k < kI; ++k) {
                const int li = wb + 32 * k;
                if (li < cnt) {
                    const uint32_t lpos = (rk[k / 2] >> (16 * (k & 1))) & 0xffffu;
                    MSC_GUARD(lpos < (uint32_t)kTile, a.status, -141) bk[lpos] = FF ? (uint32_t)(tb + li) : val[k];
                }
            }
            __syncthreads();
            // consecutive staged keys of one digit go to consecutive positions
#pragma unroll 4
            for (int k = 0; k < kI; ++k) {
                const int i = k * kT + tid;
                if (i < cnt) {
                    const uint32_t kk = bv[i];
                    const uint32_t pos = s_delta[digit_of<SHIFT>(kk)] + (uint32_t)i;
                    MSC_GUARD(pos < (uint64_t)r.n, a.status, -142) {
                        keys_out[pos] = kk;
                        vals_out[pos] = (int32_t)bk[i];
                    }
                }
            }
        } else if constexpr (OUT == kOutOrder) {
#pragma unroll
            for (int k = 0; k < kI; ++k) {
                const int li = wb + 32 * k;
                if (li < cnt) {
                    const uint32_t d = (dg[k / 4] >> (8 * (k & 3))) & 255u;
                    const uint32_t pos = s_delta[d] + wh[d] + ((rk[k / 2] >> (16 * (k & 1))) & 0xffffu);
                    const uint32_t id = bv[li];
                    MSC_GUARD(id < (uint64_t)r.n && pos < (uint64_t)r.n, a.status, -146) a.order[id] = (int32_t)pos;
                }
            }
            __syncwarp();
            for (int j = lane; j < kB / 2; j += 32) reinterpret_cast<uint32_t*>(wh)[j] = 0u;
        } else {
            // final positions straight from the ranks; (id, position) pairs
            // regrouped by id bucket, each bucket's run written with
            // consecutive lanes on consecutive slots
            uint32_t ppos[kI], prank[kI / 2];
#pragma unroll
            for (int k = 0; k < kI; ++k) {
                const int li = wb + 32 * k;
                const uint32_t d = li < cnt ? (dg[k / 4] >> (8 * (k & 3))) & 255u : 0u;
                ppos[k] = s_delta[d] + wh[d] + ((rk[k / 2] >> (16 * (k & 1))) & 0xffffu);
            }
            __syncwarp();
            for (int j = lane; j < kB / 2; j += 32) reinterpret_cast<uint32_t*>(wh)[j] = 0u;
            uint32_t id[kI];
#pragma unroll
            for (int k = 0; k < kI; ++k) {
                if (k % 2 == 0) prank[k / 2] = 0u;
                const int li = wb + 32 * k;
                id[k] = bv[li];
                if (li < cnt) {
                    const uint32_t b = id[k] >> a.bucket_shift;
                    MSC_GUARD(b < (uint32_t)kB, a.status, -143)
                    prank[k / 2] |= atomicAdd(&s_bcnt[b], 1u) << (16 * (k & 1));
                }
            }
            __syncthreads();
            {
                const uint32_t c = s_bcnt[tid];
                const uint32_t start = block_scan_256(c, s_misc + 8) - c;
                s_bbase[tid] = c ? ((uint32_t)tid << a.bucket_shift) + atomicAdd(&a.bucket_fill[tid * kOrderFillStride], c)
                                 : 0u;
                s_bcnt[tid] = start;
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < kI; ++k) {
                if (wb + 32 * k < cnt) {
                    const uint32_t j = s_bcnt[id[k] >> a.bucket_shift] + ((prank[k / 2] >> (16 * (k & 1))) & 0xffffu);
                    MSC_GUARD(j < (uint32_t)kTile, a.status, -144) {
                        bk[j] = ppos[k];
                        bv[j] = id[k];
                    }
                }
            }
            __syncthreads();
            for (int i = tid; i < cnt; i += kT) {
                const uint32_t v = bv[i];
                const uint32_t b = v >> a.bucket_shift;
                const uint32_t slot_ = s_bbase[b] + ((uint32_t)i - s_bcnt[b]);
                const uint32_t pos = bk[i];
                MSC_GUARD(slot_ < (uint64_t)r.n && pos < (uint64_t)r.n, a.status, -145) {
                    vals_out[slot_] = (int32_t)v;
                    keys_out[slot_] = pos;
                }
            }
        }
        // this buffer is refilled by a bulk copy (async proxy) two tiles on
        fence_proxy_async_smem();
        __syncthreads();
        t = tn;
    }
}

template <int OUT, int SHIFT>
int configure_down() {
    static int configured_dev = -1;  // the attribute is set once per device
    if (configured_dev != current_device().id) {
        MSC_TRY(cudaFuncSetAttribute(k_ord_down<OUT, SHIFT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDownSmem));
        configured_dev = current_device().id;
    }
    return MSC_OK;
}

// One digit pass: upsweep, scan, downsweep.
struct PassLaunch {
    DownArgs a;
    uint32_t* cnt;
    uint32_t* totals;  // [4][256]
    uint32_t* varies;
    int up_blocks, down_blocks;
    cudaStream_t s;
};

template <int OUT, int SHIFT>
int launch_pass(PassLaunch& p, const char* label) {
    const int rc = configure_down<OUT, SHIFT>();
    if (rc) return rc;
    uint32_t* total = p.totals + SHIFT / 8 * kB;
    {
        TraceScope ts_("order.up", p.s);
        k_ord_up<SHIFT><<<p.up_blocks, kT, 0, p.s>>>(p.a.bufs, p.a.r, p.cnt, total, p.varies, p.a.status);
    }
    MSC_LAUNCHED();
    {
        TraceScope ts_("order.scan", p.s);
        k_ord_scan<<<kB, kT, 0, p.s>>>(p.a.bufs, SHIFT / 8, p.cnt, total, p.a.r.supers);
    }
    MSC_LAUNCHED();
    p.a.total = total;
    {
        TraceScope ts_(label, p.s);
        k_ord_down<OUT, SHIFT><<<p.down_blocks, kT, kDownSmem, p.s>>>(p.a);
    }
    MSC_LAUNCHED();
    return MSC_OK;
}

// order[id] = position for the pairs the last pass has filed: into the
// buffer after the one it read.
__global__ void __launch_bounds__(kPermuteThreads) k_ord_permute(const Buffers bufs, int64_t n, int32_t* __restrict__ order,
                                                                 int32_t* status) {
    const int b = source_of(bufs, 3) == 0;
    permute_pairs(id_of(bufs, b), key_of(bufs, b), n, b ? bufs.aligned[1] : bufs.aligned[0], order, status);
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

// The whole sort of a small field in one cooperative launch: the sort of
// 2^18 vertices is 16 launches and fills otherwise (125 us, 93 replayed as a
// graph, against 48 here; bound by the latency of the phases, some 10 us per
// pass).  The data stays in L2 between the passes, so the last pass writes
// order[id] = position straight away.  A digit that all keys share (the low
// mantissa bits of small whole numbers) costs its count only.
struct CoopOrderArgs {
    const float* f;
    uint32_t n;
    int32_t* order;
    uint32_t* key[2];
    uint32_t* id[2];
    uint32_t* scratch;  // kCoopScratchWords
    uint32_t* barrier;  // 0 at the start
    int32_t* status;
};

template <int ITEMS>
__global__ void __launch_bounds__(kCoopThreads) k_ord_coop(const CoopOrderArgs a) {
    extern __shared__ __align__(16) uint8_t coop_smem[];
    CoopSmem<uint32_t, ITEMS>& S = *reinterpret_cast<CoopSmem<uint32_t, ITEMS>*>(coop_smem);
    GridBarrier bar{a.barrier, gridDim.x, 0};
    int src = -1;  // the buffer holding the keys; -1: the field
    bool nan = false;
#pragma unroll 1
    for (int p = 0; p < 4; ++p) {
        const bool last = p == 3;
        const uint32_t* kin = src < 0 ? nullptr : a.key[src];
        const uint32_t* vin = src < 0 ? nullptr : a.id[src];
        const int dst = src == 0;
        const CoopPass r = coop_radix_pass<uint32_t, ITEMS>(
            S, a.n, 8 * p, !last,
            [&](uint32_t i) -> uint32_t {
                if (kin) return kin[i];
                const float x = a.f[i];
                nan |= is_nan_bits(x);
                return float_key(x);
            },
            [&](uint32_t i) -> uint32_t { return vin ? vin[i] : i; },
            [&](uint32_t pos, uint32_t k, uint32_t id) {
                if (last) {
                    a.order[id] = (int32_t)pos;
                } else {
                    a.key[dst][pos] = k;
                    a.id[dst][pos] = id;
                }
            },
            a.scratch, bar, a.status);
        if (r == kPassFailed) return;
        if (r == kPassMoved) src = dst;
    }
    if (nan) record_error(a.status, MSC_ERR_NAN);
}

// Tile size of k_ord_coop for n vertices, 0 for a sort by launches.  The
// cooperative sort is the better one while every block holds one tile
// (loaded and ranked once) at two blocks per SM: 10^6 vertices 76 us against
// 116 as launches (86 replayed), 1.24 * 10^6 79 against 116 (89); with two
// tiles per block 1.5 * 10^6 take 131 against 116 (89).  Eight keys per thread
// as long as they fit: 262 144 vertices 46 us, 61 with sixteen.
int coop_tile(int64_t n) {
    const int64_t blocks = 2 * (int64_t)current_device().sms;
    if (n <= blocks * CoopSmem<uint32_t, 8>::kTile) return CoopSmem<uint32_t, 8>::kTile;
    return n <= blocks * CoopSmem<uint32_t, 16>::kTile ? CoopSmem<uint32_t, 16>::kTile : 0;
}
static_assert(kCoopScratchWords + 1 <= kOrderCntWords, "the barrier word follows the counts");

template <int ITEMS>
int launch_coop(const CoopOrderArgs& a, cudaStream_t s) {
    using Smem = CoopSmem<uint32_t, ITEMS>;
    static int configured_dev = -1;
    if (configured_dev != current_device().id) {
        MSC_TRY(cudaFuncSetAttribute(k_ord_coop<ITEMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem)));
        configured_dev = current_device().id;
    }
    int blocks = 0;
    const int r = coop_blocks(k_ord_coop<ITEMS>, kCoopThreads, sizeof(Smem),
                              std::min<int64_t>(ceil_div(a.n, Smem::kTile), kCoopMaxBlocks), s, &blocks);
    if (r) return r;
    TraceScope ts_("order.coop", s);
    return coop_launch(k_ord_coop<ITEMS>, blocks, kCoopThreads, sizeof(Smem), s, a);
}

}  // namespace

int run_order(const float* f, int64_t n, int32_t* order, uint32_t* key_a, int32_t* id_a, uint32_t* key_b,
              int32_t* id_b, const SortScratch& sc, int32_t* status, cudaStream_t s, uint32_t* barrier) {
    if (n <= 0) return MSC_OK;
    if (const int tile = coop_tile(n)) {
        if (!barrier) {
            barrier = sc.ord_cnt + kCoopScratchWords;
            MSC_TRY(cudaMemsetAsync(barrier, 0, sizeof(uint32_t), s));
        }
        const CoopOrderArgs a{f, (uint32_t)n, order, {key_a, key_b},
                              {reinterpret_cast<uint32_t*>(id_a), reinterpret_cast<uint32_t*>(id_b)}, sc.ord_cnt, barrier, status};
        return tile == CoopSmem<uint32_t, 8>::kTile ? launch_coop<8>(a, s) : launch_coop<16>(a, s);
    }
    Range rg;
    rg.n = n;
    rg.tiles = ceil_div(n, kTile);
    rg.per_super = ceil_div(rg.tiles, kOrderMaxSuper);
    rg.supers = (int)ceil_div(rg.tiles, rg.per_super);
    const int sms = current_device().sms;
    int occ = 0;
    {
        int rr = configure_down<kOutSorted, 8>();
        if (rr) return rr;
        MSC_TRY(max_blocks_per_sm(&occ, k_ord_down<kOutSorted, 8>, kT, kDownSmem));
    }
    PassLaunch p{};
    p.down_blocks = (int)std::min<int64_t>(rg.supers, (int64_t)sms * std::max(occ, 1));
    p.up_blocks = (int)std::min<int64_t>(rg.supers, (int64_t)sms * 4);
    p.s = s;
    p.cnt = sc.ord_cnt;
    p.totals = sc.ord_cnt + (size_t)kB * kOrderMaxSuper;
    uint32_t* fill = p.totals + 4 * kB;
    p.varies = fill + kOrderMaxBuckets * kOrderFillStride;
    MSC_TRY(cudaMemsetAsync(p.totals, 0, (4 * kB + kOrderMaxBuckets * kOrderFillStride + 2) * sizeof(uint32_t), s));
    DownArgs& a = p.a;
    a.bufs = Buffers{f, {key_a, key_b}, {id_a, id_b}, p.varies,
                     {aligned16(key_a) && aligned16(id_a), aligned16(key_b) && aligned16(id_b), aligned16(f)}};
    a.r = rg;
    a.base = p.cnt;
    a.status = status;
    a.order = order;
    a.bucket_fill = fill;
    a.bucket_shift = order_bucket_shift(n);
    int r;
    if ((r = launch_pass<kOutSorted, 0>(p, "order.down_first"))) return r;
    if ((r = launch_pass<kOutSorted, 8>(p, "order.down"))) return r;
    if ((r = launch_pass<kOutSorted, 16>(p, "order.down"))) return r;
    if (n <= kOrderDirectMax) return launch_pass<kOutOrder, 24>(p, "order.down_direct");
    if ((r = launch_pass<kOutBuckets, 24>(p, "order.down_last"))) return r;
    {
        TraceScope ts_("order.permute", s);
        k_ord_permute<<<(unsigned)ceil_div(n, kPermuteChunk), kPermuteThreads, 0, s>>>(a.bufs, n, order, status);
    }
    MSC_LAUNCHED();
    return MSC_OK;
}

}  // namespace msc
