// Cooperative kernels: several dependent phases in one launch, with a
// barrier across the grid between them.
//
// A stage of many short passes (the digit passes of a sort of some thousand
// keys, pointer-jumping sweeps that find nothing left to do) is bound by its
// launches, each about 4 us apart on the device and as much on the host; a
// barrier of a resident grid takes about 1.5.  Cooperative launches only:
// the runtime starts such a grid when all of its blocks fit, so every block
// is running while others wait for it.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "radix.cuh"

namespace msc {

constexpr uint32_t kBarrierLimit = 1u << 22;  // polls before a block gives up (seconds)

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// A barrier among `blocks` blocks of a cooperative launch; *count was 0 at
// its start.
struct GridBarrier {
    uint32_t* count;
    uint32_t blocks;
    uint32_t k;  // barriers passed
};

// False in every thread of a block whose wait ran out: the block then has
// to return (the others run out in turn).
__device__ __forceinline__ bool grid_barrier(GridBarrier& g, int32_t* status) {
    __shared__ int s_ok;
    if (g.blocks <= 1) {
        __syncthreads();
        return true;
    }
    ++g.k;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(g.count, 1u);
        const uint32_t want = g.k * g.blocks;
        uint32_t i = 0;
        while (ld_acquire_u32(g.count) < want && i < kBarrierLimit) {
            ++i;
            if (i > 64) __nanosleep(32);
        }
        s_ok = i < kBarrierLimit;
        if (!s_ok) record_give_up(status);
        __threadfence();
    }
    __syncthreads();
    return s_ok != 0;
}

// ----------------------------------------------------------------------------
// LSD radix sort, all passes in one launch: per pass every block counts the
// digit over its run of tiles, one warp per digit scans the blocks' counts,
// and every block ranks its tiles stably and writes them through shared
// memory in runs.

constexpr int kCoopThreads = 256;
constexpr int kCoopWarps = kCoopThreads / kWarp;
constexpr int kCoopMaxBlocks = 512;  // 16 counts per lane in the scan
constexpr int kCoopDirect = 32;      // blocks up to which every block sums the counts itself (64 blocks: 50 us a sort, 46 with the scan)

// Global scratch of a launch: counts [256][kCoopMaxBlocks], totals [256].
constexpr size_t kCoopScratchWords = (size_t)kRadixBins * kCoopMaxBlocks + kRadixBins;

// ITEMS keys per thread: 8 spread a small sort over twice the blocks, 16
// make longer runs.
template <typename KeyT, int ITEMS>
struct CoopSmem {
    static constexpr int kTile = kCoopThreads * ITEMS;
    KeyT keys[kTile];
    uint32_t vals[kTile];
    uint32_t match[kCoopWarps][kRadixBins];  // counting: the warps' histograms; ranking: lanes per digit (all 0 between keys)
    uint16_t wh[kCoopWarps][kRadixBins];     // ranking: keys per digit so far; then each warp's start in the tile
    uint32_t run[kRadixBins];                // next output position of the digit
    uint32_t delta[kRadixBins];
    uint32_t w[8];
};

enum CoopPass { kPassFailed, kPassMoved, kPassSkipped };

// One digit pass over n keys by the blocks 0 .. bar.blocks - 1.  key(i) and
// val(i) give element i; out(pos, key, val) takes an element to its position
// (called with consecutive lanes on consecutive positions of a digit's
// run).  With can_skip, a pass whose keys all share the digit moves nothing.
template <typename KeyT, int ITEMS, typename KeyF, typename ValF, typename OutF>
__device__ __forceinline__ CoopPass coop_radix_pass(CoopSmem<KeyT, ITEMS>& S, uint32_t n, int shift, bool can_skip,
                                                    KeyF key, ValF val, OutF out, uint32_t* scratch, GridBarrier& bar,
                                                    int32_t* status) {
    constexpr int kTile = CoopSmem<KeyT, ITEMS>::kTile;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t G = bar.blocks, b = blockIdx.x;
    const uint32_t tiles = (n + kTile - 1) / kTile, per = (tiles + G - 1) / G;
    const uint32_t t0 = min(tiles, b * per), t1 = min(tiles, t0 + per);
    const bool single = per == 1;  // a tile per block: loaded and ranked once, before the counts are known
    uint32_t* counts = scratch;
    uint32_t* totals = scratch + (size_t)kRadixBins * kCoopMaxBlocks;
    const uint32_t lt = lanemask_lt();
    const int wb = warp * (ITEMS * 32) + lane;
    KeyT k[ITEMS];
    uint32_t v[ITEMS], rk[ITEMS / 2];
    auto load_and_rank = [&](uint32_t tb, int cnt) {
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const int li = wb + 32 * j;
            k[j] = li < cnt ? key(tb + li) : KeyT(0);
            v[j] = li < cnt ? val(tb + li) : 0u;
        }
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint32_t d = (uint32_t)(k[j] >> shift) & 255u;
            const uint32_t r = rank_in_warp(d, wb + 32 * j < cnt, 1u << lane, lt, S.match[warp], S.wh[warp]);
            rk[j / 2] = (j & 1) ? (rk[j / 2] | r << 16) : r;
        }
        __syncthreads();
    };
    auto keys_of = [&](uint32_t t) { return t < t1 ? (int)min((uint32_t)kTile, n - t * kTile) : 0; };
#pragma unroll
    for (int w = 0; w < kCoopWarps; ++w) {
        S.match[w][tid] = 0;
        S.wh[w][tid] = 0;
    }
    __syncthreads();
    uint32_t mine = 0;  // this block's keys of digit tid
    if (single) {
        load_and_rank(t0 * kTile, keys_of(t0));
#pragma unroll
        for (int w = 0; w < kCoopWarps; ++w) mine += S.wh[w][tid];
    } else {
        constexpr int kStep = kCoopThreads * kHistRun;
        for (uint32_t i0 = t0 * kTile + tid * kHistRun; i0 < min(n, t1 * kTile); i0 += kStep) {
            KeyT x[kHistRun];
            const int cnt = (int)min((uint32_t)kHistRun, min(n, t1 * kTile) - i0);
#pragma unroll
            for (int j = 0; j < kHistRun; ++j) x[j] = j < cnt ? key(i0 + j) : KeyT(0);
            count_runs_at(x, cnt, shift, S.match[warp]);
        }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kCoopWarps; ++w) {
            mine += S.match[w][tid];
            S.match[w][tid] = 0;
        }
    }
    uint32_t before = 0, tot = mine;  // keys of digit tid in earlier blocks, in all
    if (G > 1) {
        counts[(size_t)tid * kCoopMaxBlocks + b] = mine;
        if (!grid_barrier(bar, status)) return kPassFailed;
        if (G <= (uint32_t)kCoopDirect) {
            const uint4* row = reinterpret_cast<const uint4*>(counts + (size_t)tid * kCoopMaxBlocks);
            tot = 0;
#pragma unroll
            for (int j = 0; j < kCoopDirect / 4; ++j) {
                if (4 * j >= (int)G) break;
                const uint4 c = __ldcg(row + j);  // entries past the blocks are not counted
                const uint32_t x[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (4 * j + q < (int)G) tot += x[q];
                    if (4 * j + q < (int)b) before += x[q];
                }
            }
        } else {
            // one warp per digit: exclusive positions of the blocks within the digit
            for (uint32_t d = b * kCoopWarps + warp; d < (uint32_t)kRadixBins; d += G * kCoopWarps) {
                uint32_t* row = counts + (size_t)d * kCoopMaxBlocks;
                constexpr int kPer = kCoopMaxBlocks / 32;
                uint32_t x[kPer], run = 0;
#pragma unroll
                for (int j = 0; j < kPer; ++j) x[j] = j * 32 + lane < (int)G ? __ldcg(row + j * 32 + lane) : 0u;
#pragma unroll
                for (int j = 0; j < kPer; ++j) {
                    if (j * 32 >= (int)G) break;
                    uint32_t incl = x[j];
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t q = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += q;
                    }
                    if (j * 32 + lane < (int)G) row[j * 32 + lane] = run + incl - x[j];
                    run += __shfl_sync(0xffffffffu, incl, 31);
                }
                if (lane == 0) totals[d] = run;
            }
            if (!grid_barrier(bar, status)) return kPassFailed;
            tot = __ldcg(totals + tid);
            before = __ldcg(counts + (size_t)tid * kCoopMaxBlocks + b);
        }
    }
    // (the next pass writes counts that another block may still be reading
    // only if this one ended with a barrier)
    if (__syncthreads_or(tot == n) && can_skip) {
        if (G > 1 && G <= (uint32_t)kCoopDirect && !grid_barrier(bar, status)) return kPassFailed;
        return kPassSkipped;
    }
    S.run[tid] = before + block_scan_256(tot, S.w) - tot;
    __syncthreads();
    for (uint32_t t = t0; t < t1; ++t) {
        const int cnt = keys_of(t);
        if (!single) load_and_rank(t * kTile, cnt);
        {
            uint32_t pre[kCoopWarps], sum = 0;
#pragma unroll
            for (int w = 0; w < kCoopWarps; ++w) {
                pre[w] = sum;
                sum += S.wh[w][tid];
            }
            const uint32_t excl = block_scan_256(sum, S.w) - sum;
#pragma unroll
            for (int w = 0; w < kCoopWarps; ++w) S.wh[w][tid] = (uint16_t)(excl + pre[w]);
            const uint32_t g = S.run[tid];
            S.delta[tid] = g - excl;
            S.run[tid] = g + sum;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            if (wb + 32 * j < cnt) {
                const uint32_t d = (uint32_t)(k[j] >> shift) & 255u;
                const uint32_t at = S.wh[warp][d] + ((rk[j / 2] >> (16 * (j & 1))) & 0xffffu);
                S.keys[at] = k[j];
                S.vals[at] = v[j];
            }
        }
        __syncthreads();
        for (int i = tid; i < cnt; i += kCoopThreads) {
            const KeyT kk = S.keys[i];
            out(S.delta[(uint32_t)(kk >> shift) & 255u] + (uint32_t)i, kk, S.vals[i]);
        }
#pragma unroll
        for (int w = 0; w < kCoopWarps; ++w) S.wh[w][tid] = 0;
        __syncthreads();
    }
    return grid_barrier(bar, status) ? kPassMoved : kPassFailed;
}

// ----------------------------------------------------------------------------
// host side

// Blocks of a cooperative launch on a stream: at most `want`, all resident at
// once on the SMs that the stream has.
template <typename K>
int coop_blocks(K kernel, int threads, size_t smem, int64_t want, cudaStream_t s, int* out) {
    int occ = 0;
    MSC_TRY(max_blocks_per_sm(&occ, kernel, threads, smem));
    if (occ < 1) return MSC_ERR_CUDA;
    *out = (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)stream_sms(s) * occ));
    return MSC_OK;
}

// The kernels here run on any number of blocks: a grid that the runtime finds
// too large all the same is halved until it fits.  (While a stream is being
// captured the launch is not where the size is judged: coop_blocks has to be
// right.)
template <typename... P, typename... A>
int coop_launch(void (*kernel)(P...), int blocks, int threads, size_t smem, cudaStream_t s, const A&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    for (;; blocks /= 2) {
        cfg.gridDim = dim3((unsigned)blocks);
        const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
        if (e == cudaSuccess) return MSC_OK;
        cudaGetLastError();
        if (e != cudaErrorCooperativeLaunchTooLarge || blocks <= 1) return MSC_ERR_CUDA;
    }
}

}  // namespace msc
