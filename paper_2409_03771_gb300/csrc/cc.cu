// Connected components with smallest-id labels: feature mask on a grid
// (6- or 14-connectivity) and explicit mesh adjacency (CSR).
//
// The paper (Alg. 3) points every feature vertex at its largest feature
// neighbour, compresses, hooks segment roots across segment borders
// ("d[d[v]] <- d[u]") and compresses again, first per rank and then across
// ranks.  Here the same local-then-global structure is applied to GPU
// tiles, mirrored to the smallest id, with the hooking made exact by a
// union-find on roots (hook the larger root under the smaller with
// atomicMin; retry if another thread moved it first):
//   1. k_cc_local: a 64x8x8 tile of the mask as 64 row bitmasks in shared
//      memory, x-runs labelled by bit arithmetic, runs of neighbouring rows
//      united once per overlap segment, each feature voxel written with
//      the global id of its tile-local root (the smallest id of its
//      tile-local component), -1 elsewhere;
//   2. k_cc_merge: the contacts that leave a tile through its +x, +y or +z
//      side, found on row bitmasks again and thinned to one per patch of
//      contact, unite the two roots in global memory (path halving);
//   3. k_cc_flatten: the masked voxels jump to their final root.
// The final root of a component is its smallest vertex id because every
// hook points a root at a smaller one.
//
// Mesh: union-find over the CSR edges with subgraph sampling (see the mesh
// kernels below).
#include <cuda_runtime.h>

#include <algorithm>

#include "cc.cuh"

namespace msc {
namespace {

#ifndef MSC_CC_LOCAL_MIN_BLOCKS
#define MSC_CC_LOCAL_MIN_BLOCKS 6
#endif
constexpr int CX = 64, CY = 8, CZ = 8;
constexpr int CT = CX * CY * CZ;  // 4096
constexpr int kThreads = 256;
constexpr uint32_t kUnionLimit = 1u << 20;

struct CcGrid {
    int32_t nx, ny, nz;
    int32_t tx, ty;
    int64_t ntiles;
    int conn;
    int64_t n;
};

// Root of x in a shared-memory forest whose entries point at smaller
// local indices, halving the path on the way (atomicMin: never undoes a
// hook made by another thread).
__device__ __forceinline__ int find_s(int* L, int x) {
    int p = L[x];
    while (p != x) {
        const int gp = L[p];
        if (gp == p) return p;
        atomicMin(&L[x], gp);
        x = gp;
        p = L[x];
    }
    return x;
}

// Both ends climb together until they meet or are both roots.
__device__ __forceinline__ void union_s(int* L, int a, int b) {
    for (int it = 0; it < CT * 4; ++it) {
        // both ends climb together until they meet or are both roots
        for (;;) {
            const int pa = L[a], pb = L[b];
            if (pa == pb) return;
            if (pa == a && pb == b) break;
            const int ga = L[pa], gb = L[pb];
            if (ga != pa) atomicMin(&L[a], ga);
            if (gb != pb) atomicMin(&L[b], gb);
            a = ga;
            b = gb;
        }
        if (a > b) {
            const int t = a;
            a = b;
            b = t;
        }
        const int old = atomicMin(&L[b], a);
        if (old == b) return;
        b = old;
    }
}

// Root of x in global memory, halving the path on the way.  The halving
// write is an atomicMin: labels only ever decrease (every entry points at a
// smaller or equal id of the same component), so a halving write can never
// undo a hook or overwrite a final root written by another thread.
// Cached reads: once most vertices share a root, nearly every find ends at
// its word, and reads that all go to one L2 slice serialise (mesh of 256^3
// vertices: 1.36 ms for uniting the second neighbours, 0.37 with the L1
// serving them).  A
// stale read is an older ancestor of the same component; a union that took
// it for a root learns the present value from its atomicMin and goes on from
// there.
__device__ __forceinline__ int32_t find_g(int32_t* L, int32_t x) {
    for (uint32_t it = 0; it < kUnionLimit; ++it) {
        const int32_t p = ld_cached_s32(L + x);
        if (p == x) return x;
        const int32_t gp = ld_cached_s32(L + p);
        if (gp != p) atomicMin(L + x, gp);
        x = gp;
    }
    return x;
}

__device__ __forceinline__ void union_g(int32_t* L, int32_t a, int32_t b, int32_t* status) {
    for (uint32_t it = 0; it < kUnionLimit; ++it) {
        a = find_g(L, a);
        b = find_g(L, b);
        if (a == b) return;
        if (a > b) {
            const int32_t t = a;
            a = b;
            b = t;
        }
        const int32_t old = atomicMin(L + b, a);
        if (old == b) return;
        b = old;  // below b, fresh from L2
    }
    record_error(status, MSC_ERR_INTERNAL);
}

// The same, both ends climbing together until they meet or are both roots:
// half the round trips where both paths have a few steps, as between the
// tiles of a noisy mask.
__device__ __forceinline__ void union_g_together(int32_t* L, int32_t a, int32_t b, int32_t* status) {
    for (uint32_t it = 0; it < kUnionLimit; ++it) {
        for (uint32_t hop = 0; hop < kUnionLimit; ++hop) {
            const int32_t pa = ld_cached_s32(L + a), pb = ld_cached_s32(L + b);
            if (pa == pb) return;
            if (pa == a && pb == b) break;
            const int32_t ga = ld_cached_s32(L + pa), gb = ld_cached_s32(L + pb);
            if (ga != pa) atomicMin(L + a, ga);
            if (gb != pb) atomicMin(L + b, gb);
            a = ga;
            b = gb;
        }
        if (a > b) {
            const int32_t t = a;
            a = b;
            b = t;
        }
        const int32_t old = atomicMin(L + b, a);
        if (old == b) return;
        b = old;  // below b, fresh from L2
    }
    record_error(status, MSC_ERR_INTERNAL);
}

// Eight mask bytes as eight bits: bit j set iff byte j is nonzero and
// j < valid.  Rows of any alignment load whole 4-byte words, shifted into
// place; only words wholly inside the mask are loaded, the few bytes at its
// two ends come one by one.
__device__ __forceinline__ uint32_t nonzero_bits(uint32_t lo, uint32_t hi) {
    // high bit of each byte set iff the byte is nonzero; then the four high
    // bits gathered into bits 28..31
    lo = (lo | ((lo & 0x7f7f7f7fu) + 0x7f7f7f7fu)) & 0x80808080u;
    hi = (hi | ((hi & 0x7f7f7f7fu) + 0x7f7f7f7fu)) & 0x80808080u;
    return ((lo * 0x00204081u) >> 28) | (((hi * 0x00204081u) >> 28) << 4);
}

template <bool MASK8>
__device__ __forceinline__ uint32_t mask_bits8(const uint8_t* __restrict__ mask, const CcGrid& g, int64_t off, int valid) {
    if (valid <= 0) return 0u;
    if (MASK8) {  // valid is at least 8: nx is a multiple of 8
        const uint2 w = __ldg(reinterpret_cast<const uint2*>(mask + off));
        return nonzero_bits(w.x, w.y);
    }
    const int sh = (int)((uintptr_t)(mask + off) & 3);
    const int64_t w = off - sh;
    uint32_t bits = 0;
    if (w >= 0 && w + 12 <= g.n) {
        const uint32_t* p = reinterpret_cast<const uint32_t*>(mask + w);
        const uint32_t p0 = __ldg(p), p1 = __ldg(p + 1), p2 = __ldg(p + 2);
        bits = nonzero_bits(__funnelshift_r(p0, p1, 8 * sh), __funnelshift_r(p1, p2, 8 * sh));
    } else {
#pragma unroll 1
        for (int j = 0; j < min(valid, 8); ++j)
            if (mask[off + j]) bits |= 1u << j;
    }
    return bits & (0xffu >> (8 - min(valid, 8)));
}

// Tile-local labelling, run based.  Rows are x-lines of 64 voxels, one
// 64-bit mask each.  Only the first voxel of an x-run has an entry in the
// shared forest; runs of neighbouring rows are united once per overlap
// segment (a maximal x-range where both rows' voxels are masked); then every
// voxel takes its run's root.  A diagonal contact is united only where no
// voxel on the way between its two ends is masked: otherwise edges with fewer
// steps already join them.  Bound: the label store (4 of 5 bytes per voxel);
// an empty tile stores its -1s straight after the rows are read.
// 1024^3, top 10 % of a blob field: 1.71 -> 1.04 ms (its 5.4 GB take 0.79 at the copy rate).
// Noisy masks are bound by the unions instead (a thousand contacts per tile,
// divergent finds): 512^3, half of the voxels set at random, 1.11 ms with 6
// neighbours, 1.62 with 14; with the ends' finds one after the other and run
// starts from four 64-bit shifts 1.55 and 2.27.
constexpr int kRows = CY * CZ;  // 64 rows of CX = 64 voxels

__device__ __forceinline__ uint64_t run_starts(uint64_t m) { return m & ~(m << 1); }

// First voxel of the run that holds x: the last of the row's starts up to x.
__device__ __forceinline__ int run_start(uint64_t starts, int x) { return x - __clzll((long long)(starts << (63 - x))); }

// Contacts of a row (m00) with the rows one step in y (m10), z (m01) or
// both (m11) away, where the row's voxel x meets the other row's voxel x
// (straight) or x + 1 (the s.. masks are the rows shifted down by one).
__device__ __forceinline__ uint64_t contact_x(uint64_t m, uint64_t m2, uint64_t sm, uint64_t sm2) {
    return m & sm2 & ~m2 & ~sm;  // (1,1,0), (1,0,1)
}
__device__ __forceinline__ uint64_t contact_yz(uint64_t m00, uint64_t m10, uint64_t m01, uint64_t m11) {
    return m00 & m11 & ~m10 & ~m01;  // (0,1,1)
}
__device__ __forceinline__ uint64_t contact_xyz(uint64_t m00, uint64_t m10, uint64_t m01, uint64_t m11, uint64_t s00,
                                                uint64_t s10, uint64_t s01, uint64_t s11) {
    return m00 & s11 & ~(s00 | m11 | m10 | m01 | s10 | s01);  // (1,1,1)
}

// MASK8: nx is a multiple of 8 and the mask 8-byte aligned.
template <bool MASK8>
__global__ void __launch_bounds__(kThreads, MSC_CC_LOCAL_MIN_BLOCKS) k_cc_local(const uint8_t* __restrict__ mask, const CcGrid g,
                                                       int32_t* __restrict__ label, int32_t* status) {
    __shared__ int s_l[CT];
    __shared__ int32_t s_first[kRows];  // vertex id of each row's first voxel (unused rows may wrap)
    __shared__ uint64_t s_rows[2][kRows];  // the next tile's rows may be read while this one's are in use
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (blockIdx.x == 0 && tid == 0) *status = MSC_OK;  // the merge comes after this kernel
    int slot = 0;
    const int64_t nxy = (int64_t)g.nx * g.ny;
    TileWalk tile(g.tx, g.ty, blockIdx.x, gridDim.x);
    for (int64_t t = blockIdx.x; t < g.ntiles; t += gridDim.x, tile.advance(), slot ^= 1) {
        uint64_t* s_row = s_rows[slot];
        const int x0 = tile.x * CX, y0 = tile.y * CY, z0 = tile.z * CZ;
        const int64_t tbase = x0 + (int64_t)g.nx * y0 + nxy * z0;
        // the 64 row bitmasks: 8 lanes per row, 8 mask bytes per lane
        uint32_t any = 0;
        {
            const int sub = lane & 7, r = warp * 4 + (lane >> 3), ly = r & (CY - 1), lz = r / CY;
            const int64_t off = tbase + 8 * sub + (int64_t)g.nx * ly + nxy * lz;
            const int valid = y0 + ly < g.ny ? g.nx - x0 - 8 * sub : 0;
            const uint32_t b0 = mask_bits8<MASK8>(mask, g, off, z0 + lz < g.nz ? valid : 0);
            const uint32_t b1 = mask_bits8<MASK8>(mask, g, off + 4 * nxy, z0 + lz + 4 < g.nz ? valid : 0);
            reinterpret_cast<uint8_t*>(s_row)[8 * r + sub] = (uint8_t)b0;
            reinterpret_cast<uint8_t*>(s_row)[8 * (r + 32) + sub] = (uint8_t)b1;
            any = b0 | b1;
        }
        const bool some = __syncthreads_or(any != 0);
        if (some) {  // block-uniform
            if (tid < kRows) s_first[tid] = x0 + g.nx * (y0 + (tid & (CY - 1)) + g.ny * (z0 + tid / CY));
            {   // run starts (four threads per row, a quarter of the row each)
                const int r = tid >> 2, q = tid & 3;
                const uint64_t m = s_row[r];
                uint64_t st = m & ~(m << 1) & (0xffffull << (16 * q));
                while (st) {
                    const int i = __ffsll((long long)st) - 1 + CX * r;
                    st &= st - 1;
                    s_l[i] = i;
                }
            }
            __syncthreads();
            // unite runs of neighbouring rows: a quarter of the threads per
            // direction, a thread per row
            {
                const int r = tid & (kRows - 1), dir = tid / kRows;  // y step, z step, both, both to x + 1
                const bool oy = (r & (CY - 1)) == CY - 1, oz = r / CY == CZ - 1;
                const int step = dir == 0 ? 1 : dir == 1 ? CY : CY + 1;
                if (!((dir != 1 && oy) || (dir != 0 && oz)) && (dir < 2 || g.conn == 14)) {
                    const uint64_t m = s_row[r], m2 = s_row[r + step];
                    uint64_t o = m & m2;
                    int dx = 0;
                    if (dir >= 2) {
                        const uint64_t m10 = s_row[r + 1], m01 = s_row[r + CY];
                        dx = dir == 3;
                        o = dx ? contact_xyz(m, m10, m01, m2, m >> 1, m10 >> 1, m01 >> 1, m2 >> 1)
                               : contact_yz(m, m10, m01, m2);
                    }
                    const uint64_t st = run_starts(m), st2 = run_starts(m2);
                    auto unite = [&](uint64_t contacts, int to) {
                        for (uint64_t seg = contacts & ~(contacts << 1); seg; seg &= seg - 1) {
                            const int x = __ffsll((long long)seg) - 1;
                            union_s(s_l, run_start(st, x) + CX * r, run_start(st2, x + to) + CX * (r + step));
                        }
                    };
                    unite(o, dx);
                    if (dir < 2 && g.conn == 14) unite(contact_x(m, m2, m >> 1, m2 >> 1), 1);
                }
            }
            __syncthreads();
            {   // every run start takes its root
                const int r = tid >> 2, q = tid & 3;
                const uint64_t m = s_row[r];
                uint64_t st = m & ~(m << 1) & (0xffffull << (16 * q));
                while (st) {
                    const int i = __ffsll((long long)st) - 1 + CX * r;
                    st &= st - 1;
                    s_l[i] = find_s(s_l, i);
                }
            }
            __syncthreads();
        }
        // 16 threads per row, four consecutive voxels each, starting `sh`
        // before a multiple of four so that the label words are 16-byte
        // aligned whatever the row's address; thread 0's first sh voxels wrap
        // around to the row's end
        const int i = tid & 15, ly = (tid >> 4) & (CY - 1);
        int32_t* dst = label + tbase + (int64_t)g.nx * ly + nxy * (tid >> 7);
#pragma unroll
        for (int pass = 0; pass < kRows / 16; ++pass, dst += 2 * nxy) {
            const int r = (tid >> 4) + 16 * pass;
            if (y0 + ly >= g.ny || z0 + r / CY >= g.nz) continue;
            const int sh = (int)((uintptr_t)dst >> 2) & 3, x = 4 * i - sh;
            int32_t id[4] = {-1, -1, -1, -1};
            if (some) {
                const uint64_t m = s_row[r];
                const uint32_t q = (uint32_t)((sh ? m << sh | m >> (64 - sh) : m) >> (4 * i)) & 15u;
                const uint32_t low = q & (0u - q);
                if (q && x >= 0 && !(q & (q + low))) {  // one run (nearly always)
                    const int l = s_l[run_start(run_starts(m), x + __ffs(q) - 1) + CX * r];
                    const int32_t cur = s_first[l / CX] + (l & (CX - 1));
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (q >> j & 1u) id[j] = cur;
                } else if (q) {
                    // several runs: a voxel starts its own unless the one before it is masked
                    int st[4], l[4];
                    st[0] = q & 1u ? run_start(run_starts(m), x & (CX - 1)) : 0;
#pragma unroll
                    for (int j = 1; j < 4; ++j) st[j] = (q >> (j - 1) & 1u) && x + j != 0 ? st[j - 1] : (x + j) & (CX - 1);
#pragma unroll
                    for (int j = 0; j < 4; ++j) l[j] = q >> j & 1u ? s_l[st[j] + CX * r] : 0;
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (q >> j & 1u) id[j] = s_first[l[j] / CX] + (l[j] & (CX - 1));
                }
            }
            if (x >= 0 && x0 + x + 3 < g.nx) {
                *reinterpret_cast<int4*>(dst + x) = make_int4(id[0], id[1], id[2], id[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int xj = (x + j) & (CX - 1);
                    if (x0 + xj < g.nx) dst[xj] = id[j];
                }
            }
        }
    }
}

// A warp per tile: the bitmasks of the tile's rows and of the rows one step
// beyond its +y and +z sides (9 x 9 rows of 64 voxels plus the voxel beyond
// the +x side) go to shared memory, and the contacts that leave the tile come
// from bit operations, thinned so that two components meeting across a face
// are mostly united once: of a face's contacts only those with no contact
// before them in the row or in the row before (both sides' voxels are then
// joined within their tiles), and diagonals only where no voxel between the
// ends is masked.  A tile without a masked voxel is done once its rows are
// read.  Bound: instructions of the row reading, and L2 latency of the
// unions.  1024^3, top 10 % of a blob field: 1.73 -> 0.44 ms; with
// labels compared voxel by voxel the faces cost 1.2 warp instructions per voxel
// of the grid.
constexpr int kHaloRows = (CY + 1) * (CZ + 1);  // 81, row y + 9 z
constexpr int kMergeWarps = 8;
constexpr uint32_t kMergeQueue = 256;  // contacts of a tile held before they are united

// Unites the tile-local roots of the two ends of a contact: x, y, z of the
// voxel in the tile and the offset, packed.
template <bool FEW>
__device__ __forceinline__ void merge_contact(int32_t* label, const CcGrid& g, int64_t tbase, uint32_t c, int32_t* status) {
    const int64_t nxy = (int64_t)g.nx * g.ny;
    const int64_t v = tbase + (c & 63) + (int64_t)g.nx * (c >> 6 & 7) + nxy * (c >> 9 & 7);
    const int64_t u = v + (c >> 12 & 1) + (int64_t)g.nx * (c >> 13 & 1) + nxy * (c >> 14 & 1);
    const int32_t a = ld_volatile_s32(label + v), b = ld_volatile_s32(label + u);
    if (a == b) return;
    if (FEW) union_g_together(label, a, b, status);
    else union_g(label, a, b, status);
}

// FEW: at most one tile per resident warp, so the round trips of a tile's
// unions are what the kernel takes (90^3, half of the voxels set at random: 32 ->
// 28 us with 6 neighbours).  Larger grids read rows of one tile under the
// unions of others, and the second climb's code costs the reading more than
// it saves (1024^3, top 10 %: 425 -> 447 us).
template <bool MASK8, bool FEW>
__global__ void __launch_bounds__(kMergeWarps * 32, 4) k_cc_merge(const uint8_t* __restrict__ mask, const CcGrid g,
                                                               int32_t* label, int32_t* status) {
    __shared__ uint64_t s_rows[kMergeWarps][kHaloRows];
    __shared__ uint8_t s_next[kMergeWarps][kHaloRows];  // the voxel at x0 + 64
    __shared__ uint16_t s_queue[kMergeWarps][kMergeQueue];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t* rows = s_rows[warp];
    uint8_t* next = s_next[warp];
    uint16_t* queue = s_queue[warp];
    const int64_t nxy = (int64_t)g.nx * g.ny;
    const uint32_t first = blockIdx.x * kMergeWarps + warp, step = gridDim.x * kMergeWarps;
    TileWalk tile(g.tx, g.ty, first, step);
    for (int64_t t = first; t < g.ntiles; t += step, tile.advance()) {
        const int x0 = tile.x * CX, y0 = tile.y * CY, z0 = tile.z * CZ;
        const int64_t tbase = x0 + (int64_t)g.nx * y0 + nxy * z0;
        const int sub = lane & 7;
        auto row_bits = [&](int ly, int lz) -> uint32_t {
            const int valid = y0 + ly < g.ny && z0 + lz < g.nz ? g.nx - x0 - 8 * sub : 0;
            return mask_bits8<MASK8>(mask, g, tbase + 8 * sub + (int64_t)g.nx * ly + nxy * lz, valid);
        };
        // own rows: 8 lanes per row, 4 rows per step
        uint32_t any = 0;
#pragma unroll (MASK8 ? 16 : 4)
        for (int i = 0; i < kRows / 4; ++i) {
            const int r = 4 * i + (lane >> 3), ly = r & (CY - 1), lz = r / CY;
            const uint32_t bits = row_bits(ly, lz);
            reinterpret_cast<uint8_t*>(rows)[8 * (ly + 9 * lz) + sub] = (uint8_t)bits;
            any |= bits;
        }
        if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
        for (int i = 0; i < 5; ++i) {  // the 17 rows beyond the sides: y = 8 for z 0..8, then z = 8 for y 0..7
            const int r = 4 * i + (lane >> 3);
            if (r < 17) {
                const int ly = r < 9 ? CY : r - 9, lz = r < 9 ? r : CZ;
                reinterpret_cast<uint8_t*>(rows)[8 * (ly + 9 * lz) + sub] = (uint8_t)row_bits(ly, lz);
            }
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int r = lane + 32 * i;
            if (r < kHaloRows) {
                const int ly = r % 9, lz = r / 9;
                const bool in = x0 + CX < g.nx && y0 + ly < g.ny && z0 + lz < g.nz;
                next[r] = in && __ldg(mask + tbase + CX + (int64_t)g.nx * ly + nxy * lz) != 0;
            }
        }
        __syncwarp();
        // +x face crossings as bit y + 8 z, thinned to the first of each patch
        uint64_t xheads;
        {
            const int ra = (lane & 7) + 9 * (lane >> 3);
            const uint32_t xa = __ballot_sync(0xffffffffu, (rows[ra] >> 63) && next[ra]);
            const uint32_t xb = __ballot_sync(0xffffffffu, (rows[ra + 36] >> 63) && next[ra + 36]);
            const uint64_t X = (uint64_t)xb << 32 | xa;
            xheads = X & ~((X & 0x7f7f7f7f7f7f7f7full) << 1) & ~(X << 8);
        }
        // each lane's contacts, kind by kind, into the queue; all lanes unite what it holds
        const int kinds = g.conn == 6 ? 3 : 11;
        uint32_t total = 0;
        auto drain = [&](uint32_t count) {
            __syncwarp();
            for (uint32_t i = lane; i < count; i += 32) merge_contact<FEW>(label, g, tbase, queue[i], status);
            __syncwarp();
        };
#pragma unroll 1
        for (int kind = 0; kind < kinds; ++kind) {
            uint64_t seg = 0;
            uint32_t c = 0;  // code of the contact but for x
            if (kind == 0) {  // +z face rows (lanes 0..7) and +y face rows (8..15)
                if (lane < 16) {
                    const bool zface = lane < 8;
                    const int i = lane & 7;
                    const int ly = zface ? i : CY - 1, lz = zface ? CZ - 1 : i;
                    const int r = ly + 9 * lz, step = zface ? 9 : 1, back = zface ? 1 : 9;
                    const uint64_t o = rows[r] & rows[r + step];
                    const uint64_t before = i > 0 ? rows[r - back] & rows[r - back + step] : 0ull;
                    // a segment that touches one of the row before is joined to it on both sides
                    for (uint64_t left = o & ~(o << 1); left; left &= left - 1) {
                        const uint64_t head = left & (~left + 1);
                        if (!(((o + head) ^ o) & o & before)) seg |= head;
                    }
                    c = ly << 6 | lz << 9 | (zface ? 1u << 14 : 1u << 13);
                }
            } else if (kind < 3) {
                const int i = lane + 32 * (kind - 1);
                seg = (xheads >> i & 1ull) << 63;
                c = (i & 7) << 6 | (i >> 3) << 9 | 1u << 12;
            } else {
                const int ly = lane & 7, lz = (lane >> 3) + (kind < 7 ? 0 : 4), r = ly + 9 * lz, d = (kind - 3) & 3;
                const uint64_t m00 = rows[r], m10 = rows[r + 1], m01 = rows[r + 9], m11 = rows[r + 10];
                auto shifted = [&](uint64_t m, int i) { return (m >> 1) | ((uint64_t)next[i] << 63); };
                const uint64_t s00 = shifted(m00, r), s10 = shifted(m10, r + 1), s01 = shifted(m01, r + 9),
                               s11 = shifted(m11, r + 10);
                // a contact leaves the tile through y or z, or else only at x = 63
                const bool oy = ly == CY - 1, oz = lz == CZ - 1;
                uint64_t o;
                if (d == 0) o = contact_x(m00, m10, s00, s10) & (oy ? ~0ull : 1ull << 63);
                else if (d == 1) o = contact_x(m00, m01, s00, s01) & (oz ? ~0ull : 1ull << 63);
                else if (d == 2) o = oy || oz ? contact_yz(m00, m10, m01, m11) : 0ull;
                else o = contact_xyz(m00, m10, m01, m11, s00, s10, s01, s11) & (oy || oz ? ~0ull : 1ull << 63);
                seg = o & ~(o << 1);
                c = ly << 6 | lz << 9 | (d == 0 ? 3u : d == 1 ? 5u : d == 2 ? 6u : 7u) << 12;
            }
            for (uint32_t act; (act = __ballot_sync(0xffffffffu, seg != 0ull)) != 0u; seg &= seg - 1) {
                if (total + 32 > kMergeQueue) {  // isolated voxels on both sides of the faces
                    drain(total);
                    total = 0;
                }
                if (seg) queue[total + __popc(act & lanemask_lt())] = (uint16_t)(c | (uint32_t)(__ffsll((long long)seg) - 1));
                total += __popc(act);
            }
        }
        drain(total);
    }
}

// The masked voxels jump to their roots.  A block reads kFlatChunk mask
// bytes, lists the quads of four voxels that hold any, and spreads the
// quads over its threads: labels are read only where the mask is set, all
// lanes have work, and of neighbours with one label only the first walks its
// chain.  Once every union is done the root reached is the component
// minimum, so a plain store of it cannot lose anything, and a label read
// stale is still an ancestor of the voxel.  Bound: reading the mask, and the
// labels where it is set.  1024^3, top 10 %: 1.02 (reading every label) ->
// 0.43 ms; a thread following its own eight voxels took 0.90 ms (too few
// bytes in flight, most lanes idle).
constexpr int kFlatBytes = 32;  // mask bytes per thread
constexpr int kFlatChunk = kThreads * kFlatBytes;

// Voxels v .. v + 3, of which some are masked.
__device__ __forceinline__ void flatten_quad(int32_t* label, int64_t v, int64_t n, int label16) {
    const bool whole = label16 && v + 4 <= n;
    int32_t l[4], r[4];
    if (whole) {
        const int4 x = *reinterpret_cast<const int4*>(label + v);
        l[0] = x.x, l[1] = x.y, l[2] = x.z, l[3] = x.w;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) l[j] = v + j < n ? label[v + j] : -1;
    }
    uint32_t open = 0, moved = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        r[j] = l[j];
        open |= (l[j] >= 0 && (j == 0 || l[j] != l[j - 1]) ? 1u : 0u) << j;
    }
    for (uint32_t it = 0; it < kUnionLimit && open; ++it) {  // bound only: chains are short
        int32_t up[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) up[j] = open >> j & 1u ? label[r[j]] : 0;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (open >> j & 1u) {
                if (up[j] == r[j]) open &= ~(1u << j);
                else {
                    r[j] = up[j];
                    moved |= 1u << j;
                }
            }
    }
    if (!moved) return;
#pragma unroll
    for (int j = 1; j < 4; ++j)
        if (l[j] == l[j - 1]) r[j] = r[j - 1];
    if (whole) {
        *reinterpret_cast<int4*>(label + v) = make_int4(r[0], r[1], r[2], r[3]);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (r[j] != l[j]) label[v + j] = r[j];
    }
}

// A small mask: a quad per thread, as chunks would leave most of the GPU
// without a block (48^3: fourteen of them).  48^3, half set: 14 -> 6 us; 128^3: 15
// -> 9.  Beyond, dense masks gain and sparse ones lose (203 x 150 x 177, 2 %
// set: the call 88 -> 92 us).
constexpr int64_t kFlatSmall = 1 << 21;

__global__ void __launch_bounds__(kThreads) k_cc_flatten_small(const uint8_t* __restrict__ mask, int64_t n, int mask4,
                                                               int label16, int32_t* label) {
    const int64_t v = 4 * ((int64_t)blockIdx.x * kThreads + threadIdx.x);
    uint32_t any = 0;
    if (mask4 && v + 4 <= n) {
        any = __ldg(reinterpret_cast<const uint32_t*>(mask + v));
    } else {
        for (int64_t u = v; u < min(n, v + 4); ++u) any |= mask[u];
    }
    if (any) flatten_quad(label, v, n, label16);
}

__global__ void __launch_bounds__(kThreads) k_cc_flatten(const uint8_t* __restrict__ mask, int64_t n, int mask16, int label16,
                                                         int32_t* label) {
    __shared__ uint16_t s_quad[kFlatChunk / 4];
    __shared__ uint32_t s_count;
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t stride = (int64_t)gridDim.x * kFlatChunk;
    // word h of thread tid: 16 mask bytes at (h * kThreads + tid) * 16 of the chunk
    auto load = [&](int64_t c0, uint4 (&w)[2]) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t v = c0 + (int64_t)(h * kThreads + tid) * 16;
            w[h] = make_uint4(0u, 0u, 0u, 0u);
            if (mask16 && v + 16 <= n) {
                w[h] = __ldg(reinterpret_cast<const uint4*>(mask + v));
            } else {
                uint32_t q[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll 1
                    for (int k = 0; k < 4; ++k)
                        if (v + 4 * j + k < n) q[j] |= mask[v + 4 * j + k];
                w[h] = make_uint4(q[0], q[1], q[2], q[3]);
            }
        }
    };
    int64_t c0 = (int64_t)blockIdx.x * kFlatChunk;
    uint4 w[2];
    if (c0 < n) load(c0, w);
    for (; c0 < n; c0 += stride) {
        if (tid == 0) s_count = 0;
        __syncthreads();
        const uint32_t word[8] = {w[0].x, w[0].y, w[0].z, w[0].w, w[1].x, w[1].y, w[1].z, w[1].w};
        uint32_t set = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) set |= (word[k] ? 1u : 0u) << k;
        const uint32_t cnt = __popc(set);
        uint32_t incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        uint32_t base = 0;
        if (lane == 31 && incl) base = atomicAdd(&s_count, incl);
        uint32_t at = __shfl_sync(0xffffffffu, base, 31) + incl - cnt;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (set >> k & 1u) s_quad[at++] = (uint16_t)(((k >> 2) * kThreads + tid) * 4 + (k & 3));
        __syncthreads();
        const uint32_t total = s_count;
        if (c0 + stride < n) load(c0 + stride, w);  // in flight while this chunk's quads are followed
        for (uint32_t i = tid; i < total; i += kThreads) {
            flatten_quad(label, c0 + 4 * (int64_t)s_quad[i], n, label16);
        }
        __syncthreads();
    }
}

// Mesh: pointer jumping to the roots.  A thread takes 8 labels, lane-consecutive
// (label c*2048 + j*256 + tid), and follows their chains hop by hop
// together until the warp's chains have all ended: 8 independent gathers
// in flight, and the 32 lanes of each gather read neighbouring labels,
// whose roots are mostly shared (the union-find before it halved the
// paths, so chains are short).  Once every hook is done the root reached is
// the component minimum, so a plain store of it cannot lose anything.
constexpr int kFlatPer = 8;
constexpr int kFlatHops = (int)kUnionLimit;  // bound only: a forest's chains end far sooner
constexpr int kFlatThreads = 256;

__global__ void __launch_bounds__(kFlatThreads) k_flatten(int32_t* label, int64_t n) {
    constexpr int64_t kChunk = (int64_t)kFlatThreads * kFlatPer;
    for (int64_t c = blockIdx.x; c * kChunk < n; c += gridDim.x) {
        int32_t l[kFlatPer], r[kFlatPer];
        uint32_t open = 0;
#pragma unroll
        for (int j = 0; j < kFlatPer; ++j) {
            const int64_t v = c * kChunk + (int64_t)j * kFlatThreads + threadIdx.x;
            l[j] = v < n ? label[v] : -1;
            r[j] = l[j];
            open |= (l[j] >= 0 ? 1u : 0u) << j;
        }
        // cached loads: a label read stale is still an ancestor of the
        // vertex (labels only decrease), so following it stays correct
#pragma unroll 1
        for (int h = 0; h < kFlatHops; ++h) {
            if (!__any_sync(0xffffffffu, open)) break;  // the warp's chains all ended
            int32_t w[kFlatPer];
#pragma unroll
            for (int j = 0; j < kFlatPer; ++j) w[j] = (open >> j & 1u) ? label[r[j]] : 0;
#pragma unroll
            for (int j = 0; j < kFlatPer; ++j)
                if (open >> j & 1u) {
                    if (w[j] == r[j]) open &= ~(1u << j);
                    else r[j] = w[j];
                }
        }
#pragma unroll
        for (int j = 0; j < kFlatPer; ++j) {
            const int64_t v = c * kChunk + (int64_t)j * kFlatThreads + threadIdx.x;
            if (v < n && r[j] != l[j]) label[v] = r[j];
        }
    }
}

// ----------------------------------------------------------------------------
// mesh

// Mesh kernels (subgraph sampling, after the Afforest scheme):
//   1. label[v] = v;
//   2. every vertex unites its first two neighbours, both read at once: any
//      read of a row's start fetches a good part of the row from DRAM (64
//      bytes at a time), so one launch per neighbour read the columns twice
//      (256^3 vertices, 13.7 columns each: 1.59 ms as two launches with
//      uncached finds, 0.54 with a plain hook to the first neighbour as a
//      pass of its own and cached finds, 0.38 as one launch; reading every
//      column once takes 0.14);
//   3. flatten; sample 1024 vertices and take the most frequent label --
//      on a well-connected mesh, nearly every vertex is already in that
//      component;
//   4. every vertex outside it unites all its remaining edges (8 lanes per
//      row); an edge to a vertex of the frequent component is found from
//      this side, since the adjacency is symmetric;
//   5. flatten.
// Every union hooks the larger root under the smaller, so the final root of
// a component is its smallest vertex id, whatever the order of unions.
constexpr int kRowLanes = 8;
constexpr int kSamples = 1024;

__global__ void k_mesh_init(int32_t* label, int32_t n) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        label[v] = (int32_t)v;
}

__global__ void __launch_bounds__(256) k_mesh_link(const int32_t* __restrict__ row, const int32_t* __restrict__ col,
                                                   int32_t n, int32_t* label, int32_t* status) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        const int32_t e = row[v], e1 = row[v + 1];
        const int32_t u0 = e < e1 ? col[e] : (int32_t)v, u1 = e + 1 < e1 ? col[e + 1] : (int32_t)v;
        if ((uint32_t)u0 >= (uint32_t)n || (uint32_t)u1 >= (uint32_t)n) {
            record_error(status, MSC_ERR_ARG);
            continue;
        }
        if (u0 != v) union_g(label, (int32_t)v, u0, status);
        if (u1 != v) union_g(label, (int32_t)v, u1, status);
    }
}

// The most frequent label among kSamples vertices spread over the ids
// (one block; labels sorted in shared memory, longest run wins, ties to
// the smaller label).
__global__ void __launch_bounds__(kSamples) k_mesh_sample(const int32_t* label, int32_t n, int32_t* frequent) {
    __shared__ int32_t s[kSamples];
    const int t = threadIdx.x;
    const uint64_t mixed = (uint64_t)(t + 1) * 0x9e3779b97f4a7c15ull;
    s[t] = label[(int64_t)((mixed >> 11) % (uint64_t)n)];
    __syncthreads();
    for (int k = 2; k <= kSamples; k <<= 1)  // bitonic sort
        for (int j = k >> 1; j > 0; j >>= 1) {
            const int p = t ^ j;
            if (p > t) {
                const bool up = (t & k) == 0;
                const int32_t a = s[t], b = s[p];
                if ((a > b) == up) {
                    s[t] = b;
                    s[p] = a;
                }
            }
            __syncthreads();
        }
    // each run's first entry finds its end; (length, smallest label) wins
    __shared__ unsigned long long best;
    if (t == 0) best = 0;
    __syncthreads();
    if (t == 0 || s[t - 1] != s[t]) {
        int lo = t + 1, hi = kSamples;  // first entry past the run
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (s[mid] == s[t]) lo = mid + 1;
            else hi = mid;
        }
        atomicMax(&best, (unsigned long long)(lo - t) << 32 | (uint32_t)~s[t]);
    }
    __syncthreads();
    if (t == 0) *frequent = (int32_t)~(uint32_t)best;
}

// Vertices outside the frequent component unite their remaining edges.
__global__ void __launch_bounds__(256) k_mesh_hook(const int32_t* __restrict__ row,
                                                   const int32_t* __restrict__ col, int32_t n,
                                                   const int32_t* __restrict__ frequent, int32_t* label,
                                                   int32_t* status) {
    const int lane = threadIdx.x & 31, sub = lane & (kRowLanes - 1);
    const int32_t big = *frequent;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) / 32;
    for (int64_t wbase = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32) * 32; wbase < n; wbase += warps * 32) {
        // 32 vertices' labels at once, then the rows that are wanted, four at a time
        const int64_t own = wbase + lane;
        const uint32_t want = __ballot_sync(0xffffffffu, own < n && label[own] != big);
        if (!want) continue;
#pragma unroll 1
        for (int i = 0; i < kRowLanes; ++i) {
            const int q = (32 / kRowLanes) * i + lane / kRowLanes;
            if (!(want >> q & 1u)) continue;
            const int64_t v = wbase + q;
            const int32_t e1 = row[v + 1];
            for (int32_t e = row[v] + 2 + sub; e < e1; e += kRowLanes) {
                const int32_t u = col[e];
                if ((uint32_t)u >= (uint32_t)n) {
                    record_error(status, MSC_ERR_ARG);
                    continue;
                }
                union_g(label, (int32_t)v, u, status);
            }
        }
    }
}

int cc_grid_for(int64_t work, int per_sm = 8) {
    const int64_t want = ceil_div(std::max<int64_t>(work, 1), 256);
    return (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)current_device().sms * per_sm));
}

}  // namespace

int run_cc_mask(const uint8_t* mask, msc_grid gd, int conn, int32_t* label, int32_t* status,
                cudaStream_t s) {
    CcGrid g;
    g.nx = gd.nx;
    g.ny = gd.ny;
    g.nz = gd.nz;
    g.tx = (int)ceil_div(gd.nx, CX);
    g.ty = (int)ceil_div(gd.ny, CY);
    g.ntiles = (int64_t)g.tx * g.ty * ceil_div(gd.nz, CZ);
    g.conn = conn;
    g.n = (int64_t)gd.nx * gd.ny * gd.nz;
    const bool mask8 = gd.nx % 8 == 0 && ((uintptr_t)mask & 7) == 0;
    const int sms = current_device().sms;
    auto local = mask8 ? k_cc_local<true> : k_cc_local<false>;
    const bool few = g.ntiles <= (int64_t)sms * 4 * kMergeWarps;
    auto merge = mask8 ? (few ? k_cc_merge<true, true> : k_cc_merge<true, false>)
                       : (few ? k_cc_merge<false, true> : k_cc_merge<false, false>);
    int occ = 1;
    MSC_TRY(max_blocks_per_sm(&occ, local, kThreads, 0));
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(g.ntiles, (int64_t)sms * std::max(occ, 1)));
    {
        TraceScope ts_("cc.local", s);
        local<<<grid, kThreads, 0, s>>>(mask, g, label, status);
    }
    MSC_LAUNCHED();
    {
        TraceScope ts_("cc.merge", s);
        merge<<<cc_grid_for(g.ntiles * 32), kMergeWarps * 32, 0, s>>>(mask, g, label, status);
    }
    MSC_LAUNCHED();
    {
        TraceScope ts_("cc.flatten", s);
        if (g.n <= kFlatSmall)
            k_cc_flatten_small<<<(unsigned)ceil_div(g.n, 4 * kThreads), kThreads, 0, s>>>(
                mask, g.n, ((uintptr_t)mask & 3) == 0, ((uintptr_t)label & 15) == 0, label);
        else
            k_cc_flatten<<<cc_grid_for(ceil_div(g.n, kFlatBytes), 6), kThreads, 0, s>>>(
            mask, g.n, ((uintptr_t)mask & 15) == 0, ((uintptr_t)label & 15) == 0, label);
    }
    MSC_LAUNCHED();
    return MSC_OK;
}

int run_cc_mesh(const int32_t* row, const int32_t* col, int32_t n, int32_t* label, int32_t* status,
                cudaStream_t s, int32_t* frequent) {
    if (n <= 0) return MSC_OK;
    const int grid = cc_grid_for(n);
    const int fgrid = cc_grid_for(ceil_div(n, kFlatPer));
    {
        TraceScope ts_("mesh.init", s);
        k_mesh_init<<<grid, 256, 0, s>>>(label, n);
    }
    MSC_LAUNCHED();
    {
        TraceScope ts_("mesh.link", s);
        k_mesh_link<<<grid, 256, 0, s>>>(row, col, n, label, status);
    }
    MSC_LAUNCHED();
    {
        TraceScope ts_("mesh.flatten", s);
        k_flatten<<<fgrid, kFlatThreads, 0, s>>>(label, n);
    }
    MSC_LAUNCHED();
    {
        TraceScope ts_("mesh.sample", s);
        k_mesh_sample<<<1, kSamples, 0, s>>>(label, n, frequent);
    }
    MSC_LAUNCHED();
    {
        TraceScope ts_("mesh.hook", s);
        k_mesh_hook<<<grid, 256, 0, s>>>(row, col, n, frequent, label, status);
    }
    MSC_LAUNCHED();
    {
        TraceScope ts_("mesh.flatten", s);
        k_flatten<<<fgrid, kFlatThreads, 0, s>>>(label, n);
    }
    MSC_LAUNCHED();
    return MSC_OK;
}

}  // namespace msc
