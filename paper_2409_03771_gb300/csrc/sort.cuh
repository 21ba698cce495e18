// Radix sorts: float32 -> vertex order (one field, packed fields), 64-bit keys
// with or without an int32 payload, and the ranks of a hash table's keys.
#pragma once

#include "common.cuh"

namespace msc {

struct SortScratch {
    uint32_t* ord_cnt;                // vertex order: [256][kOrderMaxSuper] super-tile counts, [4][256]
                                      // pass totals, [kOrderMaxBuckets][kOrderFillStride] bucket fills,
                                      // the bits in which the keys differ
    uint32_t* hist;                   // [8][256] digit histograms
    uint32_t* tile_counters;          // [8] dynamic tile ids, one per pass
    unsigned long long* lookback;     // [max_tiles][256] decoupled look-back words
    int64_t max_tiles;
};

constexpr int kSortTile = 4096;       // keys per onesweep tile
constexpr int kOrderMaxSuper = 8192;  // super-tiles (runs of consecutive tiles) of a vertex-order pass
constexpr int kOrderMaxBuckets = 256; // id buckets the last order pass files pairs into
constexpr int kOrderFillStride = 32;  // words between bucket fill counters (one 128-byte line each)
constexpr size_t kOrderCntWords = (size_t)256 * kOrderMaxSuper + 4 * 256 + kOrderMaxBuckets * kOrderFillStride + 64;

// Width of the id buckets of the order's last pass: 2^19 ids at least, at
// most kOrderMaxBuckets buckets.
int order_bucket_shift(int64_t n);

// Bytes of scratch (hist + counters + look-back) for up to n keys.
void size_sort_scratch(Sizer& s, int64_t n);
SortScratch carve_sort_scratch(Carver& c, int64_t n);

// order[v] = rank of (f[v], v).  Uses two (key, id) ping-pong buffers of n
// entries each.  Records MSC_ERR_NAN in status when f holds a NaN.
// `barrier` (optional): a word that is 0 now and free for this call.
int run_order(const float* f, int64_t n, int32_t* order, uint32_t* key_a, int32_t* id_a,
              uint32_t* key_b, int32_t* id_b, const SortScratch& sc, int32_t* status,
              cudaStream_t s, uint32_t* barrier = nullptr);

// Packed segments sorted independently (batched instances).  Segment i
// holds keys [off[i], off[i+1]) and tiles [tile0[i], tile0[i+1]) of
// kSortTile keys; tile_seg[t] is the segment of tile t.  Device arrays,
// built once on the host; total < 2^31.
struct SegTable {
    const int32_t* off;       // [count + 1]
    const int32_t* tile0;     // [count + 1]
    const int32_t* tile_seg;  // [tiles]
    int32_t count;
    int64_t total;
    int64_t tiles;
};

void size_seg_sort_scratch(Sizer& s, int count, int64_t tiles);
SortScratch carve_seg_sort_scratch(Carver& c, int count, int64_t tiles);

// order[v] = rank of (f[v], v) within v's segment, for every segment at
// once (4 segmented onesweep passes).  Ping-pong buffers of `total` entries.
int run_order_seg(const float* f, const SegTable& t, int32_t* order, uint32_t* key_a, int32_t* id_a,
                  uint32_t* key_b, int32_t* id_b, const SortScratch& sc, int32_t* status,
                  cudaStream_t s);

// The occupied slots of a hash table of 64-bit keys (kPairEmpty: free), ranked:
// vals[slot] = rank of the slot's key, and keys[npass & 1] the sorted keys with
// keep_keys.  On the device, ctl holds the table's capacity [2] (slots:
// capacity + kPairPad), whether there is anything to do [kPairCtlRoute] and
// two barrier words that are 0 [kPairCtlBarrier]; ctl[kPairCtlCount], 0 at the
// start, gets the number of keys.  At most n keys; buffers of n + kPairPad.
constexpr unsigned long long kPairEmpty = ~0ull;
constexpr uint32_t kPairPad = 4096;
constexpr int kPairCtlRoute = 16, kPairCtlCount = 18, kPairCtlBarrier = 40;

struct PairRanks {
    const unsigned long long* table;
    uint32_t* ctl;
    unsigned long long* keys[2];
    int32_t* slots[2];
    uint32_t* vals;
    int npass;      // 8-bit digits of the keys
    int keep_keys;  // the caller reads the sorted keys
};

int run_pair_ranks(const PairRanks& p, int64_t n, const SortScratch& sc, int32_t* status, cudaStream_t s);

// Stable sort of (keys, vals) by the low `key_bits` bits of keys.  The
// count is read on the device from *d_count (<= max_count).  Returns, via
// *result_in_alt, whether the sorted data ended in the alt buffers.  With
// vals and vals_alt both null the keys are sorted alone.
int run_sort_u64(unsigned long long* keys, int32_t* vals, unsigned long long* keys_alt,
                 int32_t* vals_alt, const int32_t* d_count, int64_t max_count, int key_bits,
                 const SortScratch& sc, int32_t* status, cudaStream_t s, bool* result_in_alt,
                 const char* hist_label, const char* pass_label);

}  // namespace msc
