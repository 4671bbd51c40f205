// Arguments and launchers of the query pipeline (query.cu), shared with the C-ABI layer.
#pragma once

#include "sfc_internal.cuh"

namespace sfc {

// Groups of 32 points per item of the scan passes (powers of two: an item's boxes are loaded in
// pairs).  2-D: four measured best (two and one: count 5.8 -> 6.6 and 9.4 ms at 10^8 mixed points);
// 3-D: two (four the same, one 1.70 -> 2.32 ms at 10^7 points and 10^6 balls).
constexpr int kItemGroups2 = 4, kItemGroups3 = 2;
inline uint64_t item_groups(int dim) { return dim == 3 ? kItemGroups3 : kItemGroups2; }

struct QueryArgs {
    int curve;
    const uint64_t* keys;        // sorted keys [n]
    const uint32_t* ids;         // ids in sorted order [n]
    const int2* xy;              // coordinates in sorted order [n] (2-D)
    const uint2* packed;         // coordinates in sorted order [n] (3-D, pack3)
    int dim;                     // 2 or 3; queries are int32[m][dim]
    uint32_t n;
    const int32_t* q;            // [m][dim]
    const int32_t* delta;        // [m]
    uint64_t m;
    const uint32_t* dir;         // key directory (boxes.cu), 2^dir_bits + 1 positions
    int dir_bits;
    const int4* box;             // bounding boxes of the groups of 32 sorted points (boxes.cu)
    // plan results, by processing rank (the order in which queries are handed out)
    uint2* ranges;               // [m][kint]: the non-empty (begin, end) array ranges, in order
    uint32_t kint;               // range slots per query (2-D: 4, 9 or 25 by the cover; 3-D: 8 or 27)
    int drop;                    // cover refinement: 0 cells(Q), 1 or 2 levels finer
    int norm;                    // SFC_NORM_DISC or SFC_NORM_SQUARE
    int4* qrec;                  // [m] x, y, delta, z (0 in 2-D)
    uint32_t* nitems;            // [m] items of the query, at least 1
    uint64_t* gbase;             // [m + 1] the query's first item
    uint8_t* ovf;                // [m] 1: some of the query's items have no record
    uint32_t* counts;            // [m] hits per query, by query index
    // the hits, per batch of 32 items: heads[b] = (rank of the first item's query, records, first
    // record, 0), bhits[b] hits, bbase their exclusive scan; a record is one group with hits: (hit
    // bits, first array position | its query's rank minus the batch's)
    uint4* heads;
    uint32_t* bhits;
    uint64_t* bbase;             // [cap_batches + 1]
    uint64_t cap_batches;        // batches that have room
    uint2* recs;
    uint64_t cap_recs;           // records that have room (< 2^32)
    uint32_t slab;               // records a warp reserves at a time
    uint32_t chunk;              // points per chunk of the statistics
    uint32_t cgrab, wgrab;       // batches taken per work-queue grab (count and write pass)
    unsigned long long* work_ctr;  // kCtrWords counters, see kCtrCount ... kCtrOverflow
    uint64_t* out_offsets;       // [m + 1]
    uint32_t* out_ids;
    uint64_t ids_capacity;
    uint64_t q_begin, q_end;     // write pass: the processing ranks to write
    uint32_t* status;
    unsigned long long* scanned;   // statistics: [0] sum of S_q over the batch, [3] chunks
    // optional processing order: queries handed out in curve order of their centres
    const uint32_t* perm;        // [m] query index at each processing rank (NULL: identity)
    uint32_t* pstart;            // [m] hits of the batch before the query's first item (with perm)
    uint64_t* dbase;             // [m] output offset minus hits before the query (with perm)
    // early-termination bitmap (NULL: off) and the cover statistics
    const uint32_t* occ;
    int occ_depth;
    unsigned long long* cells;   // [0] cells of the covers, [1] of them found empty
};

struct LearnedModelView {
    const RootParams* root;      // device memory (written by training, no host copy needed)
    const LeafParams* leaf;
    const uint64_t* fence;       // [leaves][kFence] fence keys
    const uint64_t* fence_fine;  // [leaves][kFenceFine] fine fence keys
    unsigned long long* stats;   // [3]: endpoints, misses, window sum
};

sfc_status launch_plan(const QueryArgs& a, const LearnedModelView* lm, cudaStream_t st);
int query_intervals(int dim, int drop);   // range slots per query for a cover refinement
sfc_status launch_count(const QueryArgs& a, cudaStream_t st);
// queries that scan at most this many points have no chunks in the statistics
constexpr uint32_t kSmallScan = 64;
// work counters of a query batch: the count pass's and the write pass's queues of item batches,
// the records handed out, and whether some item found no room for its record
constexpr int kCtrCount = 0, kCtrWrite = 1, kCtrRecs = 2, kCtrOverflow = 3;
constexpr int kCtrWords = 4;
// most items, and batches of 32 of them, that m queries over n points can have: a range touches at
// most two items more than its length fills
inline uint64_t max_batches(int dim, uint64_t m, uint64_t n, uint64_t kint)
{
    return m * (n / 32 / item_groups(dim) + 2 * kint + 1) / 32 + 1;
}
// Zeroes what a query batch counts in: the statistics, the work counters and the look-back words
// of its scans.
sfc_status launch_reset(unsigned long long* stats, int nstats, unsigned long long* ctr, uint64_t* flags, uint64_t nflags,
                        cudaStream_t st);
// sort keys of the processing order: (input slice, top 24 bits of the centre's curve key)
sfc_status launch_query_keys(const int32_t* q, uint64_t m, int curve, int slices, uint64_t* keys, cudaStream_t st);
// dbase from the scans (with perm)
sfc_status launch_dbase(const QueryArgs& a, cudaStream_t st);
sfc_status launch_write(const QueryArgs& a, cudaStream_t st);
sfc_status launch_ranges(const QueryArgs& a, const LearnedModelView* lm, uint64_t* lo, uint64_t* hi,
                         uint32_t* b, uint32_t* e, uint32_t* cnt, cudaStream_t st);

}  // namespace sfc
