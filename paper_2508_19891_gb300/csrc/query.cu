// Batched distance query (Alg. 1 for m queries at once).
//
//   plan_kernel    one thread per query (in curve order of the centres when the queries are
//                  reordered): bounding square Q of B_delta(q), the level l with
//                  2 delta <= 2^l < 4 delta, the <= 4 cells of cells(Q) and their key
//                  intervals [pi(C)o0, pi(C)o1] (Observation) -- or, with a refined cover,
//                  the cells one or two levels finer (<= 9 / <= 25) that meet the window;
//                  cells the early-termination bitmap shows empty are dropped -- sorted and
//                  with abutting intervals merged, then lower_bound of both ends of every
//                  interval, by binary search or by the learned model (fence bracket and
//                  error window, verified, with fallback).  It keeps the non-empty array ranges
//                  and how many items they make: group g is the 32 array positions
//                  32 g .. 32 g + 31, an item is four (3-D: two) neighbouring groups.
//   scan           exclusive scan of the item counts: the batch's scan is now one list of items,
//                  in processing order.
//   count_kernel   a warp takes a batch of 32 items, one per lane.  A lane looks its groups'
//                  bounding boxes up (boxes.cu) and so knows, for most groups, that no point or
//                  every point of them lies in the window; the warp reads the points of the
//                  remaining groups, one coalesced load per group, and applies the exact window
//                  test (disc dx^2 + dy^2 <= delta^2 in int64, square, or 3-D ball).  Each group
//                  gets a word of 32 hit bits; the non-empty ones are kept as records (word,
//                  first position, query).
//   scan           exclusive scans of the hits per batch (where each batch's ids begin, in
//                  processing order) and of the hits per query (the caller's out_offsets).
//   write_kernel   a warp takes the records of a batch and knows each one's output position from
//                  the scan, whatever query it belongs to: it reads the ids of a group with one
//                  coalesced load and stores those of the hits side by side.
//   refilter_kernel  the queries whose items did not all fit the record buffer, if there are any:
//                  one warp walks the items of one query, filters them again and writes.
//
// Items are the same work whatever the size of their query, so one query of 10^6 hits and 10^6
// queries of one spread over the warps alike.
#include <algorithm>

#include "sfc_internal.cuh"
#include "query.cuh"

namespace sfc {

namespace {

constexpr int kThreads = 256;

// Binary searches in lock step per thread, and the plan kernel's resident blocks per SM (its
// register budget) for each bound search.
constexpr int kBinaryBatch = 4, kBinaryBatch3 = 8, kLearnedBatch = 2;
constexpr int kPlanBlocksBinary = 4, kPlanBlocksLearned = 4;
// Targets a warp searches per round: the flat list of its 32 queries' interval endpoints is
// searched in rounds of at most this many (one round for nearly every warp: cover 1 averages
// about 6.5 endpoints per query).  A multiple of 32.
constexpr uint32_t kPlanCap = 256;
// Resident blocks per SM (the register budgets) of the count and the write pass.
constexpr int kCountBlocks = 6, kWriteBlocks = 7;
// Records whose ids a warp of the write pass has in flight.  Measured with the blocks that the
// registers leave, 10^6 queries over 10^7 mixed points (10^7 over 10^8): two on 8 blocks 597 us (5.77 ms),
// four on 8 588 (5.81), six on 7 553 (5.62), eight on 7 576 (5.77), on 6 632 (5.97).
constexpr uint32_t kCopyUnroll = 6;

// ------------------------------------------------------------------------------------
// Bound search: lower_bounds in lock step (independent loads in flight together)
// ------------------------------------------------------------------------------------
// E lower_bounds in lock step, the answer of search x in [base[x], base[x] + len[x]]; a search that
// has ended loads nothing more (padding all to the longest made the short ones probe cold lines
// beyond their part: the plan of 10^6 mixed queries 502 us; the learned search, whose queries run in
// curve order over lines that their neighbours hold, is the faster padded, 2.35 against 2.58 ms).
template <int E>
__device__ __forceinline__ void lower_bounds_each(const uint64_t* __restrict__ keys, const uint64_t* t, uint32_t* base,
                                                  uint32_t* len)
{
    while (true) {
        uint32_t any = 0;
#pragma unroll
        for (int x = 0; x < E; ++x) any |= len[x];
        if (!any) break;
        uint64_t k[E];
#pragma unroll
        for (int x = 0; x < E; ++x)
            if (len[x]) k[x] = __ldg(keys + base[x] + (len[x] >> 1));
#pragma unroll
        for (int x = 0; x < E; ++x) {
            if (!len[x]) continue;
            const uint32_t half = len[x] >> 1;
            const bool below = k[x] < t[x];
            base[x] = below ? base[x] + half + 1 : base[x];
            len[x] = below ? len[x] - half - 1 : half;
        }
    }
}

// E lower_bounds in lock step with one step count for all: the answer of search x lies in
// [base[x], base[x] + len] (the same len for every x, keys[base[x] .. base[x] + len) inside the
// array).  Each step halves len and moves a base past the probed key when that key is below
// the target (Khuong & Morin's branch-free search); the final probe decides between base and
// base + 1.  With one length there is no per-search bookkeeping: a step is an add, the load,
// the 64-bit compare and a select.
template <int E>
__device__ __forceinline__ void lower_bounds_uniform(const uint64_t* __restrict__ keys, const uint64_t* t,
                                                     uint32_t* base, uint32_t len)
{
    if (len == 0) return;
#pragma unroll 1
    while (len > 1) {
        const uint32_t half = len >> 1;
#pragma unroll
        for (int x = 0; x < E; ++x) base[x] = __ldg(keys + base[x] + half) < t[x] ? base[x] + half : base[x];
        len -= half;
    }
#pragma unroll
    for (int x = 0; x < E; ++x) base[x] += __ldg(keys + base[x]) < t[x] ? 1u : 0u;
}

// Per-thread counters of the learned search, summed once per block at the end of the plan.
struct BoundStats {
    unsigned long long endpoints = 0, misses = 0, window = 0;
};

// Bound search functors: search_flat gives lower_bound over the whole array of the warp's flat
// list of T targets (each lane takes targets lane, lane + 32, ...; kBatch of them in lock step).
//
// Binary search behind the key directory (boxes.cu): one lookup leaves the keys of one of 2^bits
// equal parts of the key range, so a search takes that load and about log2(n / 2^bits) steps where
// the array is evenly filled (more in a cluster) instead of log2(n).
// Measured, plan of 10^6 queries over 10^7 points: mixed, cover 1, 421 -> 261 us; Normal points,
// square windows 209 -> 112 us; 3-D balls 1371 -> 712 us (whose cells also moved from local memory to
// columns in shared memory).
template <int DIM>
struct BinaryBounds {
    static constexpr bool kStats = false;
    // (3-D: the columns of cell keys leave few warps, which need more loads in flight)
    static constexpr int kBatch = DIM == 3 ? kBinaryBatch3 : kBinaryBatch;
    static constexpr int kMinBlocks = kPlanBlocksBinary;
    const uint32_t* dir;
    int bits;
    uint64_t kmin, kmax;
    int shift;
    __device__ __forceinline__ void prepare(RootParams*, const uint64_t* keys, uint32_t n)
    {
        kmin = n ? __ldg(keys) : 0;
        kmax = n ? __ldg(keys + n - 1) : 0;
        shift = dir_shift(kmin, kmax, bits);
    }
    __device__ __forceinline__ void search_flat(const uint64_t* keys, uint32_t n, const uint64_t* tg, uint32_t* res,
                                                uint32_t T, BoundStats&) const
    {
        constexpr int E = kBatch;
#pragma unroll 1
        for (uint32_t e0 = lane_id(); e0 < T; e0 += 32 * E) {
            uint64_t t[E];
            uint32_t base[E], len[E];
#pragma unroll
            for (int x = 0; x < E; ++x) {
                const uint32_t e = e0 + 32 * x;
                t[x] = e < T ? tg[e] : 0;
                base[x] = len[x] = 0;
                if (t[x] > kmax) {
                    base[x] = n;
                } else if (t[x] > kmin) {
                    const uint32_t v = (uint32_t)((t[x] - kmin) >> shift);
                    base[x] = __ldg(dir + v);
                    len[x] = __ldg(dir + v + 1) - base[x];
                }
            }
            lower_bounds_each<E>(keys, t, base, len);
#pragma unroll
            for (int x = 0; x < E; ++x) {
                const uint32_t e = e0 + 32 * x;
                if (e < T) res[e] = base[x];
            }
        }
    }
};

struct LearnedBounds {
    static constexpr bool kStats = true;
    static constexpr int kBatch = kLearnedBatch;
    static constexpr int kMinBlocks = kPlanBlocksLearned;
    const RootParams* root;      // device; after prepare() the block's shared-memory copy
    const LeafParams* leaf;
    const uint64_t* fence;       // [leaves][kFence] coarse fence keys
    const uint64_t* fence_fine;  // [leaves][kFenceFine] fine fence keys
    unsigned long long* stats;   // [0] endpoints, [1] misses, [2] window sum
    // every thread of the block calls this, then the block synchronises
    __device__ __forceinline__ void prepare(RootParams* s, const uint64_t*, uint32_t)
    {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(root);
        uint32_t* dst = reinterpret_cast<uint32_t*>(s);
        for (unsigned i = threadIdx.x; i < sizeof(RootParams) / 4; i += blockDim.x) dst[i] = src[i];
        root = s;
    }
    // lower_bound over the whole array of the warp's flat list of T targets (each lane takes
    // targets lane, lane + 32, ...; kBatch of them in lock step); results in res.  Per target:
    //   1. the root routes it to leaf j (the keys below it lie in leaves before j, the keys
    //      above it in leaves after j, as the root is monotone);
    //   2. the leaf's line predicts its position p and the stored error window bounds it:
    //      lower_bound(t) lies in [a, b] = [p + err_lo, p + err_hi + 1] within the leaf;
    //   3. the window picks the slice of the leaf's fine fence (the keys at kFenceFine equally
    //      spaced positions of the leaf) that falls inside it, and counting the slice's keys
    //      below t brackets the target between two fence keys;
    //   4. the last-mile search runs over the bracket within the window (every search of a
    //      batch padded to the longest); an answer on the edge of its range is checked against
    //      the key beyond the edge, and a target whose window missed is searched over the whole
    //      array.
    __device__ __forceinline__ void search_flat(const uint64_t* keys, uint32_t n, const uint64_t* tg, uint32_t* res,
                                                uint32_t T, BoundStats& bs) const
    {
        constexpr int E = kBatch;
#pragma unroll 1
        for (uint32_t e0 = lane_id(); e0 < T; e0 += 32 * E) {
            uint64_t t[E];
            uint32_t lo[E], len[E], fo[E];
            int ne = 0;
            uint32_t F = 0;   // longest fence slice of the batch
#pragma unroll
            for (int x = 0; x < E; ++x) {
                const uint32_t e = e0 + 32 * x;
                ne += e < T;
                t[x] = e < T ? tg[e] : 0;
                const uint32_t j = (uint32_t)route_leaf(*root, t[x]);
                const LeafParams lp = leaf[j];
                const int64_t p = leaf_predict(lp, t[x]);
                int64_t a = p + lp.err_lo, b = p + (int64_t)lp.err_hi + 1;
                a = min(max(a, (int64_t)lp.first), (int64_t)lp.end);
                b = min(max(b, a), (int64_t)lp.end);
                lo[x] = (uint32_t)a;
                len[x] = (uint32_t)(b - a);
                // fine fence entry r sits at position first + floor(r cnt / kFenceFine): the
                // entries at positions below a are below t, those above b are not, so only
                // entries [ra, rb) need counting; ra and rb from a float estimate widened by one
                // entry on each side (its error is far below one entry)
                const uint32_t cnt = lp.end - lp.first;
                uint32_t ra = 0, rb = 0;
                if (cnt) {
                    const float scale = __fdividef((float)kFenceFine, (float)cnt);
                    const float fa = (float)(uint32_t)(a - lp.first) * scale;
                    const float fbk = (float)(uint32_t)(b - lp.first + 1) * scale;
                    ra = (uint32_t)max((int)fa - 1, 0);
                    rb = (uint32_t)min((int)fbk + 2, kFenceFine);
                }
                fo[x] = j * kFenceFine + ra;
                F = max(F, rb - ra);
            }
            // count the slice's fence keys below t: branch-free, every slice padded to the
            // batch's longest, moved left where it would run past the leaf's fence (the entries
            // it takes in on the left are below t and are counted like the others)
#pragma unroll
            for (int x = 0; x < E; ++x) {
                const uint32_t r0 = fo[x] % kFenceFine;
                fo[x] -= r0 + F > kFenceFine ? r0 + F - kFenceFine : 0;
            }
            uint32_t c[E];
#pragma unroll
            for (int x = 0; x < E; ++x) c[x] = 0;
            if (F > 0) {
                uint32_t flen = F;
#pragma unroll 1
                while (flen > 1) {
                    const uint32_t half = flen >> 1;
#pragma unroll
                    for (int x = 0; x < E; ++x) c[x] = __ldg(fence_fine + fo[x] + c[x] + half) < t[x] ? c[x] + half : c[x];
                    flen -= half;
                }
#pragma unroll
                for (int x = 0; x < E; ++x) c[x] += __ldg(fence_fine + fo[x] + c[x]) < t[x] ? 1u : 0u;
            }
            uint32_t N = 0;
            unsigned long long wsum = 0;
#pragma unroll
            for (int x = 0; x < E; ++x) {
                const uint32_t j = fo[x] / kFenceFine;
                const uint64_t first = __ldg(&leaf[j].first), cnt = __ldg(&leaf[j].end) - first;
                // r fine keys below t: lower_bound(t) lies in [P(r - 1) + 1, P(r)], P(r) the
                // position of fine key r, P(kFenceFine) = end
                const uint32_t r = cnt ? fo[x] % kFenceFine + c[x] : 0u;
                const uint64_t bl = r == 0 ? first : first + ((uint64_t)(r - 1) * cnt) / kFenceFine + 1;
                const uint64_t bh = r == 0 ? first : (r == kFenceFine ? first + cnt : first + ((uint64_t)r * cnt) / kFenceFine);
                const uint64_t nl = max((uint64_t)lo[x], bl), nh = min((uint64_t)lo[x] + len[x], bh);
                if (nl <= nh) {
                    lo[x] = (uint32_t)nl;
                    len[x] = (uint32_t)(nh - nl);
                } else {   // both hold lower_bound(t) unless the window is off: keep the bracket
                    lo[x] = (uint32_t)bl;
                    len[x] = (uint32_t)(bh - bl);
                }
                if (e0 + 32 * x < T) wsum += len[x];
                N = max(N, len[x]);
            }
            // pad every range to the longest: [lo, lo + N) still holds the answer, moved left
            // where it would run past the end of the array (a model kept over a rebuild that did not
            // fit it again may bracket more keys than there are)
            N = min(N, n);
            uint32_t lo0[E];
#pragma unroll
            for (int x = 0; x < E; ++x) {
                lo[x] = (uint64_t)lo[x] + N > n ? n - N : lo[x];
                lo0[x] = lo[x];
            }
            lower_bounds_uniform<E>(keys, t, lo, N);
            // an answer strictly inside its range has both neighbours in it, compared by the
            // search; on an edge, the key beyond the edge decides
            uint32_t miss = 0;
#pragma unroll
            for (int x = 0; x < E; ++x) {
                const uint32_t r = lo[x];
                bool ok = true;
                if (r == lo0[x] && r > 0) ok = __ldg(keys + r - 1) < t[x];
                if (r == lo0[x] + N && r < n) ok = ok && __ldg(keys + r) >= t[x];
                if (!ok && e0 + 32 * x < T) miss |= 1u << x;
            }
            if (miss) {
                uint32_t r2[E];
#pragma unroll
                for (int x = 0; x < E; ++x) r2[x] = 0;
                lower_bounds_uniform<E>(keys, t, r2, n);
#pragma unroll
                for (int x = 0; x < E; ++x) lo[x] = (miss >> x) & 1u ? r2[x] : lo[x];
            }
#pragma unroll
            for (int x = 0; x < E; ++x) {
                const uint32_t e = e0 + 32 * x;
                if (e < T) res[e] = lo[x];
            }
            bs.endpoints += ne;
            bs.misses += __popc(miss);
            bs.window += wsum;
        }
    }
};

// Inclusive prefix sum over the warp (every lane calls).
__device__ __forceinline__ uint32_t warp_incl_scan_u32(uint32_t v)
{
    const unsigned lane = lane_id();
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if ((int)lane >= o) v += t;
    }
    return v;
}

// Sum of v over the warp (every lane calls), returned to every lane.
__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ------------------------------------------------------------------------------------
// plan_kernel: range derivation and bound search, one thread per query
// ------------------------------------------------------------------------------------
template <int DIM, int DROP>
struct Cover {
    // cells per axis at most: 2 for cells(Q) (2 delta <= 2^l), 2^DROP + 1 one or two levels finer
    static constexpr int NX = DROP == 0 ? 2 : (1 << DROP) + 1;
    static constexpr int K = DIM == 3 ? NX * NX * NX : NX * NX;   // 2-D: 4, 9, 25 slots per query; 3-D: 8, 27
    // threads per block: the columns of cell keys are K words a thread
    static constexpr int kThreads = DIM == 3 ? 128 : 256;
};

// Early termination (Sec. 2.2): whether the cell of level l whose key interval starts at c may
// hold a point -- the bit of its own node when the node is within depth D, else of its
// ancestor at depth D.
__device__ __forceinline__ bool cell_occupied(const uint32_t* __restrict__ occ, int D, int l, uint64_t c)
{
    const int t = min(kOmega - l, D);
    const uint64_t b = occupancy_level_start(t) + (c >> (2 * (kOmega - t)));
    return (__ldg(occ + (b >> 5)) >> (b & 31)) & 1u;
}

// Puts key c into its place among the cnt ascending keys of the column.
__device__ __forceinline__ void insert_cell(uint64_t* col, int stride, int cnt, uint64_t c)
{
    int j = cnt;
    while (j > 0 && col[(j - 1) * stride] > c) {
        col[j * stride] = col[(j - 1) * stride];
        --j;
    }
    col[j * stride] = c;
}

// The cells of the cover, each as the key of its first point (its key interval is [c, c | span],
// Observation; every cell of a cover has the same level), sorted ascending into the thread's
// column col[0], col[stride], ... of shared memory; returns how many; *span_out = 4^l - 1.
// DROP 0: cells(Q), the cells of level l (2 delta <= 2^l < 4 delta, capped at omega) that meet
// the clipped square Q.  DROP > 0: the cells of level max(0, l - DROP) that hold an integer
// point of the closed ball (the distance from q to the cell's nearest integer point is at most
// delta; for the square window every cell meeting Q qualifies).  With the early-termination
// bitmap (occ != NULL), cells it shows empty are dropped; ncell / nempty count the cover's
// cells and the dropped ones.
template <int DROP>
__device__ __forceinline__ int derive_cells(int curve, int norm, const HilbertTables* tb, int32_t qx, int32_t qy,
                                            int32_t delta, const uint32_t* occ, int D, uint64_t* col, int stride,
                                            uint64_t* span_out, uint32_t& ncell, uint32_t& nempty)
{
    const int64_t d = delta;
    const int64_t x0 = max((int64_t)0, (int64_t)qx - d), x1 = min((int64_t)kSide - 1, (int64_t)qx + d);
    const int64_t y0 = max((int64_t)0, (int64_t)qy - d), y1 = min((int64_t)kSide - 1, (int64_t)qy + d);
    int l = 0;
    if (d > 0) {
        l = 64 - __clzll((unsigned long long)(2 * d - 1));   // bit length of 2 delta - 1
        if (l > kOmega) l = kOmega;
    }
    l = max(0, l - DROP);
    const uint64_t span = (l >= kOmega) ? kKeyMax : ((1ull << (2 * l)) - 1);
    *span_out = span;
    constexpr int NX = Cover<2, DROP>::NX;   // cells per axis at most
    const int64_t cx0 = x0 >> l, cy0 = y0 >> l;
    const int nx = (int)min((int64_t)NX, (x1 >> l) - cx0 + 1), ny = (int)min((int64_t)NX, (y1 >> l) - cy0 + 1);
    // per column: the squared distance from q to the column's nearest x and, for the Z curve,
    // the spread bits of its first x (the key of cell (cx, cy) is spread(cx 2^l) | spread(cy 2^l) << 1)
    int64_t dx2[NX];
    uint64_t sx[NX];
#pragma unroll
    for (int ix = 0; ix < NX; ++ix) {
        const int64_t cx = cx0 + ix;
        const int64_t ax0 = cx << l, ax1 = ((cx + 1) << l) - 1;
        const int64_t dx = qx < ax0 ? ax0 - qx : (qx > ax1 ? qx - ax1 : 0);
        dx2[ix] = dx * dx;
        sx[ix] = curve == SFC_CURVE_Z ? spread_bits((uint32_t)(cx << l)) : 0;
    }
    const int64_t d2 = d * d;
    int cnt = 0;
#pragma unroll
    for (int iy = 0; iy < NX; ++iy) {
        if (iy >= ny) break;
        const int64_t cy = cy0 + iy;
        const int64_t ay0 = cy << l, ay1 = ((cy + 1) << l) - 1;
        const int64_t dy = qy < ay0 ? ay0 - qy : (qy > ay1 ? qy - ay1 : 0);
        const int64_t dy2 = dy * dy;
        const uint64_t sy = curve == SFC_CURVE_Z ? spread_bits((uint32_t)(cy << l)) << 1 : 0;
#pragma unroll
        for (int ix = 0; ix < NX; ++ix) {
            if (ix >= nx) break;
            // every cell meeting Q meets a square window; a disc needs an integer point of the
            // ball in the cell
            if (DROP > 0 && norm == SFC_NORM_DISC && dx2[ix] + dy2 > d2) continue;
            const uint64_t c = (curve == SFC_CURVE_Z ? (sx[ix] | sy)
                                                     : hilbert_key(tb, (uint32_t)((cx0 + ix) << l), (uint32_t)(cy << l))) &
                               ~span;
            ++ncell;
            if (occ && !cell_occupied(occ, D, l, c)) {
                ++nempty;
                continue;
            }
            insert_cell(col, stride, cnt++, c);
        }
    }
    return cnt;
}

// The same in 3-D.  DROP 0: cells(Q), the cells of level l (2 delta <= 2^l < 4 delta, capped at 21)
// meeting the clipped cube Q.  DROP 1: the cells of level max(0, l - 1) holding an integer point of
// the closed ball.
template <int DROP>
__device__ __forceinline__ int derive_cells3(int4 w, uint64_t* col, int stride, uint64_t* span_out)
{
    constexpr int NX = Cover<3, DROP>::NX;
    const int64_t d = w.z, d2 = d * d;
    int l = 0;
    if (d > 0) {
        l = 64 - __clzll((unsigned long long)(2 * d - 1));
        if (l > kOmega3) l = kOmega3;
    }
    l = max(0, l - DROP);
    const uint64_t span = (1ull << (3 * l)) - 1;   // 3 l <= 63
    *span_out = span;
    // per axis: the first cell and the squared distance from q to each cell's nearest coordinate
    // (-1: no such cell)
    const int c[3] = {w.x, w.y, w.w};
    int first[3];
    int64_t dist2[3][NX];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int a0 = (int)max((int64_t)0, c[k] - d), a1 = (int)min((int64_t)kSide3 - 1, c[k] + d);
        first[k] = a0 >> l;
#pragma unroll
        for (int j = 0; j < NX; ++j) {
            const int64_t b0 = (int64_t)(first[k] + j) << l, b1 = b0 + ((int64_t)1 << l) - 1;
            const int64_t e = c[k] < b0 ? b0 - c[k] : (c[k] > b1 ? c[k] - b1 : 0);
            dist2[k][j] = first[k] + j <= (a1 >> l) ? e * e : -1;
        }
    }
    int cnt = 0;
#pragma unroll
    for (int iz = 0; iz < NX; ++iz) {
        if (dist2[2][iz] < 0) break;
        const uint64_t sz = spread3_bits((uint32_t)(first[2] + iz) << l) << 2;
#pragma unroll
        for (int iy = 0; iy < NX; ++iy) {
            if (dist2[1][iy] < 0) break;
            const uint64_t sy = sz | spread3_bits((uint32_t)(first[1] + iy) << l) << 1;
#pragma unroll
            for (int ix = 0; ix < NX; ++ix) {
                if (dist2[0][ix] < 0) break;
                if (DROP > 0 && dist2[0][ix] + dist2[1][iy] + dist2[2][iz] > d2) continue;
                insert_cell(col, stride, cnt++, sy | spread3_bits((uint32_t)(first[0] + ix) << l));
            }
        }
    }
    return cnt;
}

// Visits the endpoints of the merged key intervals of nc sorted cells (cells whose intervals
// abut in key order form one interval: the scan over them is identical): endpoint 2k is the
// first key of interval k, endpoint 2k + 1 one past its last key (the interval's array range is
// [lower_bound(first key), lower_bound(last key + 1))).  fn(ep, key) in order.
template <class F>
__device__ __forceinline__ void for_each_endpoint(const uint64_t* col, int stride, int nc, uint64_t span, F&& fn)
{
    uint32_t ep = 0;
    uint64_t prev_end = 0;
    for (int k = 0; k < nc; ++k) {
        const uint64_t c = col[k * stride];
        if (k == 0 || c != prev_end) fn(ep++, c);                           // an interval starts
        prev_end = c + span + 1;
        if (k + 1 == nc || col[(k + 1) * stride] != prev_end) fn(ep++, prev_end);   // ... and ends
    }
}

// Items that the range [b, e) (b < e) touches: item j is the kGroups groups of 32 array positions
// from position 32 kGroups j on.
template <int kGroups>
__device__ __forceinline__ uint32_t range_items(uint32_t b, uint32_t e)
{
    return (e - 1) / (32 * kGroups) - b / (32 * kGroups) + 1;
}

// The plan's per-query results, at the query's processing rank r: its window, its number of items
// (a query without points keeps one, an empty one, so that every query owns at least one item
// and the items' owners can be counted), zeroed hit count and overflow flag.
__device__ __forceinline__ void plan_store(const QueryArgs& a, uint64_t r, uint64_t i, int4 window, uint32_t items)
{
    a.qrec[r] = window;
    a.nitems[r] = items ? items : 1u;
    if (!items) a.ranges[(uint64_t)a.kint * r] = make_uint2(0u, 0u);
    a.counts[i] = 0;
    a.ovf[r] = 0;
}

// Statistics of a batch, one atomic per warp and counter: the scanned total, and the scan's
// chunks (a.chunk points each; queries that scan at most kSmallScan points count none).
__device__ __forceinline__ void plan_stats(const QueryArgs& a, uint64_t S)
{
    const unsigned long long t = warp_sum_u64(S);
    const unsigned long long c = warp_sum_u64(S > kSmallScan ? (S + a.chunk - 1) / a.chunk : 0);
    if (lane_id() == 0 && t) {
        atomicAdd(a.scanned, t);
        if (c) atomicAdd(a.scanned + 3, c);
    }
}

// Optional outputs of the plan (the ranges export); null in the query path.
struct PlanExport {
    uint64_t* lo;
    uint64_t* hi;
    uint32_t* b;
    uint32_t* e;
    uint32_t* cnt;
};


// Dynamic shared memory of plan_kernel<.., DIM, DROP, ..>: each thread's column of K cell keys
// (column-major, so that the lanes of a warp touch consecutive words), then per warp the flat
// target list (kPlanCap keys) and its results (kPlanCap positions).
template <int DIM, int DROP>
constexpr size_t plan_smem_bytes()
{
    constexpr int T = Cover<DIM, DROP>::kThreads;
    return (size_t)Cover<DIM, DROP>::K * T * sizeof(uint64_t) +
           (size_t)(T / 32) * kPlanCap * (sizeof(uint64_t) + sizeof(uint32_t));
}

// One thread per query for the range derivation: the cells of its cover, sorted, in shared
// memory.  The bound search runs on the warp's endpoints as one flat list in shared memory:
// lane L's query owns list positions [off_L, off_L + 2 cnt_L), the lanes take the list
// round-robin, so every lane searches about the same number of endpoints whatever the spread
// of interval counts over the warp's queries.  Then each thread writes its query's intervals'
// (begin, end) to slots 0.. of its K slots (unused slots (0, 0)), the number of chunks of its
// scan, and adds to the scanned total.  Nothing per query lives in local memory.
template <class Bounds, int DIM, int DROP, bool EXPORT>
__global__ void __launch_bounds__((Cover<DIM, DROP>::kThreads), Bounds::kMinBlocks)
plan_kernel(QueryArgs a, Bounds bounds_in, PlanExport ex)
{
    chain_start();
    constexpr int K = Cover<DIM, DROP>::K, kThreads = Cover<DIM, DROP>::kThreads;
    __shared__ HilbertTables tb;
    __shared__ RootParams s_root;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    uint64_t* col = reinterpret_cast<uint64_t*>(s_dyn) + threadIdx.x;
    const unsigned warp = threadIdx.x >> 5;
    uint64_t* tg = reinterpret_cast<uint64_t*>(s_dyn) + (size_t)K * kThreads + (size_t)warp * kPlanCap;
    uint32_t* res = reinterpret_cast<uint32_t*>(reinterpret_cast<uint64_t*>(s_dyn) + (size_t)K * kThreads +
                                                (size_t)(kThreads / 32) * kPlanCap) + (size_t)warp * kPlanCap;
    Bounds bounds = bounds_in;
    bounds.prepare(&s_root, a.keys, a.n);
    if constexpr (Bounds::kStats) __syncthreads();   // the root's shared-memory copy
    if (DIM == 2 && a.curve == SFC_CURVE_HILBERT) hilbert_tables_init(&tb);   // ends with a block barrier
    // thread r takes the query of processing rank r (curve order of the centres when a
    // processing order is given: neighbouring threads then search neighbouring keys)
    const uint64_t r = (uint64_t)blockIdx.x * kThreads + threadIdx.x;
    const bool active = r < a.m;
    const uint32_t* perm = after_wait(a.perm);
    const int32_t *qs = after_wait(a.q), *ds = after_wait(a.delta);
    const uint64_t i = active && perm ? (uint64_t)perm[r] : r;
    int4 q = make_int4(0, 0, -1, 0);   // x, y, delta, z
    if (active) {
        if (DIM == 3) {
            q.x = qs[3 * i];
            q.y = qs[3 * i + 1];
            q.w = qs[3 * i + 2];
        } else {
            const int2 c = reinterpret_cast<const int2*>(qs)[i];
            q.x = c.x;
            q.y = c.y;
        }
        q.z = ds[i];
    }
    const bool ok = active && q.z >= 0 && (DIM == 3 ? point3_in_domain(q.x, q.y, q.w) : point_in_domain(q.x, q.y));
    if (active && !ok) set_status(a.status, SFC_DEV_BAD_QUERY);
    BoundStats bs;
    uint32_t ncell = 0, nempty = 0;
    uint64_t span = 0;
    int nc = 0;
    if (ok) {
        if constexpr (DIM == 3) nc = derive_cells3<DROP>(q, col, kThreads, &span);
        else nc = derive_cells<DROP>(a.curve, a.norm, &tb, q.x, q.y, q.z, a.occ, a.occ_depth, col, kThreads, &span, ncell,
                                     nempty);
    }
    uint32_t cnt = 0;   // merged intervals
    for_each_endpoint(col, kThreads, nc, span, [&](uint32_t ep, uint64_t) { cnt += ep & 1u; });
    if (DIM == 3) ncell = cnt;
    const uint32_t ne = 2u * cnt;
    const uint32_t incl = warp_incl_scan_u32(ne);
    const uint32_t off = incl - ne;
    const uint32_t T = __shfl_sync(0xffffffffu, incl, 31);
    uint2* rp = (!EXPORT && active) ? a.ranges + (uint64_t)K * r : nullptr;
    uint32_t open = 0, items = 0;   // begin of the interval whose end comes next; items so far
    uint64_t S = 0;   // sum of e_k - b_k, gathered endpoint by endpoint
#pragma unroll 1
    for (uint32_t r0 = 0; r0 < T; r0 += kPlanCap) {   // warp-uniform
        const uint32_t r1 = min(T, r0 + kPlanCap);
        for_each_endpoint(col, kThreads, nc, span, [&](uint32_t ep, uint64_t key) {
            const uint32_t f = off + ep;
            if (f >= r0 && f < r1) tg[f - r0] = key;
        });
        __syncwarp();
        bounds.search_flat(a.keys, a.n, tg, res, r1 - r0, bs);
        __syncwarp();
        const uint32_t f0 = max(off, r0), f1 = min(off + ne, r1);
        for (uint32_t f = f0; f < f1; ++f) {
            const uint32_t ep = f - off;
            const uint32_t pos = res[f - r0];
            S += (ep & 1u) ? (uint64_t)pos : (uint64_t)0 - pos;
            if (!EXPORT) {
                if ((ep & 1u) == 0) {
                    open = pos;
                } else if (pos > open) {   // a non-empty range
                    *rp++ = make_uint2(open, pos);
                    items += range_items<DIM == 3 ? kItemGroups3 : kItemGroups2>(open, pos);
                }
            } else {
                const uint64_t o = (uint64_t)K * i + (ep >> 1);
                const uint64_t key = tg[f - r0];
                if (ep & 1u) {
                    if (ex.hi) ex.hi[o] = key - 1;
                    if (ex.e) ex.e[o] = pos;
                } else {
                    if (ex.lo) ex.lo[o] = key;
                    if (ex.b) ex.b[o] = pos;
                }
            }
        }
        __syncwarp();   // read before the next round's targets overwrite the list
    }
    // warp totals of the statistics: one atomic per warp and counter, no block barrier (a warp
    // that is done leaves without waiting for the rest of its block)
    if (a.scanned) plan_stats(a, S);
    if (a.cells) {
        const unsigned long long tc = warp_sum_u64(ncell), te = warp_sum_u64(nempty);
        if (lane_id() == 0 && tc) {
            atomicAdd(a.cells, tc);
            if (te) atomicAdd(a.cells + 1, te);
        }
    }
    if constexpr (Bounds::kStats) {
        if (bounds.stats) {
            const unsigned long long te = warp_sum_u64(bs.endpoints);
            const unsigned long long tm = warp_sum_u64(bs.misses);
            const unsigned long long tw = warp_sum_u64(bs.window);
            if (lane_id() == 0 && te) {
                atomicAdd(bounds.stats + 0, te);
                if (tm) atomicAdd(bounds.stats + 1, tm);
                atomicAdd(bounds.stats + 2, tw);
            }
        }
    }
    if (!active) return;
    if (!EXPORT) {
        plan_store(a, r, i, q, items);
    } else {
        for (uint32_t k = cnt; k < (uint32_t)K; ++k) {
            const uint64_t o = (uint64_t)K * i + k;
            if (ex.lo) ex.lo[o] = 1;
            if (ex.hi) ex.hi[o] = 0;
            if (ex.b) ex.b[o] = 0;
            if (ex.e) ex.e[o] = 0;
        }
        if (ex.cnt) ex.cnt[i] = cnt;
    }
}

// ------------------------------------------------------------------------------------
// Items: (query, group) pairs
// ------------------------------------------------------------------------------------
// The scans are specialised by geometry: the 2-D disc, the 2-D square window, and the 3-D
// ball (points packed into 8 bytes).
constexpr int kGeomDisc = SFC_NORM_DISC;
constexpr int kGeomSquare = SFC_NORM_SQUARE;
constexpr int kGeomBall3 = 2;

template <int GEOM>
struct Geom {
    using P = int2;
    static constexpr int kGroups = kItemGroups2;
    static __device__ __forceinline__ const P* points(const QueryArgs& a) { return a.xy; }
};
template <>
struct Geom<kGeomBall3> {
    using P = uint2;
    static constexpr int kGroups = kItemGroups3;
    static __device__ __forceinline__ const P* points(const QueryArgs& a) { return a.packed; }
};

// A query's window as the lanes hold it: x, y, delta, z (0 in 2-D).
using Window = int4;

// Exact window tests.  Disc (the problem statement's closed ball): |dx|, |dy| < 2^30, so each
// square is one signed 32x32 -> 64-bit multiply-add and the sum stays below 2^61; the test
// dx^2 + dy^2 <= delta^2 is taken as the sign of dx^2 + dy^2 - (delta^2 + 1), read from the
// high word alone (delta^2 + 1 <= 2^62, so nothing overflows).  Square (the experiments'
// windows): max(|dx|, |dy|) <= delta in 32-bit integers.  3-D ball: |dx|, |dy|, |dz| < 2^21,
// the sum of squares stays below 2^44, the same sign test.
// w: the window as a filter slot holds it (FilterSmem), c: the ball's -(delta^2 + 1).
template <int GEOM>
__device__ __forceinline__ bool is_hit(const int4& w, long long, int2 p)
{
    const int dx = p.x - w.x, dy = p.y - w.y;
    if (GEOM == kGeomSquare) return max(abs(dx), abs(dy)) <= w.z;
    const long long c = (long long)((unsigned long long)(uint32_t)w.w << 32 | (uint32_t)w.z);
    const long long s = (long long)dx * dx + ((long long)dy * dy + c);
    return (int)(s >> 32) < 0;
}

template <int GEOM>
__device__ __forceinline__ bool is_hit(const int4& w, long long c, uint2 packed)
{
    const int3 p = unpack3(packed);
    const int dx = p.x - w.x, dy = p.y - w.y, dz = p.z - w.z;
    const long long s = (long long)dx * dx + ((long long)dy * dy + ((long long)dz * dz + c));
    return (int)(s >> 32) < 0;
}

__device__ __forceinline__ int2 ldg_points(const int2* p) { return __ldg(p); }
__device__ __forceinline__ uint2 ldg_points(const uint2* p) { return __ldg(p); }

// Where the box of a group of points lies: out, no point of it is in the window; in, every point is;
// neither, the points have to be looked at.  The nearest and farthest points of the box are
// tested with the window's own arithmetic (the same bounds on every term).
struct BoxSide {
    bool out, in;
};

// 2-D box (x0, y0, x1, y1); d2 = delta^2.
template <int GEOM>
__device__ __forceinline__ BoxSide box_side(const Window& w, long long d2, const int4& b)
{
    const int nx = max(max(b.x - w.x, w.x - b.z), 0), fx = max(w.x - b.x, b.z - w.x);
    const int ny = max(max(b.y - w.y, w.y - b.w), 0), fy = max(w.y - b.y, b.w - w.y);
    if (GEOM == kGeomSquare) return {max(nx, ny) > w.z, max(fx, fy) <= w.z};
    return {(long long)nx * nx + (long long)ny * ny > d2, (long long)fx * fx + (long long)fy * fy <= d2};
}

// 3-D box.
__device__ __forceinline__ BoxSide box3_side(const Window& w, long long d2, const int4& lo, const int4& hi)
{
    const int nx = max(max(lo.x - w.x, w.x - hi.x), 0), fx = max(w.x - lo.x, hi.x - w.x);
    const int ny = max(max(lo.y - w.y, w.y - hi.y), 0), fy = max(w.y - lo.y, hi.y - w.y);
    const int nz = max(max(lo.z - w.w, w.w - hi.z), 0), fz = max(w.w - lo.z, hi.z - w.w);
    return {(long long)nx * nx + (long long)ny * ny + (long long)nz * nz > d2,
            (long long)fx * fx + (long long)fy * fy + (long long)fz * fz <= d2};
}

// Two neighbouring 16-byte records, 32-byte aligned, in one load: a lane's boxes lie side by side,
// so the widest load touches the fewest cache lines per instruction.
__device__ __forceinline__ void ldg_pair(const int4* p, int4& a, int4& b)
{
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
        : "l"(p));
}

// The t-th item of a query whose ranges start at rp: the range [b, e) it belongs to (0, 0 for the
// empty item of a query without points) and the first array position p0 of its groups.  Ranges
// of one query may touch the same item; each then has its own for it.
template <int kGroups>
__device__ __forceinline__ uint2 locate_item(const uint2* __restrict__ rp, uint32_t kint, uint32_t t, uint32_t& p0)
{
    p0 = 0;
    for (uint32_t k = 0; k < kint; ++k) {
        const uint2 r = __ldg(rp + k);
        if (r.y <= r.x) break;
        const uint32_t c = range_items<kGroups>(r.x, r.y);
        if (t < c) {
            p0 = (r.x / (32 * kGroups) + t) * (32 * kGroups);
            return r;
        }
        t -= c;
    }
    return make_uint2(0u, 0u);
}

// Which of an item's positions 32 u .. 32 u + 31 lie in [lo, hi) (0 <= lo, hi <= the item's length).
__device__ __forceinline__ uint32_t group_mask(int lo, int hi, int u)
{
    // ones from bit max(lo - 32 u, 0) on, none past 31 (the shift clamps at 32)
    return __funnelshift_lc(0u, 0xffffffffu, max(lo - 32 * u, 0)) & ~__funnelshift_lc(0u, 0xffffffffu, max(hi - 32 * u, 0));
}

// Per-warp shared memory of the filter: the groups whose points have to be looked at, side by
// side, and their hit words.  A slot is read with one or two broadcast loads: disc (x, y,
// -(delta^2 + 1)) and the first position apart (four positions per load), square (x, y, delta,
// position), ball (x, y, z, position) and -(delta^2 + 1).
template <int GEOM>
struct FilterSmem {
    static constexpr int kSlots = 32 * Geom<GEOM>::kGroups;   // groups per batch of items
    static_assert(Geom<GEOM>::kGroups <= 4, "a lane keeps its groups' slots in the bytes of one word");
    int4 w[kSlots];
    unsigned long long c[GEOM == kGeomBall3 ? kSlots : 1];
    alignas(16) uint32_t p[GEOM == kGeomDisc ? kSlots : 1];
    alignas(16) uint32_t hits[kSlots];
};

// Slots are read four at a time; the ones past the last hold an earlier group or, at the start,
// position 0.  Every lane of the warp calls.
template <int GEOM>
__device__ __forceinline__ void filter_init(FilterSmem<GEOM>* sm)
{
    for (uint32_t k = lane_id(); k < FilterSmem<GEOM>::kSlots; k += 32) {
        sm->w[k] = make_int4(0, 0, 0, 0);
        if (GEOM == kGeomDisc) sm->p[k] = 0;
        if (GEOM == kGeomBall3) sm->c[k] = 0;
    }
    __syncwarp();
}

// The hit bits of every lane's item: the groups at p0, p0 + 32, ... inside the range r, window w.
// Groups that need their points looked at are gathered in shared memory and taken four at a
// time, so that four coalesced loads are in flight.  The points' array is padded to whole
// groups.  Every lane of the warp calls.
// Much of the pass is instruction issue: a group's side, mask and shared-memory slot are made in one step (all
// classes first, then masks, then slots: count pass of 10^6 queries over 10^7 mixed points 586 us
// against 564, square windows over Normal points 120 against 110), with masks of two clamped shifts.
template <int GEOM>
__device__ __forceinline__ void filter_items(const QueryArgs& a, const Window& w, uint2 r, uint32_t p0,
                                             uint32_t (&word)[Geom<GEOM>::kGroups], FilterSmem<GEOM>* sm)
{
    constexpr int kGroups = Geom<GEOM>::kGroups;
    using P = typename Geom<GEOM>::P;
    const unsigned lane = lane_id();
    const P* __restrict__ pts = Geom<GEOM>::points(a) + lane;
    uint32_t cnt = 0, slots = 0;   // byte u: 0x80 | slot of group u when its points are looked at
    const bool item = r.y > r.x;
    const int lo = r.x > p0 ? (int)(r.x - p0) : 0, hi = item ? (int)min(r.y - p0, 32u * kGroups) : 0;
    const long long d2 = (long long)w.z * w.z, c = ~d2;   // -(delta^2 + 1)
    __syncwarp();   // the previous groups have been read
#pragma unroll
    for (int v = 0; v < kGroups; v += GEOM == kGeomBall3 ? 1 : 2) {
        int4 b[2] = {make_int4(0, 0, 0, 0), make_int4(0, 0, 0, 0)};   // two boxes, or the two corners of one
        if (item) ldg_pair(a.box + (GEOM == kGeomBall3 ? 2 : 1) * (uint64_t)((p0 >> 5) + v), b[0], b[1]);
#pragma unroll
        for (int u = v; u < v + (GEOM == kGeomBall3 ? 1 : 2); ++u) {
            BoxSide side;
            if constexpr (GEOM == kGeomBall3) side = box3_side(w, d2, b[0], b[1]);
            else side = box_side<GEOM>(w, d2, b[u - v]);
            word[u] = side.out ? 0u : group_mask(lo, hi, u);
            const bool look = word[u] != 0 && !side.in;
            const uint32_t edge = __ballot_sync(0xffffffffu, look);
            if (look) {
                const uint32_t s = cnt + __popc(edge & lanemask_lt()), p = p0 + 32 * u;
                slots |= (0x80u | s) << (8 * u);
                if (GEOM == kGeomDisc) {
                    sm->w[s] = make_int4(w.x, w.y, (int)c, (int)(c >> 32));
                    sm->p[s] = p;
                } else if (GEOM == kGeomSquare) {
                    sm->w[s] = make_int4(w.x, w.y, w.z, (int)p);
                } else {
                    sm->w[s] = make_int4(w.x, w.y, w.w, (int)p);
                    sm->c[s] = (unsigned long long)c;
                }
            }
            cnt += __popc(edge);
        }
    }
    if (cnt == 0) return;
    __syncwarp();
    constexpr uint32_t U = 4;
#pragma unroll 1
    for (uint32_t k = 0; k < cnt; k += U) {
        P p[U];
        if (GEOM == kGeomDisc) {
            const uint4 pos = *reinterpret_cast<const uint4*>(sm->p + k);
            p[0] = ldg_points(pts + pos.x);
            p[1] = ldg_points(pts + pos.y);
            p[2] = ldg_points(pts + pos.z);
            p[3] = ldg_points(pts + pos.w);
        } else {
#pragma unroll
            for (uint32_t u = 0; u < U; ++u) p[u] = ldg_points(pts + (uint32_t)sm->w[k + u].w);
        }
        uint32_t h[U];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
            const long long cc = GEOM == kGeomBall3 ? (long long)sm->c[k + u] : 0;
            h[u] = __ballot_sync(0xffffffffu, is_hit<GEOM>(sm->w[k + u], cc, p[u]));
        }
        if (lane == 0) *reinterpret_cast<uint4*>(sm->hits + k) = make_uint4(h[0], h[1], h[2], h[3]);
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < kGroups; ++u)
        if ((slots >> (8 * u)) & 0x80u) word[u] &= sm->hits[(slots >> (8 * u)) & 0x7fu];
}

// Warp-cooperative search: the query owning item g (largest q with base[q] <= g).  Ordinary loads: base
// is what the kernel before wrote (after_wait).
__device__ __forceinline__ uint64_t owner_query(const uint64_t* base, uint64_t m, uint64_t g)
{
    uint64_t lo = 0, hi = m;   // base[lo] <= g < base[hi]
    const unsigned lane = lane_id();
    while (hi - lo > 1) {
        const uint64_t step = (hi - lo + 31) >> 5;
        const uint64_t pos = lo + lane * step;
        const bool le = pos < hi && base[pos] <= g;
        const uint32_t bal = __ballot_sync(0xffffffffu, le);
        const int last = 31 - __clz(bal);
        const uint64_t nlo = lo + (uint64_t)last * step;
        const uint64_t nhi = min(hi, nlo + step);
        lo = nlo;
        hi = nhi;
    }
    return lo;
}

// Batches a warp takes per grab: at most `most`, and few enough that every warp of the grid takes
// four times, so that short batches spread over all of them.
__device__ __forceinline__ uint32_t grab_size(uint64_t batches, uint32_t most)
{
    const uint64_t share = batches / ((uint64_t)gridDim.x * (kThreads / 32) * 4);
    return (uint32_t)max((uint64_t)1, min(share, (uint64_t)most));
}

__device__ __forceinline__ uint32_t lanemask_le() { return lanemask_lt() | (1u << lane_id()); }

// ------------------------------------------------------------------------------------
// count_kernel
// ------------------------------------------------------------------------------------
// Bound by instruction issue and by the latency of the boxes and points, which come from L2: it issues in
// 60% of its cycles at 10^6 queries over 10^7 points and 68% at 10^7 over 10^8, and its warps wait on
// loads for most of the rest (43 of 64 resident).  So the design spends as few instructions per
// scanned point as it can: a lane settles 32 points with one box (about 12 instructions), a warp
// tests 32 points with about 10, and only where a box is cut by the window's edge.  Measured, count pass only, before (every scanned point tested, a warp per chunk
// of one query) and now: 10^7 queries over 10^8 mixed points, cover 1 (1.48*10^10 scanned points)
// 12.8 -> 5.4 ms; 10^6 over 10^7 1.20 -> 0.56 ms; 10^6 3-D balls over 10^7 3.87 -> 1.66 ms.  Blocks per
// SM, 10^6 over 10^7 mixed points / Normal points and square windows / 3-D: five 592 / 114 / 1637 us,
// six 564 / 110 / 1657, seven 637 / 146 / 1601 (spills).
//
// Every query owns at least one item, so the owners of 32 consecutive items follow from the
// owner of the first and one load of the next 32 queries' first items (past the last query the
// end of the list stands in, whose items belong to the query rank m: none).
template <int GEOM>
__global__ void __launch_bounds__(kThreads, kCountBlocks) count_kernel(QueryArgs a)
{
    chain_start();
    constexpr int kGroups = Geom<GEOM>::kGroups;
    __shared__ FilterSmem<GEOM> s_filter[kThreads / 32];
    FilterSmem<GEOM>* sm = &s_filter[threadIdx.x >> 5];
    const unsigned lane = lane_id();
    const uint32_t le = lanemask_le();
    filter_init(sm);
    const uint32_t m = (uint32_t)a.m;
    const uint64_t nb = (a.gbase[m] + 31) >> 5;
    const uint32_t grab = grab_size(nb, a.cgrab);
    uint32_t slab_pos = 0, slab_left = 0;   // this warp's part of the record buffer
    while (true) {
        uint64_t b0 = 0;
        if (lane == 0) b0 = atomicAdd(a.work_ctr + kCtrCount, (unsigned long long)grab);
        b0 = __shfl_sync(0xffffffffu, b0, 0);
        if (b0 >= nb) break;
        const uint32_t left = (uint32_t)min(nb - b0, (uint64_t)grab);
        uint32_t r0 = (uint32_t)owner_query(a.gbase, m, b0 * 32);   // owner of the batch's first item
        uint32_t t0 = (uint32_t)(b0 * 32 - __ldg(a.gbase + r0));    // ... and which of its items it is
        for (uint32_t k = 0; k < left; ++k) {
            const uint64_t b = b0 + k;
            // where the following queries begin, relative to the batch
            const uint64_t nx = __ldg(a.gbase + r0 + min(lane + 1, m - r0)) - b * 32;
            const uint32_t start = __reduce_or_sync(0xffffffffu, nx < 32 ? 1u << (uint32_t)nx : 0u);
            const bool next_starts = __any_sync(0xffffffffu, nx == 32);
            const uint32_t before = start & le;
            const uint32_t roff = __popc(before), r = r0 + roff;
            const uint32_t first = 31 - __clz(before | 1);   // the lane of this query's first item here
            Window w = make_int4(0, 0, 0, 0);
            uint2 range = make_uint2(0u, 0u);
            uint32_t p0 = 0;
            if (r < m) {
                w = __ldg(a.qrec + r);
                range = locate_item<kGroups>(a.ranges + (uint64_t)r * a.kint, a.kint, before ? lane - first : t0 + lane, p0);
            }
            uint32_t word[kGroups];
            filter_items<GEOM>(a, w, range, p0, word, sm);
            // hits and records up to each item, in the two halves of one word
            uint32_t v = 0;
#pragma unroll
            for (int u = 0; u < kGroups; ++u) v += __popc(word[u]) + (word[u] ? 1u << 16 : 0u);
            const uint32_t incl = warp_incl_scan_u32(v), excl = incl - v;
            const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
            // hits per query: the last item of each query's run adds the run's sum
            const uint32_t sum = (incl - __shfl_sync(0xffffffffu, excl, first)) & 0xffffu;
            if ((lane == 31 || ((start >> 1) >> lane) & 1u) && sum)
                atomicAdd(a.counts + (a.perm ? __ldg(a.perm + r) : r), sum);
            if (a.pstart && (lane == 0 ? t0 == 0 : (start >> lane) & 1u) && r < m) a.pstart[r] = excl & 0xffffu;
            // the batch's records
            const uint32_t cnt = total >> 16;
            bool kept = b < a.cap_batches;
            if (kept && cnt > slab_left) {
                unsigned long long p = 0;
                if (lane == 0) p = atomicAdd(a.work_ctr + kCtrRecs, (unsigned long long)a.slab);
                p = __shfl_sync(0xffffffffu, p, 0);
                kept = p + a.slab <= a.cap_recs;
                slab_pos = (uint32_t)p;
                slab_left = kept ? a.slab : 0;
            }
            if (b < a.cap_batches && lane == 0) {
                a.heads[b] = make_uint4(r0, kept ? cnt : 0u, slab_pos, 0u);
                a.bhits[b] = total & 0xffffu;
            }
            if (kept) {
                uint32_t s = slab_pos + (excl >> 16);
#pragma unroll
                for (int u = 0; u < kGroups; ++u)
                    if (word[u]) a.recs[s++] = make_uint2(word[u], (p0 + 32 * u) | roff);
                slab_pos += cnt;
                slab_left -= cnt;
            } else {   // the queries of this batch are written by refilter_kernel
                if (r < m) a.ovf[r] = 1;
                if (lane == 0) a.work_ctr[kCtrOverflow] = 1;
            }
            t0 = start ? 32 - (31 - __clz(start)) : t0 + 32;
            r0 += __popc(start);
            if (next_starts) {
                ++r0;
                t0 = 0;
            }
        }
    }
}

// ------------------------------------------------------------------------------------
// write_kernel
// ------------------------------------------------------------------------------------
// Per-warp shared memory of a copy: up to 32 records (hit word, first position, output
// pointer).  A slot past the last has an empty word.
struct CopySmem {
    ulonglong2 it[32 + kCopyUnroll];
};

// Writes the ids of every lane's record (hit word, first position p0) to out_ids[dst ...), the
// hits in order; with !fits, ids whose slot is past the capacity are dropped.  Six records at a
// time: the id loads of their 32 positions are in flight together.  Lanes [0, cnt) have records.
// Every lane calls.
__device__ __forceinline__ void copy_records(const QueryArgs& a, bool fits, uint32_t cnt, uint32_t word, uint32_t p0,
                                             uint64_t dst, CopySmem* sm)
{
    const unsigned lane = lane_id();
    const uint32_t lt = lanemask_lt(), bit = 1u << lane;
    constexpr uint32_t U = kCopyUnroll;
    __syncwarp();   // the previous records have been read
    if (lane < cnt)
        sm->it[lane] = make_ulonglong2((unsigned long long)p0 << 32 | word,
                                       fits ? reinterpret_cast<unsigned long long>(a.out_ids + dst) : dst);
    if (lane < U) sm->it[cnt + lane] = make_ulonglong2(0, 0);
    __syncwarp();
    const uint32_t* __restrict__ ids = a.ids + lane;
    if (fits) {
#pragma unroll 1
        for (uint32_t k = 0; k < cnt; k += U) {
            uint32_t wd[U], id[U];
            unsigned long long o[U];
#pragma unroll
            for (uint32_t u = 0; u < U; ++u) {
                const ulonglong2 it = sm->it[k + u];
                wd[u] = (uint32_t)it.x;
                o[u] = it.y;
                if (wd[u] & bit) id[u] = __ldg(ids + (uint32_t)(it.x >> 32));
            }
#pragma unroll
            for (uint32_t u = 0; u < U; ++u)
                if (wd[u] & bit) __stcs(reinterpret_cast<uint32_t*>(o[u]) + __popc(wd[u] & lt), id[u]);
        }
        return;
    }
    for (uint32_t k = 0; k < cnt; ++k) {
        const ulonglong2 it = sm->it[k];
        const uint32_t wd = (uint32_t)it.x;
        const uint64_t d = it.y + __popc(wd & lt);
        if ((wd & bit) && d < a.ids_capacity) a.out_ids[d] = __ldg(ids + (uint32_t)(it.x >> 32));
    }
}

// The records of the items of the queries of processing ranks [q_begin, q_end).  Bound by the
// latency of record, id and store (most ids are read from the L2, all are written once to HBM, 3.6
// TB/s) about as much as by issue (66% of its cycles at 10^6 queries over 10^7 points, with 62 of 64
// warps resident; the L1 at 73% of its rate): 4.25*10^9 ids of 10^7 queries over 10^8 mixed points in 5.6 ms, 6.1 TB/s of id reads and
// writes, 1.0 warp instructions per id (11.4 ms and 2.2 with one warp per query,
// whose dependent loads and per-hit shared-memory store set the time); 129 windows of 2*10^5 ids
// 48.8 ms -> 0.07 ms, as no warp owns a query.
__global__ void __launch_bounds__(kThreads, kWriteBlocks) write_kernel(QueryArgs a)
{
    chain_start();
    __shared__ CopySmem s_copy[kThreads / 32];
    CopySmem* sm = &s_copy[threadIdx.x >> 5];
    const unsigned lane = lane_id();
    const bool fits = a.out_offsets[a.m] <= a.ids_capacity;
    if (blockIdx.x == 0 && threadIdx.x == 0 && !fits) set_status(a.status, SFC_DEV_CAPACITY);
    const uint32_t ra = (uint32_t)a.q_begin, rb = (uint32_t)a.q_end;
    const bool all = ra == 0 && rb == (uint32_t)a.m;
    const uint64_t first = a.gbase[ra] >> 5, nb = min((a.gbase[rb] + 31) >> 5, a.cap_batches);
    const uint64_t todo = nb > first ? nb - first : 0;
    const uint32_t grab = grab_size(todo, a.wgrab);
    while (true) {
        uint64_t b0 = 0;
        if (lane == 0) b0 = atomicAdd(a.work_ctr + kCtrWrite, (unsigned long long)grab);
        b0 = __shfl_sync(0xffffffffu, b0, 0);
        if (b0 >= todo) {
            // Every warp fails to grab once, at todo rounded up and `grab` further for each that failed
            // before it.  The last one puts the queue back to its start for the next write: of another
            // slice, of the same batch again, or of a replayed capture that holds no count.
            const uint64_t others = (uint64_t)gridDim.x * (kThreads / 32) - 1;
            if (lane == 0 && b0 >= todo + others * grab) a.work_ctr[kCtrWrite] = 0;
            break;
        }
        b0 += first;
        const uint32_t left = (uint32_t)min(nb - b0, (uint64_t)grab);
        const uint4* heads = a.heads + b0;
        const uint64_t* bbase = a.bbase + b0;
        // the next batch's head, then its first records, are loaded while one is copied
        uint4 head = __ldg(heads);
        uint2 rec = lane < head.y ? __ldg(a.recs + head.z + lane) : make_uint2(0u, 0u);
        for (uint32_t k = 0; k < left; ++k) {
            const uint4 nhead = k + 1 < left ? __ldg(heads + k + 1) : make_uint4(0u, 0u, 0u, 0u);
            uint64_t base = __ldg(bbase + k);
            for (uint32_t k0 = 0;; k0 += 32) {
                const bool last = k0 + 32 >= head.y;
                const uint32_t cnt = last ? head.y - k0 : 32;
                const uint32_t r = head.x + (rec.y & 31u);
                uint64_t dst = base + (a.dbase && lane < cnt ? __ldg(a.dbase + r) : 0);
                const uint4 h2 = last ? nhead : head;
                const uint32_t l2 = last ? lane : k0 + 32 + lane;
                const uint2 nrec = l2 < h2.y ? __ldg(a.recs + h2.z + l2) : make_uint2(0u, 0u);
                const uint32_t h = __popc(rec.x);
                const uint32_t incl = warp_incl_scan_u32(h);
                dst += incl - h;
                base += __shfl_sync(0xffffffffu, incl, 31);
                copy_records(a, fits, cnt, all || (r >= ra && r < rb) ? rec.x : 0u, rec.y & ~31u, dst, sm);
                rec = nrec;
                if (last) break;
            }
            head = nhead;
        }
    }
}

// Queries of processing ranks [q_begin, q_end) whose items did not all get records (their
// other items' ids, which write_kernel has written, are written again with the same values).
template <int GEOM>
__global__ void __launch_bounds__(kThreads) refilter_kernel(QueryArgs a)
{
    chain_start();
    constexpr int kGroups = Geom<GEOM>::kGroups;
    __shared__ FilterSmem<GEOM> s_filter[kThreads / 32];
    __shared__ CopySmem s_copy[kThreads / 32];
    if (a.work_ctr[kCtrOverflow] == 0) return;
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    filter_init(&s_filter[warp]);
    const uint64_t warps = (uint64_t)gridDim.x * (kThreads / 32);
    for (uint64_t r = a.q_begin + (uint64_t)blockIdx.x * (kThreads / 32) + warp; r < a.q_end; r += warps) {
        if (!a.ovf[r]) continue;
        const uint64_t q = a.perm ? __ldg(a.perm + r) : r;
        uint32_t left = __ldg(a.counts + q);
        uint64_t dst = a.out_offsets[q];
        const uint32_t items = (uint32_t)(__ldg(a.gbase + r + 1) - __ldg(a.gbase + r));
        const bool fits = a.out_offsets[a.m] <= a.ids_capacity;
        const Window w = __ldg(a.qrec + r);
        for (uint32_t t0 = 0; t0 < items && left; t0 += 32) {
            uint2 range = make_uint2(0u, 0u);
            uint32_t p0 = 0, word[kGroups];
            if (t0 + lane < items) range = locate_item<kGroups>(a.ranges + r * a.kint, a.kint, t0 + lane, p0);
            filter_items<GEOM>(a, w, range, p0, word, &s_filter[warp]);
            uint32_t h = 0;
#pragma unroll
            for (int u = 0; u < kGroups; ++u) h += __popc(word[u]);
            const uint32_t incl = warp_incl_scan_u32(h);
            uint64_t d = dst + (incl - h);
#pragma unroll
            for (int u = 0; u < kGroups; ++u) {
                copy_records(a, fits, 32, word[u], p0 + 32 * u, d, &s_copy[warp]);
                d += __popc(word[u]);
            }
            const uint32_t sum = __shfl_sync(0xffffffffu, incl, 31);
            dst += sum;
            left -= sum;
        }
    }
}

// Curve order: the records' ids are counted in processing order (bbase), the output is in query
// order.  dbase[r] moves the ids of rank r from one to the other: the query's output offset
// minus the hits before its first item.
__global__ void dbase_kernel(QueryArgs a)
{
    chain_start();
    for (uint64_t r = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; r < a.m; r += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t b = a.gbase[r] >> 5;
        if (b < a.cap_batches)
            a.dbase[r] = a.out_offsets[a.perm[r]] - (a.bbase[b] + a.pstart[r]);
    }
}

// Sort key of each query for the processing order: the input slice (slices > 1: the queries are
// cut into [floor(m s / slices), floor(m (s + 1) / slices))), then the curve key of its centre.
__global__ void query_keys_kernel(const int32_t* __restrict__ q, uint64_t m, int curve, int slices, uint64_t* keys)
{
    chain_start();
    __shared__ HilbertTables tb;
    if (curve == SFC_CURVE_HILBERT) hilbert_tables_init(&tb);
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < m; i += (uint64_t)gridDim.x * blockDim.x) {
        const int2 c = reinterpret_cast<const int2*>(q)[i];
        // the top 24 of the 60 key bits (cells of side 2^18) order the queries well enough: three
        // radix passes (the sort skips the constant high digits); at 10^7 queries over 10^8
        // points, 32 bits (four passes) gave the same plan and count times and a 0.1 ms longer sort
        const uint64_t k = point_in_domain(c.x, c.y) ? curve_key(curve, &tb, (uint32_t)c.x, (uint32_t)c.y) >> 36 : (1ull << 24) - 1;
        uint64_t s = 0;
        for (int t = 1; t < slices; ++t) s += i >= m * (uint64_t)t / (uint64_t)slices;
        keys[i] = s << 24 | k;
    }
}

__global__ void reset_kernel(unsigned long long* stats, int nstats, unsigned long long* ctr, uint64_t* flags,
                             uint64_t nflags)
{
    chain_start();
    const uint64_t i = blockIdx.x * (uint64_t)kThreads + threadIdx.x;
    if (i < (uint64_t)nstats) stats[i] = 0;
    if (i < (uint64_t)kCtrWords) ctr[i] = 0;
    for (uint64_t w = i; w < nflags; w += (uint64_t)gridDim.x * kThreads) flags[w] = 0;
}

int persistent_grid(const void* fn)
{
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kThreads, 0) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    return per_sm * num_sms();
}

// Persistent grid of at most g blocks, no more than the batch's items can use.
unsigned batch_grid(const QueryArgs& a, int g)
{
    return (unsigned)std::min<uint64_t>((uint64_t)g, max_batches(a.dim, a.m, a.n, a.kint) / (kThreads / 32) + 1);
}

// Whether items of this batch can be left without a record (the launch of refilter_kernel is
// saved when they cannot): more batches than heads, or more records than the buffer holds even
// if every slab but a warp's last is left with as many free records as can be.
bool may_overflow(const QueryArgs& a)
{
    const uint64_t batches = max_batches(a.dim, a.m, a.n, a.kint), per_batch = 32 * item_groups(a.dim);
    if (batches > a.cap_batches) return true;
    if (a.slab < 2 * per_batch) return batches * a.slab > a.cap_recs;
    return 2 * batches * per_batch + (uint64_t)num_sms() * 64 * a.slab > a.cap_recs;
}

template <int GEOM>
void launch_count_geom(const QueryArgs& a, cudaStream_t st)
{
    static const int g = persistent_grid((const void*)count_kernel<GEOM>);
    launch_chain(count_kernel<GEOM>, batch_grid(a, g), kThreads, 0, st, a);
    count_launch();
}

template <int GEOM>
void launch_write_geom(const QueryArgs& a, cudaStream_t st)
{
    static const int g = persistent_grid((const void*)write_kernel);
    launch_chain(write_kernel, batch_grid(a, g), kThreads, 0, st, a);
    count_launch();
    if (may_overflow(a)) {
        launch_chain(refilter_kernel<GEOM>, num_sms() * 4, kThreads, 0, st, a);
        count_launch();
    }
}

}  // namespace

// Launches plan_kernel<Bounds, DIM, DROP, EXPORT>, opted into its dynamic shared memory (more
// than 48 KB for the finest covers) once per instantiation and device.
template <class Bounds, int DIM, int DROP, bool EXPORT>
static void plan_dispatch(const QueryArgs& a, const Bounds& bounds, const PlanExport& ex, cudaStream_t st)
{
    static bool done[64] = {false};
    constexpr size_t smem = plan_smem_bytes<DIM, DROP>();
    constexpr int T = Cover<DIM, DROP>::kThreads;
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 && !done[dev]) {
        cudaFuncSetAttribute(plan_kernel<Bounds, DIM, DROP, EXPORT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        done[dev] = true;
    }
    launch_chain(plan_kernel<Bounds, DIM, DROP, EXPORT>, (unsigned)((a.m + T - 1) / T), T, smem, st, a, bounds, ex);
    count_launch();
}

template <class Bounds, bool EXPORT>
static void plan_launch2(const QueryArgs& a, const Bounds& bounds, const PlanExport& ex, cudaStream_t st)
{
    if (a.drop == 0) plan_dispatch<Bounds, 2, 0, EXPORT>(a, bounds, ex, st);
    else if (a.drop == 1) plan_dispatch<Bounds, 2, 1, EXPORT>(a, bounds, ex, st);
    else plan_dispatch<Bounds, 2, 2, EXPORT>(a, bounds, ex, st);
}

template <bool EXPORT>
static sfc_status plan_launch(const QueryArgs& a, const LearnedModelView* lm, const PlanExport& ex, cudaStream_t st)
{
    if (a.m == 0) return SFC_OK;
    if (a.dim == 3) {
        const BinaryBounds<3> binary{a.dir, a.dir_bits, 0, 0, 0};
        if (a.drop == 0) plan_dispatch<BinaryBounds<3>, 3, 0, EXPORT>(a, binary, ex, st);
        else plan_dispatch<BinaryBounds<3>, 3, 1, EXPORT>(a, binary, ex, st);
    } else if (lm) {
        plan_launch2<LearnedBounds, EXPORT>(a, LearnedBounds{lm->root, lm->leaf, lm->fence, lm->fence_fine, lm->stats}, ex,
                                            st);
    } else {
        plan_launch2<BinaryBounds<2>, EXPORT>(a, BinaryBounds<2>{a.dir, a.dir_bits, 0, 0, 0}, ex, st);
    }
    return launch_status();
}

sfc_status launch_plan(const QueryArgs& a, const LearnedModelView* lm, cudaStream_t st)
{
    return plan_launch<false>(a, lm, PlanExport{}, st);
}

int query_intervals(int dim, int drop)
{
    if (dim == 3) return drop == 0 ? Cover<3, 0>::K : Cover<3, 1>::K;
    return drop == 0 ? Cover<2, 0>::K : (drop == 1 ? Cover<2, 1>::K : Cover<2, 2>::K);
}

static unsigned flat_grid(uint64_t m)
{
    uint64_t g = (m + kThreads - 1) / kThreads;
    const uint64_t cap = (uint64_t)num_sms() * 16;
    return (unsigned)(g < 1 ? 1 : (g > cap ? cap : g));
}

sfc_status launch_query_keys(const int32_t* q, uint64_t m, int curve, int slices, uint64_t* keys, cudaStream_t st)
{
    if (m == 0) return SFC_OK;
    launch_chain(query_keys_kernel, flat_grid(m), kThreads, 0, st, q, m, curve, slices, keys);
    count_launch();
    return launch_status();
}

sfc_status launch_reset(unsigned long long* stats, int nstats, unsigned long long* ctr, uint64_t* flags, uint64_t nflags,
                        cudaStream_t st)
{
    launch_chain(reset_kernel, flat_grid(nflags), kThreads, 0, st, stats, nstats, ctr, flags, nflags);
    count_launch();
    return launch_status();
}

sfc_status launch_dbase(const QueryArgs& a, cudaStream_t st)
{
    if (a.m == 0 || !a.dbase) return SFC_OK;
    launch_chain(dbase_kernel, flat_grid(a.m), kThreads, 0, st, a);
    count_launch();
    return launch_status();
}

sfc_status launch_count(const QueryArgs& a, cudaStream_t st)
{
    if (a.m == 0) return SFC_OK;
    if (a.dim == 3) launch_count_geom<kGeomBall3>(a, st);
    else if (a.norm == SFC_NORM_SQUARE) launch_count_geom<kGeomSquare>(a, st);
    else launch_count_geom<kGeomDisc>(a, st);
    return launch_status();
}

sfc_status launch_write(const QueryArgs& a, cudaStream_t st)
{
    if (a.m == 0) return SFC_OK;
    if (a.dim == 3) launch_write_geom<kGeomBall3>(a, st);
    else if (a.norm == SFC_NORM_SQUARE) launch_write_geom<kGeomSquare>(a, st);
    else launch_write_geom<kGeomDisc>(a, st);
    return launch_status();
}

sfc_status launch_ranges(const QueryArgs& a, const LearnedModelView* lm, uint64_t* lo, uint64_t* hi,
                         uint32_t* b, uint32_t* e, uint32_t* cnt, cudaStream_t st)
{
    QueryArgs x = a;
    x.ranges = nullptr;
    x.scanned = nullptr;
    x.cells = nullptr;
    return plan_launch<true>(x, lm, PlanExport{lo, hi, b, e, cnt}, st);
}

}  // namespace sfc
