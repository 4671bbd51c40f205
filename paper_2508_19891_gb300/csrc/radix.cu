// Construction sort: stable radix sort of (key, id) pairs by curve key ("sort them once",
// Sec. 3.1.1), one-sweep style (Adinets & Merrill, 2022), over the leading digits only.
//
// n keys of 60 bits are told apart by far fewer: the sort runs its least-significant-digit
// passes over the top bits of the keys, as many as leave only short runs of equal top bits, and
// a last local step puts each run in order.
//
//   1. sample_kernel   2,048 keys (16,384 of 2^22 or more) at hashed positions; for each number of
//                      passes, how many sampled pairs agree in the bits those passes sort
//                      estimates the mean length of the runs left over.
//                      The fewest passes with short runs are chosen (all of them if none is).
//   2. hist_kernel     one read of the input: the keys of the points are computed and written
//                      out, and the 256-bin histograms of all digits are accumulated at once.
//   3. plan_kernel     exclusive scan of each histogram (global digit offsets) and the pass
//                      plan: a digit that is the same for every key is skipped, and the
//                      source/destination of each remaining pass is chosen on the device, so
//                      the host never waits (the sort can be captured in a CUDA graph).
//   4. onesweep_kernel, once per digit: persistent blocks take tiles of 4096 keys, rank the keys
//                      per digit inside each warp (stable: item order, then lane order), combine
//                      warps in shared memory, publish the tile's digit counts, reorder the tile
//                      in shared memory by digit, start loading the next tile's keys, learn the
//                      tile's global digit offsets by decoupled look-back over earlier tiles and
//                      write the tile out in contiguous runs.  After a sort over all digits the
//                      last pass writes the final arrays and decodes each key back into its
//                      coordinates.
//   5. fix_kernel      (fewer digits) every key looks at its neighbours with equal top bits: those
//                      before it that are larger and those after it that are smaller give its
//                      final place; writes the final arrays and decodes the coordinates, which
//                      replaces a random gather xy[id] by a streaming write.
//   6. long_kernel     runs too long for that (many equal points, or what the sample missed): one
//                      block sorts each by the remaining bits.
//
// Look-back words are tagged with a per-pass epoch, so stale words from earlier passes or
// sorts read as "not ready" and the buffer never needs clearing.  The epoch counter lives in
// device memory and is advanced by plan_kernel, so a sort replayed from a CUDA graph still
// gets fresh epochs.  Every wait is bounded (SFC_DEV_TIMEOUT).
#include <algorithm>

#include "sfc_internal.cuh"
#include "sizes.cuh"

namespace sfc {

namespace {

constexpr int kBits = 8;
constexpr int kRadix = 1 << kBits;
constexpr int kPasses = 8;
// threads of a pass's block, keys per thread of a tile, and resident blocks per SM (the register
// budget)
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kSortBlocks = 3;
constexpr int kLookBack = 4;                    // earlier tiles' words that a thread has in flight
constexpr int kItems = 16;                      // keys per thread: tiles of 4096 ...
constexpr int kItemsSmall = 4;                  // ... and of 1024 while those do not fill the GPU
static_assert(kThreads >= kRadix && kItems % 2 == 0, "thread d owns digit d; two ranks per word");
constexpr int kHistThreads = 1024;
// Sample: keys looked at (large arrays; smaller ones), and the mean number of others in a key's run
// up to which fewer passes are made (a run of L keys costs each of them L comparisons in shared
// memory, a pass 24 bytes of traffic and the ranking).
constexpr int kSampleLarge = 16384, kSampleSmall = 2048;
constexpr uint64_t kSampleLargeFrom = 1ull << 22;
constexpr uint64_t kSampleMin = 8192;           // shorter arrays are sorted by all digits
// Fewer passes were faster at every mean measured: builds of 10^6 uniform points in runs of 16 78.9 us,
// 88.2 with a pass more, of 1.6*10^6 in runs of 24 96.4 and 105.6; sorts of 1.7*10^7 keys in runs of 16 599 and
// 666 us, of 3.4*10^7 in runs of 32 1195 and 1250.  The line is lower, as the estimate scatters by 8 to
// 20% and the runs of uneven points are partly much longer than the mean.
constexpr uint64_t kMeanRun = 20;
// Longest run that fix_kernel orders.
constexpr uint32_t kMaxRun = 512;   // a power of two

struct PassPlan {
    uint32_t active;
    uint32_t src;   // 0 = sort source, 1 = tmp 0, 2 = tmp 1
    uint32_t dst;   // 1 = tmp 0, 2 = tmp 1, 3 = final destination
    uint32_t shift;
};

struct Small {
    uint32_t hist[kPasses][kRadix];
    uint32_t offs[kPasses][kRadix];
    PassPlan plan[kPasses];
    uint32_t tile_ctr[kPasses];
    uint32_t epoch_base;   // epoch of pass 0 of this sort (pass p uses epoch_base + p)
    uint32_t passes;       // chosen by the sample (0: all)
    uint32_t low;          // bits below the sorted ones, for fix_kernel to order by
    uint32_t from;         // where they lie before it: 1 = tmp 0, 2 = tmp 1
    uint32_t runs;         // long runs
    uint32_t run_ctr;      // ... taken
};

constexpr uint64_t kFlagAgg = 1ull << 32;
constexpr uint64_t kFlagPrefix = 2ull << 32;

// word = value (32 bits) | flag (2 bits) << 32 | epoch (30 bits) << 34
__device__ __forceinline__ uint64_t lb_word(uint32_t value, uint64_t flag, uint32_t epoch)
{
    return (uint64_t)value | flag | ((uint64_t)epoch << 34);
}

// Lowest bit that a sort of `passes` digits of a key of `bits` bits looks at.
__device__ __forceinline__ int low_bits(int bits, int passes) { return max(bits - kBits * passes, 0); }

template <int CURVE>
__device__ __forceinline__ uint64_t source_key(const SortSource& s, const HilbertTables* tb, uint64_t i)
{
    if (s.points) {
        int2 p = __ldg(s.points + i);
        return curve_key(CURVE, tb, (uint32_t)p.x & (kSide - 1), (uint32_t)p.y & (kSide - 1));
    }
    return __ldg(s.keys + i);
}

// Chooses the number of passes (one block).  Of S sampled keys, C pairs agree in their top bits: the
// run of a key is about n * 2 C / S^2 keys long, itself counted (a position may be drawn twice): at most
// kMeanRun others and itself.
template <int CURVE, int SAMPLE>
__global__ void __launch_bounds__(1024) sample_kernel(SortSource src, uint64_t n, Small* sm)
{
    chain_start();
    __shared__ HilbertTables tb;
    __shared__ uint32_t s_pairs, s_live[2];   // 32-bit words: 64-bit shared atomics retry under contention
    constexpr uint32_t kSlots = 2 * SAMPLE;
    extern __shared__ uint32_t s_slots[];            // kSlots fingerprints, then their 16-bit counts
    uint32_t* s_count = s_slots + kSlots;
    if (CURVE == SFC_CURVE_HILBERT && src.points) hilbert_tables_init(&tb);
    constexpr int K = SAMPLE / 1024;
    uint64_t key[K], live = 0;
#pragma unroll
    for (int i = 0; i < K; ++i) key[i] = source_key<CURVE>(src, &tb, sample_position(i * 1024 + threadIdx.x, SAMPLE, n));
    // bits in which the sampled keys differ: passes above them leave one run
    const uint64_t first = source_key<CURVE>(src, &tb, 0);
#pragma unroll
    for (int i = 0; i < K; ++i) live |= key[i] ^ first;
    if (threadIdx.x < 2) s_live[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t l0 = __reduce_or_sync(0xffffffffu, (uint32_t)live), l1 = __reduce_or_sync(0xffffffffu, (uint32_t)(live >> 32));
    if (lane_id() == 0) {
        atomicOr(&s_live[0], l0);
        atomicOr(&s_live[1], l1);
    }
    __syncthreads();
    live = (uint64_t)s_live[1] << 32 | s_live[0];
    const int all = (src.bits + kBits - 1) / kBits;
    const int top = live ? 63 - __clzll((long long)live) : 0;
    // pairs of short runs (all pairs there are: SAMPLE^2 / 2 < 2^27)
    const uint32_t most = (uint32_t)min((kMeanRun + 1) * SAMPLE * SAMPLE / (2 * n), (uint64_t)SAMPLE * SAMPLE);
    int passes = 2;
    for (; passes < all; ++passes) {
        const int low = low_bits(src.bits, passes);
        // 2^(top + 1 - low) values of the sorted bits cannot keep n keys apart
        if (top + 1 <= low || (top + 1 - low < 32 && (kMeanRun << (top + 1 - low)) < n)) continue;
        for (uint32_t i = threadIdx.x; i < kSlots + kSlots / 2; i += 1024) s_slots[i] = 0;
        if (threadIdx.x == 0) s_pairs = 0;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < K; ++i) {
            if (*(volatile uint32_t*)&s_pairs > most) break;   // long runs, however many more
            // 32-bit fingerprint of the top bits (multiplicative hashing), never 0
            const uint64_t h = (key[i] >> low) * 0x9e3779b97f4a7c15ull;
            const uint32_t f = (uint32_t)(h >> 32) | 1u;
            uint32_t at = (uint32_t)(h >> 40) & (kSlots - 1);
            for (uint32_t t = 0; t < kSlots; ++t) {
                uint32_t old = *(volatile uint32_t*)(s_slots + at);
                if (old == 0u) old = atomicCAS(&s_slots[at], 0u, f);
                if (old == 0u || old == f) break;
                at = (at + 1) & (kSlots - 1);
            }
            const uint32_t sh = 16 * (at & 1);
            const uint32_t earlier = (atomicAdd(&s_count[at >> 1], 1u << sh) >> sh) & 0xffffu;
            if (earlier) atomicAdd(&s_pairs, earlier);
        }
        __syncthreads();
        if (s_pairs <= most) break;
        __syncthreads();
    }
    if (threadIdx.x == 0) sm->passes = (uint32_t)passes;
}

// Digit counts of a block: a row per digit with a 16-bit counter per lane (two lanes a word), so
// the 32 lanes' increments meet at most two deep whatever the digits are (one counter per digit
// takes random digits three to four deep and equal ones one by one).  A block counts at most
// 2^21 keys, a lane's counter at most 2^16 - 1.
constexpr int kHistRow = 16;
constexpr uint64_t kHistMost = 65000ull * 32;

// Histograms of the sorted digits, one read of the input; the keys of a sort of points are written
// out for the first pass.  16 bytes per key: 10^8 points, four digits 0.59 -> 0.47 ms, 3.4 TB/s (one shared counter
// per digit, keys computed again by the first pass).
template <int CURVE>
__global__ void __launch_bounds__(kHistThreads) hist_kernel(SortSource src, uint64_t n, uint64_t* keys_out, Small* sm,
                                                            uint32_t* status)
{
    chain_start();
    __shared__ HilbertTables tb;
    extern __shared__ uint32_t s_rows[];   // [passes][kRadix][kHistRow]
    if (CURVE == SFC_CURVE_HILBERT && src.points) hilbert_tables_init(&tb);
    const int passes = sm->passes ? (int)sm->passes : (src.bits + kBits - 1) / kBits;
    const int low = low_bits(src.bits, passes);
    for (int i = threadIdx.x; i < passes * kRadix * kHistRow; i += kHistThreads) s_rows[i] = 0;
    __syncthreads();
    uint32_t* mine = s_rows + (lane_id() & 15);
    const uint32_t one = lane_id() & 16 ? 1u << 16 : 1u;
    bool bad = false;
    const uint64_t stride = (uint64_t)gridDim.x * kHistThreads;
    // four elements of the grid stride per iteration, their loads issued together
    for (uint64_t i0 = (uint64_t)blockIdx.x * kHistThreads + threadIdx.x; i0 < n; i0 += 4 * stride) {
        uint64_t kk[4];
        if (src.points) {
            int2 pt[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint64_t i = i0 + u * stride;
                pt[u] = i < n ? __ldcs(src.points + i) : make_int2(0, 0);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint64_t i = i0 + u * stride;
                bad |= i < n && !point_in_domain(pt[u].x, pt[u].y);
                kk[u] = curve_key(CURVE, &tb, (uint32_t)pt[u].x & (kSide - 1), (uint32_t)pt[u].y & (kSide - 1));
                if (i < n) keys_out[i] = kk[u];
            }
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint64_t i = i0 + u * stride;
                kk[u] = i < n ? __ldg(src.keys + i) : 0;
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (i0 + u * stride >= n) break;
            const uint64_t k = kk[u] >> low;
#pragma unroll
            for (int p = 0; p < kPasses; ++p) {
                if (p >= passes) break;
                const uint32_t d = (uint32_t)(k >> (kBits * p)) & (kRadix - 1);
                atomicAdd(mine + (p * kRadix + d) * kHistRow, one);
            }
        }
    }
    if (bad) set_status(status, SFC_DEV_BAD_POINT);
    __syncthreads();
    for (int i = threadIdx.x; i < passes * kRadix; i += kHistThreads) {
        uint32_t c = 0;
#pragma unroll
        for (int j = 0; j < kHistRow; ++j) {
            const uint32_t w = s_rows[i * kHistRow + ((j + i) & (kHistRow - 1))];
            c += (w & 0xffffu) + (w >> 16);
        }
        if (c) atomicAdd(&(&sm->hist[0][0])[i], c);
    }
}

// One block of 256 threads (thread = digit).
__global__ void __launch_bounds__(kRadix) plan_kernel(Small* sm, uint64_t n, int bits, uint32_t* epoch_ctr)
{
    chain_start();
    if (threadIdx.x == 0) {
        // 30-bit epochs, never 0 (the value of a cleared word); wraps after 2^27 sorts
        uint32_t e = *epoch_ctr;
        if (e + kPasses >= (1u << 30)) e = 0;
        sm->epoch_base = e + 1;
        *epoch_ctr = e + kPasses;
    }
    __shared__ uint32_t s_const[kPasses];
    __shared__ uint32_t s_w[kRadix / 32];
    const int d = threadIdx.x, lane = d & 31, warp = d >> 5;
    const int passes = sm->passes ? (int)sm->passes : (bits + kBits - 1) / kBits;
    const int low = low_bits(bits, passes);
    for (int p = 0; p < passes; ++p) {
        uint32_t c = sm->hist[p][d];
        uint32_t full = __syncthreads_or(c == (uint32_t)n);
        if (d == 0) s_const[p] = full;
        // block exclusive scan of the 256 counts
        uint32_t v = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += t;
        }
        if (lane == 31) s_w[warp] = v;
        __syncthreads();
        uint32_t wo = 0;
        for (int w = 0; w < warp; ++w) wo += s_w[w];
        sm->offs[p][d] = wo + v - c;
        __syncthreads();
    }
    if (d == 0) {
        int act[kPasses], k = 0;
        for (int p = 0; p < passes; ++p)
            if (!s_const[p]) act[k++] = p;
        if (k == 0) act[k++] = 0;   // every digit constant: one pass still copies the data
        for (int p = 0; p < kPasses; ++p) sm->plan[p] = PassPlan{0, 0, 0, 0};
        sm->low = (uint32_t)low;
        for (int j = 0; j < k; ++j) {
            PassPlan pl;
            pl.active = 1;
            pl.src = j == 0 ? 0u : 1u + ((j - 1) & 1);
            pl.dst = j == k - 1 && low == 0 ? 3u : 1u + (j & 1);
            pl.shift = (uint32_t)(low + kBits * act[j]);
            sm->from = pl.dst;
            sm->plan[act[j]] = pl;
        }
    }
}

struct PassArgs {
    SortSource src;
    uint64_t* tmp_keys[2];
    uint32_t* tmp_vals[2];
    SortDest dst;
    uint64_t* lookback;   // [tile][digit]
    uint2* runs;          // long runs: first position, length
    Small* sm;
    uint64_t n;
    uint32_t* status;
    int pass;
};

// Shared memory of a pass's block.
template <int ITEMS>
struct PassSmem {
    static constexpr int kTile = kThreads * ITEMS;
    uint64_t keys[kTile];
    uint32_t vals[kTile];
    uint32_t hist[kWarps][kRadix];
    uint32_t match[kWarps][kRadix];
    uint32_t gbase[kRadix];   // global start of the digit's run minus its tile-local start
    uint32_t w[kRadix / 32];  // warp totals of the tile-local scan
    uint32_t tile;
    HilbertTables tb;
};

// Keys of a tile in the order of the ranking: item i of lane l is key wbase + 32 i + l.
template <int ITEMS>
__device__ __forceinline__ void load_keys(const PassArgs& a, const PassPlan& pl, uint32_t wbase, uint64_t (&key)[ITEMS])
{
    constexpr uint32_t kTile = kThreads * ITEMS;
    const uint32_t n = (uint32_t)a.n;
    const uint64_t* kin = pl.src == 0 ? a.src.keys : a.tmp_keys[pl.src - 1];
    const bool full = (uint64_t)wbase - wbase % kTile + kTile <= n;   // block-uniform
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const uint32_t idx = wbase + (uint32_t)(i * 32) + lane_id();
        key[i] = full || idx < n ? __ldcs(kin + idx) : ~0ull;
    }
}

// Ranks a warp's keys by the digit at `shift`, stable (item order, then lane order): rank[i] (two
// per word) is how many of the warp's earlier keys share key i's digit; wh counts the warp's keys
// per digit (zero on entry).  The lanes that share a digit find each other in wm[digit], where
// each sets its bit (all zero on entry and exit): about 16 instructions per key and warp, where
// comparing digits bit by bit with eight ballots took 36 (10^7 keys: a pass 85 -> 81 us).  Keys at
// or past n are not counted.
template <bool FULL, int ITEMS>
__device__ __forceinline__ void rank_keys(const uint64_t (&key)[ITEMS], int shift, uint32_t wbase, uint32_t n, uint32_t* wh,
                                          uint32_t* wm, uint32_t (&rank)[ITEMS / 2])
{
    const uint32_t lt = lanemask_lt();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const bool valid = FULL || wbase + (uint32_t)(i * 32) + lane_id() < n;
        const uint32_t d = (uint32_t)(key[i] >> shift) & (kRadix - 1);
        if (valid) atomicOr(wm + d, 1u << lane_id());
        __syncwarp();
        const uint32_t peers = *(volatile uint32_t*)(wm + d);
        const uint32_t before = __popc(peers & lt);
        const uint32_t basec = wh[d];
        __syncwarp();
        if (valid && before == 0) {
            wh[d] = basec + __popc(peers);
            wm[d] = 0;
        }
        __syncwarp();
        if (i & 1) rank[i / 2] |= (basec + before) << 16;
        else rank[i / 2] = basec + before;
    }
}

// Bound by shared memory (its pipe at 74% of its rate, more than half of its wavefronts bank conflicts)
// and by the latency of the key loads with 24 warps per SM, not yet by HBM (24 bytes per key and pass:
// 10^8 keys 0.70 ms, 3.4 TB/s; 0.83 ms with one block per tile, ballots and one look-back word at a time).
// Measured at 10^8 mixed points (build): 256 threads of 16 keys 5.5 ms, 512 of 8 6.1, of 16 8.2 (two
// blocks per SM), 256 of 24 6.0; the next tile's keys loaded during the look-back 5.5 instead of
// 5.9; the values loaded before the warps are combined 5.9.
template <int CURVE, int ITEMS>
__global__ void __launch_bounds__(kThreads, kSortBlocks) onesweep_kernel(PassArgs a)
{
    chain_start();
    const PassPlan pl = a.sm->plan[a.pass];
    if (!pl.active) return;
    const uint32_t epoch = a.sm->epoch_base + (uint32_t)a.pass;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PassSmem<ITEMS>& S = *reinterpret_cast<PassSmem<ITEMS>*>(smem_raw);
    constexpr int kTile = kThreads * ITEMS, kWarpSpan = 32 * ITEMS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t n = (uint32_t)a.n;
    const uint32_t tiles = tiles_of(a.n, kTile);
    const int shift = (int)pl.shift;
    if (CURVE == SFC_CURVE_HILBERT && pl.dst == 3 && a.dst.xy) hilbert_tables_init(&S.tb);
    uint32_t *wh = S.hist[warp], *wm = S.match[warp];
    for (int d = lane; d < kRadix; d += 32) wh[d] = wm[d] = 0;
    if (tid == 0) S.tile = atomicAdd(&a.sm->tile_ctr[a.pass], 1u);
    __syncthreads();
    uint32_t tile = S.tile;
    if (tile >= tiles) return;
    const uint32_t* vin = pl.src == 0 ? a.src.vals : a.tmp_vals[pl.src - 1];
    uint64_t* kout = pl.dst == 3 ? a.dst.keys : a.tmp_keys[pl.dst - 1];
    uint32_t* vout = pl.dst == 3 ? a.dst.vals : a.tmp_vals[pl.dst - 1];
    int2* xyout = pl.dst == 3 ? a.dst.xy : nullptr;
    uint64_t key[ITEMS];
    load_keys(a, pl, tile * (uint32_t)kTile + (uint32_t)(warp * kWarpSpan), key);
    while (true) {
        const uint32_t tbase = tile * (uint32_t)kTile;
        const uint32_t wbase = tbase + (uint32_t)(warp * kWarpSpan);
        const bool full = (uint64_t)tbase + kTile <= n;
        uint32_t rank[ITEMS / 2], val[ITEMS];
        if (full) rank_keys<true>(key, shift, wbase, n, wh, wm, rank);
        else rank_keys<false>(key, shift, wbase, n, wh, wm, rank);
        __syncthreads();
        // ---- combine warps: thread d < 256 owns digit d ----
        uint32_t tcount = 0, local = 0;
        uint64_t* lbw = a.lookback + (uint64_t)tile * kRadix + tid;
        if (tid < kRadix) {
#pragma unroll
            for (int w = 0; w < kWarps; ++w) tcount += S.hist[w][tid];
            atomicExch(reinterpret_cast<unsigned long long*>(lbw),
                       lb_word(tcount, tile == 0 ? kFlagPrefix : kFlagAgg, epoch));
            // tile-local exclusive scan over digits
            uint32_t v = tcount;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += t;
            }
            if (lane == 31) S.w[warp] = v;
            local = v - tcount;
        }
        if (tid == kThreads - 1) S.tile = atomicAdd(&a.sm->tile_ctr[a.pass], 1u);   // this block's next tile
        __syncthreads();
        if (tid < kRadix) {
            // hist[w][d] becomes the tile-local position of warp w's first key of digit d
#pragma unroll
            for (int w = 0; w < kRadix / 32; ++w) local += w < warp ? S.w[w] : 0u;
            uint32_t run = local;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const uint32_t cw = S.hist[w][tid];
                S.hist[w][tid] = run;
                run += cw;
            }
        }
        __syncthreads();
        // (the values are loaded only now: the ranking holds no registers for them)
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const uint32_t idx = wbase + (uint32_t)(i * 32) + lane;
            val[i] = vin == nullptr ? a.src.val_base + idx : (full || idx < n ? __ldcs(vin + idx) : 0u);
        }
        // ---- reorder the tile by digit in shared memory ----
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if (full || wbase + (uint32_t)(i * 32) + lane < n) {
                const uint32_t d = (uint32_t)(key[i] >> shift) & (kRadix - 1);
                const uint32_t lp = wh[d] + ((rank[i / 2] >> (16 * (i & 1))) & 0xffffu);
                S.keys[lp] = key[i];
                S.vals[lp] = val[i];
            }
        }
        const uint32_t next = S.tile;
        if (next < tiles)
            load_keys(a, pl, next * (uint32_t)kTile + (uint32_t)(warp * kWarpSpan), key);
        // ---- decoupled look-back for digit tid, four tiles at a time ----
        if (tid < kRadix) {
            uint32_t excl = 0;
            if (tile > 0) {
                const uint64_t* words = a.lookback + tid;
                uint32_t t = tile, spins = 0;   // tiles below t are still to be added
                bool done = false;
                while (!done && t > 0) {
                    uint64_t w[kLookBack];
#pragma unroll
                    for (int u = 0; u < kLookBack; ++u) {
                        const uint32_t at = t > (uint32_t)u + 1 ? t - 1 - u : 0;
                        w[u] = *reinterpret_cast<const volatile uint64_t*>(words + (uint64_t)at * kRadix);
                    }
#pragma unroll
                    for (int u = 0; u < kLookBack; ++u) {
                        if (done || t == 0) break;
                        const uint32_t fl = (uint32_t)(w[u] >> 34) == epoch ? (uint32_t)(w[u] >> 32) & 3u : 0u;
                        if (fl == 0) {   // not published yet
                            if (++spins > kSpinLimit) {
                                set_status(a.status, SFC_DEV_TIMEOUT);
                                done = true;
                            } else if (u == 0) {
                                __nanosleep(32);   // leave the issue slots to other warps
                            }
                            break;
                        }
                        excl += (uint32_t)w[u];
                        done = fl == 2;
                        --t;
                    }
                }
                atomicExch(reinterpret_cast<unsigned long long*>(lbw), lb_word(excl + tcount, kFlagPrefix, epoch));
            }
            // global position of tile-local position j of digit d: gbase[d] + j (mod 2^32)
            S.gbase[tid] = a.sm->offs[a.pass][tid] + excl - local;
        }
        __syncthreads();
        // ---- write contiguous digit runs ----
        for (int d = lane; d < kRadix; d += 32) wh[d] = 0;
        const uint32_t valid_n = full ? (uint32_t)kTile : n - tbase;
#pragma unroll 4
        for (uint32_t j = tid; j < valid_n; j += kThreads) {
            const uint64_t k = S.keys[j];
            const uint32_t d = (uint32_t)(k >> shift) & (kRadix - 1);
            const uint32_t g = S.gbase[d] + j;
            if (g >= n) continue;   // only after a look-back timeout (already flagged)
            kout[g] = k;
            vout[g] = S.vals[j];
            if (xyout) {
                uint32_t x, y;
                if (CURVE == SFC_CURVE_HILBERT) hilbert_decode(&S.tb, k, x, y);
                else morton_decode(k, x, y);
                xyout[g] = make_int2((int)x, (int)y);
            }
        }
        if (next >= tiles) return;
        tile = next;
        __syncthreads();   // the tile's shared memory is free
    }
}

// Final place of one entry.
template <int CURVE>
__device__ __forceinline__ void store_final(const SortDest& dst, const HilbertTables* tb, uint32_t at, uint64_t k, uint32_t v)
{
    dst.keys[at] = k;
    dst.vals[at] = v;
    if (dst.xy) {
        uint32_t x, y;
        if (CURVE == SFC_CURVE_HILBERT) hilbert_decode(tb, k, x, y);
        else morton_decode(k, x, y);
        dst.xy[at] = make_int2((int)x, (int)y);
    }
}

constexpr int kFixThreads = 256, kFixBlocks = 4;   // four blocks per SM
constexpr int kFixItems = 8;
constexpr int kFixTile = kFixThreads * kFixItems;
constexpr int kFixHalo = 64;                         // neighbours kept on each side of the tile
constexpr int kFixSpan = kFixTile + 2 * kFixHalo;
constexpr int kFixWords = kFixSpan / 32;
constexpr int kFixAt = 12;                           // bits of a place in the span
static_assert(kFixSpan <= 1 << kFixAt && kFixHalo * 2 <= kFixThreads, "");

// Orders the runs of keys that agree in the sorted bits.  A bit per key marks where a run begins;
// a key of a run of one keeps its place, any other counts the keys of its run that come before it
// (all lanes of a run read the same shared-memory word: the low bits, then the place, so that one
// comparison decides ties too).  Bound by the issue of the counting (72%
// of its cycles, the integer pipe at 70%) before HBM (12 bytes read, 20 written per key, 3.7 TB/s):
// 10^8 mixed points in runs of up to 16 on average 0.89 ms.
template <int CURVE>
__global__ void __launch_bounds__(kFixThreads, kFixBlocks) fix_kernel(PassArgs a)
{
    chain_start();
    const uint32_t low = a.sm->low;
    if (low == 0) return;   // sorted by all digits
    __shared__ HilbertTables tb;
    __shared__ uint64_t s_keys[kFixSpan];
    __shared__ uint32_t s_head[kFixWords];
    if (CURVE == SFC_CURVE_HILBERT && a.dst.xy) hilbert_tables_init(&tb);
    const uint32_t n = (uint32_t)a.n;
    const uint64_t* keys = a.tmp_keys[a.sm->from - 1];
    const uint32_t* vals = a.tmp_vals[a.sm->from - 1];
    const uint32_t tiles = tiles_of(a.n, kFixTile);
    const uint64_t mask = (1ull << low) - 1;   // low <= 48: at least two digits are sorted
    const int tid = threadIdx.x;
    // place in the span of this thread's halo key
    const int hx = tid < kFixHalo ? tid : (tid < 2 * kFixHalo ? kFixTile + tid : -1);
    for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int64_t g0 = (int64_t)tile * kFixTile - kFixHalo;   // array position of s_keys[0]
        // the part of the array that lies in the span: [lo, hi)
        const int lo = g0 < 0 ? (int)-g0 : 0, hi = (int)min((int64_t)kFixSpan, (int64_t)n - g0);
        uint64_t key[kFixItems], hkey = 0;
        uint32_t val[kFixItems];
#pragma unroll
        for (int i = 0; i < kFixItems; ++i) {
            const int x = kFixHalo + i * kFixThreads + tid;
            key[i] = x < hi ? __ldg(keys + (g0 + x)) : 0;
        }
        if (hx >= lo && hx < hi) hkey = __ldg(keys + (g0 + hx));
#pragma unroll
        for (int i = 0; i < kFixItems; ++i) {
            const int x = kFixHalo + i * kFixThreads + tid;
            val[i] = x < hi ? __ldcs(vals + (g0 + x)) : 0u;
        }
        __syncthreads();   // the previous tile has been read
#pragma unroll
        for (int i = 0; i < kFixItems; ++i) s_keys[kFixHalo + i * kFixThreads + tid] = key[i];
        if (hx >= 0) s_keys[hx] = hkey;
        __syncthreads();
        // run begins: the array's first position and the one past its last are some too, the
        // span's ends are not
        for (int x = tid; x < kFixSpan; x += kFixThreads) {
            const bool head = x == lo ? g0 + lo == 0 : (x > lo && x < hi ? ((s_keys[x] ^ s_keys[x - 1]) >> low) != 0 : x == hi);
            const uint32_t w = __ballot_sync(0xffffffffu, head);
            if (lane_id() == 0) s_head[x >> 5] = w;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kFixItems; ++i) {
            const int x = kFixHalo + i * kFixThreads + tid;
            s_keys[x] = (key[i] & mask) << kFixAt | (uint32_t)x;
        }
        if (hx >= 0) s_keys[hx] = (hkey & mask) << kFixAt | (uint32_t)hx;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kFixItems; ++i) {
            const int x = kFixHalo + i * kFixThreads + tid;
            if (x >= hi) continue;
            // the run's first position s and one past its last e in the span (-1: beyond it)
            int w = x >> 5;
            uint32_t bits = s_head[w] & (0xffffffffu >> (31 - (x & 31)));
            while (!bits && w > 0) bits = s_head[--w];
            const int s = bits ? w * 32 + 31 - __clz(bits) : -1;
            w = x >> 5;
            bits = s_head[w] & (0xfffffffeu << (x & 31));
            while (!bits && w + 1 < kFixWords) bits = s_head[++w];
            const int e = bits ? w * 32 + __ffs(bits) - 1 : (hi < kFixSpan ? hi : -1);
            const uint64_t k = key[i];
            const uint32_t at = (uint32_t)(g0 + x);
            if (s >= 0 && e >= 0 && e - s <= (int)kMaxRun) {
                int place = x;
                if (e - s > 1) {
                    const uint64_t c = (k & mask) << kFixAt | (uint32_t)x;
                    place = s;
#pragma unroll 4
                    for (int j = s; j < e; ++j) place += s_keys[j] < c;
                }
                store_final<CURVE>(a.dst, &tb, (uint32_t)(g0 + place), k, val[i]);
                continue;
            }
            // the run reaches past the span: how many of the kMaxRun keys on each side are in it
            uint32_t before = 0, after = 0;
            for (uint32_t step = kMaxRun; step; step >>= 1) {
                const uint32_t l = min(before + step, kMaxRun), r = min(after + step, kMaxRun);
                if (l <= at && !((__ldg(keys + (at - l)) ^ k) >> low)) before = l;
                if (r < n - at && !((__ldg(keys + (at + r)) ^ k) >> low)) after = r;
            }
            if (before + after < kMaxRun) {
                uint32_t more = 0, less = 0;
                for (uint32_t j = 1; j <= before; ++j) more += __ldg(keys + (at - j)) > k;
                for (uint32_t j = 1; j <= after; ++j) less += __ldg(keys + (at + j)) < k;
                store_final<CURVE>(a.dst, &tb, at - more + less, k, val[i]);
            } else if (before == 0) {   // the first of a long run finds its end and lists it
                uint32_t l = at + 1, len = n - l;
                while (len > 0) {
                    const uint32_t half = len >> 1;
                    const bool in = !((__ldg(keys + l + half) ^ k) >> low);
                    l = in ? l + half + 1 : l;
                    len = in ? len - half - 1 : half;
                }
                a.runs[atomicAdd(&a.sm->runs, 1u)] = make_uint2(at, l - at);
            }
        }
    }
}

// Sorts the long runs by their low bits, one block per run: a stable radix sort between the two
// temporary arrays in the run's own range, then the copy to the final arrays.  A run that is in
// order already (equal points) is copied only.
template <int CURVE>
__global__ void __launch_bounds__(kThreads) long_kernel(PassArgs a)
{
    chain_start();
    const uint32_t runs = a.sm->runs;
    if (runs == 0) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PassSmem<kItems>& S = *reinterpret_cast<PassSmem<kItems>*>(smem_raw);
    constexpr int kTile = kThreads * kItems, kWarpSpan = 32 * kItems;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t *wh = S.hist[warp], *wm = S.match[warp];
    if (CURVE == SFC_CURVE_HILBERT && a.dst.xy) hilbert_tables_init(&S.tb);
    const int low = (int)a.sm->low;
    for (int d = lane; d < kRadix; d += 32) wm[d] = 0;
    while (true) {
        __syncthreads();
        if (tid == 0) S.tile = atomicAdd(&a.sm->run_ctr, 1u);
        __syncthreads();
        if (S.tile >= runs) return;
        const uint2 run = a.runs[S.tile];
        const uint64_t first = run.x, len = run.y;
        int cur = (int)a.sm->from - 1;
        bool ordered = true;
        for (uint64_t j = tid; j + 1 < len; j += kThreads)
            ordered &= a.tmp_keys[cur][first + j] <= a.tmp_keys[cur][first + j + 1];
        if (!__syncthreads_and(ordered)) {
            for (int shift = 0; shift < low; shift += kBits) {
                // digit counts of the run, then each digit's next position in it
                if (tid < kRadix) S.gbase[tid] = 0;
                __syncthreads();
                for (uint64_t j = tid; j < len; j += kThreads)
                    atomicAdd(&S.gbase[(uint32_t)(a.tmp_keys[cur][first + j] >> shift) & (kRadix - 1)], 1u);
                __syncthreads();
                uint32_t v = 0, c = 0;
                if (tid < kRadix) {
                    v = c = S.gbase[tid];
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
                        if (lane >= o) v += t;
                    }
                    if (lane == 31) S.w[warp] = v;
                }
                __syncthreads();
                if (tid < kRadix) {
                    for (int w = 0; w < warp; ++w) v += S.w[w];
                    S.gbase[tid] = v - c;
                }
                for (uint64_t t0 = 0; t0 < len; t0 += kTile) {
                    // places in the tile, which holds `left` keys
                    const uint32_t wbase = (uint32_t)(warp * kWarpSpan);
                    const uint32_t left = (uint32_t)min(len - t0, (uint64_t)kTile);
                    uint64_t key[kItems];
                    uint32_t rank[kItems / 2];
#pragma unroll
                    for (int i = 0; i < kItems; ++i) {
                        const uint32_t j = wbase + (uint32_t)(i * 32) + lane;
                        key[i] = j < left ? a.tmp_keys[cur][first + t0 + j] : ~0ull;
                    }
                    for (int d = lane; d < kRadix; d += 32) wh[d] = 0;
                    __syncwarp();
                    rank_keys<false>(key, shift, wbase, left, wh, wm, rank);
                    __syncthreads();
                    if (tid < kRadix) {
                        uint32_t next = S.gbase[tid];
                        for (int w = 0; w < kWarps; ++w) {
                            const uint32_t cw = S.hist[w][tid];
                            S.hist[w][tid] = next;
                            next += cw;
                        }
                        S.gbase[tid] = next;
                    }
                    __syncthreads();
#pragma unroll
                    for (int i = 0; i < kItems; ++i) {
                        const uint32_t j = wbase + (uint32_t)(i * 32) + lane;
                        if (j >= left) continue;
                        const uint64_t at = first + wh[(uint32_t)(key[i] >> shift) & (kRadix - 1)] +
                                            ((rank[i / 2] >> (16 * (i & 1))) & 0xffffu);
                        a.tmp_keys[cur ^ 1][at] = key[i];
                        a.tmp_vals[cur ^ 1][at] = a.tmp_vals[cur][first + t0 + j];
                    }
                    __syncthreads();
                }
                cur ^= 1;
            }
        }
        for (uint64_t j = tid; j < len; j += kThreads)
            store_final<CURVE>(a.dst, &S.tb, (uint32_t)(first + j), a.tmp_keys[cur][first + j], a.tmp_vals[cur][first + j]);
    }
}

// Opts a kernel into more than 48 KB of dynamic shared memory, once per device.
void allow_smem(const void* fn, size_t bytes, bool (&done)[64])
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || done[dev]) return;
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    done[dev] = true;
}

template <int CURVE, int SAMPLE>
void launch_sample(const PassArgs& a, cudaStream_t st)
{
    static bool ok[64] = {false};
    constexpr size_t smem = 3 * SAMPLE * sizeof(uint32_t);
    allow_smem((const void*)sample_kernel<CURVE, SAMPLE>, smem, ok);
    launch_chain(sample_kernel<CURVE, SAMPLE>, 1, 1024, smem, st, a.src, a.n, a.sm);
    count_launch();
}

template <int CURVE, int ITEMS>
void launch_pass(const PassArgs& a, cudaStream_t st)
{
    static bool ok[64] = {false};
    allow_smem((const void*)onesweep_kernel<CURVE, ITEMS>, sizeof(PassSmem<ITEMS>), ok);
    const uint32_t tiles = tiles_of(a.n, kThreads * ITEMS);
    const unsigned grid = (unsigned)std::min<uint64_t>(tiles, (uint64_t)num_sms() * kSortBlocks);
    launch_chain(onesweep_kernel<CURVE, ITEMS>, grid, kThreads, sizeof(PassSmem<ITEMS>), st, a);
    count_launch();
}

// Tiles of 1024 keys while they are all resident at once: a pass is then one short chain per
// block.
bool small_tiles(uint64_t n) { return n <= (uint64_t)kThreads * kItemsSmall * num_sms() * kSortBlocks; }

template <int CURVE>
sfc_status run_sort(const PassArgs& args, uint32_t* epoch, cudaStream_t st)
{
    PassArgs a = args;
    const int all = (a.src.bits + kBits - 1) / kBits;
    const bool sample = a.src.partial && a.n >= kSampleMin && all > 2;
    if (sample) {
        if (a.n >= kSampleLargeFrom) launch_sample<CURVE, kSampleLarge>(a, st);
        else launch_sample<CURVE, kSampleSmall>(a, st);
    }
    static bool hist_ok[64] = {false};
    const size_t hsmem = (size_t)all * kRadix * kHistRow * sizeof(uint32_t);
    allow_smem((const void*)hist_kernel<CURVE>, (size_t)kPasses * kRadix * kHistRow * sizeof(uint32_t), hist_ok);
    const uint64_t hgrid = std::min<uint64_t>((a.n + kHistThreads * 4 - 1) / (kHistThreads * 4),
                                              std::max<uint64_t>(num_sms(), a.n / kHistMost + 1));
    uint64_t* keys_out = a.src.keys_out ? a.src.keys_out : a.tmp_keys[1];
    launch_chain(hist_kernel<CURVE>, (unsigned)hgrid, kHistThreads, hsmem, st, a.src, a.n, keys_out, a.sm, a.status);
    if (a.src.points) {   // the passes read the keys
        a.src.points = nullptr;
        a.src.keys = keys_out;
    }
    launch_chain(plan_kernel, 1, kRadix, 0, st, a.sm, a.n, a.src.bits, epoch);
    count_launch(2);
    for (int p = 0; p < all; ++p) {
        a.pass = p;
        if (small_tiles(a.n)) launch_pass<CURVE, kItemsSmall>(a, st);
        else launch_pass<CURVE, kItems>(a, st);
    }
    if (sample) {
        static bool ok[64] = {false};
        const uint32_t ftiles = tiles_of(a.n, kFixTile);
        launch_chain(fix_kernel<CURVE>, (unsigned)std::min<uint64_t>(ftiles, (uint64_t)num_sms() * 8), kFixThreads, 0, st, a);
        allow_smem((const void*)long_kernel<CURVE>, sizeof(PassSmem<kItems>), ok);
        const unsigned lgrid = (unsigned)std::min<uint64_t>(a.n / kMaxRun + 1, (uint64_t)num_sms());
        launch_chain(long_kernel<CURVE>, lgrid, kThreads, sizeof(PassSmem<kItems>), st, a);
        count_launch(2);
    }
    return launch_status();
}

}  // namespace

void release_sort_ws(SortWorkspace& ws, cudaStream_t st)
{
    for (int i = 0; i < 2; ++i) {
        ws.tmp_keys[i].release(st);
        ws.tmp_vals[i].release(st);
    }
    ws.lookback.release(st);
    ws.small.release(st);
    ws.runs.release(st);
    ws.epoch_dev.release(st);
}

sfc_status reserve_sort(SortWorkspace& ws, uint64_t n, cudaStream_t st)
{
    // the look-back words of the small tiles' longest array cover shorter ones with larger tiles
    const uint64_t per = kThreads * (small_tiles(n) ? kItemsSmall : kItems);
    const uint64_t most = (uint64_t)num_sms() * kSortBlocks;   // small tiles at their limit
    const uint64_t tiles = std::max((n + per - 1) / per, std::min((n + kThreads * kItemsSmall - 1) / (kThreads * kItemsSmall), most));
    for (int i = 0; i < 2; ++i) {
        SFC_TRY(ws.tmp_keys[i].ensure(n * sizeof(uint64_t), st));
        SFC_TRY(ws.tmp_vals[i].ensure(n * sizeof(uint32_t), st));
    }
    const size_t lb_bytes = tiles * kRadix * sizeof(uint64_t);
    if (!ws.epoch_dev.ptr) {
        SFC_TRY(ws.epoch_dev.ensure(sizeof(uint32_t), st));
        SFC_CUDA_TRY(cudaMemsetAsync(ws.epoch_dev.ptr, 0, sizeof(uint32_t), st));
    }
    if (lb_bytes > ws.lookback.bytes) {
        // new words start cleared; older epochs stay distinct from future ones
        SFC_TRY(ws.lookback.ensure(lb_bytes, st));
        SFC_CUDA_TRY(cudaMemsetAsync(ws.lookback.ptr, 0, ws.lookback.bytes, st));
    }
    SFC_TRY(ws.small.ensure(sizeof(Small), st));
    SFC_TRY(ws.runs.ensure((n / kMaxRun + 1) * sizeof(uint2), st));
    return SFC_OK;
}

sfc_status radix_sort(const SortSource& src, uint64_t n, const SortDest& dst, SortWorkspace& ws,
                      uint32_t* status, cudaStream_t st)
{
    if (n == 0) return SFC_OK;
    if (n >= 0xffffffffull) return SFC_ERR_INVALID;
    if (src.points && dst.curve != src.curve) return SFC_ERR_INVALID;
    SFC_TRY(reserve_sort(ws, n, st));
    Small* sm = ws.small.as<Small>();
    SFC_CUDA_TRY(cudaMemsetAsync(sm, 0, sizeof(Small), st));
    PassArgs a;
    a.src = src;
    a.src.curve = src.points ? src.curve : dst.curve;
    for (int i = 0; i < 2; ++i) {
        a.tmp_keys[i] = ws.tmp_keys[i].as<uint64_t>();
        a.tmp_vals[i] = ws.tmp_vals[i].as<uint32_t>();
    }
    a.dst = dst;
    a.lookback = ws.lookback.as<uint64_t>();
    a.runs = ws.runs.as<uint2>();
    a.sm = sm;
    a.n = n;
    a.status = status;
    a.pass = 0;
    if (a.src.curve == SFC_CURVE_HILBERT) return run_sort<SFC_CURVE_HILBERT>(a, ws.epoch_dev.as<uint32_t>(), st);
    return run_sort<SFC_CURVE_Z>(a, ws.epoch_dev.as<uint32_t>(), st);
}

}  // namespace sfc
