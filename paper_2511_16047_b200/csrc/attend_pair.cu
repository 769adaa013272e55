// Tensor-core attention for sm_100a, paired form: softmax(scale * Q K^T) V over the resident
// token ranges of one layer, both products on tcgen05 with every accumulator in tensor memory.
//
// A CTA is persistent and walks "pairs".  A pair is two streams, A and B, each a (row, head,
// 128-query tile) that runs through the same number of 64-token key/value tiles:
//   * more than 128 query tokens: the two streams are two query tiles of ONE item, so each
//     key/value tile is fetched into shared memory once and used by both;
//   * at most 128 query tokens: the two streams are two different items with their own tiles.
// Stream B is absent when the pair has no second member.
//   warps 0-3    softmax group of stream A: one query row per thread (row = TMEM lane)
//   warps 4-7    softmax group of stream B
//   warp 8       TMA producer of the key/value tiles (ring of stages, 16 tokens per bulk copy so a
//                range's tail tile reads only the 16-token groups it needs)
//   warp 9       issues tcgen05.mma for both streams, alternating between them
// In the split form two CTAs (a cluster) share the key tiles of each pair of a launch's last round and merge O, references and
// sums through distributed shared memory.
// Per stream and tile: S = Q K^T (128 x 64 fp32 in TMEM) -> the group reads S with tcgen05.ld,
// exponentiates in exp2 form against a reference maximum, packs P to bf16 and writes it back
// over S with tcgen05.st -> O += P V with P read from TMEM.  S and P share their columns, so
// there is no shared-memory tile for P.  While one group exponentiates, the tensor pipe works
// for the other.  The reference maximum of a row is the maximum of its first tile; O and the
// row sum are rescaled only when a later tile exceeds it by more than 2^8, so for
// well-conditioned logits they are never touched.  Launches of three key tiles or more (kLazy)
// do not even take the later tiles' maxima: a tile is exponentiated against the reference as it
// stands, and only a row whose tile sum leaves the range (beyond 2^64, or not a number) makes
// its warp take the true maxima, rescale and form the tile again.  The first lane of each group fetches its
// next query tile as soon as the last S of the current one has landed.
// Every wait is bounded: one that gives up records a status code and sets a flag, its role stops, and so do the others at
// their next wait for it.  Copies and products still under way then are awaited, and the tensor memory is freed.
#include <algorithm>
#include <type_traits>

#include "kernels.cuh"
#include "sm100_ptx.cuh"

namespace amskv {

namespace {

constexpr int kQRows = 128;       // query rows per tile = TMEM lanes
constexpr int kMaxDenRuns = 16;   // runs of attended tokens a density launch can tell apart
constexpr int kQBoxRows = 32;     // query rows per bulk copy
constexpr int kKT = 64;           // key/value tokens per tile
constexpr int kKVBoxRows = 16;    // tokens per bulk copy
constexpr int kGroupWarps = 4;
constexpr int kProducerWarp = 8;
constexpr int kMmaWarp = 9;        // first MMA-issuing warp; Cfg<D>::kMmaWarps of them
constexpr int kMaxStages = 4;
constexpr float kRescaleLog2 = 8.f;
constexpr int kQSplitRows = 64;   // query tiles of at most this many rows are double-buffered inside their slot
constexpr float kLazySumLimit = 1.8446744e19f;   // 2^64: see the kLazy form of the softmax loop
// Every 6th pair of exponentials goes to the FMA pipe (0: none); swept 2, 3, 4, 6, 8.  None in density launches: a run of few keys
// shows the polynomial's error (8e-4 at most), the more where it is not in the tile whose maximum is the reference.  Masses of 480
// items, T = 256, peaked rows: off by 2.5e-5 with it (8e-6 when every run had tiles of its own and the first run the first), 4e-8
// without.  512 items, T = 256: 51.4 -> 51.8 us a call, 128 channels 81.8 -> 83.0.
constexpr int kPolyEvery = 6;

// kWide: one CTA per SM with two S buffers per stream and an issuing warp per stream (below): the form
// 128 channels use, and 64 channels in launches of at most one unit per SM; with more units 64 channels use the
// two-CTA form.
// kDen: the launch also accumulates the attention density (below): two CTAs per SM then run with three
// key/value stages, the fourth stage's 16 KB holding the per-row sums.
template <int D, bool kWide, bool kDen = false>
struct Cfg {
    static_assert(D == 64 || kWide, "128 channels always use the wide form");
    static constexpr int kHalves = D / 64;                      // 128-byte swizzle atoms per row
    static constexpr int kStages = (kDen && !kWide) ? 3 : 4;
    static constexpr uint32_t kQBytes = kQRows * D * 2;         // one query tile
    static constexpr uint32_t kQHalfBytes = kQRows * 128;
    static constexpr uint32_t kKVBytes = kKT * D * 2;           // one K (or V) tile
    static constexpr uint32_t kKVHalfBytes = kKT * 128;
    static constexpr uint32_t kStageBytes = 2 * kKVBytes;
    static constexpr uint32_t kDenBytes = kDen ? 2u * kMaxDenRuns * kQRows * 4u : 0u;   // [stream][run][row] fp32
    static constexpr uint32_t kTileBytes = 2 * kQBytes + kStages * kStageBytes + kDenBytes;
    static constexpr uint32_t kSmemBytes = 4096 + kTileBytes;   // barriers, tile table and alignment slack in front
    // Score buffers per stream.  With 64 channels two CTAs share the SM's 512 tensor-memory columns and a
    // stream has one S buffer (S and O of two streams: 256 columns).  With 128 channels one CTA has all
    // 512 columns and a stream has two S buffers used alternately, so that S of the next tile is computed
    // while the softmax of the current one runs (2 x 2 x 64 for S, 2 x 128 for O).
    static constexpr int kSBufs = kWide ? 2 : 1;
    // MMA-issuing warps.  One thread issuing for both streams is enough with 64 channels (two CTAs per SM
    // share the tensor pipe).  With 128 channels a stream's tile is 12 instructions of 50-65 clocks of issue
    // each plus three barrier waits, and a single issuer for both streams was what bound the kernel: each
    // stream gets its own issuing warp (one CTA per SM, so the registers are there).
    static constexpr int kMmaWarps = kWide ? 2 : 1;
    static constexpr int kThreads = (kMmaWarp + kMmaWarps) * 32;
    static constexpr uint32_t kTmemCols = kWide ? 512 : 256;
    static constexpr uint32_t kSCol = 0, kOCol = 2 * kSBufs * kKT;
    static constexpr int kCtasPerSm = kWide ? 1 : 2;
    // Extents every address in the kernel is derived from, checked at compile time:
    //  - tensor memory: S buffers of both streams, then O of both streams, inside the allocation, and the
    //    allocations of all CTAs of an SM inside its 512 columns (otherwise tcgen05.alloc would block; a CTA of
    //    another form, from the launch before or behind, may make it block until one of the two ends, which both
    //    do: a launch lets the next one in only when all its CTAs own their columns);
    //  - shared memory: the CTAs of an SM (each with 1 KB reserved by the system) inside 228 KB;
    //  - matrix descriptors: a start address is 14 bits of 16-byte units (256 KB), so adding a stage, half
    //    or K-step offset to the low descriptor word can never carry into the field above it.
    static_assert(kOCol + 2 * D <= kTmemCols, "S and O of both streams must fit the tensor-memory allocation");
    static_assert((kTmemCols & (kTmemCols - 1)) == 0 && kTmemCols >= 32 && kCtasPerSm * kTmemCols <= 512,
                  "tensor-memory allocations of an SM's CTAs");
    static_assert(kCtasPerSm * (kSmemBytes + 1024) <= 228 * 1024, "shared memory of an SM's CTAs");
    static_assert(kKVHalfBytes % 1024 == 0 && kQHalfBytes % 1024 == 0 && kStageBytes % 1024 == 0 && kQBytes % 1024 == 0,
                  "swizzle atoms must stay 1024-byte aligned");
    static_assert(228 * 1024 <= (1 << 18), "descriptor start-address field covers all of shared memory");
    static_assert(kStages <= kMaxStages, "barrier arrays");
};

constexpr int kTileTab = 256;     // tiles whose (first token, valid tokens) are tabulated in shared memory

struct Barriers {
    uint64_t q_full[2][2];     // [stream][half]: see kQSplitRows
    uint64_t kv_full[kMaxStages], kv_empty[kMaxStages];
    uint64_t s_full[2][2], p_full[2][2];   // [stream][S buffer]
    uint64_t o_full[2], pv_done[2], drained[2];
    uint32_t tmem_base;
    uint32_t issued;           // stages the producer has filled, for the end of a launch that gave up
    int abort_flag;
    int2 tile_tab[kTileTab];
};

static_assert(sizeof(Barriers) + 1024 <= 4096, "barrier block must fit in front of the 1024-byte aligned tiles");

// How the pairs (units of two streams) of one launch are formed; shared by every role.  The first
// n_shared pairs are two consecutive query tiles of one item, which share every key/value tile in
// shared memory; an item with an odd number of query tiles has one tile left over, and the left-over
// tiles of two consecutive items form a pair whose streams fetch their own key/value tiles (with one
// query tile per item every pair is of that kind).
struct PairPlan {
    int32_t nqt;          // query tiles per item
    int32_t npi;          // shared pairs per item = nqt / 2
    int32_t n_items;
    int32_t n_shared;     // = n_items * npi
    int32_t n_pairs;      // n_shared + ceil(n_items * (nqt & 1) / 2)
    int32_t full;         // kSplit form: whole pairs per CTA; the pairs left over are shared by clusters of two CTAs
    int32_t kind;         // 0: no pair is shared, 1: every pair is, 2: both kinds (so that the common cases test a launch constant),
                          // 3: a pair is one query tile, stream B absent
};

// The current scale read from the caller's K/V tensors instead of the cache: the last entry of the
// range list stands for it (start 0, len T).  With `store` every tile fetched that way is also written
// to the scale's place in the cache (the append fused into attention).
constexpr int32_t kExtFlag = 1 << 30;   // marks such a tile's first token in the tile table
struct ExtArgs {
    CUtensorMap k64, v64, k16, v16;   // rank-4 maps of the caller's K and V (64- and 16-token boxes)
    CUtensorMap k_store, v_store;     // the layer's region, clipped at the end of the scale's place (64-token boxes)
    int32_t range;                    // index of the range that stands for the current scale
    int32_t store;
    int32_t dst;                      // first position of the scale in the per-item region
    int3 pos;                         // coordinate slots of token, head and row in the rank-4 maps
    __nv_bfloat16* region;            // the layer's region, for rows written one by one
    int32_t capacity;
    int32_t n_pieces, last_piece;     // kPieces form: the scale's place is several pieces (a ring that wraps inside it, say);
    Piece piece[LayerLayout::kMaxPieces];   // last_piece holds its last token, and the store maps end where that piece does
    int32_t rider_tok, rider_valid;   // older cache tokens that ride in the spare box of the scale's last tile
};

// Attention density as a by-product (Sec. 4.1): the range list of such a launch has one entry per piece of a
// run of attended tokens (never merged across runs), and every 16-token box of a key tile belongs to one run, so
// a row's un-normalised probability mass per run is a running sum of the box sums the softmax computes anyway.
// The whole 64-token tiles of the ranges come first; what is left of each range, up to four boxes with the last
// partly filled, is packed four boxes to a mixed tile, whatever the runs.  (With every tile cut at the runs, T = 100 of a
// cache-demanding layer of the 680-token schedule was nine tiles; it is five.  With the epilogue below: 512 items, T = 64, 100,
// 169, 256: 22.9 / 31.1 / 48.6 / 64.8 -> 19.9 / 27.9 / 44.2 / 62.3 us per call, copy of the append included.)
struct MixedTile {
    uint64_t keep;                     // a bit per column that holds a key
    int32_t tok[4];                    // first token of each box
    uint32_t runs;                     // run of each box, a byte each
    int32_t boxes;
};
template <bool kDen>   // (without the tables for the launches that do not need them)
struct DenArgs {
    double* out;                       // [heads][n_runs], accumulated with atomic adds
    int32_t n_runs;
    int32_t n_whole;                   // whole tiles; the mixed ones are the tiles behind them
    float weight[kDen ? kMaxDenRuns : 1];         // 1 / (rows * tokens of the run)
    int8_t run_of_range[kDen ? kMaxRanges : 1];
    MixedTile mixed[kDen ? kMaxRanges : 1];       // (a range leaves at most four boxes)
};
constexpr int32_t kMixedFlag = 1 << 16;   // in a tile's second word; its first is then the index of the mixed tile

struct Stream {
    int32_t item;
    int32_t qt;
    bool valid;
};

__device__ __forceinline__ bool pair_is_shared(const PairPlan& pp, int32_t pair)
{
    return pp.kind == 2 ? pair < pp.n_shared : pp.kind == 1;
}

// (kSolo: the kernel form knows pairs of one query tile, kind 3)
template <bool kSolo>
__device__ __forceinline__ Stream stream_of(const PairPlan& pp, int32_t pair, int g)
{
    Stream s;
    if (pair_is_shared(pp, pair)) {
        s.item = pp.npi == 1 ? pair : pair / pp.npi;
        s.qt = 2 * (pair - s.item * pp.npi) + g;
        s.valid = true;
    } else if (kSolo && pp.kind == 3) {
        s.item = pp.nqt == 1 ? pair : pair / pp.nqt;
        s.qt = pair - s.item * pp.nqt;
        s.valid = g == 0;
    } else {
        s.item = 2 * (pair - pp.n_shared) + g;
        s.qt = pp.nqt - 1;
        s.valid = s.item < pp.n_items;
    }
    return s;
}

using namespace ptx;


// Tile j of the resident ranges: first token and number of valid tokens (<= 64).
// A tile of range `ext_range` (the current scale in the caller's tensors) carries kExtFlag in t0.
__device__ __forceinline__ void tile_at(const RangeList& rl, int j, int32_t& t0, int32_t& valid, int ext_range = -1)
{
    int r = 0;
    for (; r < rl.n - 1; ++r) {
        const int nt = (rl.r[r].len + kKT - 1) / kKT;
        if (j < nt) break;
        j -= nt;
    }
    t0 = rl.r[r].start + j * kKT;
    valid = min(kKT, rl.r[r].start + rl.r[r].len - t0);
    if (r == ext_range) t0 |= kExtFlag;
}

// The same for a density launch: (first token, 64 | run << 8) of a whole tile, (index, 16 * boxes | kMixedFlag) of a mixed one.
__device__ __forceinline__ void density_tile_at(const RangeList& rl, const DenArgs<true>& den, int j, int32_t& t0, int32_t& word)
{
    if (j >= den.n_whole) {
        t0 = j - den.n_whole;
        word = den.mixed[t0].boxes * kKVBoxRows | kMixedFlag;
        return;
    }
    int r = 0;
    for (; r < rl.n - 1; ++r) {
        const int nt = rl.r[r].len / kKT;
        if (j < nt) break;
        j -= nt;
    }
    t0 = rl.r[r].start + j * kKT;
    word = kKT | ((int32_t)den.run_of_range[r] << 8);
}

// ---------------------------------------------------------------- kernel
template <int D, bool kExt, bool kWide, bool kDen, bool kLazy, bool kShort, bool kPieces, bool kSplit>
__global__ void __launch_bounds__(Cfg<D, kWide, kDen>::kThreads, Cfg<D, kWide, kDen>::kCtasPerSm)
attend_pair_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
                   const __grid_constant__ CUtensorMap v_map, const __grid_constant__ CUtensorMap k_map64,
                   const __grid_constant__ CUtensorMap v_map64, const __grid_constant__ ExtArgs ext,
                   __nv_bfloat16* __restrict__ O, int64_t o_row,
                   int64_t o_head, int64_t o_tok, const RangeList ranges, int32_t T, int32_t heads,
                   const PairPlan pp, int32_t n_tiles, int3 qpos, float scale_log2, int* __restrict__ status,
                   const __grid_constant__ DenArgs<kDen> den)
{
    static_assert(!(kDen && kExt), "the density form serves the plain attend call");
    const int ext_range = kExt ? ext.range : -1;
    using C = Cfg<D, kWide, kDen>;
    extern __shared__ uint8_t smem_raw[];
    Barriers* bars = reinterpret_cast<Barriers*>(smem_raw);
    volatile int* abort_flag = &bars->abort_flag;
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t tiles = (raw + (uint32_t)sizeof(Barriers) + 1023u) & ~1023u;
    const uint32_t q_smem = tiles;
    const uint32_t kv_smem = q_smem + 2 * C::kQBytes;
    // the warp index is taken through a shuffle so that the compiler knows it to be the same in every
    // lane: role branches are then uniform branches and the issuing warps keep their operands uniform
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;

    const bool layout_ok = (tiles + C::kTileBytes) <= (raw + C::kSmemBytes);
    if (threadIdx.x == 0) {
        bars->abort_flag = 0;
        for (int g = 0; g < 2; ++g) {
            mbar_init(smem_u32(&bars->q_full[g][0]), 1);
            mbar_init(smem_u32(&bars->q_full[g][1]), 1);
            for (int b = 0; b < 2; ++b) {
                mbar_init(smem_u32(&bars->s_full[g][b]), 1);
                mbar_init(smem_u32(&bars->p_full[g][b]), kGroupWarps);
            }
            mbar_init(smem_u32(&bars->pv_done[g]), 1);
            mbar_init(smem_u32(&bars->o_full[g]), 1);
            mbar_init(smem_u32(&bars->drained[g]), 1);
        }
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(smem_u32(&bars->kv_full[s]), 1);
            mbar_init(smem_u32(&bars->kv_empty[s]), C::kMmaWarps);   // one arrival per issuing warp
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (!layout_ok) report(status, kStatusSyncTimeout, abort_flag);
    }
    for (int j = threadIdx.x; j < n_tiles && j < kTileTab; j += C::kThreads) {
        int32_t t0, valid;
        if constexpr (kDen) density_tile_at(ranges, den, j, t0, valid);
        else tile_at(ranges, j, t0, valid, ext_range);
        bars->tile_tab[j] = make_int2(t0, valid);
    }
    if (layout_ok) {
        // query rows a tile does not cover keep whatever the slot held before; start them at zero
        uint4* qz = reinterpret_cast<uint4*>(smem_raw + (q_smem - raw));
        for (uint32_t i = threadIdx.x; i < 2 * C::kQBytes / 16; i += C::kThreads) qz[i] = make_uint4(0, 0, 0, 0);
        if constexpr (kDen) {
            uint4* dz = reinterpret_cast<uint4*>(smem_raw + (kv_smem - raw) + C::kStages * C::kStageBytes);
            for (uint32_t i = threadIdx.x; i < C::kDenBytes / 16; i += C::kThreads) dz[i] = make_uint4(0, 0, 0, 0);
        }
        fence_async_smem();
    }
    // Everything up to a role's first load touches only this CTA's own memory, so it runs while the kernel before this one
    // ends: the threads that issue this CTA's loads wait for that kernel right before the first of them, and what the others
    // read or write follows from those loads.  By then the code up to there, its launch parameters and its tensor maps have
    // been fetched.  With one wait for all here, a launch issued its first loads 2 000 to 3 800 clocks after it.  us a call, before
    // and after (neutral at large launches):
    //   64 channels, 60 items      T = 100   6.86 -> 6.05    T = 169  9.55 -> 8.95    T = 256  11.1 -> 10.0
    //   64 channels, 256 items     T =  64   9.05 -> 8.76    T = 100  11.6 -> 11.0
    //   64 channels, 1 920 items   T =  25   19.1 -> 17.3    T =  36  23.7 -> 22.6
    //   128 channels, 32 items     T = 144   8.74 -> 7.8     T = 400  16.5 -> 15.7
    // Tensor memory is owned before the roles split, but in the two-CTA form's long launches (kOwnLate), where the producer
    // allocates behind its preparations and the other warps meet it there, the softmax warps after the wait:
    //   where it is done so        256 items, T = 169  14.8 -> 14.3, T = 256  21.3 -> 20.6;  2 304 items, T = 324  223 -> 218
    //   in the other forms         60 items, T = 100   6.05 -> 6.88;  256 items, T = 64  8.76 -> 8.95
    constexpr bool kOwnLate = !kWide && !kShort;
    uint32_t tmem = 0;
    auto allocate = [&]() {
        __syncwarp();   // (an aligned instruction; loops and a branch of one lane lie before)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars->tmem_base)),
                     "r"(C::kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    };
    if (!kOwnLate && warp == kProducerWarp) allocate();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (!kOwnLate) tmem = __shfl_sync(0xffffffffu, bars->tmem_base, 0);
    auto own_late = [&]() {   // (once by every warp)
        if (!kOwnLate) return;
        if (warp == kProducerWarp) allocate();
        tc_fence_before();
        barrier_of(1, C::kThreads);
        tc_fence_after();
        tmem = __shfl_sync(0xffffffffu, bars->tmem_base, 0);
    };
    // (in a density launch `valid` also carries the tile's run, or that the tile is a mixed one; tile_run() strips that)
    auto tile_of = [&](int j, int32_t& t0, int32_t& valid) {
        if (j < kTileTab) {
            const int2 e = bars->tile_tab[j];
            t0 = e.x;
            valid = e.y;
        } else {
            if constexpr (kDen) density_tile_at(ranges, den, j, t0, valid);
            else tile_at(ranges, j, t0, valid, ext_range);
        }
    };
    auto tile_run = [](int32_t& valid) -> int {   // run of a whole tile, -1 for a mixed one
        const int run = !kDen ? 0 : (valid & kMixedFlag) ? -1 : (valid >> 8);
        if (kDen) valid &= 0xff;
        return run;
    };

    const uint32_t q_full0 = smem_u32(&bars->q_full[0][0]);   // [g][half] at + 16 * g + 8 * half
    // With at most 64 query tokens a query tile fills half of its slot, so the slot holds the tiles of two
    // consecutive units and the next unit's queries are fetched a whole unit ahead.  The MMA reads 128
    // rows from wherever the tile starts; what it reads past the tile only reaches dead rows of S.
    const bool q_split = T <= kQSplitRows;
    constexpr uint32_t kQHalfSlot = kQSplitRows * 128;   // bytes from the first to the second tile of a slot
    const uint32_t s_full0 = smem_u32(&bars->s_full[0][0]), p_full0 = smem_u32(&bars->p_full[0][0]);   // + 16 g + 8 buffer
    const uint32_t pv_done0 = smem_u32(&bars->pv_done[0]);
    // S buffer and barrier phase of a stream's flat tile index: with two buffers they alternate, and each
    // buffer's barriers see every other tile
    auto buf_of = [](uint32_t t) -> uint32_t { return C::kSBufs == 2 ? (t & 1u) : 0u; };
    auto par_of = [](uint32_t t) -> uint32_t { return C::kSBufs == 2 ? ((t >> 1) & 1u) : (t & 1u); };
    const uint32_t o_full0 = smem_u32(&bars->o_full[0]);
    const uint32_t kv_full0 = smem_u32(&bars->kv_full[0]), kv_empty0 = smem_u32(&bars->kv_empty[0]);

    // pairs of this CTA: p = blockIdx.x + n * gridDim.x, n = 0 .. my_pairs-1.  In the split form that gives every CTA pp.full
    // pairs, and of the pairs left over each cluster of two CTAs takes one, its CTAs one half of the key tiles each.
    const uint32_t rank = kSplit ? cluster_rank() : 0u;
    const int32_t split_pair = kSplit ? pp.full * (int32_t)gridDim.x + (int32_t)(blockIdx.x >> 1) : 0;
    const bool has_split = kSplit && split_pair < pp.n_pairs;
    const uint32_t my_pairs = kSplit ? (uint32_t)pp.full + (has_split ? 1u : 0u)
                                     : ((int32_t)blockIdx.x < pp.n_pairs ? ((uint32_t)pp.n_pairs - 1u - blockIdx.x) / gridDim.x + 1u : 0u);
    auto pair_at = [&](uint32_t n) -> int32_t {
        return kSplit && n == (uint32_t)pp.full ? split_pair : (int32_t)(blockIdx.x + n * gridDim.x);
    };
    auto tiles_begin = [&](uint32_t n) -> int { return kSplit && n == (uint32_t)pp.full && rank == 1u ? n_tiles / 2 : 0; };
    auto tiles_end = [&](uint32_t n) -> int { return kSplit && n == (uint32_t)pp.full && rank == 0u ? n_tiles / 2 : n_tiles; };
    float m_ref = 0.f, l = 0.f;   // softmax warps: a row's reference maximum and sum

    // The producer and the MMA issuer run their loops with the whole warp converged and let one
    // elected lane issue: addresses, descriptors and coordinates then stay warp-uniform values,
    // which keeps the per-instruction issue cost of the TMA and tcgen05 instructions low.
    if (layout_ok && warp == kProducerWarp) {
        // ------------------------------------------------------------ TMA producer of K/V tiles
        uint32_t sq = 0;  // stages issued so far
        bool ok = true;
        // Fused append: a tile of the current scale is written to the cache two stages after it was
        // requested (it has landed by then, so the wait costs nothing), by lane 0, as one bulk group per
        // stage; before a stage is refilled, every group but the two newest has finished reading it.
        const bool storing = kExt && ext.store != 0;
        if (lane == 0) {
            prefetch_tensormap(&k_map);
            prefetch_tensormap(&v_map);
            prefetch_tensormap(&k_map64);
            prefetch_tensormap(&v_map64);
            if (kExt) {
                prefetch_tensormap(&ext.k64);
                prefetch_tensormap(&ext.v64);
                prefetch_tensormap(&ext.k16);
                prefetch_tensormap(&ext.v16);
                if (storing) {
                    prefetch_tensormap(&ext.k_store);
                    prefetch_tensormap(&ext.v_store);
                }
            }
        }
        own_late();
        uint32_t st_sq[2] = {0, 0};
        int32_t st_tok[2] = {0, 0}, st_item[2] = {0, 0};
        int st_n = 0;
        auto store_front = [&]() -> bool {
            const uint32_t stage = st_sq[0] % C::kStages, use = st_sq[0] / C::kStages;
            if (!warp_wait(kv_full0 + 8 * stage, use & 1u, abort_flag)) return false;
            const uint32_t k_src = kv_smem + stage * C::kStageBytes, v_src = k_src + C::kKVBytes;
            if constexpr (kPieces) {
                // Of every piece the tile's share: with one bulk store where it is the whole tile (up to the end of the scale,
                // where the map clips the box), else row by row (a box that starts or ends inside the tile cannot be told
                // to the copy engine: the swizzle wants it to start on eight rows, and a clipped start is not allowed).
                const int32_t first = st_tok[0], end = min(first + kKT, T);
                for (int i = 0; i < ext.n_pieces; ++i) {
                    const int32_t lo = max(first, ext.piece[i].src), hi = min(end, ext.piece[i].src + ext.piece[i].len);
                    if (lo >= hi) continue;
                    const int32_t dst = ext.piece[i].dst + lo - ext.piece[i].src;
                    if (lo == first && (hi - lo == kKT || (hi == T && i == ext.last_piece))) {
                        if (lane == 0) {
#pragma unroll
                            for (int h = 0; h < C::kHalves; ++h) {
                                tma_store_3d(hi - lo < kKT ? &ext.k_store : &k_map64, k_src + h * C::kKVHalfBytes, h * 64, dst, st_item[0]);
                                tma_store_3d(hi - lo < kKT ? &ext.v_store : &v_map64, v_src + h * C::kKVHalfBytes, h * 64, dst, st_item[0]);
                            }
                        }
                    } else {
                        const uint8_t* tile = smem_raw + (k_src - raw);
                        uint4* kd = reinterpret_cast<uint4*>(ext.region + ((int64_t)st_item[0] * 2 * ext.capacity + dst) * D);
                        for (int32_t c = lane; c < (hi - lo) * (D / 8); c += 32) {
                            const int32_t r = c / (D / 8), p = c % (D / 8), row = lo - first + r;
                            const uint32_t off = (uint32_t)((p >> 3) * C::kKVHalfBytes + row * 128 + (((p & 7) ^ (row & 7)) << 4));
                            kd[(int64_t)r * (D / 8) + p] = *reinterpret_cast<const uint4*>(tile + off);
                            kd[((int64_t)r + ext.capacity) * (D / 8) + p] = *reinterpret_cast<const uint4*>(tile + C::kKVBytes + off);
                        }
                    }
                }
                __syncwarp();
            } else if (lane == 0) {
#pragma unroll
                for (int h = 0; h < C::kHalves; ++h) {
                    tma_store_3d(&ext.k_store, k_src + h * C::kKVHalfBytes, h * 64, ext.dst + st_tok[0], st_item[0]);
                    tma_store_3d(&ext.v_store, v_src + h * C::kKVHalfBytes, h * 64, ext.dst + st_tok[0], st_item[0]);
                }
            }
            st_sq[0] = st_sq[1];
            st_tok[0] = st_tok[1];
            st_item[0] = st_item[1];
            --st_n;
            return true;
        };
        for (uint32_t n = 0; ok && n < my_pairs; ++n) {
            const int32_t pair = pair_at(n);
            const int j_begin = tiles_begin(n), j_end = tiles_end(n);
            const Stream sa = stream_of<kWide>(pp, pair, 0), sb = stream_of<kWide>(pp, pair, 1);
            const bool shared = pair_is_shared(pp, pair);
            const int per_tile = (!shared && sb.valid) ? 2 : 1;
            // one unit per item writes the item's tiles: the unit of its first query tiles
            const bool unit_stores = storing && (shared || (kWide && pp.kind == 3) ? sa.qt == 0 : pp.nqt == 1);
            for (int j = j_begin; ok && j < j_end; ++j) {
                int32_t t0, valid;
                tile_of(j, t0, valid);
                const bool mixed = tile_run(valid) < 0;
                const bool from_ext = kExt && (t0 & kExtFlag) != 0;
                t0 &= ~kExtFlag;
                const int nch = (valid + 15) >> 4;
                const bool rider = kExt && ext.rider_valid > 0 && j == n_tiles - 1;   // one more box, from the cache
                for (int g = 0; g < per_tile; ++g, ++sq) {
                    const int item = g == 0 ? sa.item : sb.item;
                    const uint32_t stage = sq % C::kStages, use = sq / C::kStages;
                    if (storing) {
                        if (st_n > 0 && st_sq[0] + 2 <= sq && !store_front()) {
                            ok = false;
                            break;
                        }
                        if (lane == 0) {
                            bulk_commit();
                            bulk_wait_read<2>();
                        }
                        __syncwarp();
                    }
                    if (!warp_wait(kv_empty0 + 8 * stage, (use & 1u) ^ 1u, abort_flag)) {
                        ok = false;
                        break;
                    }
                    if (sq == 0) {
                        wait_for_previous();
                        // The next kernel comes in only now that this CTA owns its tensor memory.  Let in earlier, a CTA of it could take
                        // columns that this one is still waiting for, and keep them while it waits for this launch to end.
                        let_next_start();
                    }
                    const uint32_t full = kv_full0 + 8 * stage;
                    const uint32_t k_dst = kv_smem + stage * C::kStageBytes, v_dst = k_dst + C::kKVBytes;
                    // A tile of the caller's tensors that no rider shares its stage with is one 64-token box whatever
                    // its length: the tokens past the end of the scale are outside the tensor, cost no traffic and
                    // arrive as zeros (the products never read their rows, the fused write is clipped at the scale's end).
                    const bool whole_box = !mixed && (nch == kKT / kKVBoxRows || (kShort && from_ext && !rider));
                    if (whole_box) {
                        if (elect_one()) {
                            mbar_expect_tx(full, (uint32_t)kKT * D * 2 * 2);
                            if (from_ext) {
                                const int32_t row = item / heads, head = item - row * heads;
                                int c[4] = {0, 0, 0, 0};
                                c[ext.pos.y] = head;
                                c[ext.pos.z] = row;
                                c[ext.pos.x] = t0;
#pragma unroll
                                for (int h = 0; h < C::kHalves; ++h) {
                                    tma_load_4d(k_dst + h * C::kKVHalfBytes, &ext.k64, full, h * 64, c[1], c[2], c[3]);
                                    tma_load_4d(v_dst + h * C::kKVHalfBytes, &ext.v64, full, h * 64, c[1], c[2], c[3]);
                                }
                            } else {
#pragma unroll
                                for (int h = 0; h < C::kHalves; ++h) {
                                    tma_load_3d(k_dst + h * C::kKVHalfBytes, &k_map64, full, h * 64, t0, item);
                                    tma_load_3d(v_dst + h * C::kKVHalfBytes, &v_map64, full, h * 64, t0, item);
                                }
                            }
                        }
                    } else if (!kShort && !kDen) {
                        // 16-token boxes (and the rider's box), issued by one lane
                        if (elect_one()) {
                            mbar_expect_tx(full, (uint32_t)(nch + (rider ? 1 : 0)) * kKVBoxRows * D * 2 * 2);
                            if (rider) {
#pragma unroll
                                for (int h = 0; h < C::kHalves; ++h) {
                                    tma_load_3d(k_dst + h * C::kKVHalfBytes + nch * kKVBoxRows * 128, &k_map, full, h * 64,
                                                ext.rider_tok, item);
                                    tma_load_3d(v_dst + h * C::kKVHalfBytes + nch * kKVBoxRows * 128, &v_map, full, h * 64,
                                                ext.rider_tok, item);
                                }
                            }
                            if (from_ext) {
                                const int32_t row = item / heads, head = item - row * heads;
                                int c[4] = {0, 0, 0, 0};
                                c[ext.pos.y] = head;
                                c[ext.pos.z] = row;
                                for (int bx = 0; bx < nch; ++bx) {
                                    c[ext.pos.x] = t0 + bx * kKVBoxRows;
#pragma unroll
                                    for (int h = 0; h < C::kHalves; ++h) {
                                        tma_load_4d(k_dst + h * C::kKVHalfBytes + bx * kKVBoxRows * 128, &ext.k16, full, h * 64,
                                                    c[1], c[2], c[3]);
                                        tma_load_4d(v_dst + h * C::kKVHalfBytes + bx * kKVBoxRows * 128, &ext.v16, full, h * 64,
                                                    c[1], c[2], c[3]);
                                    }
                                }
                            } else {
                                for (int bx = 0; bx < nch; ++bx) {
#pragma unroll
                                    for (int h = 0; h < C::kHalves; ++h) {
                                        tma_load_3d(k_dst + h * C::kKVHalfBytes + bx * kKVBoxRows * 128, &k_map, full, h * 64,
                                                    t0 + bx * kKVBoxRows, item);
                                        tma_load_3d(v_dst + h * C::kKVHalfBytes + bx * kKVBoxRows * 128, &v_map, full, h * 64,
                                                    t0 + bx * kKVBoxRows, item);
                                    }
                                }
                            }
                        }
                    } else {
                        // Short units (at most four key tiles) and mixed tiles: one lane per bulk copy, all issued by one instruction.  A
                        // lane issuing six or eight copies one after the other is what such units wait for (the issuing
                        // warp of a 36-token scale spent half its time waiting for tiles).
                        if (lane == 0) mbar_expect_tx(full, (uint32_t)(nch + (rider ? 1 : 0)) * kKVBoxRows * D * 2 * 2);
                        __syncwarp();
                        const int n_main = 2 * C::kHalves * nch, n_ops = n_main + (rider ? 2 * C::kHalves : 0);
                        if (lane < n_ops) {
                            const bool is_rider = lane >= n_main;
                            const int o = is_rider ? lane - n_main : lane;
                            const int h = o % C::kHalves, kv = (o / C::kHalves) & 1, bx = is_rider ? nch : o / (2 * C::kHalves);
                            const uint32_t dst = (kv ? v_dst : k_dst) + h * C::kKVHalfBytes + bx * kKVBoxRows * 128;
                            if (from_ext && !is_rider) {
                                const int32_t row = item / heads, head = item - row * heads;
                                int c[4] = {0, 0, 0, 0};
                                c[ext.pos.y] = head;
                                c[ext.pos.z] = row;
                                c[ext.pos.x] = t0 + bx * kKVBoxRows;
                                tma_load_4d(dst, kv ? &ext.v16 : &ext.k16, full, h * 64, c[1], c[2], c[3]);
                            } else {
                                const int32_t tok = is_rider ? ext.rider_tok : kDen && mixed ? den.mixed[t0].tok[bx] : t0 + bx * kKVBoxRows;
                                tma_load_3d(dst, kv ? &v_map : &k_map, full, h * 64, tok, item);
                            }
                        }
                    }
                    __syncwarp();
                    if (from_ext && unit_stores) {
                        st_sq[st_n] = sq;
                        st_tok[st_n] = t0;
                        st_item[st_n] = item;
                        ++st_n;
                    }
                }
            }
        }
        if (storing) {
            while (ok && st_n > 0) ok = store_front();
            if (lane == 0) {
                bulk_commit();
                bulk_wait_all();   // the writes are complete, and the stages no longer read, before the CTA ends
            }
            __syncwarp();
        }
        if (lane == 0) {
            if (!ok) report(status, kStatusTmaTimeout, abort_flag);
            bars->issued = sq;
        }
    } else if (layout_ok && warp >= kMmaWarp) {
        // ------------------------------------------------------------ MMA issuer(s)
        // With two issuing warps, warp kMmaWarp + g issues for stream g only; both walk the same loop, so the
        // stage counter advances alike in both.  A commit covers the issuing thread's own instructions only,
        // hence a key/value stage is released by one arrival per issuing warp: each commits its own P V on a
        // shared tile, and the one stream that uses a tile of its own commits twice.
        //
        // A warp's own instructions are what a tile costs here: a satisfied wait in the other roles' form 220 clocks, a branch into
        // the elected lane and back 130, the bookkeeping of a tile 500, against 320 (64 channels) and 640 clocks of products.  So
        // a satisfied wait is a poll, a vote and a branch, a product's instructions and commits are one predicated block, and a
        // tile's length is fetched a tile ahead.  Eight images, T = 4 096, 128 channels: 4 836 -> 4 717 us a call at the same
        // power; one image, T = 576 and 1 600: 35.7 -> 31.5 and 98.3 -> 93.4; 64 channels, 256 items, T = 64 and 100: 9.35 -> 9.05
        // and 11.9 -> 11.6, and no change where the softmax warps fill the SM.  (Those without the votes, by which the warp stops
        // as one behind a wait that gives up: they cost 0.3 to 0.8 % of a pass of few items.  Lanes that each remember how their
        // waits ended, and predicates on that in the blocks: 7 130 -> 7 550 us a 256x256 pass of 15 360 items, three layers.)
        const int my_g = C::kMmaWarps == 2 ? warp - kMmaWarp : 0;
        if (my_pairs > 0) {
            constexpr int kStreams = C::kMmaWarps == 2 ? 1 : 2;   // streams this warp issues for
            const uint32_t idesc_pv = make_idesc(kQRows, D, 1);
            const uint32_t k_lo0 = desc_lo(kv_smem, 16);                             // K tile of stage 0, K-major
            const uint32_t v_lo0 = desc_lo(kv_smem + C::kKVBytes, C::kKVHalfBytes);  // V tile of stage 0, MN-major
            const uint32_t q_lo0 = desc_lo(q_smem, 16);
            constexpr uint32_t kStageLo = C::kStageBytes >> 4, kQLo = C::kQBytes >> 4;
            auto await = [&](const uint32_t bar, const uint32_t parity) -> bool {
                return warp_wait_lean(bar, parity, status, kStatusMmaTimeout, abort_flag);
            };
            // per stream: the tile whose S was issued last and whose P V is still to be issued
            uint32_t pv_stage[kStreams] = {}, pv_nch[kStreams] = {}, pv_first[kStreams] = {}, pv_last[kStreams] = {},
                     pv_release[kStreams] = {}, pv_twice[kStreams] = {};
            bool pv_live[kStreams] = {};
            uint32_t tcount[kStreams] = {};   // tiles issued per stream
            uint32_t ucount[kStreams] = {};   // units started per stream
            uint32_t q_half[kStreams] = {};   // half of the query slot the current unit of each stream uses
            uint32_t sq = 0;
            bool owned = !kOwnLate;

            // O (+)= P V : M = 128, N = D channels, K = 16 * nch tokens; P from TMEM (packed over S),
            // V read MN-major from its stage
            auto issue_pv = [&](const int i) -> bool {
                const int g = kStreams == 2 ? i : my_g;
                const uint32_t t = tcount[i] - 1u;  // flat tile index of this stream
                if (!await(p_full0 + 16 * g + 8 * buf_of(t), par_of(t))) return false;
                // (a unit's first P V overwrites O: every warp of the group arrives on p_full for that tile
                // only after its epilogue of the previous unit, so O has been read by then)
                tc_fence_after();
                const uint32_t empty = kv_empty0 + 8 * pv_stage[i];
                umma_pv(tmem + C::kOCol + g * D, tmem + C::kSCol + (g * C::kSBufs + buf_of(t)) * kKT,
                        v_lo0 + pv_stage[i] * kStageLo, kDescHi, idesc_pv, pv_first[i] ^ 1u, pv_nch[i], pv_release[i], empty,
                        pv_last[i], o_full0 + 8 * g);
                if (C::kMmaWarps == 2) {
                    if (pv_twice[i]) umma_commit_elected(empty);
                    umma_commit_elected(pv_done0 + 8 * g);   // read by the (rare) rescale of O only
                }
                return true;
            };
            auto tile_steps = [&](const int j) -> uint32_t {   // 16-token steps of tile j
                int32_t t0, valid;
                tile_of(j, t0, valid);
                (void)tile_run(valid);
                return ((uint32_t)(valid + 15) >> 4) + ((kExt && ext.rider_valid > 0 && j == n_tiles - 1) ? 1u : 0u);
            };

            for (uint32_t n = 0; n < my_pairs; ++n) {
                const int32_t pair = pair_at(n);
                const int j_begin = tiles_begin(n), j_end = tiles_end(n);
                const bool shared = pair_is_shared(pp, pair);
                const bool two = shared || (!(kWide && pp.kind == 3) && 2 * (pair - pp.n_shared) + 1 < pp.n_items);   // stream B is there
                // One S buffer: the pending P V of the previous tile goes first, because this S overwrites its P.  Two buffers: this S
                // goes first and runs on the tensor pipe while the softmax of the previous tile finishes (streams with
                // tiles of their own keep the first order: they need their key/value stages back sooner).
                const bool s_first = C::kSBufs == 2 && (shared || pp.kind == 3);
                const uint32_t per_tile = shared || !two ? 1u : 2u;
                uint32_t nch = tile_steps(j_begin);
                for (int j = j_begin; j < j_end; ++j, sq += per_tile) {
                    const uint32_t idesc_s = make_idesc(kQRows, nch * 16, 0);
#pragma unroll
                    for (int i = 0; i < kStreams; ++i) {
                        const int g = kStreams == 2 ? i : my_g;
                        if (g == 1 && !two) {
                            // the stream is absent from this pair: its last P V of the previous pair must not
                            // wait for a next S that is not coming soon (it also holds a key/value stage)
                            if (pv_live[i] && !issue_pv(i)) goto stopped;
                            pv_live[i] = false;
                            continue;
                        }
                        // S = Q K^T for (stream g, tile j).  Its operands are waited for first: they have
                        // almost always landed, and this keeps the two waits out of the P -> P V -> S chain.
                        const uint32_t seq = shared ? sq : sq + g;
                        const uint32_t stage = seq % C::kStages, use = seq / C::kStages;
                        if (!owned) {
                            own_late();
                            owned = true;
                        }
                        if (j == j_begin) {
                            if (tcount[i] == 0) wait_for_previous();   // (the waits that follow have a limit, the launch before has none)
                            const uint32_t u = ucount[i]++;
                            q_half[i] = q_split ? (u & 1u) : 0u;
                            if (!await(q_full0 + 16 * g + 8 * q_half[i], (q_split ? u >> 1 : u) & 1u)) goto stopped;
                        }
                        // (one issuer: the second stream of a shared tile finds it landed)
                        if (!(shared && i == 1) && !await(kv_full0 + 8 * stage, use & 1u)) goto stopped;
                        if (!s_first && pv_live[i] && !issue_pv(i)) goto stopped;
                        tc_fence_after();
                        const uint32_t buf = buf_of(tcount[i]);
                        umma_s<D, C::kQHalfBytes, C::kKVHalfBytes>(tmem + C::kSCol + (g * C::kSBufs + buf) * kKT,
                                                                  q_lo0 + g * kQLo + q_half[i] * (kQHalfSlot >> 4), k_lo0 + stage * kStageLo,
                                                                  kDescHi, idesc_s, s_full0 + 16 * g + 8 * buf);
                        if (s_first && pv_live[i] && !issue_pv(i)) goto stopped;
                        pv_live[i] = true;
                        pv_stage[i] = stage;
                        pv_nch[i] = nch;
                        pv_first[i] = j == j_begin;
                        pv_last[i] = j == j_end - 1;
                        pv_release[i] = !(shared && kStreams == 2 && i == 0);
                        pv_twice[i] = !shared;
                        ++tcount[i];
                    }
                    if (j + 1 < j_end) nch = tile_steps(j + 1);
                }
            }
#pragma unroll
            for (int i = 0; i < kStreams; ++i)
                if (pv_live[i] && !issue_pv(i)) goto stopped;
        stopped:
            if (!owned) own_late();
        } else {
            own_late();
        }
    } else if (layout_ok) {
        // ------------------------------------------------------------ softmax + epilogue (warps 0-7)
        const int g = warp >> 2, wq = warp & 3;
        const uint32_t lane_base = ((uint32_t)(wq * 32)) << 16;
        const int r = wq * 32 + lane;  // query row inside the tile = TMEM lane
        const uint32_t o_full = o_full0 + 8 * g;
        const bool q_loader = (wq == 0 && lane == 0);
        // the output rows start on 32-byte boundaries (the interface only promises 16)
        const bool o_sectors = ((reinterpret_cast<uintptr_t>(O) | (uintptr_t)(2 * o_row) | (uintptr_t)(2 * o_head) | (uintptr_t)(2 * o_tok)) & 31u) == 0;
        // density: [run][row] sums of this stream, in the shared memory the fourth key/value stage would take
        // (every thread only ever touches the entries of its own row; they were zeroed before the roles split)
        float* den_rows = reinterpret_cast<float*>(smem_raw + (kv_smem - raw) + C::kStages * C::kStageBytes) + g * kMaxDenRuns * kQRows;
        uint32_t q_armed = 0;     // query tiles requested so far
        uint32_t q_next_n = 0;    // first pair index not yet searched for a query tile

        // request the query tile of this stream's next unit not yet requested (first lane of the group only)
        if (q_loader) prefetch_tensormap(&q_map);
        auto load_next_q = [&]() {
            for (; q_next_n < my_pairs; ++q_next_n) {
                const int32_t pair = pair_at(q_next_n);
                const Stream s = stream_of<kWide>(pp, pair, g);
                if (!s.valid) continue;
                const int32_t row = s.item / heads, head = s.item - row * heads;
                const int32_t valid_rows = min(kQRows, T - s.qt * kQRows);
                const int qboxes = (valid_rows + kQBoxRows - 1) / kQBoxRows;
                const uint32_t half = q_split ? (q_armed & 1u) : 0u;
                const uint32_t bar = q_full0 + 16 * g + 8 * half;
                const uint32_t dst = q_smem + g * C::kQBytes + half * kQHalfSlot;
                if (q_armed == 0) wait_for_previous();
                mbar_expect_tx(bar, (uint32_t)qboxes * kQBoxRows * D * 2);
                int c[4] = {0, 0, 0, 0};
                c[qpos.y] = head;
                c[qpos.z] = row;
                for (int bx = 0; bx < qboxes; ++bx) {
                    c[qpos.x] = s.qt * kQRows + bx * kQBoxRows;
#pragma unroll
                    for (int h = 0; h < C::kHalves; ++h)
                        tma_load_4d(dst + h * C::kQHalfBytes + bx * kQBoxRows * 128, &q_map, bar, h * 64, c[1], c[2], c[3]);
                }
                ++q_armed;
                ++q_next_n;
                return;
            }
        };
        if (q_loader) {
            load_next_q();
            if (q_split) load_next_q();
        }
        __syncwarp();
        own_late();
        if (kOwnLate) wait_for_previous();
        const uint32_t s_tmem0 = tmem + C::kSCol + g * C::kSBufs * kKT + lane_base;   // + kKT per S buffer
        const uint32_t o_tmem = tmem + C::kOCol + g * D + lane_base;

        uint32_t t = 0;   // flat tile counter of this stream
        uint32_t un = 0;  // units done by this stream
        bool ok = true;
        for (uint32_t n = 0; ok && n < my_pairs; ++n) {
            const int32_t pair = pair_at(n);
            const int j_begin = tiles_begin(n), j_end = tiles_end(n);
            const Stream st = stream_of<kWide>(pp, pair, g);
            if (!st.valid) continue;
            const int32_t valid_rows = min(kQRows, T - st.qt * kQRows);
            const bool warp_live = wq * 32 < valid_rows;
            m_ref = 0.f;
            l = 0.f;
            float nb = 0.f;
            float run_mass = 0.f;   // density: this row's un-normalised mass on the run the tiles are in
            int cur_run = -1;
            for (int j = j_begin; j < j_end; ++j, ++t) {
                int32_t t0, valid;
                tile_of(j, t0, valid);
                const int run = tile_run(valid);
                const uint32_t s_tmem = s_tmem0 + buf_of(t) * kKT;
                const uint32_t s_full = s_full0 + 16 * g + 8 * buf_of(t), p_full = p_full0 + 16 * g + 8 * buf_of(t);
                // (the first wait may span the end of the launch before; the issuing warp's limit, through the abort flag, ends it too)
                if (!__all_sync(0xffffffffu, mbar_wait(s_full, par_of(t), abort_flag, !kOwnLate && t == 0 ? ~0u : kSpinLimit))) {
                    report(status, kStatusSyncTimeout, abort_flag);
                    ok = false;
                    break;
                }
                tc_fence_after();
                // the last S of this unit has landed, so its query tile is no longer read
                if (j == j_end - 1 && q_loader) load_next_q();
                if (warp_live) {
                    uint32_t sr[kKT];
                    tmem_ld64(s_tmem, sr);
                    if (valid < kKT || (kDen && run < 0)) {
                        // (a rider occupies the box behind the tile's own: its tokens stay, the gap before them goes)
                        // as a bit per column, so that each column costs one test of a constant bit
                        uint64_t keep;
                        if (kDen) keep = den.mixed[t0].keep;   // (every other tile of a density launch is whole)
                        else keep = (1ull << valid) - 1ull;
                        if (kExt && ext.rider_valid > 0 && j == n_tiles - 1)
                            keep |= ((1ull << ext.rider_valid) - 1ull) << ((valid + 15) & ~15);
                        const uint32_t keep_lo = (uint32_t)keep, keep_hi = (uint32_t)(keep >> 32);
#pragma unroll
                        for (int i = 0; i < kKT; ++i)
                            if ((((i < 32 ? keep_lo : keep_hi) >> (i & 31)) & 1u) == 0u) sr[i] = 0xff800000u;  // -inf
                    }
                    // row maximum with four independent chains
                    auto row_max = [&]() -> float {
                        float mx[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            mx[c] = max3(__uint_as_float(sr[c]), __uint_as_float(sr[4 + c]), __uint_as_float(sr[8 + c]));
#pragma unroll
                        for (int i = 12; i < kKT - 4; i += 8) {
#pragma unroll
                            for (int c = 0; c < 4; ++c)
                                mx[c] = max3(mx[c], __uint_as_float(sr[i + c]), __uint_as_float(sr[i + 4 + c]));
                        }
#pragma unroll
                        for (int c = 0; c < 4; ++c) mx[c] = fmaxf(mx[c], __uint_as_float(sr[kKT - 4 + c]));
                        return fmaxf(max3(mx[0], mx[1], mx[2]), mx[3]);
                    };
                    // rare: bring O and the row sum to a new reference (rows with `grow`).  The previous P V must
                    // be done.  One S buffer: it was issued before this tile's S, whose arrival covers every
                    // earlier product.  Two buffers: this S may have been issued first, so wait for the
                    // product's own completion (one arrival per P V; at most one phase can be ahead,
                    // because the next P V needs the P this tile has not written yet).
                    auto rescale = [&](const bool grow, const float mt) -> bool {
                        if (C::kSBufs == 2 && !__all_sync(0xffffffffu, mbar_wait(pv_done0 + 8 * g, (t - 1u) & 1u, abort_flag))) {
                            report(status, kStatusSyncTimeout, abort_flag);
                            return false;
                        }
                        if (C::kSBufs == 2) tc_fence_after();
                        float alpha = 1.f;
                        if (grow) {
                            alpha = fast_exp2((m_ref - mt) * scale_log2);
                            m_ref = mt;
                            nb = -mt * scale_log2;
                            l *= alpha;
                            if (kDen) {
                                run_mass *= alpha;
                                for (int rn = 0; rn < den.n_runs; ++rn) den_rows[rn * kQRows + r] *= alpha;
                            }
                        }
#pragma unroll 1
                        for (int cblk = 0; cblk < D / 8; ++cblk) {
                            uint32_t o[8];
                            tmem_ld8(o_tmem + cblk * 8, o);
#pragma unroll
                            for (int i = 0; i < 8; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                            tmem_st8(o_tmem + cblk * 8, o);
                        }
                        return true;
                    };
                    if (j == j_begin) {
                        const float mt = row_max();
                        m_ref = mt;
                        nb = -mt * scale_log2;
                    } else if (!kLazy) {
                        const float mt = row_max();
                        const bool grow = fmaf(mt, scale_log2, nb) > kRescaleLog2;
                        if (__any_sync(0xffffffffu, grow) && !rescale(grow, mt)) {
                            ok = false;
                            break;
                        }
                    }
                    // P over S: columns 0..31 receive the 64 probabilities as bf16 pairs, 16 tokens per store.
                    // A partly filled tile only exponentiates the 16-token groups the products will read (the
                    // P V is issued for as many 16-token steps): the columns behind them keep stale bits.
                    int groups = kKT / 16;
                    if (valid < kKT) groups = ((valid + 15) >> 4) + ((kExt && ext.rider_valid > 0 && j == n_tiles - 1) ? 1 : 0);
                    // (`whole`: all four groups as one straight piece of code, whose instructions overlap from group to group; 64
                    // channels in the wide form only, where a warp has its scheduler nearly to itself: 1 000 -> 860 clocks a
                    // tile; 3 to 12 % slower elsewhere)
                    constexpr bool kStraight = kWide && D == 64;
                    float box_sum[4] = {0.f, 0.f, 0.f, 0.f};   // kDen form only
                    auto exp_tile = [&](auto whole) -> float {
                        float sum0 = 0.f, sum1 = 0.f;
#pragma unroll
                        for (int grp = 0; grp < kKT / 16; ++grp) {
                            if (kDen) sum0 = sum1 = 0.f;
                            if (decltype(whole)::value || grp < groups) {   // (the same for the whole warp)
                                uint32_t pk[8];
#pragma unroll
                                for (int ii = 0; ii < 8; ++ii) {
                                    const int i = (grp & 1) * 8 + ii;   // pair index within its 32-token half, as before
                                    const int c = grp * 16 + 2 * ii;
                                    // (but in density launches) every kPolyEvery-th pair takes its exponentials from a polynomial on the FMA pipe:
                                    // the special-function unit (16 results per clock per SM) is the narrowest resource
                                    float x0, x1, p0, p1;
                                    fma2(x0, x1, __uint_as_float(sr[c]), __uint_as_float(sr[c + 1]), scale_log2, scale_log2, nb, nb);
                                    if (!kDen && kPolyEvery > 0 && (i % (kPolyEvery > 0 ? kPolyEvery : 1)) == 0) {
                                        exp2_poly2(p0, p1, x0, x1);
                                    } else {
                                        p0 = fast_exp2(x0);
                                        p1 = fast_exp2(x1);
                                    }
                                    add2(sum0, sum1, sum0, sum1, p0, p1);
                                    const __nv_bfloat162 h = __floats2bfloat162_rn(p0, p1);
                                    pk[ii] = *reinterpret_cast<const uint32_t*>(&h);
                                }
                                tmem_st8_nowait(s_tmem + grp * 8, pk);
                            }
                            if (kDen) box_sum[grp] = sum0 + sum1;
                        }
                        if (kDen) return (box_sum[0] + box_sum[1]) + (box_sum[2] + box_sum[3]);
                        return sum0 + sum1;
                    };
                    float tile_sum = kStraight && groups == kKT / 16 ? exp_tile(std::bool_constant<kStraight>{}) : exp_tile(std::false_type{});
                    if (kLazy && j > j_begin) {
                        // No maximum was taken for this tile: its exponentials were formed against the row's reference
                        // as it stood (the maximum of the unit's first tile, or of the last tile that was redone).
                        // That is exact as long as nothing overflows.  A row whose tile sum is beyond the limit (or
                        // not a number) has outgrown its reference by more than 2^58; the warp then takes the tile's
                        // true maxima, rescales and forms the tile again before it announces P.  The polynomial
                        // saturates at 2^126, so it cannot hide such a row.
                        const bool over = !(tile_sum <= kLazySumLimit);
                        if (__any_sync(0xffffffffu, over)) {
                            tmem_wait_st();
                            const float mt = row_max();
                            const bool grow = over || fmaf(mt, scale_log2, nb) > kRescaleLog2;
                            if (!rescale(grow, mt)) {
                                ok = false;
                                break;
                            }
                            tile_sum = exp_tile(std::false_type{});
                        }
                    }
                    l += tile_sum;
                    if constexpr (kDen) {
                        // (runs are the same for every thread: tiles and their boxes are launch constants)
                        auto add_mass = [&](const int to, const float mass) {
                            if (to != cur_run) {
                                if (cur_run >= 0) den_rows[cur_run * kQRows + r] += run_mass;
                                run_mass = 0.f;
                                cur_run = to;
                            }
                            run_mass += mass;
                        };
                        if (run >= 0) {
                            add_mass(run, tile_sum);
                        } else {
                            const uint32_t runs = den.mixed[t0].runs;
#pragma unroll
                            for (int b = 0; b < kKT / kKVBoxRows; ++b)
                                if (b < groups) add_mass((int)((runs >> (8 * b)) & 0xffu), box_sum[b]);
                        }
                    }
                    tmem_wait_st();
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(p_full);
            }
            if (!ok) break;
            // epilogue: out = O / l once the last P V of the unit is done
            if (!__all_sync(0xffffffffu, mbar_wait(o_full, un & 1u, abort_flag))) {
                report(status, kStatusSyncTimeout, abort_flag);
                ok = false;
                break;
            }
            tc_fence_after();
            if (kSplit && n == (uint32_t)pp.full) {   // (always the last pair) the two CTAs merge their halves below
                ++un;
                break;
            }
            if (warp_live) {
                const float inv = 1.f / l;
                const int32_t row = st.item / heads, head = st.item - row * heads;
                __nv_bfloat16* dst = O + row * o_row + head * o_head + (int64_t)(st.qt * kQRows + r) * o_tok;
#pragma unroll
                for (int cblk = 0; cblk < D / 32; ++cblk) {
                    uint32_t o[32];
                    tmem_ld32(o_tmem + cblk * 32, o);
                    if (r < valid_rows) {
                        uint32_t w[16];
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(o[2 * i]) * inv, __uint_as_float(o[2 * i + 1]) * inv);
                            w[i] = *reinterpret_cast<const uint32_t*>(&h);
                        }
                        if (o_sectors) {
                            // whole 32-byte sectors per thread: half the store instructions, no partly written sector
                            st_global_32B(dst + cblk * 32, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
                            st_global_32B(dst + cblk * 32 + 16, w[8], w[9], w[10], w[11], w[12], w[13], w[14], w[15]);
                        } else {
#pragma unroll
                            for (int c = 0; c < 4; ++c)
                                reinterpret_cast<uint4*>(dst + cblk * 32)[c] = make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
                        }
                    }
                }
            }
            if (kDen && warp_live) {
                // The row's share of every run, normalised by its row sum, added up over the warp's rows and then,
                // weighted by 1 / (rows * tokens of the run), into the head's entry of the result.  Lane (half, run) adds
                // up 16 of the 32 rows, each lane starting at another row, so that no two read the same bank; the
                // warp's runs then go out as one request, neighbouring lanes to neighbouring addresses.  (A run at a
                // time, with a reduction by shuffles and an atomic of its own: 512 items, L = 274 and 424, 48.2 against
                // 45.3 us per call.)
                if (cur_run >= 0) den_rows[cur_run * kQRows + r] += run_mass;
                __syncwarp();
                const float inv = (r < valid_rows) ? 1.f / l : 0.f;
                static_assert(kMaxDenRuns == 16, "a lane per run and half of the rows");
                const int rn = lane & 15;
                float v = 0.f;
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const int row = (lane & 16) + ((i + rn) & 15);
                    float* e = den_rows + rn * kQRows + wq * 32 + row;
                    v = fmaf(*e, __shfl_sync(0xffffffffu, inv, row), v);
                    *e = 0.f;   // the next unit starts from zero
                }
                v += __shfl_xor_sync(0xffffffffu, v, 16);
                if (lane < den.n_runs)
                    atomicAdd(den.out + (int64_t)(st.item % heads) * den.n_runs + lane, (double)v * (double)den.weight[lane]);
                __syncwarp();
            }
            tc_fence_before();   // orders the reads of O before the arrival on p_full for the next unit's first tile
            ++un;
        }
        // wind down: query tiles requested but never consumed must land before the CTA exits
        if (q_loader) {
            for (uint32_t q = un; q < q_armed; ++q) {
                const uint32_t half = q_split ? (q & 1u) : 0u;
                const uint32_t parity = q_split ? ((q >> 1) & 1u) : (q & 1u);
                for (uint32_t i = 0; i < kSpinLimit; ++i)
                    if (mbar_try_wait(q_full0 + 16 * g + 8 * half, parity)) break;
            }
        }
    }

    if constexpr (kSplit) {
        if (has_split) {   // (the same for both CTAs of a cluster)
            // -------------------------------------------------------- merge of the two halves of the pair's keys
            // Each CTA holds O of both query tiles against its own references and sums, and finishes one half of the
            // channels: it sends the other CTA its columns of the other half (fp32) with its references and sums, into that
            // CTA's key/value ring, which nobody reads any more once every role of both CTAs is done (first barrier).  Columns
            // in groups of four, one row per lane: 16-byte accesses without bank conflicts.
            constexpr uint32_t W = D / 2, kMl = 2u * W * kQRows * 4u;   // references and sums behind the columns
            static_assert(kMl + 2u * kQRows * 8u <= C::kStages * C::kStageBytes, "exchange fits the ring");
            const int g = warp >> 2, wq = warp & 3, r = wq * 32 + lane;
            const Stream st = g < 2 ? stream_of<kWide>(pp, split_pair, g) : Stream{0, 0, false};
            const int32_t valid_rows = st.valid ? min(kQRows, T - st.qt * kQRows) : 0;
            const bool warp_live = wq * 32 < valid_rows;
            const uint32_t o_tmem = tmem + C::kOCol + g * D + (((uint32_t)(wq * 32)) << 16);
            auto col_off = [&](uint32_t c4) -> uint32_t { return ((g * (W / 4u) + c4) * kQRows + r) * 16u; };
            __syncwarp();
            cluster_sync();
            if (warp_live) {
                tc_fence_after();
                const uint32_t to = map_to_rank(kv_smem, rank ^ 1u);
#pragma unroll
                for (uint32_t cb = 0; cb < W; cb += 16) {
                    uint32_t o[16];
                    tmem_ld16(o_tmem + (rank ^ 1u) * W + cb, o);
#pragma unroll
                    for (int i = 0; i < 4; ++i) st_cluster_16B(to + col_off(cb / 4u + i), o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
                }
                st_cluster_8B(to + kMl + (g * kQRows + r) * 8u, m_ref, l);
            }
            cluster_sync();
            if (warp_live) {
                const uint8_t* ring = smem_raw + (kv_smem - raw);
                const float2 other = reinterpret_cast<const float2*>(ring + kMl)[g * kQRows + r];
                const float M = fmaxf(m_ref, other.x);
                float f_own = fast_exp2((m_ref - M) * scale_log2), f_other = fast_exp2((other.x - M) * scale_log2);
                const float inv = 1.f / fmaf(l, f_own, other.y * f_other);
                f_own *= inv;
                f_other *= inv;
                const bool o_sectors = ((reinterpret_cast<uintptr_t>(O) | (uintptr_t)(2 * o_row) | (uintptr_t)(2 * o_head) | (uintptr_t)(2 * o_tok)) & 31u) == 0;
                const int32_t row = st.item / heads, head = st.item - row * heads;
                __nv_bfloat16* dst = O + row * o_row + head * o_head + (int64_t)(st.qt * kQRows + r) * o_tok + rank * W;
#pragma unroll
                for (uint32_t cb = 0; cb < W; cb += 16) {
                    uint32_t o[16], w[8];
                    tmem_ld16(o_tmem + rank * W + cb, o);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 x = *reinterpret_cast<const float4*>(ring + col_off(cb / 4u + i));
                        const __nv_bfloat162 a = __floats2bfloat162_rn(fmaf(x.x, f_other, __uint_as_float(o[4 * i]) * f_own),
                                                                       fmaf(x.y, f_other, __uint_as_float(o[4 * i + 1]) * f_own));
                        const __nv_bfloat162 b = __floats2bfloat162_rn(fmaf(x.z, f_other, __uint_as_float(o[4 * i + 2]) * f_own),
                                                                       fmaf(x.w, f_other, __uint_as_float(o[4 * i + 3]) * f_own));
                        w[2 * i] = *reinterpret_cast<const uint32_t*>(&a);
                        w[2 * i + 1] = *reinterpret_cast<const uint32_t*>(&b);
                    }
                    if (r < valid_rows) {
                        if (o_sectors) {
                            st_global_32B(dst + cb, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
                        } else {
                            reinterpret_cast<uint4*>(dst + cb)[0] = make_uint4(w[0], w[1], w[2], w[3]);
                            reinterpret_cast<uint4*>(dst + cb)[1] = make_uint4(w[4], w[5], w[6], w[7]);
                        }
                    }
                }
            }
        }
    }

    // ---------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (layout_ok && *abort_flag) {   // (the same for all threads: no role is left to set it)
        // A launch that gave up.  Nothing is issued any more; what nobody may have waited for, the newest copy into each stage and
        // the products, ends before shared and tensor memory are given back (query tiles: at the end of the softmax role).
        auto until = [](const uint32_t bar, const uint32_t parity) {
            for (uint32_t i = 0; i < kSpinLimit; ++i)
                if (mbar_try_wait(bar, parity)) break;
        };
        if (warp == kProducerWarp) {
            const uint32_t issued = bars->issued;
            for (uint32_t q = issued > (uint32_t)C::kStages ? issued - C::kStages : 0u; q < issued; ++q)
                until(kv_full0 + 8 * (q % C::kStages), (q / C::kStages) & 1u);
        } else if (warp >= kMmaWarp) {
            const uint32_t drained = smem_u32(&bars->drained[warp - kMmaWarp]);
            umma_commit_elected(drained);
            until(drained, 0u);
        }
        __syncthreads();
    }
    if (warp == kProducerWarp && (layout_ok || !kOwnLate)) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::kTmemCols) : "memory");
    }
}

// ---------------------------------------------------------------- host side
template <int D, bool kExt, bool kWide, bool kDen, bool kLazy, bool kShort, bool kPieces, bool kSplit = false>
cudaError_t launch(const CUtensorMap& qm, const CUtensorMap& km, const CUtensorMap& vm, const CUtensorMap& km64,
                   const CUtensorMap& vm64, const ExtArgs& ext, const Strided& O,
                   const RangeList& ranges, int32_t T, int32_t heads, const PairPlan& pp, int32_t n_tiles, int3 qpos,
                   float scale_log2, int* status, int sm_count, cudaStream_t stream, const DenArgs<true>& den_tables)
{
    using C = Cfg<D, kWide, kDen>;
    DenArgs<kDen> den;
    if constexpr (kDen) den = den_tables;
    else memset(&den, 0, sizeof(den));
    static SharedMemoryOptIn opt_in;
    const cudaError_t oe = opt_in.ensure(attend_pair_kernel<D, kExt, kWide, kDen, kLazy, kShort, kPieces, kSplit>, (int)C::kSmemBytes);
    if (oe != cudaSuccess) return oe;
    int64_t grid = (int64_t)sm_count * C::kCtasPerSm;
    if (kSplit) grid = pp.full > 0 ? ((int64_t)sm_count * C::kCtasPerSm) & ~1ll : 2ll * pp.n_pairs;
    else if (grid > pp.n_pairs) grid = pp.n_pairs;
    // Where SMs hold two CTAs and an eighth to two thirds of the CTAs have a unit in the last round, it matters that those do not
    // share SMs: launched onto an idle chip they do not, but onto SMs that come free one by one they do.  us per call, with /
    // without the overlap, fused: 400 items (1.35 rounds), T = 256 32.9 / 28.2; 180 items (2.43), T = 1 024 119.6 / 105.4; 1 024 items (3.46),
    // T = 169 41.7 / 39.7, T = 256 57.3 / 52.3; 512 items (2.59), T = 361 67.6 / 65.8; 1 920 items (6.49), T = 256 95.3 / 92.3.  With shorter units
    // the launch latency that is hidden is worth more (700 items, 1.18 rounds, T = 36 11.9 / 13.2, T = 100, three key tiles, 21.2 / 22.0; 1 920
    // items, 3.24 rounds, T = 64 27.6 / 29.2), and with fewer or more units in the last round (300 items, 1.01 rounds, T = 169 19.1 / 20.3,
    // T = 256 25.3 / 26.3; 512 items, 1.73, T = 256 32.2 / 32.5).
    // Behind a copy, which leaves SMs one by one: up to a unit per SM, 80 units (T = 576) 29.8 / 24.9, 111 (T = 361) 25.0 / 22.6, 144 (T = 361) 27.1 /
    // 23.3, but 90 (T = 324) 17.5 / 18.9; beyond, 180 (T = 225) 22.9 / 23.6, 256 (T = 121) 20.4 / 22.2; 350 (T = 100) 29.4 / 30.4, 384 (T = 1 024) 90.2 /
    // 79.1, 400 (T = 169, 225, 256) 34.5 / 33.1, 37.6 / 35.6, 51.9 / 46.6; 512 (T = 256) 52.7 / 55.6.  (A density launch follows the small kernel that
    // zeroes its result, on an idle chip.)
    const int64_t slots = (int64_t)sm_count * C::kCtasPerSm, rest = pp.n_pairs % slots;
    const bool uneven = !kWide && n_tiles >= 5 && pp.n_pairs > slots && 8 * rest > slots && 3 * rest <= 2 * slots;
    const bool overlap = kDen || (kExt ? !uneven
                                       : overlaps_append(pp.n_items, T, D, sm_count) && (kWide || pp.n_pairs > sm_count) &&
                                         (pp.n_pairs <= slots || 2 * (int64_t)pp.n_pairs > 3 * slots));
    return launch_kernel(overlap, attend_pair_kernel<D, kExt, kWide, kDen, kLazy, kShort, kPieces, kSplit>, dim3((unsigned)grid), dim3(C::kThreads),
                         KernelMemory(C::kSmemBytes, kSplit ? 2u : 1u), stream, qm, km, vm, km64, vm64, ext, (__nv_bfloat16*)O.ptr, O.row, O.head, O.token,
                         ranges, T, heads, pp, n_tiles, qpos, scale_log2, status, den);
}

}  // namespace

cudaError_t launch_attend_pair(const Strided& Q, const Strided& O, const void* k_map, const void* v_map,
                               const void* k_map64, const void* v_map64, const RangeList& ranges, int32_t T, int32_t rows, int32_t heads, int32_t D,
                               float softmax_scale, int* status, int sm_count, cudaStream_t stream,
                               const CurrentScaleSource* cur, const PairDensity* density, bool fixed_form)
{
    if (ranges.n < 1 || ranges.total < 1 || T < 1) return cudaErrorInvalidValue;
    DenArgs<true> den;
    memset(&den, 0, sizeof(den));
    if (density) {
        static_assert(kPairMaxDensityRuns == kMaxDenRuns, "interface and kernel disagree");
        if (cur || density->n_runs < 1 || density->n_runs > kMaxDenRuns || !density->out) return cudaErrorInvalidValue;
        den.out = density->out;
        den.n_runs = density->n_runs;
        for (int i = 0; i < density->n_runs; ++i) den.weight[i] = (float)density->weight[i];
        for (int i = 0; i < ranges.n; ++i) {
            if (density->run_of_range[i] < 0 || density->run_of_range[i] >= density->n_runs) return cudaErrorInvalidValue;
            den.run_of_range[i] = density->run_of_range[i];
        }
    }
    ExtArgs ext;
    memset(&ext, 0, sizeof(ext));
    ext.range = -1;
    if (cur) {
        // the last range stands for the current scale, whose tokens come from the caller's tensors
        if (ranges.r[ranges.n - 1].start != 0 || ranges.r[ranges.n - 1].len != T) return cudaErrorInvalidValue;
        int kp[3], vp[3];
        if (!tc_encode_q_map(cur->K, T, rows, heads, D, kKT, &ext.k64, kp) ||
            !tc_encode_q_map(cur->V, T, rows, heads, D, kKT, &ext.v64, vp) ||
            !tc_encode_q_map(cur->K, T, rows, heads, D, kKVBoxRows, &ext.k16, kp) ||
            !tc_encode_q_map(cur->V, T, rows, heads, D, kKVBoxRows, &ext.v16, vp))
            return cudaErrorNotSupported;
        if (kp[0] != vp[0] || kp[1] != vp[1] || kp[2] != vp[2]) return cudaErrorNotSupported;
        ext.pos = make_int3(kp[0], kp[1], kp[2]);
        ext.range = ranges.n - 1;
        ext.store = cur->store ? 1 : 0;
        ext.dst = cur->dst;
        if (cur->rider_valid > 0) {
            const int32_t tail = T % kKT;
            if (cur->rider_valid > kKVBoxRows || tail < 1 || tail > kKT - kKVBoxRows) return cudaErrorInvalidValue;
            ext.rider_tok = cur->rider_tok;
            ext.rider_valid = cur->rider_valid;
        }
        int32_t place_end = cur->dst + T;
        if (cur->n_pieces > 0) {
            if (cur->n_pieces > LayerLayout::kMaxPieces || !cur->store) return cudaErrorInvalidValue;
            ext.region = cur->region.base;
            ext.capacity = cur->region.capacity;
            ext.n_pieces = cur->n_pieces;
            ext.last_piece = -1;
            for (int i = 0; i < cur->n_pieces; ++i) {
                ext.piece[i] = cur->piece[i];
                if (cur->piece[i].src + cur->piece[i].len == T) {
                    ext.last_piece = i;   // (the last of them, should there be two)
                    place_end = cur->piece[i].dst + cur->piece[i].len;
                }
            }
            if (ext.last_piece < 0) place_end = cur->region.capacity;   // (no piece ends the scale: the maps are not used)
        }
        if (cur->store &&
            !tc_encode_kv_store_maps(cur->region, (int64_t)rows * heads, D, kKT, place_end, &ext.k_store, &ext.v_store))
            return cudaErrorNotSupported;
    }
    CUtensorMap qm;
    int pos[3];
    if (!tc_encode_q_map(Q, T, rows, heads, D, kQBoxRows, &qm, pos)) return cudaErrorNotSupported;
    CUtensorMap km, vm, km64, vm64;
    memcpy(&km, k_map, sizeof(km));
    memcpy(&vm, v_map, sizeof(vm));
    memcpy(&km64, k_map64, sizeof(km64));
    memcpy(&vm64, v_map64, sizeof(vm64));
    PairPlan pp;
    pp.full = 0;
    pp.nqt = (T + kQRows - 1) / kQRows;
    pp.npi = pp.nqt / 2;
    if ((int64_t)rows * heads > 0x3fffffffll) return cudaErrorInvalidValue;
    pp.n_items = rows * heads;
    const int64_t n_shared = (int64_t)pp.n_items * pp.npi;
    const int64_t n_pairs = n_shared + ((pp.nqt & 1) ? ((int64_t)pp.n_items + 1) / 2 : 0);
    if (n_pairs > 0x7fffffffll) return cudaErrorInvalidValue;
    pp.n_shared = (int32_t)n_shared;
    pp.n_pairs = (int32_t)n_pairs;
    pp.kind = pp.npi == 0 ? 0 : ((pp.nqt & 1) ? 2 : 1);
    // When every query tile of the launch can have an SM of its own, it gets one: what such a call takes is a stream's serial
    // chain, and two streams on the same SM sub-partitions lengthen it (64 channels 2 090 -> 1 500 clocks a key tile with
    // the form below; the second fetch of K and V comes from L2).  us per call, before / after: 64 channels, 60 items: T = 100
    // 10.1 / 7.7, T = 169 11.1 / 9.6, T = 256 14.2 / 11.7; 32 items, T = 256 13.2 / 10.9; 128 channels, 32 items: T = 144 12.9 /
    // 10.3, T = 256 14.5 / 12.3, T = 400 23.6 / 20.7; 16 items, T = 576 35.3 / 22.6.  With more tiles than SMs the pairs win (128
    // channels, 32 items, T = 576, 160 tiles: 38.3 / 40.9).
    if (!density && !fixed_form && pair_one_tile_per_sm(pp.n_items, T, sm_count)) {
        pp.kind = 3;
        pp.n_shared = 0;
        pp.n_pairs = pp.n_items * pp.nqt;
    }
    int32_t n_tiles = 0;
    for (int i = 0; i < ranges.n; ++i) n_tiles += density ? ranges.r[i].len / kKT : (ranges.r[i].len + kKT - 1) / kKT;
    if (density) {
        den.n_whole = n_tiles;
        int boxes = 0;
        for (int i = 0; i < ranges.n; ++i) {
            for (int32_t at = ranges.r[i].len / kKT * kKT; at < ranges.r[i].len; at += kKVBoxRows, ++boxes) {
                MixedTile& m = den.mixed[boxes / 4];
                const int b = boxes % 4;
                m.keep |= ((1ull << std::min(kKVBoxRows, ranges.r[i].len - at)) - 1ull) << (b * kKVBoxRows);
                m.tok[b] = ranges.r[i].start + at;
                m.runs |= (uint32_t)den.run_of_range[i] << (8 * b);
                m.boxes = b + 1;
            }
        }
        n_tiles += (boxes + 3) / 4;
    }
    const int3 qpos = make_int3(pos[0], pos[1], pos[2]);
    const float scale_log2 = softmax_scale * 1.4426950408889634f;
    // 64 channels take the two-CTA form once there are units for it: the wide form was measured on the tensor-bound launches
    // of a 2 240-token schedule (T = 576 and 1 024, 36 heads, 64 rows) and lost there too (26.3 vs 20.8 and 64.2 vs 53.9 ms):
    // two streams per SM do not keep the tensor pipe as busy as four, even with the chain broken.
#define AMSKV_PAIR_LAUNCH(DD, EXT, WIDE, DEN, LAZY, SHORT, ...)                                                     \
    return launch<DD, EXT, WIDE, DEN, LAZY, SHORT, __VA_ARGS__>(qm, km, vm, km64, vm64, ext, O, ranges, T, heads, pp, n_tiles, qpos,  \
                                                   scale_log2, status, sm_count, stream, den)
    // Launches of three key tiles or more take the row maximum of a unit's first tile only (the kLazy form of the
    // softmax loop: 1.7 % of a 256x256-shaped pass, 6 % of a 1024x1024-shaped one); with fewer tiles there is next
    // to nothing to skip and the plain form is the faster code.  Launches of at most four key tiles (kShort, 64
    // channels) have a producer that issues a tile's bulk copies from several lanes at once and fetches a partly
    // filled tile of the caller's tensors as one box; the long launches keep the one-lane producer (its smaller code
    // measured 2 % faster there).
    // Writes in several pieces are instantiated for the lazy form only.
    constexpr int lazy_min = 3, lazy128_min = 3, short_max = 4, split_min = 12;
    if (D == 128 && !density && !fixed_form && ext.n_pieces == 0 && pp.kind != 3) {
        // The last round of units often leaves most SMs idle.  Where at most half of them have a unit in it (and there is
        // something to halve: a merge costs about five key tiles), two CTAs share each of its units.  us per call, before /
        // after: 32 items, T = 1 600 (208 units on 148 SMs) 139 / 105, T = 4 096 (512) 535 / 491; 48 items, T = 1 024 (192) 82 / 68;
        // 64 items, T = 576 (160) 61 / 50; 128 items, T = 576 (320) 88 / 77; 256 items, T = 400 (512, 11 to 15 tiles) 89 / 86.
        // (64 channels have two CTAs per SM, and the one that is left alone in the last round runs a third faster.)
        const int32_t slots = sm_count & ~1, rest = pp.n_pairs % slots;
        if (rest > 0 && 2 * rest <= slots && n_tiles >= split_min) {
            pp.full = pp.n_pairs / slots;
            if (cur) AMSKV_PAIR_LAUNCH(128, true, true, false, true, false, false, true);
            AMSKV_PAIR_LAUNCH(128, false, true, false, true, false, false, true);
        }
    }
    if (D == 128) {
        if (density) AMSKV_PAIR_LAUNCH(128, false, true, true, false, false, false);
        if (n_tiles >= lazy128_min || ext.n_pieces > 0) {
            if (ext.n_pieces > 0) AMSKV_PAIR_LAUNCH(128, true, true, false, true, false, true);
            if (cur) AMSKV_PAIR_LAUNCH(128, true, true, false, true, false, false);
            AMSKV_PAIR_LAUNCH(128, false, true, false, true, false, false);
        }
        if (cur) AMSKV_PAIR_LAUNCH(128, true, true, false, false, false, false);
        AMSKV_PAIR_LAUNCH(128, false, true, false, false, false, false);
    }
    if (density) AMSKV_PAIR_LAUNCH(64, false, false, true, false, false, false);
    // A launch of at most one unit per SM takes the wide form: nobody shares the SM, so the second S buffer, which takes S of
    // the next tile off the chain, costs no parallelism (T = 256, 60 items 13.8 -> 12.8 us, 128 items 15.2 -> 14.6; T = 1 024, 36
    // items, 144 units 37.9 -> 33.4; with 256 units 21.0 -> 24.3).  Not for launches of both kinds of pairs (T = 576, 36 items:
    // 23.6 -> 24.7).
    if (!fixed_form && pp.n_pairs <= sm_count && pp.kind != 2) {
        if (ext.n_pieces > 0) AMSKV_PAIR_LAUNCH(64, true, true, false, true, true, true);
        if (cur) AMSKV_PAIR_LAUNCH(64, true, true, false, true, true, false);
        AMSKV_PAIR_LAUNCH(64, false, true, false, true, true, false);
    }
    if (n_tiles > short_max) {
        if (ext.n_pieces > 0) AMSKV_PAIR_LAUNCH(64, true, false, false, true, false, true);
        if (cur) AMSKV_PAIR_LAUNCH(64, true, false, false, true, false, false);
        AMSKV_PAIR_LAUNCH(64, false, false, false, true, false, false);
    }
    if (n_tiles >= lazy_min || ext.n_pieces > 0) {
        if (ext.n_pieces > 0) AMSKV_PAIR_LAUNCH(64, true, false, false, true, true, true);
        if (cur) AMSKV_PAIR_LAUNCH(64, true, false, false, true, true, false);
        AMSKV_PAIR_LAUNCH(64, false, false, false, true, true, false);
    }
    if (cur) AMSKV_PAIR_LAUNCH(64, true, false, false, false, true, false);
    AMSKV_PAIR_LAUNCH(64, false, false, false, false, true, false);
#undef AMSKV_PAIR_LAUNCH
}

}  // namespace amskv
