// Internal interface between the C ABI (api.cu) and the kernels.  Not installed.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "policy.hpp"

namespace amskv {

constexpr int kMaxRanges = 32;

// Token ranges of one layer's per-item region that an attention call reads; passed by value.
struct RangeList {
    int32_t n;
    int32_t total;  // sum of len
    Range r[kMaxRanges];
};

// A [rows, heads, tokens, D] bf16 tensor described by element strides (D contiguous).
struct Strided {
    const void* ptr;
    int64_t row, head, token;
};

// One layer's KV region: item i (= row * heads + head) owns 2 * capacity * D bf16 values,
// keys first ([capacity][D]) and values right behind them.
struct LayerRegion {
    __nv_bfloat16* base;
    int32_t capacity;  // tokens per item
};

// Device status codes written (first one wins) when a bounded wait gives up.
enum DeviceStatus : int {
    kStatusOk = 0,
    kStatusTmaTimeout = 1,
    kStatusMmaTimeout = 2,
    kStatusSyncTimeout = 3,
};

cudaError_t launch_append(const Strided& K, const Strided& V, const LayerRegion& region, int32_t token_offset,
                          int32_t T, int32_t rows, int32_t heads, int32_t D, bool bulk, int* status, int sm_count,
                          cudaStream_t stream);

// The current scale taken from the caller's K/V tensors instead of the cache: the last entry of the
// range list given with it stands for that scale (start 0, len T).  With `store`, the kernel also
// writes the scale to position `dst` of every item's part of `region` (the append fused into attention).
// `rider`: up to 16 older tokens of the cache (positions rider_tok .. rider_tok + rider_valid - 1) that are
// not in the range list but ride in the free 16-token box of the scale's last, partly filled key tile, so
// that they do not cost a tile of their own (rider_valid = 0: none; the scale's last tile must then have
// a box to spare: (T mod 64) in 1..48).
struct CurrentScaleSource {
    Strided K, V;
    bool store;
    int32_t dst;
    LayerRegion region;
    int32_t rider_tok = 0, rider_valid = 0;
    const Piece* piece = nullptr;   // the place is `n_pieces` pieces instead of T tokens from `dst` (the paired kernel)
    int32_t n_pieces = 0;
};

// (the CUDA-core kernel takes a current-scale source without `store` only)
cudaError_t launch_attend_simt(const Strided& Q, const Strided& O, const LayerRegion& region, const RangeList& ranges,
                               int32_t T, int32_t rows, int32_t heads, int32_t D, float softmax_scale,
                               cudaStream_t stream, const CurrentScaleSource* cur = nullptr);

constexpr int kSimilarityMaxBlocks = 2048;
cudaError_t launch_similarity(const __nv_bfloat16* K_prev, int32_t side_prev, const __nv_bfloat16* K_cur,
                              int32_t side_cur, int64_t items, int32_t D, double* out_ss, double* partials,
                              cudaStream_t stream);

// Tensor-core path.  The tensor maps are built on the host by the caller of launch_attend_tc.
struct TcMaps;  // defined in attend_tc.cu
bool tc_supported(int32_t D);
// Encodes the tensor maps a layer needs for its K and V streams; returns false on failure.
// (box = 64 channels x box_rows tokens of one item)
bool tc_encode_kv_maps(const LayerRegion& region, int64_t items, int32_t D, int box_rows, void* k_map_out,
                       void* v_map_out);
cudaError_t launch_attend_tc(const Strided& Q, const Strided& O, const LayerRegion& region, const void* k_map,
                             const void* v_map, const RangeList& ranges, int32_t T, int32_t rows, int32_t heads,
                             int32_t D, float softmax_scale, int* status, int sm_count, cudaStream_t stream);

// Encodes the rank-4 tensor map of a strided Q tensor (box = 64 channels x box_rows tokens).
bool tc_encode_q_map(const Strided& Q, int32_t T, int32_t rows, int32_t heads, int32_t D, int box_rows, void* map_out,
                     int pos[3]);
// The layer's region as store targets (box = 64 channels x box_rows tokens) whose token extent ends at
// `token_extent`, so that a box reaching past it is clipped by the copy engine.
bool tc_encode_kv_store_maps(const LayerRegion& region, int64_t items, int32_t D, int box_rows, int32_t token_extent,
                             void* k_map_out, void* v_map_out);

// Attention density as a by-product of a paired-kernel launch: `ranges` then has one entry per piece of a run
// of attended tokens (run_of_range[i] = the run of entry i; entries are never merged across runs), and the
// launch adds weight[r] * (sum over the item's queries of the normalised probability mass on run r) to
// out[head * n_runs + r] with atomic adds (out is zeroed by the caller, on the same stream).
constexpr int kPairMaxDensityRuns = 16;
struct PairDensity {
    double* out;
    int32_t n_runs;
    double weight[kPairMaxDensityRuns];
    int8_t run_of_range[kMaxRanges];
};

// Whether the paired kernel gives every 128-query tile of a launch a CTA and an SM of its own.
inline bool pair_one_tile_per_sm(int64_t items, int32_t T, int sm_count) { return items * ((T + 127) / 128) <= sm_count; }
// Units of a launch that pairs query tiles: two of one item, or the left-over ones of two items.
inline int64_t pair_units(int64_t items, int32_t T)
{
    const int64_t nqt = (T + 127) / 128;
    return items * (nqt / 2) + ((nqt & 1) ? (items + 1) / 2 : 0);
}

// Paired tensor-core kernel: two softmax groups per CTA, probabilities kept in tensor memory.  fixed_form: the form is chosen by the
// scale alone (two query tiles per CTA), so that an item's result does not depend on the number of items.
cudaError_t launch_attend_pair(const Strided& Q, const Strided& O, const void* k_map16, const void* v_map16,
                               const void* k_map64, const void* v_map64, const RangeList& ranges, int32_t T, int32_t rows, int32_t heads, int32_t D,
                               float softmax_scale, int* status, int sm_count, cudaStream_t stream,
                               const CurrentScaleSource* cur = nullptr, const PairDensity* density = nullptr, bool fixed_form = false);

// Warp-per-item kernel for the coarse scales: every retained key in one register tile.
constexpr int kSmallMaxKeys = 32;
constexpr int kSmallMaxQueries = 16;
bool small_supported(int32_t T, int32_t total_keys);
// With `cur`, `ranges` lists the cached keys only and the current scale's T tokens come from the caller's
// tensors (and are written to position cur->dst of the region when cur->store is set): T plus the cached
// keys must fit the limits.  A single-token scale that is its own only key is served by a copy kernel.
cudaError_t launch_attend_small(const Strided& Q, const Strided& O, const LayerRegion& region, const RangeList& ranges,
                                int32_t T, int32_t rows, int32_t heads, int32_t D, float softmax_scale,
                                int sm_count, cudaStream_t stream, const CurrentScaleSource* cur = nullptr);

// Kernel for calls of few items or few queries (attend_mid.cu): a CTA per item and group of query blocks, warp-level matrix
// instructions.  With `cur`, `ranges` lists the cached keys only and the current scale's tokens come from the caller's
// tensors; `piece` says where they go in the region (n_pieces = 0: nowhere).  With `density` (then without `cur`) an entry
// of `ranges` belongs to one run, as for the paired kernel.
bool mid_preferred(int32_t T, int32_t total_keys, int64_t items, int32_t D, int sm_count, bool density, bool copies);
cudaError_t launch_attend_mid(const Strided& Q, const Strided& O, const LayerRegion& region, const RangeList& ranges, int32_t T,
                              int32_t rows, int32_t heads, int32_t D, float softmax_scale, int sm_count, cudaStream_t stream,
                              const CurrentScaleSource* cur = nullptr, const Piece* piece = nullptr, int32_t n_pieces = 0,
                              const PairDensity* density = nullptr);

// Attention density: the pieces of the per-item region that hold the attended tokens, each with the run
// (of the attended-token list) it belongs to and the weight 1 / (tokens of that run).
constexpr int kMaxDensityPieces = 96;
struct DensityPieces {
    int32_t n, n_runs;
    int32_t start[kMaxDensityPieces], len[kMaxDensityPieces], run[kMaxDensityPieces];
    double weight[kMaxDensityPieces];
};
cudaError_t launch_zero(double* p, size_t n, cudaStream_t stream);
cudaError_t launch_density(const Strided& Q, const LayerRegion& region, const DensityPieces& pieces, int32_t T,
                           int32_t rows, int32_t heads, int32_t D, float softmax_scale, double* out, cudaStream_t stream);

// One warp whose bounded wait runs out after `limit` iterations (nothing ever arrives): records
// kStatusSyncTimeout in *status and returns normally.
cudaError_t launch_wait_gives_up(uint32_t limit, int* status, cudaStream_t stream);

void count_launch(int n = 1);

// Launches a kernel that may start while the kernel before it in the stream drains (programmatic stream
// serialisation).  Such a kernel waits (overlap_with_previous) before its first access to global memory until the kernel
// before it has ended and its writes are visible; what is hidden is launch latency and set-up (barriers, tensor memory,
// tables): 30 layers of one image 2 339 -> 2 082 us in a graph, a layer called step by step 84 -> 65 us; launches of
// several hundred microseconds are unchanged.  It lets the next kernel in only after its own wait: released before it,
// kernels pile up two and three deep, and the CTAs of the later ones take the free SMs (T = 256, 60 items: 14.6 -> 15.3 us
// a call; released after it: 13.2).
// overlap = false launches the ordinary way: all but the smallest append copies, and the attention of amskv_attend, which
// normally follows its scale's append, where that copy is large (overlaps_append).  Copies that start on SMs still
// configured for the attention kernel's shared memory keep their small L1, which is where their loads in flight are held,
// and attention CTAs placed beside the last blocks of a copy find an SM with its shared-memory split, which only an idle SM
// can change (T = 256, 1 920 items, a copy before each: +4 to +9 %).
struct KernelMemory {     // dynamic shared memory, and the CTAs of a cluster (1: no clusters)
    size_t bytes;
    unsigned cluster;
    KernelMemory(size_t n, unsigned c = 1) : bytes(n), cluster(c) {}
};
template <typename... P, typename... A>
cudaError_t launch_kernel(bool overlap, void (*kernel)(P...), dim3 grid, dim3 block, KernelMemory smem, cudaStream_t stream, const A&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem.bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    unsigned n = 0;
    if (overlap) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (smem.cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = smem.cluster;
        attr[n].val.clusterDim.y = 1;
        attr[n++].val.clusterDim.z = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, P(args)...);
    if (e == cudaSuccess) count_launch();
    return e;
}
#ifdef __CUDACC__
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// A kernel that allocates tensor memory calls this behind a barrier that follows the allocation: the CTAs it lets in may
// allocate at once, and then hold their columns until this launch has ended.
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void overlap_with_previous()
{
    wait_for_previous();
    let_next_start();
}
__device__ __forceinline__ float fast_exp2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Loads of what an earlier launch wrote or the caller passed.  A kernel that is alive while its predecessor still writes may not
// use the read-only path (ld.global.nc, which __ldg and const __restrict__ pointers lead to: the data must not change while
// the kernel runs, and the compiler may move such a load above the wait).  These are ordinary loads that stay behind it.
__device__ __forceinline__ uint4 load_16B(const void* p)
{
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint4 load_16B_once(const void* p)   // (data that no other load wants)
{
    uint4 v;
    asm volatile("ld.global.cs.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ double load_double(const double* p)
{
    double v;
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}
#endif

// The attention of amskv_attend overlaps the copy of its scale's append where all blocks of that copy are resident at once
// (eight per SM): us per append and attend, 64 channels: 60 items T = 100 11.5 -> 9.7, 256 items T = 64 12.5 -> 11.7, 512 items
// T = 169 34.7 -> 33.2, 1 110 items T = 100 32.7 -> 31.3; beyond, 1 920 items T = 256 140 -> 147, 3 840 items T = 361 567 -> 591.
constexpr int kAppendBlockChunks = 1024;   // 16-byte chunks of K (and of V) a block of the copy moves
inline bool overlaps_append(int64_t items, int32_t T, int32_t D, int sm_count)
{
    return items * T * (D / 8) <= 8ll * kAppendBlockChunks * sm_count;
}

// A kernel's dynamic shared-memory limit is a per-device setting: raised once per device and kernel,
// from whichever host thread gets there first (setting it twice is harmless).
struct SharedMemoryOptIn {
    std::atomic<uint64_t> done{0};   // bit d: set on device d
    template <typename Kernel>
    cudaError_t ensure(Kernel* kernel, int bytes)
    {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64 && ((done.load(std::memory_order_acquire) >> dev) & 1u)) return cudaSuccess;
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e == cudaSuccess && dev >= 0 && dev < 64) done.fetch_or(1ull << dev, std::memory_order_release);
        return e;
    }
};

}  // namespace amskv
