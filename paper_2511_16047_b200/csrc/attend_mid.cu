// Attention for calls of few (row, head) items or few queries, which the paired tensor-memory kernel spends on its
// set-up and on its per-tile chain rather than on memory or arithmetic.
//
// A CTA serves up to NW / 2 sixteen-row query blocks of one item with warp-level matrix instructions (mma.sync), two warps
// per query block, each with half of the keys of every chunk.  Keys are one packed sequence -- the retained ranges of the
// cache first, then (append fused in) the current scale in the caller's tensors -- cut into 64-key chunks with no regard
// to where a range ends.  K and V of a chunk go to a stage of shared memory by 16-byte asynchronous copies of all threads, up
// to kStages chunks ahead, so the whole key set of a coarse scale is in flight after a few hundred clocks; there is no
// tensor map, no tensor memory to allocate and no role to hand data to.  The thread that copied a piece of the current
// scale also writes it to its place in the cache, after the output where the stage can wait that long.
//
// S = Q K^T takes both operands as 16-byte pieces used directly as fragment registers (the contraction order inside a
// piece is permuted alike on both sides); K pieces are swizzled by the row's lowest bit for conflict-free 16-byte
// reads, V pieces by its three lowest bits for ldmatrix.trans.  A row's reference maximum moves only when a chunk exceeds
// it by more than 2^8; the two halves of the keys are merged through shared memory at the end.
//
// Attention density (kDen): the mass of a row on each of up to 16 runs of keys is P times a 0/1 matrix of run membership,
// two more column tiles of the second product.  P enters as the sum of three bf16 numbers, which hold all 24 bits of the fp32
// probabilities; a step's products go into accumulators of their own, added up in fp32 with rounding (the tensor pipe
// truncates), and rows are added up in fp64.  With two terms, one accumulator and fp32 sums and weights the masses were off by
// 1.4e-7 (480 items, T = 4) and 4.6e-7 (32 items; 1.7e-6 at a single entry); with these by 6e-9 and 1.5e-8, the CUDA-core pass by
// 6e-9 and 2.4e-8.  512 items, T = 16: 8.9 -> 9.2 us a call.
#include <cstring>

#include "kernels.cuh"

namespace amskv {

namespace {

constexpr int kChunk = 64;            // keys per stage
constexpr int kSplits = 2;            // warps per query block
constexpr float kRescaleLog2 = 8.f;
constexpr int kMaxDenRuns = kPairMaxDensityRuns;

template <int D, bool kDen>
struct MidCfg {
    static constexpr int kStages = D == 64 ? 4 : 2;
    static constexpr int kRowBytes = D * 2;
    static constexpr int kTileBytes = kChunk * kRowBytes;       // one of K, V
    static constexpr int kStageBytes = 2 * kTileBytes;
    static constexpr int kMergeBytes = (16 * D + 32 + (kDen ? 256 : 0)) * 4;   // O, maxima and sums (and masses) of 16 rows
};

struct MidExt {
    const __nv_bfloat16* K;
    const __nv_bfloat16* V;
    int64_t row, head, tok;            // element strides, the same for K and V
    int32_t len;                       // tokens of the current scale read from there (0: none)
    int32_t n_pieces;                  // where they go in the per-item region
    Piece piece[LayerLayout::kMaxPieces];
};
struct MidDen {
    double* out;
    int32_t n_runs;
    double weight[kMaxDenRuns];
    int8_t run_of_range[kMaxRanges];
};

__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                          uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
// 16 bytes global -> shared
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ float max3(float a, float b, float c)
{
    float y;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
    return y;
}
// a * b + c and d + a on two packed fp32 lanes
__device__ __forceinline__ void fma2(float& d0, float& d1, float a0, float a1, float b, float c)
{
    asm("{\n"
        ".reg .b64 ra, rb, rc, rd;\n"
        "mov.b64 ra, {%2, %3};\n"
        "mov.b64 rb, {%4, %4};\n"
        "mov.b64 rc, {%5, %5};\n"
        "fma.rn.f32x2 rd, ra, rb, rc;\n"
        "mov.b64 {%0, %1}, rd;\n"
        "}\n"
        : "=f"(d0), "=f"(d1)
        : "f"(a0), "f"(a1), "f"(b), "f"(c));
}
__device__ __forceinline__ void add2(float (&d)[2], float a0, float a1)
{
    asm("{\n"
        ".reg .b64 ra, rd;\n"
        "mov.b64 ra, {%2, %3};\n"
        "mov.b64 rd, {%0, %1};\n"
        "add.rn.f32x2 rd, rd, ra;\n"
        "mov.b64 {%0, %1}, rd;\n"
        "}\n"
        : "+f"(d[0]), "+f"(d[1])
        : "f"(a0), "f"(a1));
}

// 4x4 transpose of 32-bit words among the four lanes of a quad: lane q's w[j] becomes lane j's w[q]
__device__ __forceinline__ void quad_transpose(uint32_t (&w)[4], int q)
{
    const bool odd = q & 1, high = q & 2;
    {
        const uint32_t s0 = odd ? w[0] : w[1], s1 = odd ? w[2] : w[3];
        const uint32_t r0 = __shfl_xor_sync(0xffffffffu, s0, 1), r1 = __shfl_xor_sync(0xffffffffu, s1, 1);
        if (odd) { w[0] = r0; w[2] = r1; } else { w[1] = r0; w[3] = r1; }
    }
    {
        const uint32_t s0 = high ? w[0] : w[2], s1 = high ? w[1] : w[3];
        const uint32_t r0 = __shfl_xor_sync(0xffffffffu, s0, 2), r1 = __shfl_xor_sync(0xffffffffu, s1, 2);
        if (high) { w[0] = r0; w[1] = r1; } else { w[2] = r0; w[3] = r1; }
    }
}

template <int N>
__device__ __forceinline__ void scale_rows(float (&o)[N][4], float f_a, float f_b)
{
#pragma unroll
    for (int n = 0; n < N; ++n) {
        o[n][0] *= f_a;
        o[n][1] *= f_a;
        o[n][2] *= f_b;
        o[n][3] *= f_b;
    }
}

template <int D, int NW, bool kDen>
__global__ void __launch_bounds__(NW * 32, D == 64 ? 16 / NW : 2)
attend_mid_kernel(const __nv_bfloat16* Q, int64_t q_row, int64_t q_head, int64_t q_tok,
                  __nv_bfloat16* __restrict__ O, int64_t o_row, int64_t o_head, int64_t o_tok,
                  __nv_bfloat16* __restrict__ region, int32_t capacity, const __grid_constant__ RangeList ranges,
                  int32_t T, int32_t heads, int32_t parts, int32_t n_rb, int32_t n_stages, float scale_log2,
                  const __grid_constant__ MidExt ext, const __grid_constant__ MidDen den)
{
    using C = MidCfg<D, kDen>;
    constexpr int kPieces = D / 32;            // 16-byte pieces of a token row per lane in fragment order
    constexpr int kTokPieces = D / 8;          // 16-byte pieces of a token row
    constexpr int kWarpKeys = kChunk / kSplits, kTiles = kWarpKeys / 8;
    constexpr int kDenTiles = kDen ? 2 : 1;    // (one unused register tile otherwise)
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ int8_t key_run[kDen ? C::kStages : 1][kChunk];
    __shared__ double den_sum[kDen ? kMaxDenRuns : 1];
    const uint32_t smem0 = (uint32_t)__cvta_generic_to_shared(smem);
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int g = lane >> 2, q = lane & 3;
    const int ks = warp % kSplits, rb = warp / kSplits;
    const int32_t item = blockIdx.x / parts, part = blockIdx.x - item * parts;
    const int32_t row = item / heads, head = item - row * heads;
    const int32_t m0 = (part * n_rb + rb) * 16;                 // first query row of this warp
    const bool live = rb < n_rb && m0 < T;                      // (a warp without a query block only copies)
    const int32_t Lc = ranges.total, L = Lc + ext.len;
    const int32_t n_chunks = (L + kChunk - 1) / kChunk;
    __nv_bfloat16* kbase = region + (int64_t)item * (2ll * capacity * D);
    const int64_t v_shift = (int64_t)capacity * D;

    // This thread's part of the copies: one 16-byte column of every kStep-th row.  kStep is a multiple of 8, so the
    // swizzle of a thread's rows is the same for all of them.
    constexpr int kStep = NW * 32 / kTokPieces, kRows = kChunk / kStep;
    static_assert(kStep % 8 == 0 && kChunk % kStep == 0, "copy mapping");
    const int cp_piece = (int)threadIdx.x % kTokPieces, cp_row0 = (int)threadIdx.x / kTokPieces;
    const uint32_t k_slot = (uint32_t)cp_row0 * C::kRowBytes + (uint32_t)((cp_piece ^ ((cp_row0 & 1) << 2)) << 4);
    const uint32_t v_slot = C::kTileBytes + (uint32_t)cp_row0 * C::kRowBytes + (uint32_t)((cp_piece ^ (cp_row0 & 7)) << 4);

    // The source of keys src_first .. src_end - 1; walks forward as the chunks do.
    int src_range = -1;
    int32_t src_first = 0, src_end = 0;
    const __nv_bfloat16 *src_k = nullptr, *src_v = nullptr;   // of key src_first
    int64_t src_tok = D;
    auto next_source = [&]() {
        ++src_range;
        src_first = src_end;
        if (src_range < ranges.n) {
            src_k = kbase + (int64_t)ranges.r[src_range].start * D;
            src_v = src_k + v_shift;
            src_end = src_first + ranges.r[src_range].len;
        } else {
            src_k = ext.K + row * ext.row + head * ext.head;
            src_v = ext.V + row * ext.row + head * ext.head;
            src_tok = ext.tok;
            src_end = L;
        }
    };
    auto load_chunk = [&](int c, int stage) {
        const uint32_t st = smem0 + (uint32_t)stage * C::kStageBytes;
        const int32_t first = c * kChunk, end = min(first + kChunk, L);
        // one pass per source the chunk draws from (nearly always one)
        for (int32_t at = first; at < end;) {
            while (at >= src_end) next_source();
            const int32_t stop = min(src_end, end);
            const __nv_bfloat16* kp = src_k + (int64_t)(first + cp_row0 - src_first) * src_tok + cp_piece * 8;
            const __nv_bfloat16* vp = src_v + (int64_t)(first + cp_row0 - src_first) * src_tok + cp_piece * 8;
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                const int32_t key = first + cp_row0 + i * kStep;
                if (key >= at && key < stop) {
                    cp_async16(st + k_slot + i * kStep * C::kRowBytes, kp + (int64_t)(i * kStep) * src_tok);
                    cp_async16(st + v_slot + i * kStep * C::kRowBytes, vp + (int64_t)(i * kStep) * src_tok);
                    if (kDen && cp_piece == 0) key_run[stage][cp_row0 + i * kStep] = den.run_of_range[src_range];
                }
            }
            at = stop;
        }
        if (end - first < kChunk) {   // rows past the last key: finite, and of no run
#pragma unroll
            for (int i = 0; i < kRows; ++i)
                if (first + cp_row0 + i * kStep >= end) {
                    uint8_t* dst = smem + stage * C::kStageBytes + i * kStep * C::kRowBytes;
                    *reinterpret_cast<uint4*>(dst + k_slot) = make_uint4(0, 0, 0, 0);
                    *reinterpret_cast<uint4*>(dst + v_slot) = make_uint4(0, 0, 0, 0);
                    if (kDen && cp_piece == 0) key_run[stage][cp_row0 + i * kStep] = -1;
                }
        }
    };
    // the append: this thread's own pieces of chunk c's share of the current scale, from the stage to their place in the
    // cache (the item's CTAs share the chunks)
    auto store_chunk = [&](int c, int stage) {
        if (ext.n_pieces == 0 || (c + 1) * kChunk <= Lc || c % parts != part) return;
        const uint8_t* tile = smem + stage * C::kStageBytes;
#pragma unroll 1
        for (int i = 0; i < kRows; ++i) {
            const int32_t j = c * kChunk + cp_row0 + i * kStep - Lc;
            if (j < 0 || j >= ext.len) continue;
            const uint4 kv = *reinterpret_cast<const uint4*>(tile + k_slot + i * kStep * C::kRowBytes);
            const uint4 vv = *reinterpret_cast<const uint4*>(tile + v_slot + i * kStep * C::kRowBytes);
            // (a token can have two places: in the ring or its head, and in the slot of a scale that is attended from there)
            for (int n = 0; n < ext.n_pieces; ++n) {
                if (j < ext.piece[n].src || j >= ext.piece[n].src + ext.piece[n].len) continue;
                __nv_bfloat16* kd = kbase + (int64_t)(ext.piece[n].dst + j - ext.piece[n].src) * D + cp_piece * 8;
                *reinterpret_cast<uint4*>(kd) = kv;
                *reinterpret_cast<uint4*>(kd + v_shift) = vv;
            }
        }
    };

    next_source();   // (reads launch parameters only)
    const __nv_bfloat16* qbase = Q + row * q_row + head * q_head;
    const uint4* q0 = reinterpret_cast<const uint4*>(qbase + min(m0 + g, T - 1) * q_tok + 8 * q);
    const uint4* q1 = reinterpret_cast<const uint4*>(qbase + min(m0 + g + 8, T - 1) * q_tok + 8 * q);
    overlap_with_previous();
    // query pieces of rows m0 + g and m0 + g + 8 (clamped; rows past T are not stored)
    uint4 qa0[kPieces], qa1[kPieces];
#pragma unroll
    for (int h = 0; h < kPieces; ++h) {
        qa0[h] = load_16B(q0 + 4 * h);
        qa1[h] = load_16B(q1 + 4 * h);
    }
#pragma unroll 1
    for (int c = 0; c < C::kStages; ++c) {
        if (c < n_chunks) load_chunk(c, c);   // (n_stages = min(kStages, n_chunks))
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    if (kDen && threadIdx.x < kMaxDenRuns) den_sum[threadIdx.x] = 0.0;

    float o[D / 8][4];
#pragma unroll
    for (int n = 0; n < D / 8; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;
    float od[kDenTiles][4];
#pragma unroll
    for (int n = 0; n < kDenTiles; ++n) od[n][0] = od[n][1] = od[n][2] = od[n][3] = 0.f;
    float m_a = -INFINITY, m_b = -INFINITY, nb_a = 0.f, nb_b = 0.f;
    float l2_a[2] = {0.f, 0.f}, l2_b[2] = {0.f, 0.f};   // row sums of the even and of the odd keys

    int stage = 0;
#pragma unroll 1
    for (int c = 0; c < n_chunks; ++c) {
        asm volatile("cp.async.wait_group %0;" ::"n"(C::kStages - 1) : "memory");
        __syncthreads();
        const uint8_t* tile = smem + stage * C::kStageBytes;
        const int32_t key0 = c * kChunk + ks * kWarpKeys;
        if (live && key0 < L) {
            const uint8_t* kt = tile + (ks * kWarpKeys + g) * C::kRowBytes;
            const int kx = (q ^ ((g & 1) << 2)) << 4;
            float s[kTiles][4];
#pragma unroll
            for (int t = 0; t < kTiles; ++t) {
                s[t][0] = s[t][1] = s[t][2] = s[t][3] = 0.f;
#pragma unroll
                for (int h = 0; h < kPieces; ++h) {
                    const uint4 kk = *reinterpret_cast<const uint4*>(kt + t * 8 * C::kRowBytes + (kx ^ (h << 6)));
                    mma_16816(s[t], qa0[h].x, qa1[h].x, qa0[h].y, qa1[h].y, kk.x, kk.y);
                    mma_16816(s[t], qa0[h].z, qa1[h].z, qa0[h].w, qa1[h].w, kk.z, kk.w);
                }
            }
            if (key0 + kWarpKeys > L) {
#pragma unroll
                for (int t = 0; t < kTiles; ++t)
#pragma unroll
                    for (int e = 0; e < 2; ++e)
                        if (key0 + t * 8 + 2 * q + e >= L) s[t][e] = s[t][2 + e] = -INFINITY;
            }
            float mx_a = fmaxf(s[0][0], s[0][1]), mx_b = fmaxf(s[0][2], s[0][3]);
#pragma unroll
            for (int t = 1; t < kTiles; ++t) {
                mx_a = max3(mx_a, s[t][0], s[t][1]);
                mx_b = max3(mx_b, s[t][2], s[t][3]);
            }
            mx_a = fmaxf(mx_a, __shfl_xor_sync(0xffffffffu, mx_a, 1));
            mx_b = fmaxf(mx_b, __shfl_xor_sync(0xffffffffu, mx_b, 1));
            mx_a = fmaxf(mx_a, __shfl_xor_sync(0xffffffffu, mx_a, 2));
            mx_b = fmaxf(mx_b, __shfl_xor_sync(0xffffffffu, mx_b, 2));
            // (the first chunk always moves the reference: it starts at minus infinity)
            const bool grow_a = (mx_a - m_a) * scale_log2 > kRescaleLog2, grow_b = (mx_b - m_b) * scale_log2 > kRescaleLog2;
            if (__any_sync(0xffffffffu, grow_a || grow_b)) {
                const float f_a = grow_a ? fast_exp2((m_a - mx_a) * scale_log2) : 1.f;
                const float f_b = grow_b ? fast_exp2((m_b - mx_b) * scale_log2) : 1.f;
                if (grow_a) { m_a = mx_a; nb_a = -mx_a * scale_log2; }
                if (grow_b) { m_b = mx_b; nb_b = -mx_b * scale_log2; }
                l2_a[0] *= f_a;
                l2_a[1] *= f_a;
                l2_b[0] *= f_b;
                l2_b[1] *= f_b;
                scale_rows(o, f_a, f_b);
                if (kDen) scale_rows(od, f_a, f_b);
            }
            // ---- P V, 16 keys at a time
            const int vkey = ks * kWarpKeys + (lane & 15);
            const uint32_t vt = smem0 + (uint32_t)stage * C::kStageBytes + C::kTileBytes + (uint32_t)vkey * C::kRowBytes;
            const uint32_t vx = (uint32_t)(((lane >> 4) ^ (vkey & 7)) << 4);
#pragma unroll
            for (int step = 0; step < kTiles / 2; ++step) {
                uint32_t p[4];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    float (&x)[4] = s[2 * step + u];
                    fma2(x[0], x[1], x[0], x[1], scale_log2, nb_a);
                    fma2(x[2], x[3], x[2], x[3], scale_log2, nb_b);
#pragma unroll
                    for (int e = 0; e < 4; ++e) x[e] = fast_exp2(x[e]);
                    add2(l2_a, x[0], x[1]);
                    add2(l2_b, x[2], x[3]);
                    p[2 * u] = pack_bf16(x[0], x[1]);
                    p[2 * u + 1] = pack_bf16(x[2], x[3]);
                }
#pragma unroll
                for (int j = 0; j < D / 16; ++j) {
                    uint32_t v[4];
                    ldmatrix_x4_trans(v, vt + step * 16 * C::kRowBytes + ((uint32_t)(j << 5) ^ vx));
                    mma_16816(o[2 * j], p[0], p[1], p[2], p[3], v[0], v[1]);
                    mma_16816(o[2 * j + 1], p[0], p[1], p[2], p[3], v[2], v[3]);
                }
                if (kDen) {
                    uint32_t mid[4], lo[4];   // what P leaves, and what that leaves (differences are exact)
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float (&x)[4] = s[2 * step + u / 2];
                        const float a = x[2 * (u & 1)] - bf16_lo(p[u]), b = x[2 * (u & 1) + 1] - bf16_hi(p[u]);
                        mid[u] = pack_bf16(a, b);
                        lo[u] = pack_bf16(a - bf16_lo(mid[u]), b - bf16_hi(mid[u]));
                    }
                    const int8_t* kr = &key_run[kDen ? stage : 0][ks * kWarpKeys + step * 16 + 2 * q];
#pragma unroll
                    for (int n = 0; n < kDenTiles; ++n) {
                        const int run = n * 8 + g;
                        const uint32_t b0 = (kr[0] == run ? 0x3f80u : 0u) | (kr[1] == run ? 0x3f800000u : 0u);
                        const uint32_t b1 = (kr[8] == run ? 0x3f80u : 0u) | (kr[9] == run ? 0x3f800000u : 0u);
                        float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f}, d2[4] = {0.f, 0.f, 0.f, 0.f};
                        mma_16816(d0, p[0], p[1], p[2], p[3], b0, b1);
                        mma_16816(d1, mid[0], mid[1], mid[2], mid[3], b0, b1);
                        mma_16816(d2, lo[0], lo[1], lo[2], lo[3], b0, b1);
#pragma unroll
                        for (int e = 0; e < 4; ++e) od[n][e] += d0[e] + (d1[e] + d2[e]);
                    }
                }
            }
        }
        if (c + C::kStages < n_chunks) {
            store_chunk(c, stage);
            __syncthreads();
            load_chunk(c + C::kStages, stage);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        stage = stage + 1 == n_stages ? 0 : stage + 1;
    }

    // row sums: a row is spread over the four lanes of a quad
    float l_a = l2_a[0] + l2_a[1], l_b = l2_b[0] + l2_b[1];
    l_a += __shfl_xor_sync(0xffffffffu, l_a, 1);
    l_b += __shfl_xor_sync(0xffffffffu, l_b, 1);
    l_a += __shfl_xor_sync(0xffffffffu, l_a, 2);
    l_b += __shfl_xor_sync(0xffffffffu, l_b, 2);

    // ---- merge the two halves of the keys: the second warp leaves its part in shared memory, the first adds it
    float* other = reinterpret_cast<float*>(smem + n_stages * C::kStageBytes + rb * C::kMergeBytes);
    float4* other4 = reinterpret_cast<float4*>(other);
    float* other_ml = other + 16 * D;
    float4* other_den = reinterpret_cast<float4*>(other + 16 * D + 32);
    if (ks > 0 && live) {
#pragma unroll
        for (int n = 0; n < D / 8; ++n) other4[n * 32 + lane] = make_float4(o[n][0], o[n][1], o[n][2], o[n][3]);
        if (q == 0) {
            other_ml[g] = m_a;
            other_ml[8 + g] = m_b;
            other_ml[16 + g] = l_a;
            other_ml[24 + g] = l_b;
        }
        if (kDen) {
#pragma unroll
            for (int n = 0; n < kDenTiles; ++n) other_den[n * 32 + lane] = make_float4(od[n][0], od[n][1], od[n][2], od[n][3]);
        }
    }
    __syncthreads();
    if (ks == 0 && live) {
        const float om_a = other_ml[g], om_b = other_ml[8 + g];
        const float M_a = fmaxf(m_a, om_a), M_b = fmaxf(m_b, om_b);
        const float f_a = fast_exp2((m_a - M_a) * scale_log2), f_b = fast_exp2((m_b - M_b) * scale_log2);
        const float e_a = fast_exp2((om_a - M_a) * scale_log2), e_b = fast_exp2((om_b - M_b) * scale_log2);
        l_a = fmaf(other_ml[16 + g], e_a, l_a * f_a);
        l_b = fmaf(other_ml[24 + g], e_b, l_b * f_b);
        scale_rows(o, f_a, f_b);
#pragma unroll
        for (int n = 0; n < D / 8; ++n) {
            const float4 x = other4[n * 32 + lane];
            o[n][0] = fmaf(x.x, e_a, o[n][0]);
            o[n][1] = fmaf(x.y, e_a, o[n][1]);
            o[n][2] = fmaf(x.z, e_b, o[n][2]);
            o[n][3] = fmaf(x.w, e_b, o[n][3]);
        }
        if (kDen) {
            scale_rows(od, f_a, f_b);
#pragma unroll
            for (int n = 0; n < kDenTiles; ++n) {
                const float4 x = other_den[n * 32 + lane];
                od[n][0] = fmaf(x.x, e_a, od[n][0]);
                od[n][1] = fmaf(x.y, e_a, od[n][1]);
                od[n][2] = fmaf(x.z, e_b, od[n][2]);
                od[n][3] = fmaf(x.w, e_b, od[n][3]);
            }
        }
        // ---- out = O / l: after a transpose among the quad a lane holds 8 consecutive channels of its rows
        const float inv_a = 1.f / l_a, inv_b = 1.f / l_b;
        const bool st_a = m0 + g < T, st_b = m0 + g + 8 < T;
        __nv_bfloat16* obase = O + row * o_row + head * o_head + (int64_t)(m0 + g) * o_tok + 8 * q;
#pragma unroll
        for (int h = 0; h < kPieces; ++h) {
            uint32_t w[4], x[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                w[j] = pack_bf16(o[4 * h + j][0] * inv_a, o[4 * h + j][1] * inv_a);
                x[j] = pack_bf16(o[4 * h + j][2] * inv_b, o[4 * h + j][3] * inv_b);
            }
            quad_transpose(w, q);
            quad_transpose(x, q);
            if (st_a) *reinterpret_cast<uint4*>(obase + 32 * h) = make_uint4(w[0], w[1], w[2], w[3]);
            if (st_b) *reinterpret_cast<uint4*>(obase + 8 * o_tok + 32 * h) = make_uint4(x[0], x[1], x[2], x[3]);
        }
        if (kDen) {
            // normalised by the sum of the row's masses, which is l added up in another order: their shares add up to one
            float d_a = (od[0][0] + od[0][1]) + (od[kDenTiles - 1][0] + od[kDenTiles - 1][1]);
            float d_b = (od[0][2] + od[0][3]) + (od[kDenTiles - 1][2] + od[kDenTiles - 1][3]);
            d_a += __shfl_xor_sync(0xffffffffu, d_a, 1);
            d_b += __shfl_xor_sync(0xffffffffu, d_b, 1);
            d_a += __shfl_xor_sync(0xffffffffu, d_a, 2);
            d_b += __shfl_xor_sync(0xffffffffu, d_b, 2);
            d_a = 1.f / d_a;
            d_b = 1.f / d_b;
#pragma unroll
            for (int n = 0; n < kDenTiles; ++n)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    double v = (double)(st_a ? od[n][e] * d_a : 0.f) + (double)(st_b ? od[n][2 + e] * d_b : 0.f);
                    v += __shfl_xor_sync(0xffffffffu, v, 4);
                    v += __shfl_xor_sync(0xffffffffu, v, 8);
                    v += __shfl_xor_sync(0xffffffffu, v, 16);
                    if (g == 0) atomicAdd(&den_sum[kDen ? n * 8 + 2 * q + e : 0], v);
                }
        }
    }
    // chunks whose stages were never refilled (a thread reads back its own copies only)
    for (int c = max(0, n_chunks - C::kStages); c < n_chunks; ++c) store_chunk(c, c % n_stages);
    if (kDen) {
        __syncthreads();
        if ((int)threadIdx.x < den.n_runs)
            atomicAdd(den.out + (int64_t)head * den.n_runs + threadIdx.x, den_sum[kDen ? threadIdx.x : 0] * den.weight[threadIdx.x]);
    }
}

template <int D, int NW, bool kDen>
cudaError_t launch(bool overlap, const Strided& Q, const Strided& O, const LayerRegion& region, const RangeList& ranges, int32_t T,
                   int32_t heads, int64_t items, float scale_log2, const MidExt& ext, const MidDen& den, cudaStream_t stream)
{
    using C = MidCfg<D, kDen>;
    const int n_rb_all = (T + 15) / 16;
    const int parts = (n_rb_all + NW / kSplits - 1) / (NW / kSplits);
    const int n_rb = (n_rb_all + parts - 1) / parts;
    if (items * parts > 0x7fffffffll) return cudaErrorInvalidValue;
    const int n_chunks = (ranges.total + ext.len + kChunk - 1) / kChunk;
    const int n_stages = n_chunks < C::kStages ? n_chunks : C::kStages;
    static SharedMemoryOptIn opt_in;
    const cudaError_t oe = opt_in.ensure(attend_mid_kernel<D, NW, kDen>, C::kStages * C::kStageBytes + NW / kSplits * C::kMergeBytes);
    if (oe != cudaSuccess) return oe;
    return launch_kernel(overlap, attend_mid_kernel<D, NW, kDen>, dim3((unsigned)(items * parts)), dim3(NW * 32),
                         (size_t)(n_stages * C::kStageBytes + n_rb * C::kMergeBytes), stream, (const __nv_bfloat16*)Q.ptr, Q.row,
                         Q.head, Q.token, (__nv_bfloat16*)O.ptr, O.row, O.head, O.token, region.base, region.capacity, ranges, T,
                         heads, (int32_t)parts, (int32_t)n_rb, (int32_t)n_stages, scale_log2, ext, den);
}

}  // namespace

// Where this kernel serves a call, in units of work (16 queries x 64 keys of one item) per SM.  Below the lines the paired kernel
// costs 5 to 9 us whatever the size (and the copy before it, where the append is not fused into that); above them the warp-level
// matrix instructions, a quarter of the tensor pipe's rate, are what the call takes.
//   64 channels   19 units; above 32 queries no more CTAs (of eight warps, two to an SM) than are resident at once; 7 units above 81
//                 queries where the paired kernel has an SM for every query tile, 19 there too for an append of several copies
//   128 channels  6 units; none above 64 queries where the paired kernel has an SM for every tile, but for several copies
// us per call, this kernel / the paired one, in a graph, append included: f fused, s a call of its own, c of several copies.
//     T   64 channels                                                 128 channels
//    25   f 60 items 3.6 / 5.9, 512 6.1 / 8.6, 1 024 (13.8 units)     f 60 4.7 / 6.8, 512 (6.9 units) 12.6 / 12.8, 700 17.4 / 16.2
//         11.1 / 12.4, 1 920 (25.9) 19.4 / 17.6
//    36   f 60 4.4 / 4.7, 256 5.9 / 7.0, 300 (second wave) 9.5 / 8.0  f 8 5.6 / 4.8, 60 5.7 / 5.2, 96 6.4 / 6.3, 148 (6.0) 6.9 / 7.8
//                                                                     s 32 6.8 / 7.5, 96 8.2 / 8.2, 148 8.3 / 9.3, 200 12.6 / 10.8
//    49   f 60 4.4 / 4.9, 256 7.0 / 7.5, 300 11.1 / 8.3               f 60 5.5 / 5.4, 120 7.1 / 7.2
//    64   f 60 4.7 / 4.7, 148 5.5 / 6.7, 200 (10.8) 7.5 / 7.2,        f 8 5.9 / 4.9, 60 6.0 / 5.4, 148 (8.0) 8.7 / 8.2
//         256 8.3 / 7.6; s 200 9.1 / 9.9, 256 9.8 / 10.7
//    81   f 8 5.4 / 4.9, 60 5.9 / 5.2, 148 7.7 / 7.4;                 f 8 7.3 / 5.7, 60 8.5 / 6.1
//         s 32 (3.9) 6.4 / 7.2, 60 (7.3) 8.2 / 7.2
//   100   f 8 5.4 / 5.2, 60 (8.5) 6.0 / 5.4, 148 8.8 / 7.8;           f 8 7.2 / 5.9; c 32 (4.5) 7.6 / 8.0, 60 (8.5) 9.6 / 8.5
//         s 32 7.0 / 7.5, 60 9.0 / 7.6; c 120 (17) 8.4 / 8.8, 148 (21) 9.0 / 9.3
//   121   s 32 (6.9) 7.7 / 8.0, 60 10.6 / 8.5; c 60 (13) 7.4 / 8.5, 96 (20.8) 9.9 / 9.6
//   169   f 8 6.8 / 6.7, 32 8.0 / 7.0; s 16 (5.9) 7.7 / 8.5,          c 8 (3.0) 7.5 / 8.0, 32 (7.1) 9.2 / 8.5
//         32 (11.9) 9.0 / 8.7; c 96 (21.4) 8.8 / 9.3, 120 (26.8) 13.9 / 9.5
// The lines were drawn when the paired kernel took 0.5 to 1.5 us more behind another launch than it does in this table.  Fused
// appends by which it would now win below them (by up to 17 %) stay here all the same: they keep this kernel's weights (every
// exponential from the special-function unit, the reference a maximum over 32 keys of each half, where the paired kernel's may be
// that of a tile of 21; peaked rows, off exact sums: T = 36, 57 keys, 128 channels 1.67e-3 / 1.97e-3, T = 64, 105 keys, 64
// channels 1.84e-3 / 1.96e-3, at 134 and more the same), and fused and separate appends of one copy choose alike.
// With the density 20 and 7 units (times with the append and the zeroed result): T = 25: 18.2 / 18.7
// (1 024 items), 27.8 / 29.3 (1 920, 25.9 units); T = 36: 10.4 / 12.4 (240), 15.0 / 13.1 (300); T = 64: 12.3 / 15.1 (240), 18.2 / 16.7 (300); T = 81:
// 12.6 / 16.2 (148, 18 units), 18.0 / 16.9 (180); 128 channels: T = 25: 18.2 / 20.1 (512, 6.9 units), 23.6 / 25.3 (700), 49 / 49 (1 920); T = 36: 11.6 /
// 13.6 (148), 17.4 / 14.0 (180); T = 64: 12.8 / 15.9 (120, 6.5), 20.7 / 17.1 (180).  Up to 16 queries with no more keys
// than the warp-per-item kernel takes the alternative is the attention call plus the CUDA-core density pass, whose time grows
// with the queries: always this one (T = 4, 9, 16 at 3 840 items: 23.3 / 27.1, 26.7 / 49.8, 31.8 / 90.5; 128 channels, T = 9 and 16:
// 63.7 / 74.2 and 74.4 / 149), but for a single token up to 10 items per SM (1 024 items 10.0 / 11.4, 1 920 13.4 / 12.7) and, with 128
// channels, where an SM holds two of its CTAs, up to two items per SM for a single token (300 items 10.8 / 11.6, 400 11.3 / 11.2,
// 3 840 53.5 / 18.9) and five for four (700 items 15.9 / 16.3, 1 024 19.8 / 17.7, 3 840 58 / 37).  With more keys the alternative is the
// paired kernel's one launch (T = 16, 916 keys: 400 items 28.9 / 41.0, 3 840 items 225 / 240; 128 channels 340 / 344).
// Without the density the warp-per-item kernel keeps its scales (T = 9: 2.6 / 3.5).
bool mid_preferred(int32_t T, int32_t total_keys, int64_t items, int32_t D, int sm_count, bool density, bool copies)
{
    if (density && T <= kSmallMaxQueries) {
        if (!small_supported(T, total_keys) || (T > 1 && D == 64) || T > 4) return true;
        return items <= (int64_t)sm_count * (T > 1 ? 5 : D == 64 ? 10 : 2);
    }
    if (!density && small_supported(T, total_keys)) return false;
    const int64_t units = items * ((T + 15) / 16) * (((int64_t)total_keys + kChunk - 1) / kChunk);
    int line = D == 64 ? 19 : 6;
    if (density) line = D == 64 ? 20 : 7;
    else if (!copies && pair_one_tile_per_sm(items, T, sm_count)) line = D == 64 ? (T > 81 ? 7 : 19) : (T > 64 ? 0 : 6);
    const bool one_wave = D == 128 || T <= 32 || items * ((T + 63) / 64) <= 2 * (int64_t)sm_count;   // (of CTAs of 64 queries)
    return units <= (int64_t)sm_count * line && one_wave;
}

cudaError_t launch_attend_mid(const Strided& Q, const Strided& O, const LayerRegion& region, const RangeList& ranges, int32_t T,
                              int32_t rows, int32_t heads, int32_t D, float softmax_scale, int sm_count, cudaStream_t stream,
                              const CurrentScaleSource* cur, const Piece* piece, int32_t n_pieces, const PairDensity* density)
{
    MidExt ext;
    memset(&ext, 0, sizeof(ext));
    if (cur) {
        if (cur->V.row != cur->K.row || cur->V.head != cur->K.head || cur->V.token != cur->K.token) return cudaErrorNotSupported;
        if (n_pieces < 0 || n_pieces > LayerLayout::kMaxPieces) return cudaErrorInvalidValue;
        ext.K = (const __nv_bfloat16*)cur->K.ptr;
        ext.V = (const __nv_bfloat16*)cur->V.ptr;
        ext.row = cur->K.row;
        ext.head = cur->K.head;
        ext.tok = cur->K.token;
        ext.len = T;
        ext.n_pieces = n_pieces;
        for (int i = 0; i < n_pieces; ++i) ext.piece[i] = piece[i];
    }
    MidDen den;
    memset(&den, 0, sizeof(den));
    if (density) {
        if (cur || density->n_runs < 1 || density->n_runs > kMaxDenRuns) return cudaErrorInvalidValue;
        den.out = density->out;
        den.n_runs = density->n_runs;
        for (int i = 0; i < density->n_runs; ++i) den.weight[i] = density->weight[i];
        for (int i = 0; i < ranges.n; ++i) den.run_of_range[i] = density->run_of_range[i];
    }
    if (T < 1 || ranges.total + ext.len < 1) return cudaErrorInvalidValue;
    const int64_t items = (int64_t)rows * heads;
    const float scale_log2 = softmax_scale * 1.4426950408889634f;
    const bool overlap = cur || density || overlaps_append(items, T, D, sm_count);   // (a density launch follows the kernel that zeroes its result)
#define AMSKV_MID_LAUNCH(DD, NN, DEN) return launch<DD, NN, DEN>(overlap, Q, O, region, ranges, T, heads, items, scale_log2, ext, den, stream)
    if (D == 128) {
        if (density) AMSKV_MID_LAUNCH(128, 4, true);
        AMSKV_MID_LAUNCH(128, 4, false);
    }
    // Densities of one query block: a CTA of four warps has two idle, which matters once an SM's share of the items is more than the
    // four such CTAs it holds (T = 4, 9, 16: 1 920 items 17.7 / 20.3 / 22.4 us with four warps, 14.6 / 17.0 / 18.8 with two; 7 680
    // items 54 / 60 / 68 and 40 / 45 / 51); below, twice the threads fetch the keys sooner (256 items 7.9 / 8.1 / 8.4 and 8.2 / 8.4 /
    // 8.9).
    if (density && T <= 16 && items > 4ll * sm_count) AMSKV_MID_LAUNCH(64, 2, true);
    // Four query blocks per CTA; two where there are no more, or where that still gives no SM a second CTA (T = 25, 512 items:
    // 6.3 us with 4 warps, 8.6 with 8; T = 64, 60 items: 5.1 and 5.8; T = 64, 256 items: 9.3 and 8.9).
    if (T <= 32 || items * ((T + 31) / 32) <= sm_count) {
        if (density) AMSKV_MID_LAUNCH(64, 4, true);
        AMSKV_MID_LAUNCH(64, 4, false);
    }
    if (density) AMSKV_MID_LAUNCH(64, 8, true);
    AMSKV_MID_LAUNCH(64, 8, false);
#undef AMSKV_MID_LAUNCH
}

}  // namespace amskv
