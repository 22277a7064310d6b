// Bit-stream kernels: C^(i) and sum_i D^(i) for every feature count and code width that the Int4 kernels for
// multiples of 8 do not take -- code widths other than 4 bits (the method "at lower and higher precision", paper
// Section 4 / Figure 3), and any E, k or row stride (k = E/64 is a multiple of 8 for few widths E).
//
// A token's codes are L*B bits long (L = E - k slots of B bits), so rows start at any bit of the code stream and
// the 8 adjacent slots of a group lie across its words.  All four kernels work on a group of 8 slots per thread, as
// the Int4 kernels do; an unaligned field costs one funnel shift out of shared memory or of a neighbour's register:
//   quantize_stream       rows that bulk copies can fetch: a ring of stages, warps that pack the codes of their own
//                         groups and write the words of the stream that start there, an edge warp for the words in
//                         which one row ends and the next begins; no barrier between warps; with a push mode
//   quantize_stream_tile  any other rows: a block quantises 8 rows into bit strings in shared memory, then writes the
//                         tile's bytes (8*L*B bits are a whole number of bytes) as words funnelled out of the strings
//   dequant_stream_rows   up to four devices, and five to eight where it is ahead: the row kernel, code rows by bulk copies into
//                         a ring, one block or two to a run of rows
//   dequant_stream        any others: a block's panel of code words comes in by 16-byte copies from the aligned place at or
//                         below each row's first bit
// Which calls they serve is decided in tpq_api.cu, by the rules at the end of this file.
// Arithmetic as everywhere: u = fl(x * inv_s), clamp, round to nearest even; acc = fma(code, s, acc) over the
// devices in ascending order.
#include <cuda_bf16.h>

#include "tpq_internal.h"

#include <type_traits>

namespace {

__device__ __forceinline__ uint32_t lop3_and_or(uint32_t x, uint32_t mask, uint32_t magic)
{
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(x), "r"(mask), "r"(magic));
    return d;
}

// ----------------------------------------------------------------------------------------------
// Quantise + pack
// ----------------------------------------------------------------------------------------------
constexpr int QS_MAX_BATCH = 16;  // shards of one launch
constexpr int QS_ROWS = 8;        // rows of a tile: 8*L*B bits are whole bytes for every L and B
constexpr int QS_THREADS = 320;   // most threads of a block; four blocks share an SM, so that one's barriers hide
                                  // behind the others' loads

struct QSParams {
    const uint16_t *y[QS_MAX_BATCH];
    uint8_t *payload[QS_MAX_BATCH];
    int64_t T, stride, lp_bytes, n_tiles;
    int E, k, L, n_holes;
    int row_words;       // words of a row's bit string in shared memory (even)
    const float *inv_s;  // [n][E], first shard of the batch
    const uint32_t *grp;
    const int32_t *hp_idx, *hole, *filler;
};

__host__ __device__ inline int qs_row_words(int L, int B) { return ((((L + 7) / 8) * B + 3) / 4 + 2) & ~1; }
inline size_t qt_smem_bytes(int L, int B) { return (size_t)QS_ROWS * qs_row_words(L, B) * 4; }

// the code of one value in the low bits (two's complement; bits above B are garbage)
template <int B>
__device__ __forceinline__ uint32_t qs_code(float x, float inv)
{
    constexpr float lo = -(float)(1 << (B - 1)), hi = (float)((1 << (B - 1)) - 1);
    const float u = fminf(fmaxf(__fmul_rn(x, inv), lo), hi);
    return __float_as_uint(__fadd_rn(u, 12582912.0f));  // + 1.5 * 2^23: nearest even, the code in the low bits
}

// 8 values -> 8 codes of B bits, four in each of two halves (two's complement, packed from bit 0).  inv: the reciprocal
// steps in pairs (i, i + 4): the two halves run side by side in packed instructions.
//
// Per value u = fl(x * inv), clamped, r = fl(u + 1.5 * 2^23): nearest even, an integer code on top of the magic number.
// From 6 bits on both clamps are minima and maxima and the shifted patterns are summed as integers.  Up to 5 bits the
// upper clamp and the packing move to the FMA pipe, which runs at twice the integer pipe's rate: t = sat(r / 2^B + c) with
// c such that t = 1 at the highest code (exact: every value in range is a multiple of 2^-B); 2^B t - 1 = code + 2^(B-1) is
// the code's digit with the sign bit flipped, and four digits are put together by FMAs as an integer below 2^20 on
// top of 2^23.  (18 integer-pipe instructions per 8 codes instead of 34; at 8 bits, where pairs of digits
// would be needed, it measured slower.)  NaN gives the lowest code (the lower clamp drops
// it), infinities saturate.
__device__ __forceinline__ float qs_sat_fma(float a, float b, float c)
{
    float d;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
template <int B>
__device__ __forceinline__ void qs_quant_halves(const uint4 v, const float2 (&inv)[4], uint32_t (&half)[2])
{
    constexpr float lo = -(float)(1 << (B - 1)), hi = (float)((1 << (B - 1)) - 1), scale = 1.0f / (float)(1 << B);
    constexpr float c = 1.0f - (12582912.0f + hi) * scale;
    constexpr uint32_t ones = 1u + (1u << B) + (1u << (2 * B)) + (1u << (3 * B));
    constexpr uint32_t sign = ones << (B - 1);
    constexpr float base = 8388608.0f - (float)ones;
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    float2 s = make_float2(base, base);
    uint32_t n[2] = {0u, 0u};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t a = w[i >> 1], b = w[2 + (i >> 1)];
        const float2 x = (i & 1) ? make_float2(__uint_as_float(a & 0xFFFF0000u), __uint_as_float(b & 0xFFFF0000u))
                                 : make_float2(__uint_as_float(a << 16), __uint_as_float(b << 16));
        float2 u = __fmul2_rn(x, inv[i]);
        u.x = fmaxf(u.x, lo);
        u.y = fmaxf(u.y, lo);
        if constexpr (B > 5) {
            u.x = fminf(u.x, hi);
            u.y = fminf(u.y, hi);
        }
        const float2 r = __fadd2_rn(u, make_float2(12582912.0f, 12582912.0f));
        if constexpr (B <= 5) {
            constexpr float unit = (float)(1 << B);
            const float at = unit * (float)(1 << (i * B));  // (the digit's place, times 2^B)
            s = __ffma2_rn(make_float2(qs_sat_fma(r.x, scale, c), qs_sat_fma(r.y, scale, c)), make_float2(at, at), s);
        } else {
            n[0] += __float_as_uint(r.x) << (i * B);
            n[1] += __float_as_uint(r.y) << (i * B);
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
        half[h] = B <= 5 ? __float_as_uint(h ? s.y : s.x) ^ (0x4B000000u | sign)  // the exponent goes, the sign bits flip
                         : (n[h] - 0x4B400000u * ones + sign) ^ sign;            // likewise, with the patterns' constant part
}

// A group's 8 codes in registers: one word of 8B bits up to 4 bits, else two words of 4B bits.
__host__ __device__ constexpr int qs_group_words(int B) { return B <= 4 ? 1 : 2; }
template <int B>
__device__ __forceinline__ void qs_quant8(const uint4 v, const float2 (&inv)[4], uint32_t (&w)[qs_group_words(B)])
{
    uint32_t half[2];
    qs_quant_halves<B>(v, inv, half);
    if constexpr (B == 4) {
        w[0] = __byte_perm(half[0], half[1], 0x5410);
    } else if constexpr (B < 4) {
        w[0] = half[0] | half[1] << (4 * B);
    } else {
        w[0] = half[0];
        w[1] = half[1];
    }
}
// code n of a group: which word, and its field there
template <int B>
__device__ __forceinline__ uint32_t qs_field_shift(int n) { return (uint32_t)((B <= 4 ? n : n & 3) * B); }
template <int B>
__device__ __forceinline__ bool qs_field_in(int n, int word) { return B <= 4 || (n >> 2) == word; }

// B bytes of codes -> shared memory, B-byte aligned
template <int B>
__device__ __forceinline__ void qs_store_group(uint8_t *dst, const uint32_t (&w)[qs_group_words(B)])
{
    if constexpr (B == 8) {
        *reinterpret_cast<uint2 *>(dst) = make_uint2(w[0], w[1]);
    } else if constexpr (B == 4) {
        *reinterpret_cast<uint32_t *>(dst) = w[0];
    } else {
        uint64_t bits = w[0];
        if constexpr (B > 4) bits |= (uint64_t)w[1] << (4 * B);
        if constexpr (B % 2 == 0) {
#pragma unroll
            for (int j = 0; j < B / 2; ++j) reinterpret_cast<uint16_t *>(dst)[j] = (uint16_t)(bits >> (16 * j));
        } else {
#pragma unroll
            for (int j = 0; j < B; ++j) dst[j] = (uint8_t)(bits >> (8 * j));
        }
    }
}

// A tile's bit strings (rows of LB bits, RW words apart) -> bytes from b0 on of a payload's code section.  Row r's
// words are those that start in it: from its bit o on, all funnelled by the same shift; the last one takes its upper
// bits from the next row (rows are at least 32 bits long).  A word shared with a neighbouring tile is written by
// bytes; the last tile writes the section's zero padding.
__device__ __forceinline__ void qs_write_tile(uint8_t *pl, const uint32_t *strings, int RW, int LB, int64_t b0, int rows, bool last,
                                              int64_t lp_bytes, int tid, int NT)
{
    const int lead = (int)(b0 & 3);  // bytes of the first word that belong to the tile before
    uint32_t *out = reinterpret_cast<uint32_t *>(pl) + ((b0 + 3) >> 2);
    if (lead && tid < 4 - lead) pl[b0 + tid] = (uint8_t)(strings[0] >> (8 * tid));
    int o = (32 - 8 * lead) & 31;
    for (int r = 0; r < rows; ++r) {
        const uint32_t *const s = strings + r * RW;
        const int n = (LB - o + 31) >> 5;  // words that start in the row
        for (int j = tid; j < n; j += NT) {
            const int at = o + 32 * j, left = LB - at;
            uint32_t v = __funnelshift_r(s[at >> 5], s[(at >> 5) + 1], at & 31);
            if (left < 32) {
                v &= (1u << left) - 1u;
                if (r + 1 < rows) {
                    v |= s[RW] << left;
                } else if (!last) {  // the tile's last word is the next tile's first one
                    for (int c = 0; c < left >> 3; ++c) reinterpret_cast<uint8_t *>(out + j)[c] = (uint8_t)(v >> (8 * c));
                    continue;
                }
            }
            out[j] = v;
        }
        out += n;
        o += 32 * n - LB;
    }
    if (last)
        for (uint32_t *w = out + tid; w < reinterpret_cast<uint32_t *>(pl + lp_bytes); w += NT) *w = 0u;
}

// Any E and row stride (and rows too long for the ring of the pipelined kernel below).
// One tile of QS_ROWS rows of one shard per block (grid = (tiles, shards)); a row's bit string is written to shared
// memory group by group, the fillers' codes are put into the holes, and the strings leave as words of the stream.
// VEC: rows are 16-byte aligned and whole groups long (E and stride multiples of 8).
template <int B, bool VEC>
__global__ void __launch_bounds__(QS_THREADS, VEC ? 4 : 2) quantize_stream_tile(const QSParams p)
{
    extern __shared__ __align__(16) uint32_t qs_smem[];  // QS_ROWS bit strings
    const int tid = threadIdx.x, NT = blockDim.x;
    const int E = p.E, k = p.k, L = p.L, G = (L + 7) >> 3, RW = p.row_words, n_holes = p.n_holes;
    const int LB = L * B;  // bits of a row
    const int64_t tile = blockIdx.x, t0 = tile * QS_ROWS;
    const int rows = (int)(p.T - t0 < QS_ROWS ? p.T - t0 : QS_ROWS);
    const uint16_t *const y = p.y[blockIdx.y] + t0 * p.stride;
    uint8_t *const pl = p.payload[blockIdx.y];
    const float *const inv_s = p.inv_s + (size_t)blockIdx.y * E;
    tpq_grid_dep_launch();

    // this thread's first item of each kind: a hole's filler value, a selected feature's value
    const int f_r = n_holes ? tid / n_holes : QS_ROWS, f_h = n_holes ? tid - f_r * n_holes : 0;
    int f_col = 0, f_slot = 0;
    float f_inv = 0.0f;
    if (f_r < rows) {
        f_col = __ldg(p.filler + f_h);
        f_slot = __ldg(p.hole + f_h);
        f_inv = __ldg(inv_s + f_col);
    }
    const int s_r = k ? tid / k : QS_ROWS;
    const int s_col = s_r < rows ? __ldg(p.hp_idx + (tid - s_r * k)) : 0;

    tpq_grid_dep_wait();  // the input and the payload buffer may still be in use by the kernel ahead
    uint32_t f_x = 0;
    uint16_t s_x = 0;
    if (f_r < rows) f_x = y[f_r * p.stride + f_col];
    if (s_r < rows) s_x = y[s_r * p.stride + s_col];
    for (int g = tid; g < G; g += NT) {
        float2 inv[4];
        if (VEC) {
            const float4 a = __ldg(reinterpret_cast<const float4 *>(inv_s + 8 * g));
            const float4 b = __ldg(reinterpret_cast<const float4 *>(inv_s + 8 * g + 4));
            inv[0] = make_float2(a.x, b.x); inv[1] = make_float2(a.y, b.y);
            inv[2] = make_float2(a.z, b.z); inv[3] = make_float2(a.w, b.w);
        } else {
#pragma unroll
            for (int n = 0; n < 4; ++n)
                inv[n] = make_float2(8 * g + n < E ? __ldg(inv_s + 8 * g + n) : 0.0f, 8 * g + n + 4 < E ? __ldg(inv_s + 8 * g + n + 4) : 0.0f);
        }
        const uint32_t mask = __ldg(p.grp + g) & 0xFFu;
        const uint16_t *src = y + 8 * g;
        uint8_t *dst = reinterpret_cast<uint8_t *>(qs_smem) + g * B;
#pragma unroll
        for (int r0 = 0; r0 < QS_ROWS; r0 += 4) {
            if (r0 >= rows) break;
            uint4 v[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {  // all loads first; rows past the end re-read the last row
                if (VEC) {
                    v[r] = *reinterpret_cast<const uint4 *>(src);  // (not __ldg: the kernel ahead may have written it)
                } else {
                    uint32_t x[8];
#pragma unroll
                    for (int n = 0; n < 8; ++n) x[n] = 8 * g + n < E ? src[n] : 0u;
                    v[r] = make_uint4(x[0] | x[1] << 16, x[2] | x[3] << 16, x[4] | x[5] << 16, x[6] | x[7] << 16);
                }
                if (r0 + r + 1 < rows) src += p.stride;
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                uint32_t w[qs_group_words(B)];
                qs_quant8<B>(v[r], inv, w);
                if (mask) {  // the holes' codes come later
#pragma unroll
                    for (int n = 0; n < 8; ++n)
                        if (mask & (1u << n)) w[B <= 4 ? 0 : n >> 2] &= ~(((1u << B) - 1u) << qs_field_shift<B>(n));
                }
                qs_store_group<B>(dst + (r0 + r) * RW * 4, w);
            }
        }
    }
    __syncthreads();
    // fillers' codes into the holes (two holes may share a word), selected features to the BF16 block
    auto fill = [&](int r, int slot, uint32_t x, float inv) {
        const uint32_t q = qs_code<B>(__uint_as_float(x << 16), inv) & ((1u << B) - 1u);
        const uint32_t bit = (uint32_t)slot * B, sh = bit & 31;
        uint32_t *const w = qs_smem + r * RW + (bit >> 5);
        atomicOr(w, q << sh);
        if (32 % B != 0 && sh + B > 32) atomicOr(w + 1, q >> (32 - sh));
    };
    if (f_r < rows) fill(f_r, f_slot, f_x, f_inv);
    for (int i = tid + NT; i < rows * n_holes; i += NT) {
        const int r = i / n_holes, h = i - r * n_holes, f = __ldg(p.filler + h);
        fill(r, __ldg(p.hole + h), y[r * p.stride + f], __ldg(inv_s + f));
    }
    uint16_t *const hp_out = reinterpret_cast<uint16_t *>(pl + p.lp_bytes) + t0 * k;
    if (s_r < rows) hp_out[tid] = s_x;
    for (int i = tid + NT; i < rows * k; i += NT) {
        const int r = i / k;
        hp_out[i] = y[r * p.stride + __ldg(p.hp_idx + (i - r * k))];
    }
    __syncthreads();
    qs_write_tile(pl, qs_smem, RW, LB, tile * (int64_t)LB, rows, tile == p.n_tiles - 1, p.lp_bytes, tid, NT);
}

template <int B>
cudaError_t launch_quantize_tile(const QSParams &p, bool vec, int threads, dim3 grid, cudaStream_t st)
{
    const size_t smem = qt_smem_bytes(p.L, B);
    auto kern = vec ? quantize_stream_tile<B, true> : quantize_stream_tile<B, false>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return tpq_launch_pdl(kern, grid, dim3(threads), smem, st, p);
}

// The pipelined kernel for rows that bulk copies can fetch (E and stride multiples of 8) and whose ring fits.
// As the Int4 kernel for multiples of 8 (quantize.cu): one persistent block per SM on a run of adjacent rows, a
// producer warp that streams stages of QS_STAGE rows into a ring, consumer lanes that own a group of 8 features with
// its steps in registers, holes patched through warp shuffles.  There is no barrier between the warps:
//   a consumer warp packs its 32 groups' codes of a row into a bit string of its own in shared memory and writes the
//   words of the stream that START in its groups; it needs up to 31 bits more for the last one, so its last one or two
//   groups (qs_ahead) are the next warp's first ones, packed by both;
//   the edge warp writes the words in which one row ends and the next begins (one code per lane: 16 of a row's last
//   and 16 of its first, or-ed together), for every row of the block and the row ahead of it.
// A block may therefore start at any row.  Measured at 4 x 2048 x 5120, 51 selected, back to back: 23.1 us against 16.3 us
// for its bytes at the copy rate (strings of whole tiles with a barrier of all consumers per 4 rows 43 us; one tile of 8 rows
// per block, four blocks per SM, 29.5 us; the shape-generic kernel 114 us); 3 bits 24.5 us, 6 bits 26.9 us, 8 x 1000 x 4608 at
// 8 bits 23.8 us.  Nearest limit: instruction issue.  A warp executes 103 instructions per 32 groups and row at 4 bits, 113 at 3,
// 126 at 8, which take 71 to 74 % of the issue slots of the launch, with DRAM at a third.
constexpr int QS_STAGE = 4;             // rows of a stage
constexpr int QS_MAX_THREADS = 768;     // 80 registers a thread
constexpr int QS_MAX_GPT = 2;           // groups of a consumer lane
constexpr int QS_MAX_STAGES = 6;
constexpr int QS_PREFETCH_ROWS = 8;     // rows whose bytes a block asks L2 for ahead of the dependency wait

__host__ __device__ constexpr int qs_ahead(int B) { return B < 4 ? 2 : 1; }  // groups whose bits cover 31
// words of a warp's bit string of one row (even; a funnel may look one word past the last group)
__host__ __device__ constexpr int qs_warp_words(int B) { return 8 * B + 2; }

struct QPipeParams {
    QSParams q;
    int bps;                 // blocks per shard
    int nstage;
    int64_t rows_per_block;
    int *status;
    // push mode (one shard, n_dst copies of its payload: q.payload[0 .. n_dst))
    int n_dst;
    uint32_t epoch;
    uint32_t *arrived[QS_MAX_BATCH];
    unsigned int *done;
};

// consumer warps for rows of G groups, gpt per lane
inline int qs_warps(int G, int B, int gpt)
{
    const int own = (32 - qs_ahead(B)) * gpt;
    return (G + own - 1) / own;
}
inline size_t qs_pipe_bytes(int E, int B, int warps, int gpt, int nstage)
{
    return (size_t)nstage * QS_STAGE * E * 2 + (size_t)warps * gpt * QS_STAGE * qs_warp_words(B) * 4 + (size_t)nstage * 16 +
           256;  // (the failure flag; lanes with no word to write may look up to 64 words past their string's start)
}

template <int B, int GPT, bool PUSH>
__global__ void __launch_bounds__(QS_MAX_THREADS, 1) quantize_stream(const QPipeParams pp)
{
    constexpr int OWN = 32 - qs_ahead(B), WW = qs_warp_words(B);
    extern __shared__ __align__(128) uint8_t qs_pipe[];
    const QSParams &p = pp.q;
    // warp 0 is the producer, warp 1 the edge warp, then come the NT consumers: where several warps of a scheduler can
    // issue, the first goes first, and the few instructions of these two must not wait behind the consumers' many
    // (as last warps it measured 1 % longer)
    const int NT = blockDim.x - 64, tid = (int)threadIdx.x - 64;
    const int E = p.E, k = p.k, L = p.L, G = (L + 7) >> 3, nstage = pp.nstage;
    const int LB = L * B;  // bits of a row
    const int sb = blockIdx.x / pp.bps, bx = blockIdx.x - sb * pp.bps;
    const uint16_t *const y = p.y[sb];
    const float *const inv_s = p.inv_s + (size_t)sb * E;
    const uint32_t row_bytes = (uint32_t)E * 2u, stage_bytes = QS_STAGE * row_bytes;
    uint8_t *const ring = qs_pipe;
    uint32_t *const strings = reinterpret_cast<uint32_t *>(ring + (size_t)nstage * stage_bytes);
    uint64_t *const full = reinterpret_cast<uint64_t *>(strings + (size_t)(NT / 32) * GPT * QS_STAGE * WW);
    uint64_t *const empty = full + nstage;
    // (push mode) a wait of this block ran out; in the slack behind the barriers, not a static variable: that would count
    // against the block's limit beside a ring that may fill it to the last byte
    int *const failed = reinterpret_cast<int *>(empty + nstage);
    if (PUSH && threadIdx.x == 0) *failed = 0;  // (ordered before any use by the barrier of the prologue)
    const int64_t t_begin = (int64_t)bx * pp.rows_per_block;
    const int rows_mine = (int)(p.T - t_begin < pp.rows_per_block ? p.T - t_begin : pp.rows_per_block);
    const int lane = threadIdx.x & 31;

    tpq_grid_dep_launch();
    if (threadIdx.x < 32) {
        // ---------------- producer warp
        if (lane == 0) {
            for (int s = 0; s < nstage; ++s) {
                mbar_init(smem_u32(&full[s]), 1);
                mbar_init(smem_u32(&empty[s]), NT / 32 + 1);
            }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        __syncwarp();
        asm volatile("bar.arrive 1, %0;" ::"r"(blockDim.x) : "memory");  // the barriers exist
        if (lane == 0 && p.stride == E) {  // a hint only: L2 is the point of coherence
            const int rows = rows_mine < QS_PREFETCH_ROWS ? rows_mine : QS_PREFETCH_ROWS;
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(y + t_begin * p.stride), "r"(rows * row_bytes) : "memory");
        }
        tpq_grid_dep_wait();  // the input and the payload buffer may still be in use by the kernel ahead
        int st = 0;
        uint32_t parity = 1;
        for (int it = 0, r0 = 0; r0 < rows_mine; ++it, r0 += QS_STAGE) {
            const int rows = rows_mine - r0 < QS_STAGE ? rows_mine - r0 : QS_STAGE;
            const uint32_t bar = smem_u32(&full[st]);
            int ok = 1;
            if (lane == 0) {
                if (it >= nstage && !mbar_wait(smem_u32(&empty[st]), parity)) {
                    atomicExch(pp.status, (int)TPQ_ERR_TIMEOUT);
                    ok = 0;
                } else {
                    mbar_expect_tx(bar, rows * row_bytes);
                }
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) break;
            const uint32_t dst = smem_u32(ring + (size_t)st * stage_bytes);
            const uint16_t *const src = y + (t_begin + r0) * p.stride;
            if (p.stride == E) {
                if (lane == 0) bulk_g2s(dst, src, rows * row_bytes, bar);
            } else if (lane < rows) {
                bulk_g2s(dst + lane * row_bytes, src + lane * p.stride, row_bytes, bar);
            }
            if (++st == nstage) {
                st = 0;
                parity ^= 1u;
            }
        }
        return;
    }

    int st = 0;
    uint32_t parity = 0;
    if (tid < 0) {
        // ---------------- edge warp: lanes 0..15 hold a row's last 16 codes, lanes 16..31 its first 16
        const int slot = lane < 16 ? L - 16 + lane : lane - 16;
        const bool on = slot >= 0 && slot < L;
        int f = 0;
        float inv = 0.0f;
        if (on) {  // the feature in the slot: itself, or the filler of a hole
            const uint32_t gd = __ldg(p.grp + (slot >> 3));
            f = slot;
            if (gd >> (slot & 7) & 1u) f = __ldg(p.filler + (int)(gd >> 8) + __popc(gd & ((1u << (slot & 7)) - 1u)));
            inv = __ldg(inv_s + f);
        }
        asm volatile("bar.sync 1, %0;" ::"r"(blockDim.x) : "memory");
        auto code = [&](uint32_t x) { return on ? qs_code<B>(__uint_as_float(x << 16), inv) & ((1u << B) - 1u) : 0u; };
        // the word in which a row ends after `in` bits (its codes `last` in lanes 0..15) and the next begins (`first`)
        auto edge = [&](int in, int64_t w, uint32_t last, uint32_t first) {
            const int at = lane < 16 ? in - (16 - lane) * B : in + (lane - 16) * B;  // the code's place in the word
            const uint32_t q = lane < 16 ? last : first;
            const uint32_t part = at >= 32 || at <= -B ? 0u : at >= 0 ? q << at : q >> -at;
            const uint32_t word = __reduce_or_sync(0xffffffffu, part);
            if (in && lane < (PUSH ? pp.n_dst : 1)) reinterpret_cast<uint32_t *>(p.payload[PUSH ? lane : sb])[w] = word;
        };
        uint32_t last = 0;
        bool dead = false;
        for (int r0 = 0; r0 < rows_mine; r0 += QS_STAGE) {
            const int rows = rows_mine - r0 < QS_STAGE ? rows_mine - r0 : QS_STAGE;
            if (!mbar_wait(smem_u32(&full[st]), parity)) {
                atomicExch(pp.status, (int)TPQ_ERR_TIMEOUT);
                if (PUSH) *failed = 1;
                dead = true;
            }
            if (__any_sync(0xffffffffu, dead)) {
                dead = true;
                break;
            }
            if (r0 == 0 && t_begin > 0) {
                tpq_grid_dep_wait();  // (the kernel ahead may have written the row: a load of this warp's own, so a wait of its own)
                last = code(y[(t_begin - 1) * p.stride + f]);
            }
            const uint16_t *const stage = reinterpret_cast<const uint16_t *>(ring + (size_t)st * stage_bytes);
            const int64_t bit0 = (t_begin + r0) * LB, w_stage = bit0 >> 5;
            const int in0 = (int)(bit0 & 31);
            uint32_t q[QS_STAGE];
#pragma unroll
            for (int r = 0; r < QS_STAGE; ++r) q[r] = stage[r * E + f];  // (rows past the stage's end: old bytes, unused)
#pragma unroll
            for (int r = 0; r < QS_STAGE; ++r) {
                if (r >= rows) break;
                const uint32_t first = code(q[r]);
                if (r0 + r > 0 || t_begin > 0) edge((in0 + r * LB) & 31, w_stage + ((in0 + r * LB) >> 5), last, first);
                last = first;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&empty[st]));
            if (++st == nstage) {
                st = 0;
                parity ^= 1u;
            }
        }
        if (t_begin + rows_mine == p.T && !dead) {  // the shard's last word and the section's zero padding
            edge((int)((p.T * (int64_t)LB) & 31), (p.T * (int64_t)LB) >> 5, last, 0u);
            const int64_t w0 = (p.T * (int64_t)LB + 31) >> 5;
            for (int d = 0; d < (PUSH ? pp.n_dst : 1); ++d)
                if (w0 + lane < p.lp_bytes / 4) reinterpret_cast<uint32_t *>(p.payload[PUSH ? d : sb])[w0 + lane] = 0u;
        }
        if (PUSH) asm volatile("bar.sync 2, %0;" ::"r"(NT + 32) : "memory");
        return;
    }

    // ---------------- consumers: constants (see quantize_tiled)
    const int warp = tid >> 5;  // consumer warp
    float2 inv[GPT][4];
    constexpr int NW = qs_group_words(B);
    uint32_t mask[GPT], w_off[GPT], f_sh[GPT][2], field[GPT][2][NW], keep[GPT][NW];
    int hb[GPT], src0[GPT];
    float w_inv[GPT];
    int most[GPT];  // most holes of a lane of the warp; above 8: the warp's holes outnumber its lanes (serial path)
    const int my_hp = tid < k ? __ldg(p.hp_idx + tid) : 0;
#pragma unroll
    for (int a = 0; a < GPT; ++a) {
        const int g = (warp + a * (NT / 32)) * OWN + lane;
        mask[a] = 0;
        hb[a] = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) inv[a][i] = make_float2(0.0f, 0.0f);
        if (g < G) {
            const float4 i0 = __ldg(reinterpret_cast<const float4 *>(inv_s + 8 * g));
            const float4 i1 = __ldg(reinterpret_cast<const float4 *>(inv_s + 8 * g + 4));
            const uint32_t gd = __ldg(p.grp + g);
            inv[a][0] = make_float2(i0.x, i1.x); inv[a][1] = make_float2(i0.y, i1.y);  // (pairs: see qs_quant_halves)
            inv[a][2] = make_float2(i0.z, i1.z); inv[a][3] = make_float2(i0.w, i1.w);
            mask[a] = gd & 0xFFu;
            if (8 * g + 8 > L) mask[a] &= (1u << (L - 8 * g)) - 1u;  // (features at or above L have no slot)
            hb[a] = (int)(gd >> 8);
        }
        const int nh = __popc(mask[a]);
        int incl = nh;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += o;
        }
        src0[a] = incl - nh;
        const int n_wh = __shfl_sync(0xffffffffu, incl, 31);  // holes of the warp
        const int hb_warp = __shfl_sync(0xffffffffu, hb[a], 0);
        most[a] = n_wh > 32 ? 9 : __reduce_max_sync(0xffffffffu, nh);
        w_off[a] = 0;
        w_inv[a] = 0.0f;
        if (lane < n_wh && n_wh <= 32) {
            const int f = __ldg(p.filler + hb_warp + lane);
            w_off[a] = (uint32_t)f * 2u;
            w_inv[a] = __ldg(inv_s + f);
        }
        uint32_t m = mask[a];
#pragma unroll
        for (int j = 0; j < NW; ++j) keep[a][j] = 0xFFFFFFFFu;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int n = m ? __ffs(m) - 1 : 0;
            f_sh[a][h] = qs_field_shift<B>(n);
#pragma unroll
            for (int j = 0; j < NW; ++j) {
                field[a][h][j] = m && qs_field_in<B>(n, j) ? ((1u << B) - 1u) << f_sh[a][h] : 0u;
                keep[a][j] &= ~field[a][h][j];
            }
            m &= m - 1;
        }
    }
    asm volatile("bar.sync 1, %0;" ::"r"(blockDim.x) : "memory");  // the producer has set up the barriers

    for (int r0 = 0; r0 < rows_mine; r0 += QS_STAGE) {
        const int rows = rows_mine - r0 < QS_STAGE ? rows_mine - r0 : QS_STAGE;
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&full[st]), parity))) {
            atomicExch(pp.status, (int)TPQ_ERR_TIMEOUT);
            if (PUSH) *failed = 1;
            break;
        }
        const uint8_t *const stage8 = ring + (size_t)st * stage_bytes;
        const int64_t bit0 = (t_begin + r0) * LB, w_stage = bit0 >> 5;  // the stage's first bit, the word it lies in ...
        const int in0 = (int)(bit0 & 31);                               // ... and its place there
#pragma unroll
        for (int a = 0; a < GPT; ++a) {
            const int wg = warp + a * (NT / 32);  // this warp's place among the row's
            const int g = wg * OWN + lane;
            const uint8_t *const src = stage8 + (g < G ? 16 * g : 0);
            uint32_t *const ws = strings + (size_t)(warp * GPT + a) * (QS_STAGE * WW);
            // the words that start in this warp's own groups and end in the row, relative to the stage's first word:
            // string bit `o` is the first word boundary, the same for every lane
            const int a0 = wg * (OWN * 8 * B);  // the string's first bit in the row
            const int a1 = a0 + OWN * 8 * B < LB - 31 ? a0 + OWN * 8 * B : LB - 31;
            auto put = [&](int r, int j, int o, uint32_t word) {
                if (a0 + o + 32 * (lane + 32 * j) < a1) {
                    const uint32_t w = ((uint32_t)(in0 + r * LB + a0 + 31) >> 5) + lane + 32 * j;
                    for (int d = 0; d < (PUSH ? pp.n_dst : 1); ++d)
                        (reinterpret_cast<uint32_t *>(p.payload[PUSH ? d : sb]) + w_stage)[w] = word;
                }
            };
            auto row_o = [&](int r) { return 31 - ((in0 + r * LB + a0 + 31) & 31); };
            // a row's codes: at 4 bits a group is a word, so its neighbour's comes by a shuffle; else to the bit string
            auto emit = [&](int r, const uint32_t (&wd)[NW], bool store) {
                if constexpr (B == 4) {
                    const uint32_t next = __shfl_down_sync(0xffffffffu, wd[0], 1);
                    const int o = row_o(r);
                    if (store) put(r, 0, o, __funnelshift_r(wd[0], next, o));
                } else {
                    qs_store_group<B>(reinterpret_cast<uint8_t *>(ws + r * WW) + lane * B, wd);
                }
            };
            // QS_STAGE independent rows (a short stage's missing ones hold old bytes and are never written)
            // (DEEP: a warp that has a lane with more than two holes, see quantize_tiled: 4 x 2048 x 5120 of 51 selected 36.4 us a
            // launch on the serial path, 23.2 so; 8 x 1000 x 4608 at 8 bits 38.1 and 26.6.  What it works out of the mask is kept
            // from the compiler: moved out of the loop over the stages it cost every warp of two groups a lane its registers,
            // 8 x 2048 x 8192 at 8 bits 99.7 us without this path, 106.9 with it, 101 so)
            auto rows_fast = [&](auto deep_tag) {
                constexpr bool DEEP = decltype(deep_tag)::value;
                uint4 v[QS_STAGE];
                uint32_t fx[QS_STAGE], wd[QS_STAGE][NW];
#pragma unroll
                for (int r = 0; r < QS_STAGE; ++r) {
                    v[r] = *reinterpret_cast<const uint4 *>(src + r * row_bytes);
                    fx[r] = *reinterpret_cast<const uint16_t *>(stage8 + r * row_bytes + w_off[a]);
                }
#pragma unroll
                for (int r = 0; r < QS_STAGE; ++r) {
                    qs_quant8<B>(v[r], inv[a], wd[r]);
                    if (DEEP || most[a]) {  // uniform over the warp
                        const uint32_t qv = qs_code<B>(__uint_as_float(fx[r] << 16), w_inv[a]) & ((1u << B) - 1u);
                        const uint32_t c0 = __shfl_sync(0xffffffffu, qv, src0[a]) << f_sh[a][0];
#pragma unroll
                        for (int j = 0; j < NW; ++j) wd[r][j] = (wd[r][j] & keep[a][j]) | (c0 & field[a][0][j]);
                        if (DEEP || most[a] > 1) {
                            const uint32_t c1 = __shfl_sync(0xffffffffu, qv, src0[a] + 1) << f_sh[a][1];
#pragma unroll
                            for (int j = 0; j < NW; ++j) wd[r][j] |= c1 & field[a][1][j];
                        }
                        if (DEEP) fx[r] = qv;
                    }
                    if (!DEEP) emit(r, wd[r], r < rows);
                }
                if constexpr (DEEP) {  // the third and further holes
                    uint32_t m = mask[a];
                    int s0 = src0[a];
                    asm volatile("" : "+r"(m), "+r"(s0));
                    m &= m - 1;
                    m &= m - 1;
                    for (int h = 2; h < most[a]; ++h, m &= m - 1) {
                        const int n = m ? __ffs(m) - 1 : 0;
                        const uint32_t sh = qs_field_shift<B>(n);
#pragma unroll
                        for (int r = 0; r < QS_STAGE; ++r) {
                            const uint32_t c = __shfl_sync(0xffffffffu, fx[r], s0 + h);
#pragma unroll
                            for (int j = 0; j < NW; ++j) {
                                const uint32_t fm = m && qs_field_in<B>(n, j) ? ((1u << B) - 1u) << sh : 0u;
                                wd[r][j] = (wd[r][j] & ~fm) | (c << sh & fm);
                            }
                        }
                    }
#pragma unroll
                    for (int r = 0; r < QS_STAGE; ++r) emit(r, wd[r], r < rows);
                }
            };
            if (most[a] <= 2) {
                rows_fast(std::false_type());
            } else if (most[a] <= 8) {
                rows_fast(std::true_type());
            } else {
                for (int r = 0; r < rows; ++r) {  // a warp on the serial path: every hole patched by its owner
                    uint32_t wd[NW];
                    qs_quant8<B>(*reinterpret_cast<const uint4 *>(src + r * row_bytes), inv[a], wd);
                    uint32_t m = mask[a];
                    for (int h = 0; m; ++h) {
                        const int n = __ffs(m) - 1;
                        m &= m - 1;
                        const int f = __ldg(p.filler + hb[a] + h);
                        const uint32_t x = *reinterpret_cast<const uint16_t *>(stage8 + r * row_bytes + 2 * f);
                        const uint32_t c = qs_code<B>(__uint_as_float(x << 16), __ldg(inv_s + f)) & ((1u << B) - 1u);
                        const uint32_t sh = qs_field_shift<B>(n);
#pragma unroll
                        for (int j = 0; j < NW; ++j) {
                            const uint32_t fm = qs_field_in<B>(n, j) ? ((1u << B) - 1u) << sh : 0u;
                            wd[j] = (wd[j] & ~fm) | (c << sh & fm);
                        }
                    }
                    __syncwarp();
                    emit(r, wd, true);
                }
            }
            if (B != 4) {
                __syncwarp();
#pragma unroll
                for (int r = 0; r < QS_STAGE; ++r) {
                    if (r >= rows) break;
                    const int o = row_o(r);
                    const uint32_t *const s = ws + r * WW + lane;
#pragma unroll
                    for (int j = 0; j < (OWN * 8 * B + 1023) / 1024; ++j)
                        put(r, j, o, __funnelshift_r(s[32 * j], s[32 * j + 1], o));
                }
                __syncwarp();
            }
        }
        for (int h = tid; h < k; h += NT) {
            const uint16_t *const x = reinterpret_cast<const uint16_t *>(stage8) + (h == tid ? my_hp : __ldg(p.hp_idx + h));
            const int64_t at = (t_begin + r0) * k + h;
            for (int d = 0; d < (PUSH ? pp.n_dst : 1); ++d) {
                uint16_t *const o = reinterpret_cast<uint16_t *>(p.payload[PUSH ? d : sb] + p.lp_bytes) + at;
                for (int r = 0; r < rows; ++r) o[r * k] = x[r * E];
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&empty[st]));
        if (++st == nstage) {
            st = 0;
            parity ^= 1u;
        }
    }
    if constexpr (PUSH) {
        // publication, as quantize_tiled: the block that counts last has observed every block's stores
        asm volatile("bar.sync 2, %0;" ::"r"(NT + 32) : "memory");
        if (tid == 0) {
            __threadfence();
            const unsigned int prev = atomicAdd(pp.done, *failed ? 0x10001u : 1u);
            if ((prev & 0xFFFFu) == gridDim.x - 1) {
                *pp.done = 0u;
                if ((prev >> 16) == 0 && !*failed) {
                    __threadfence_system();
                    for (int d = 0; d < pp.n_dst; ++d)
                        asm volatile("st.relaxed.sys.global.u32 [%0], %1;" ::"l"(pp.arrived[d]), "r"(pp.epoch) : "memory");
                }
            }
        }
    }
}

// groups per lane and ring depth of the pipelined kernel; false: the shape is the tile kernel's
bool qs_pipe_plan(const tpq_ctx *c, int64_t stride, int *gpt_out, int *warps_out, int *nstage_out)
{
    const int E = c->E, G = (E - c->k + 7) / 8;
    if (E % 8 || stride % 8) return false;
    for (int gpt = 1; gpt <= QS_MAX_GPT; ++gpt) {
        const int warps = qs_warps(G, c->bits, gpt);
        if (warps * 32 + 64 > QS_MAX_THREADS) continue;
        for (int n = QS_MAX_STAGES; n > 1; --n)
            if (qs_pipe_bytes(E, c->bits, warps, gpt, n) <= (size_t)c->smem_optin) {
                *gpt_out = gpt; *warps_out = warps; *nstage_out = n;
                return true;
            }
    }
    return false;
}

template <int B>
cudaError_t launch_quantize_pipe(const QPipeParams &pp, bool push, int gpt, int threads, unsigned grid, size_t smem, cudaStream_t st)
{
    auto kern = gpt == 1 ? (push ? quantize_stream<B, 1, true> : quantize_stream<B, 1, false>)
                         : (push ? quantize_stream<B, 2, true> : quantize_stream<B, 2, false>);
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return tpq_launch_pdl(kern, dim3(grid), dim3(threads), smem, st, pp);
}

// ----------------------------------------------------------------------------------------------
// Dequantise + reduce
//
// The layout of the copy-ring panel kernel (dequant.cu): a block owns a panel of CG groups and walks chunks of RC
// rows; the panel's steps of all devices sit in shared memory in slot order; the code words of a step (NB devices
// x RC rows) come by 16-byte asynchronous copies into a ring, one block barrier per step; a hole's lane holds its
// filler feature's sum, which an item thread moves to its own column after the chunk's stores.  What differs is
// the alignment: a segment starts at any bit, so the copies start at the 16-byte boundary at or below it and a
// thread funnels its 8*B bits out of two (three) words; the shift is the same for all devices, so it is worked
// out once per chunk and row.  Blocks are half the size, two to an SM, so that one's barrier hides behind the other's work.
// 5 x 1000 x 4608 at 8 bits 12.0 us back to back (5.0 us for its bytes at the copy rate), 8 devices 15.4 (one block of 512 threads
// per SM 22.1).  With 8 devices 61 instructions per warp of 32 groups and device take 52 % of the issue slots: 14 warps an SM (109
// registers a thread) leave one eligible a cycle between the chunk's barriers.
// ----------------------------------------------------------------------------------------------
constexpr int DS_THREADS = 256;  // two blocks share an SM, so that one's barrier hides behind the other's work
constexpr int DS_CG = 64;        // groups of a panel
constexpr int DS_R = 4;       // rows per thread
constexpr int DS_STAGES = 4;  // ring depth (steps)

__host__ __device__ constexpr int ds_nb(int B) { return B <= 4 ? 4 : 2; }  // devices per step

struct DSParams {
    const uint8_t *pl[TPQ_MAX_SHARDS];
    int N, E, k, L;
    int64_t T, lp_bytes, out_stride, n_chunks;
    const float *s_slot;  // [N][E] steps in slot order
    const uint32_t *grp;
    const int32_t *lp_idx, *hp_idx, *filler;
    int n_holes, panels, gy;
    bool vec;  // 8 adjacent outputs are 16-byte aligned (E and the output stride multiples of 8)
    void *out;
    const float *bias;  // [E] added after the sum, or NULL
    tpq_arrivals arr;   // arrival words to wait for before the first payload read (words == NULL: none)
};

__host__ __device__ constexpr int ds_seg_pieces(int B) { return DS_CG * B / 16 + 1; }
__host__ __device__ constexpr size_t ds_stage_bytes(int B)
{
    return (size_t)ds_nb(B) * (DS_THREADS / DS_CG * DS_R) * ds_seg_pieces(B) * 16;
}
__host__ __device__ constexpr size_t ds_smem_bytes(int B, int N)
{
    return (size_t)N * DS_CG * 32 + DS_STAGES * ds_stage_bytes(B) + 16;  // (a funnel may look one word past the ring)
}

// bit position, inside the float's mantissa, at which code n of a half is decoded
__host__ __device__ constexpr int ds_pos(int B, int n) { return (B <= 5 ? (n & 3) : B == 8 ? 0 : (n & 1)) * B; }

// 4 codes of a half (x: the half's bits from bit 0 on, more above), accumulated: (x & mask) | 0x4B000000 is the
// float 2^23 + (code + 2^(B-1)) 2^pos once the sign bits are flipped; subtracting 2^23 + 2^(B-1+pos) is exact and the
// steps are pre-divided by 2^pos, so the FMA rounds exactly like fma(code, s, acc).  A code must end below bit 23:
// up to 5 bits all four do, 6 and 7 bits take codes 2 and 3 from the half shifted down, and at 8 bits a byte permute
// puts every code at bit 0 in one instruction.
//
// DSConsts: masks, exponent pattern and bias pairs.  KEEP makes them opaque to the compiler, which then keeps them in
// registers instead of rebuilding them at every use (where the kernel has the registers for it).
template <int B>
struct DSConsts {
    uint32_t magic, mask[4];
    float2 bias[2];
    template <bool KEEP>
    __device__ __forceinline__ void init()
    {
        magic = 0x4B000000u;
#pragma unroll
        for (int n = 0; n < 4; ++n) mask[n] = ((1u << B) - 1u) << ds_pos(B, n);
#pragma unroll
        for (int h = 0; h < 2; ++h)
            bias[h] = make_float2(-(8388608.0f + (float)(1u << (B - 1 + ds_pos(B, 2 * h)))),
                                  -(8388608.0f + (float)(1u << (B - 1 + ds_pos(B, 2 * h + 1)))));
        if (KEEP) {
            asm volatile("" : "+r"(magic));
#pragma unroll
            for (int n = 0; n < (B == 8 ? 0 : B <= 5 ? 4 : 2); ++n) asm volatile("" : "+r"(mask[n]));
#pragma unroll
            for (int h = 0; h < (B <= 5 ? 2 : 1); ++h) asm volatile("" : "+f"(bias[h].x), "+f"(bias[h].y));
        }
    }
};
// FIRST: the accumulators start here (what fma(code, step, +0) gives, but for the sign of a zero where a step is 0: the lane
// of a selected feature, whose sum is never kept)
template <int B, bool FIRST = false>
__device__ __forceinline__ void ds_decode4(uint32_t x, const float2 s01, const float2 s23, float2 &a01, float2 &a23, const DSConsts<B> &c)
{
    constexpr uint32_t sign = (1u << (B - 1)) * (1u + (1u << B) + (1u << (2 * B)) + (1u << (3 * B)));
    x ^= sign;
    float2 f01, f23;
    if constexpr (B == 8) {
        f01 = make_float2(__uint_as_float(__byte_perm(x, c.magic, 0x7440)), __uint_as_float(__byte_perm(x, c.magic, 0x7441)));
        f23 = make_float2(__uint_as_float(__byte_perm(x, c.magic, 0x7442)), __uint_as_float(__byte_perm(x, c.magic, 0x7443)));
    } else {
        const uint32_t x2 = B <= 5 ? x : x >> (2 * B);
        constexpr int m2 = B <= 5 ? 2 : 0;
        f01 = make_float2(__uint_as_float(lop3_and_or(x, c.mask[0], c.magic)), __uint_as_float(lop3_and_or(x, c.mask[1], c.magic)));
        f23 = make_float2(__uint_as_float(lop3_and_or(x2, c.mask[m2], c.magic)), __uint_as_float(lop3_and_or(x2, c.mask[m2 + 1], c.magic)));
    }
    const float2 d01 = __fadd2_rn(f01, c.bias[0]), d23 = __fadd2_rn(f23, c.bias[B <= 5 ? 1 : 0]);
    a01 = FIRST ? __fmul2_rn(d01, s01) : __ffma2_rn(d01, s01, a01);
    a23 = FIRST ? __fmul2_rn(d23, s23) : __ffma2_rn(d23, s23, a23);
}

// the 8 codes that begin at bit sh of the first of a group's words (w1: the second one, w2: the third, read from 5 bits on)
template <int B, bool FIRST = false>
__device__ __forceinline__ void ds_decode8(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t sh, const float2 (&sc)[4], float2 (&acc)[4],
                                           const DSConsts<B> &c)
{
    const uint32_t lo = __funnelshift_r(w0, w1, sh);
    uint32_t hi;  // codes 4..7
    if constexpr (B <= 4) {
        hi = lo >> (4 * B);
    } else {
        const uint32_t up = __funnelshift_r(w1, w2, sh);
        hi = B == 8 ? up : __funnelshift_r(lo, up, 4 * B & 31);
    }
    ds_decode4<B, FIRST>(lo, sc[0], sc[1], acc[0], acc[1], c);
    ds_decode4<B, FIRST>(hi, sc[2], sc[3], acc[2], acc[3], c);
}

__device__ __forceinline__ void ds_cp16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

template <bool FP32OUT>
__device__ __forceinline__ void ds_store_one(void *out, int64_t off, float v)
{
    if (FP32OUT)
        static_cast<float *>(out)[off] = v;
    else
        static_cast<__nv_bfloat16 *>(out)[off] = __float2bfloat16_rn(v);
}

template <int B, bool FP32OUT>
__global__ void __launch_bounds__(DS_THREADS, 2) dequant_stream(const DSParams p)
{
    extern __shared__ __align__(128) uint8_t ds_smem[];
    constexpr int NB = ds_nb(B), CG = DS_CG;
    constexpr int RS = DS_THREADS / CG, RC = RS * DS_R;
    constexpr int SEGC = ds_seg_pieces(B), SEGW = SEGC * 4;
    constexpr int PIECES = NB * RC * SEGC;
    constexpr int NCP = (PIECES + DS_THREADS - 1) / DS_THREADS;
    constexpr uint32_t STAGE_BYTES = PIECES * 16;

    if (p.arr.words) {  // (first thing, with no load of its own in flight)
        tpq_block_wait_arrivals(p.arr);
        __syncthreads();
    }
    const int N = p.N, E = p.E, k = p.k, L = p.L;
    const uint32_t LB = (uint32_t)L * B;
    const int tid = threadIdx.x;
    float4 *const steps = reinterpret_cast<float4 *>(ds_smem);  // [N][2][CG]
    uint8_t *const ring = ds_smem + (size_t)N * CG * 32;
    const uint32_t ring_s = smem_u32(ring);
    const int panel = blockIdx.x % p.panels, by = blockIdx.x / p.panels;
    const int cg = tid & (CG - 1), rs = tid / CG;
    const int g = panel * CG + cg;
    const int lanes = L - 8 * g < 8 ? L - 8 * g : 8;  // slots of the thread's group (the last one may be short)
    const uint32_t panel_bit = (uint32_t)panel * (CG * 8 * B);

    // copy side: piece c = tid + j * DS_THREADS of a step is piece `within` of segment (device, row) and lands at
    // byte 16 c of the stage
    int cp_dev[NCP];
    uint32_t cp_bit[NCP], cp_in[NCP];  // first bit of the segment relative to the chunk, byte inside the segment
#pragma unroll
    for (int j = 0; j < NCP; ++j) {
        const int c = tid + j * DS_THREADS;
        const int seg = c / SEGC, within = c - seg * SEGC;
        const int i = seg / RC, row = seg - i * RC;
        cp_dev[j] = c < PIECES ? i : -1;
        cp_bit[j] = (uint32_t)row * LB + panel_bit;
        cp_in[j] = (uint32_t)within * 16u;
    }
    int64_t ich = by;
    int ib = 0;
    const int nbatch = (N + NB - 1) / NB;
    uint32_t idst = ring_s + (uint32_t)tid * 16u;
    auto issue = [&]() {
        if (ich < p.n_chunks) {
            const int64_t bit = ich * RC * (int64_t)LB;
            const int64_t base = (bit >> 3) & ~(int64_t)15;        // the chunk's 16-byte aligned start ...
            const uint32_t rem = (uint32_t)(bit - base * 8);       // ... and its first bit behind it
            const int64_t left = p.lp_bytes - base;
            const uint32_t lim = (uint32_t)(left < (int64_t)0x7FFFFFF0 ? left : (int64_t)0x7FFFFFF0);
            const int i0 = ib * NB;
#pragma unroll
            for (int j = 0; j < NCP; ++j) {
                // pieces past the end of the code section (a multiple of 16 bytes) and devices past N are skipped;
                // what they would have filled is never stored
                const uint32_t at = ((((rem + cp_bit[j]) >> 3) & ~15u) + cp_in[j]);
                if (cp_dev[j] >= 0 && i0 + cp_dev[j] < N && at + 16u <= lim)
                    ds_cp16(idst + (uint32_t)(j * DS_THREADS * 16), p.pl[i0 + cp_dev[j]] + base + at);
            }
            if (++ib == nbatch) {
                ib = 0;
                ich += p.gy;
            }
            idst += STAGE_BYTES;
            if (idst == ring_s + (uint32_t)tid * 16u + DS_STAGES * STAGE_BYTES) idst = ring_s + (uint32_t)tid * 16u;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");  // (possibly empty: keeps the count in step with the consumer)
    };
    for (int a = tid; a < N * CG; a += DS_THREADS) {
        const int i = a / CG, c = a & (CG - 1), c0 = 8 * (panel * CG + c);
        float s[8];
        const float *const src = p.s_slot + (size_t)i * E + c0;
        if (p.vec && c0 < L) {
            const float4 u = __ldg(reinterpret_cast<const float4 *>(src)), v = __ldg(reinterpret_cast<const float4 *>(src) + 1);
            s[0] = u.x; s[1] = u.y; s[2] = u.z; s[3] = u.w; s[4] = v.x; s[5] = v.y; s[6] = v.z; s[7] = v.w;
        } else {
#pragma unroll
            for (int n = 0; n < 8; ++n) s[n] = c0 + n < L ? __ldg(src + n) : 0.0f;
        }
#pragma unroll
        for (int n = 0; n < 8; ++n) s[n] *= 1.0f / (float)(1u << ds_pos(B, n));
        steps[(2 * i) * CG + c] = make_float4(s[0], s[1], s[2], s[3]);
        steps[(2 * i + 1) * CG + c] = make_float4(s[4], s[5], s[6], s[7]);
    }
    tpq_grid_dep_wait();  // the payloads and the output buffer may still be in use by the kernel ahead
    tpq_grid_dep_launch();
#pragma unroll
    for (int s = 0; s < DS_STAGES - 1; ++s) issue();
    const float4 *const my_steps = steps + cg;
    const uint32_t *const ring_w = reinterpret_cast<const uint32_t *>(ring);
    const uint32_t *sw = ring_w;

    // Items (one per row of the chunk and selected feature): the panel's holes, ranks [hs, he); the last panel also
    // takes the selected features at or above L, ranks [n_holes, k).
    const int n_holes = p.n_holes;
    const int hs = (int)(__ldg(p.grp + panel * CG) >> 8);
    const int he = (panel == p.panels - 1) ? k : (int)(__ldg(p.grp + (panel + 1) * CG) >> 8);
    const int n_it = he - hs;
    const int items = RC * n_it;
    const int my_r = (tid < items) ? tid / n_it : 0;
    const int my_h = (tid < items) ? hs + (tid - my_r * n_it) : 0;
    const int my_col = (tid < items) ? __ldg(p.hp_idx + my_h) : 0;
    const int my_fcol = (tid < items && my_h < n_holes) ? __ldg(p.filler + my_h) : -1;
    auto read_out = [&](int64_t at) -> float {  // the bits of an output element
        if (FP32OUT) return __ldcg(static_cast<const float *>(p.out) + at);
        return __uint_as_float((uint32_t)__ldcg(static_cast<const uint16_t *>(p.out) + at));
    };
    auto write_out = [&](int64_t at, float bits) {
        if (FP32OUT)
            static_cast<float *>(p.out)[at] = bits;
        else
            static_cast<uint16_t *>(p.out)[at] = (uint16_t)__float_as_uint(bits);
    };
    // an item's read of the hole's column is issued a step ahead of its stores (a store right behind the read of
    // the same address would hold up the memory pipe until the read is done)
    bool fl_on = false;
    float fl_f = 0.0f, fl_v = 0.0f;
    int64_t fl_row = 0;
    auto flush = [&]() {
        if (fl_on) {
            if (my_fcol >= 0) write_out(fl_row + my_fcol, fl_f);
            ds_store_one<FP32OUT>(p.out, fl_row + my_col, p.bias ? __fadd_rn(fl_v, p.bias[my_col]) : fl_v);
            fl_on = false;
        }
    };
    auto fixup = [&](int64_t tcp, bool on, float v) {
        if (on) {
            fl_row = (tcp + my_r) * p.out_stride;
            if (my_fcol >= 0) fl_f = read_out(fl_row + my_col);
            fl_v = v;
            fl_on = true;
        }
        for (int a = tid + DS_THREADS; a < items; a += DS_THREADS) {  // panels with more items than threads
            const int r = a / n_it, h = hs + (a - r * n_it);
            if (tcp + r >= p.T) break;
            const int64_t off = p.lp_bytes + ((tcp + r) * k + h) * 2, orow = (tcp + r) * p.out_stride;
            float u = 0.0f;
            for (int i = 0; i < N; ++i)
                u = __fadd_rn(u, __uint_as_float((uint32_t)__ldcs(reinterpret_cast<const uint16_t *>(p.pl[i] + off)) << 16));
            const int col = __ldg(p.hp_idx + h);
            if (h < n_holes) write_out(orow + __ldg(p.filler + h), read_out(orow + col));
            ds_store_one<FP32OUT>(p.out, orow + col, p.bias ? __fadd_rn(u, p.bias[col]) : u);
        }
    };
    bool pend = false, pend_on = false;
    float pend_v = 0.0f;
    int64_t pend_tc = 0;
    DSConsts<B> dc;
    dc.template init<false>();  // (in registers: 18.1 us instead of 17.8 at 16 x 500 x 4416)

    for (int64_t ch = by; ch < p.n_chunks; ch += p.gy) {
        const int64_t tc = ch * RC, t0 = tc + rs * DS_R;
        const bool it_on = tid < items && tc + my_r < p.T;
        const int64_t it_off = p.lp_bytes + ((tc + my_r) * k + my_h) * 2;
        float hv = 0.0f;
        uint16_t hvv[NB] = {};
        float2 acc[DS_R][4];
        int wofs[DS_R];       // this thread's first word of row r inside a device's part of a stage ...
        uint32_t wsh[DS_R];   // ... and the bit it starts at
        const uint32_t rem = (uint32_t)((ch * RC * (int64_t)LB) & 127);
#pragma unroll
        for (int r = 0; r < DS_R; ++r) {
            const int rowc = rs * DS_R + r;
            const uint32_t bit = ((rem + (uint32_t)rowc * LB + panel_bit) & 127u) + (uint32_t)cg * (8 * B);
            wofs[r] = rowc * SEGW + (int)(bit >> 5);
            wsh[r] = bit & 31u;
#pragma unroll
            for (int h = 0; h < 4; ++h) acc[r][h] = make_float2(0.0f, 0.0f);
        }
        const float4 *st4 = my_steps;
        for (int i0 = 0; i0 < N; i0 += NB, st4 += NB * 2 * CG) {
            asm volatile("cp.async.wait_group %0;" ::"n"(DS_STAGES - 2) : "memory");
            __syncthreads();  // the step has landed for everybody; the stage consumed last is free
            issue();
            flush();
            if (pend) {  // (first step of a chunk) the barrier above is also behind the previous chunk's row stores
                if (n_it > 0) fixup(pend_tc, pend_on, pend_v);
                pend = false;
            }
            if (it_on) {  // add the values loaded a step ago (ascending device order), then load this step's
                if (i0 > 0) {
#pragma unroll
                    for (int i = 0; i < NB; ++i) hv = __fadd_rn(hv, __uint_as_float((uint32_t)hvv[i] << 16));
                }
#pragma unroll
                for (int i = 0; i < NB; ++i)
                    if (i0 + i < N) hvv[i] = __ldcs(reinterpret_cast<const uint16_t *>(p.pl[i0 + i] + it_off));
            }
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                if (i0 + i >= N) break;
                const float4 a = st4[(2 * i) * CG], b = st4[(2 * i + 1) * CG];
                const float2 sc[4] = {make_float2(a.x, a.y), make_float2(a.z, a.w), make_float2(b.x, b.y), make_float2(b.z, b.w)};
#pragma unroll
                for (int r = 0; r < DS_R; ++r) {
                    const uint32_t *const s = sw + i * RC * SEGW + wofs[r];
                    ds_decode8<B>(s[0], s[1], B > 4 ? s[2] : 0u, wsh[r], sc, acc[r], dc);
                }
            }
            sw += STAGE_BYTES / 4;
            if (sw == ring_w + DS_STAGES * (STAGE_BYTES / 4)) sw = ring_w;
        }
        if (it_on) {  // the last step's values (a partial batch has fewer than NB of them)
            const int nl = N - (N - 1) / NB * NB;
#pragma unroll
            for (int i = 0; i < NB; ++i)
                if (i < nl) hv = __fadd_rn(hv, __uint_as_float((uint32_t)hvv[i] << 16));
        }
        if (p.bias && lanes > 0) {
            const uint32_t holes = __ldg(p.grp + g) & 0xFFu;
            float b[8];  // lane n belongs to feature 8g+n, or, at a hole, to the filler whose codes sit in the slot
#pragma unroll
            for (int n = 0; n < 8; ++n)
                b[n] = n < lanes ? p.bias[(holes & (1u << n)) ? __ldg(p.lp_idx + 8 * g + n) : 8 * g + n] : 0.0f;
#pragma unroll
            for (int r = 0; r < DS_R; ++r)
#pragma unroll
                for (int h = 0; h < 4; ++h) acc[r][h] = __fadd2_rn(acc[r][h], make_float2(b[2 * h], b[2 * h + 1]));
        }
#pragma unroll
        for (int r = 0; r < DS_R; ++r) {
            if (t0 + r >= p.T) break;
            const int64_t o = (t0 + r) * p.out_stride + 8 * (int64_t)g;
            if (p.vec && lanes >= 8) {
                if (FP32OUT) {
                    float4 *const dst = reinterpret_cast<float4 *>(static_cast<float *>(p.out) + o);
                    __stcs(dst, make_float4(acc[r][0].x, acc[r][0].y, acc[r][1].x, acc[r][1].y));
                    __stcs(dst + 1, make_float4(acc[r][2].x, acc[r][2].y, acc[r][3].x, acc[r][3].y));
                } else {
                    uint32_t w[4];
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const __nv_bfloat162 v = __floats2bfloat162_rn(acc[r][h].x, acc[r][h].y);
                        w[h] = *reinterpret_cast<const uint32_t *>(&v);
                    }
                    __stcs(reinterpret_cast<uint4 *>(static_cast<uint16_t *>(p.out) + o), make_uint4(w[0], w[1], w[2], w[3]));
                }
            } else {
#pragma unroll
                for (int n = 0; n < 8; ++n)
                    if (n < lanes) ds_store_one<FP32OUT>(p.out, o + n, (n & 1) ? acc[r][n >> 1].y : acc[r][n >> 1].x);
            }
        }
        pend = true;
        pend_on = it_on;
        pend_v = hv;
        pend_tc = tc;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    flush();
    if (pend) {
        __syncthreads();
        if (n_it > 0) fixup(pend_tc, pend_on, pend_v);
        flush();
    }
}

template <int B>
cudaError_t launch_dequant_stream(const DSParams &p, int fp32_out, cudaStream_t st)
{
    const size_t smem = ds_smem_bytes(B, p.N);
    auto kern = fp32_out ? dequant_stream<B, true> : dequant_stream<B, false>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return tpq_launch_pdl(kern, dim3((unsigned)(p.panels * p.gy)), dim3(DS_THREADS), smem, st, p);
}

// ----------------------------------------------------------------------------------------------
// Dequantise + reduce for up to eight devices: the row kernel (dequant.cu) at bit granularity.  (When it is taken: dw_stages.)
//
// One persistent block per SM on a run of adjacent rows, DW_ROWS at a time (fewer in the first stage, which lands sooner); for
// rows of six to eight devices whose steps one block has no registers for, two blocks to a run (SPLIT below).
// Warp 0 streams the devices' code rows and BF16 rows into a ring (two bulk copies per device and stage, between 16-byte
// boundaries).  A main thread owns a group of 8 features with the steps of all devices in registers (0 at selected
// features), funnels its bits out of two (three) words, stores the whole group and then overwrites the lanes of selected
// features with the sums the auxiliary warps left in shared memory (same thread, same address: ordered).  An auxiliary
// thread per rank h adds up the devices' BF16 values of selected feature h and decodes column L + h of the output where that
// is a filler feature.  No warp waits for another's global stores.
// Four devices: 48 (4 bits) and 49 (3 bits) instructions per warp of 32 groups and device take 61 to 63 % of the issue slots and the
// ALU pipe half of its cycles, with 1.7 to 1.8 eligible warps; the rest is the prologue and the drain.  Two blocks to a run, eight
// devices at 8 bits: 41 instructions, 40 % of the slots, 0.7 eligible warps: 13 warps an SM (128 registers a thread) that wait
// for loads.  Back to back, with the BF16 values loaded from memory a stage ahead, general loops in the auxiliary warps and a
// device count read at run time, against this form: 4 x 2048 x 5120, 51 selected 15.0 and 12.0 us, 3 bits 14.6 and 11.7, 8 bits
// 16.3 and 13.8; two devices 3 bits 11.1 and 8.3; three 12.8 and 10.3 (6.5, 5.8, 9.7, 4.5 and 5.1 us for the bytes; the Int4 row
// kernel 10.8).  Either half alone loses: the staged values behind general loops take 15.9 us, the compile-time device count
// without them 15.2.
// ----------------------------------------------------------------------------------------------
constexpr int DW_ROWS = 4, DW_AUX = 96, DW_MAX_K = 384;
// most groups of a row, by the devices whose steps a main thread keeps in registers
__host__ __device__ constexpr int dw_main(int nd) { return nd > 4 ? 320 : 640; }

struct DWParams {
    DSParams d;
    const float *s_k;      // [N][E] steps, 0 at selected features
    const int32_t *pos;    // [E]
    int nstage;
    int half_groups;       // (two blocks to a run of rows) groups of the first block
    uint32_t dev_bytes;    // a device's code words in a stage ...
    uint32_t hp_bytes;     // ... and its BF16 values
    int first;             // rows of a block's first stage
    int64_t rows_per_block;
    int *status;
};

__host__ __device__ inline uint32_t dw_dev_bytes(int L, int B) { return (uint32_t)(((DW_ROWS * L * B + 127 + 127) / 128 + 1) * 16); }
// (two blocks to a run of rows) a row's half in a stage
__host__ __device__ inline uint32_t dw_pitch(int half_groups, int B) { return (uint32_t)((half_groups * 8 * B + 127 + 127) / 128 * 16); }
__host__ __device__ inline uint32_t dw_hp_bytes(int k) { return k ? (uint32_t)(DW_ROWS * k * 2 + 14 + 15) & ~15u : 0u; }
inline size_t dw_smem_bytes(int nd, uint32_t dev_bytes, int k, int nstage)
{
    return (size_t)nstage * ((size_t)nd * (dev_bytes + dw_hp_bytes(k)) + (size_t)DW_ROWS * k * 4 + 24) + 16;
}

__device__ __forceinline__ uint32_t dw_lds32(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t dw_lds16(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void dw_sts32(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }

// ROWS rows of a stage, from its row r0 on, for one main thread.  stage: its address, rem: the bit of its first 16 bytes at which
// its first row begins, g_bit: the first bit of the thread's group in a row.
// ND devices, a number that the compiler knows: straight-line code, every device's words at the same place in its part.
// SPLIT: a row's half lies by itself, DW_ROWS of them `pitch` bytes apart.
template <bool SPLIT>
__device__ __forceinline__ uint32_t dw_row_bit(uint32_t rem, int r, uint32_t LB, uint32_t pitch)
{
    return SPLIT ? (uint32_t)r * pitch * 8u + ((rem + (uint32_t)r * LB) & 127u) : rem + (uint32_t)r * LB;
}

template <int B, int ND, bool SPLIT, int ROWS, bool FP32OUT, bool HAS_BIAS>
__device__ __forceinline__ void dw_rows(const uint8_t *stage, uint32_t dev_bytes, uint32_t rem, int r0, uint32_t LB, uint32_t pitch, uint32_t g_bit,
                                        const float2 (&sc)[ND][4], const float2 (&b)[4], const DSConsts<B> &dc, uint8_t *out,
                                        int64_t out_row_bytes, int lanes)
{
#pragma unroll
    for (int r = 0; r < ROWS; ++r, out += out_row_bytes) {
        const uint32_t bit = dw_row_bit<SPLIT>(rem, r0 + r, LB, pitch) + g_bit;
        const uint8_t *w = stage + (bit >> 5) * 4;
        float2 acc[4];
#pragma unroll
        for (int i = 0; i < ND; ++i, w += dev_bytes) {
            const uint32_t *const q = reinterpret_cast<const uint32_t *>(w);
            if (i == 0) ds_decode8<B, true>(q[0], q[1], B > 4 ? q[2] : 0u, bit & 31u, sc[i], acc, dc);
            else ds_decode8<B>(q[0], q[1], B > 4 ? q[2] : 0u, bit & 31u, sc[i], acc, dc);
        }
        if (HAS_BIAS) {  // (a selected feature's lane is overwritten later)
#pragma unroll
            for (int h = 0; h < 4; ++h) acc[h] = __fadd2_rn(acc[h], b[h]);
        }
        if (lanes >= 8) {
            if (FP32OUT) {
                __stcs(reinterpret_cast<float4 *>(out), make_float4(acc[0].x, acc[0].y, acc[1].x, acc[1].y));
                __stcs(reinterpret_cast<float4 *>(out) + 1, make_float4(acc[2].x, acc[2].y, acc[3].x, acc[3].y));
            } else {
                uint32_t x[4];
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const __nv_bfloat162 t = __floats2bfloat162_rn(acc[h].x, acc[h].y);
                    x[h] = *reinterpret_cast<const uint32_t *>(&t);
                }
                __stcs(reinterpret_cast<uint4 *>(out), make_uint4(x[0], x[1], x[2], x[3]));
            }
        } else {
#pragma unroll
            for (int n = 0; n < 8; ++n)
                if (n < lanes) ds_store_one<FP32OUT>(out, n, (n & 1) ? acc[n >> 1].y : acc[n >> 1].x);
        }
    }
}

// first row (within the block's run) of the block's it-th stage: a short first stage lands sooner
__device__ __forceinline__ int dw_stage_row(int it, int first) { return it == 0 ? 0 : first + (it - 1) * DW_ROWS; }

// ND: 2, 3, 4, 6 or 8, at least the number of devices.  A stage has room for ND; where there are fewer, the last ones have steps of 0
// and whatever bits lie in their part: every pattern decodes to a finite code, and fma(code, 0, acc) is acc (never -0).
//
// SPLIT (six to eight devices on rows of more than 320 groups): two blocks share a run of rows.  Each stages its half of every row (a
// copy per device and row) and the BF16 rows, decodes its groups, adds up the selected features that lie among them (the
// second block also those at or above L) and decodes the columns whose codes lie there.
template <int B, int ND, bool SPLIT, bool FP32OUT, bool HAS_BIAS>
__global__ void __launch_bounds__(dw_main(ND) + DW_AUX + 32, 1) dequant_stream_rows(const DWParams pp)
{
    extern __shared__ __align__(128) uint8_t dw_smem[];
    const DSParams &p = pp.d;
    const int N = p.N, E = p.E, k = p.k, L = p.L, G = (L + 7) >> 3, nstage = pp.nstage;
    const uint32_t LB = (uint32_t)L * B;
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t stage_bytes = (uint32_t)ND * (pp.dev_bytes + pp.hp_bytes);
    uint32_t *const sums = reinterpret_cast<uint32_t *>(dw_smem + (size_t)nstage * stage_bytes);  // [nstage][DW_ROWS][k]
    uint64_t *const full = reinterpret_cast<uint64_t *>(dw_smem + (((size_t)nstage * (stage_bytes + (size_t)DW_ROWS * k * 4) + 15) & ~(size_t)15));
    uint64_t *const empty = full + nstage, *const sums_ready = empty + nstage;
    const int64_t t_begin = (int64_t)(SPLIT ? blockIdx.x >> 1 : blockIdx.x) * pp.rows_per_block;
    const int rows_mine = (int)(p.T - t_begin < pp.rows_per_block ? p.T - t_begin : pp.rows_per_block);
    const int half = SPLIT ? (int)(blockIdx.x & 1u) : 0;
    const int g0 = half * pp.half_groups, g1 = SPLIT ? (half ? G : pp.half_groups) : G;  // this block's groups
    const uint32_t bit0 = SPLIT ? (uint32_t)g0 * (8 * B) : 0u;                              // their first bit in a row
    const uint32_t pitch = SPLIT ? dw_pitch(pp.half_groups, B) : 0u;

    tpq_grid_dep_launch();
    if (p.arr.words) {
        tpq_block_wait_arrivals(p.arr);
        __syncthreads();
    }
    if (tid < 32) {
        // ---------------- producer warp: lane i copies device i's code rows, lane ND + i its BF16 rows.  Those begin and
        // end anywhere: the copy runs between 16-byte boundaries, and the values in the payload's last, incomplete 16 bytes
        // (none where T k is a multiple of 8) are loaded and put into the stage by the warp, behind its copies and ahead of the
        // arrival that the stage's readers wait for.  (Read by the auxiliary threads, device after device once the stage had
        // landed: 148 x 2048 of 21 selected 2.2 to 2.8 us for one to four devices, 1.8 to 2.3 so; 148 x 3072 of 31 2.3 to 3.1, 2.1 to 2.8.)
        if (lane == 0) {
            for (int s = 0; s < nstage; ++s) {
                mbar_init(smem_u32(&full[s]), 1);
                mbar_init(smem_u32(&empty[s]), (blockDim.x - 32) / 32);
                mbar_init(smem_u32(&sums_ready[s]), DW_AUX / 32);
            }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        __syncwarp();
        asm volatile("bar.arrive 1, %0;" ::"r"(blockDim.x) : "memory");  // the barriers exist
        if (lane < N) {  // the first rows may start their way to L2 (a hint only: L2 is the point of coherence)
            const int rows = rows_mine < DW_ROWS ? rows_mine : DW_ROWS;
            const int64_t bit = t_begin * (int64_t)LB, from = (bit >> 3) & ~(int64_t)15;
            const int64_t to = ((bit + (int64_t)rows * LB + 127) >> 7) << 4;
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p.pl[lane] + from), "r"((uint32_t)(to - from)) : "memory");
        }
        tpq_grid_dep_wait();  // the payloads and the output buffer may still be in use by the kernel ahead
        int st = 0;
        uint32_t parity = 1;
        for (int it = 0, r0 = 0; r0 < rows_mine; r0 = dw_stage_row(++it, pp.first)) {
            const int cap = it == 0 ? pp.first : DW_ROWS, rows = rows_mine - r0 < cap ? rows_mine - r0 : cap;
            const int64_t bit = (t_begin + r0) * (int64_t)LB, from = (bit >> 3) & ~(int64_t)15;
            const int64_t to = ((bit + (int64_t)rows * LB + 127) >> 7) << 4;  // (the code section is a multiple of 16 bytes)
            const uint32_t bytes = (uint32_t)(to - from), bar = smem_u32(&full[st]);
            // SPLIT: lane 8 r + i copies device i's half of row r
            uint32_t c_bytes = 0;
            int64_t c_from = 0;
            const int c_dev = lane & 7, c_row = lane >> 3;
            if (SPLIT && c_dev < N && c_row < rows) {
                const int64_t b0 = (t_begin + r0 + c_row) * (int64_t)LB + bit0;
                const uint32_t n = half ? LB - bit0 : (uint32_t)pp.half_groups * (8 * B);
                c_from = (b0 >> 3) & ~(int64_t)15;
                c_bytes = (uint32_t)((((b0 + n + 127) >> 7) << 4) - c_from);
            }
            const uint32_t all = SPLIT ? __reduce_add_sync(0xffffffffu, c_bytes) : (uint32_t)N * bytes;
            const int64_t h_from = ((t_begin + r0) * k * 2) & ~(int64_t)15, h_all = (p.T * k * 2) & ~(int64_t)15;
            int64_t h_to = ((t_begin + r0 + rows) * k * 2 + 15) & ~(int64_t)15;
            if (h_to > h_all) h_to = h_all;
            const uint32_t h_bytes = h_to > h_from ? (uint32_t)(h_to - h_from) : 0u;
            const int left = (t_begin + r0 + rows) * k * 2 > h_all ? (int)(p.T * k - h_all / 2) : 0;  // values that no copy brings
            int ok = 1;
            if (lane == 0) {
                if (it >= nstage && !mbar_wait(smem_u32(&empty[st]), parity)) {
                    atomicExch(pp.status, (int)TPQ_ERR_TIMEOUT);
                    ok = 0;
                } else if (left == 0) {
                    mbar_expect_tx(bar, all + (uint32_t)N * h_bytes);
                }
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) break;
            const uint32_t stage = smem_u32(dw_smem) + (uint32_t)st * stage_bytes;
            const int h_lane = SPLIT ? lane : lane - ND;
            if (SPLIT) {
                if (c_bytes) bulk_g2s(stage + (uint32_t)c_dev * pp.dev_bytes + (uint32_t)c_row * pitch, p.pl[c_dev] + c_from, c_bytes, bar);
            } else if (lane < N) {
                bulk_g2s(stage + (uint32_t)lane * pp.dev_bytes, p.pl[lane] + from, bytes, bar);
            }
            if (h_lane >= 0 && h_lane < N && h_bytes)
                bulk_g2s(stage + ND * pp.dev_bytes + (uint32_t)h_lane * pp.hp_bytes, p.pl[h_lane] + p.lp_bytes + h_from, h_bytes, bar);
            if (left) {  // lane 8 a + b: value b of devices a and a + 4 (those of rows of another stage as well: there is room)
                const int b = lane & 7;
                uint16_t v[(ND + 3) / 4];
#pragma unroll
                for (int u = 0; u < (ND + 3) / 4; ++u)
                    if ((lane >> 3) + 4 * u < N && b < left)
                        v[u] = __ldcs(reinterpret_cast<const uint16_t *>(p.pl[(lane >> 3) + 4 * u] + p.lp_bytes + h_all) + b);
#pragma unroll
                for (int u = 0; u < (ND + 3) / 4; ++u)
                    if ((lane >> 3) + 4 * u < N && b < left)
                        asm volatile("st.shared.u16 [%0], %1;" ::"r"(stage + ND * pp.dev_bytes + ((lane >> 3) + 4 * u) * pp.hp_bytes +
                                                                     (uint32_t)(h_all - h_from) + 2u * b),
                                     "h"(v[u])
                                     : "memory");
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // (a later stage's copies may land on them)
                __syncwarp();
                if (lane == 0) mbar_expect_tx(bar, all + (uint32_t)N * h_bytes);  // (release: the values are in the stage)
            }
            if (++st == nstage) {
                st = 0;
                parity ^= 1u;
            }
        }
        return;
    }
    int st = 0;
    uint32_t parity = 0;
    if (tid < 32 + DW_AUX) {
        // ---------------- auxiliary warps: thread `at` adds up selected feature `at` and decodes column L + at, row by row in
        // short rolled loops over what it has loaded once (this code runs once per stage and nobody else runs it, so that
        // straight-line code would pay an instruction fetch for every few instructions)
        const int at = tid - 32;
        // (SPLIT: whether a feature below L, or a slot, lies among this block's groups; the second block takes the features above)
        auto mine = [&](int c) { return !SPLIT || (c < L ? (c >> 3) >= g0 && (c >> 3) < g1 : half == 1); };
        const int s_col = at < k ? __ldg(p.hp_idx + at) : 0;                    // rank `at`: its feature
        const bool on = at < k && mine(s_col);
        int ps = at < k ? __ldg(pp.pos + L + at) : -1;                          // column L + at: its slot (< 0: selected)
        if (ps >= 0 && !mine(ps)) ps = -1;
        float c_s[ND];
#pragma unroll
        for (int i = 0; i < ND; ++i) c_s[i] = i < N && ps >= 0 ? __ldg(pp.s_k + (size_t)i * E + L + at) : 0.0f;
        asm volatile("bar.sync 1, %0;" ::"r"(blockDim.x) : "memory");
        if (HAS_BIAS) tpq_grid_dep_wait();  // (the kernel ahead may be writing it; the payloads come through the producer warp only)
        float s_b = HAS_BIAS && on ? p.bias[s_col] : 0.0f, c_b = HAS_BIAS && ps >= 0 ? p.bias[L + at] : 0.0f;
        uint32_t c_bit = ps >= 0 ? (uint32_t)ps * B - bit0 : 0u;
        asm volatile("" : "+r"(c_bit), "+f"(s_b), "+f"(c_b));
#pragma unroll
        for (int i = 0; i < ND; ++i) asm volatile("" : "+f"(c_s[i]));
        constexpr int ESIZE = FP32OUT ? 4 : 2;
        const int64_t out_row_bytes = p.out_stride * ESIZE;
        auto bits_of = [&](float v) { return FP32OUT ? __float_as_uint(v) : (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v)); };
        // the code of the slot whose first bit is bit `bit` of a device's part of the stage
        auto code = [&](uint32_t dev, uint32_t bit) {
            const uint32_t a = dev + (bit >> 5) * 4u;
            const uint32_t w = __funnelshift_r(dw_lds32(a), dw_lds32(a + 4u), bit & 31u) & ((1u << B) - 1u);
            return __fsub_rn(__uint_as_float((w ^ (1u << (B - 1))) | 0x4B000000u), 8388608.0f + (float)(1 << (B - 1)));
        };
        for (int it = 0, r0 = 0; r0 < rows_mine; r0 = dw_stage_row(++it, pp.first)) {
            const int cap = it == 0 ? pp.first : DW_ROWS, rows = rows_mine - r0 < cap ? rows_mine - r0 : cap;
            const int64_t t0 = t_begin + r0;
            // (the stage's previous sums have been read by everybody when its next copies land)
            if (!mbar_wait(smem_u32(&full[st]), parity)) {
                atomicExch(pp.status, (int)TPQ_ERR_TIMEOUT);
                break;
            }
            const uint32_t stage = smem_u32(dw_smem) + (uint32_t)st * stage_bytes;
            const uint32_t sum0 = smem_u32(sums) + (uint32_t)(st * DW_ROWS * k) * 4u;  // the stage's sums
            uint8_t *const out0 = static_cast<uint8_t *>(p.out) + t0 * out_row_bytes;
            // the sums of the selected features, out of the stage
            const uint32_t hp = stage + ND * pp.dev_bytes + (uint32_t)((t0 * k * 2) & 15);
            if (on) {
                uint32_t a = hp + 2u * at, o = sum0 + 4u * at;
                uint8_t *og = out0 + (int64_t)s_col * ESIZE;
#pragma unroll 1
                for (int r = 0; r < rows; ++r, a += 2u * k, o += 4u * k, og += out_row_bytes) {
                    float v = 0.0f;
#pragma unroll
                    for (int i = 0; i < ND; ++i)
                        if (i < N) v = __fadd_rn(v, __uint_as_float(dw_lds16(a + (uint32_t)i * pp.hp_bytes) << 16));
                    if (HAS_BIAS) v = __fadd_rn(v, s_b);
                    if (s_col < L) dw_sts32(o, bits_of(v));
                    else ds_store_one<FP32OUT>(og, 0, v);
                }
            }
            for (int h = at + DW_AUX; h < k; h += DW_AUX) {  // (more selected features than threads)
                const int col = __ldg(p.hp_idx + h);
                if (!mine(col)) continue;
                for (int r = 0; r < rows; ++r) {
                    const int e = r * k + h;
                    float v = 0.0f;
                    for (int i = 0; i < N; ++i) v = __fadd_rn(v, __uint_as_float(dw_lds16(hp + (uint32_t)i * pp.hp_bytes + 2u * e) << 16));
                    if (HAS_BIAS) v = __fadd_rn(v, p.bias[col]);
                    if (col < L) dw_sts32(sum0 + 4u * e, bits_of(v));
                    else ds_store_one<FP32OUT>(out0 + r * out_row_bytes, col, v);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sums_ready[st]));  // (release: the sums are visible to whoever waits)
            // the last k columns: filler features, decoded from the holes' slots that carry them
            const uint32_t rem = (uint32_t)((t0 * (int64_t)LB + bit0) & 127);
            if (ps >= 0) {
                uint8_t *og = out0 + (int64_t)(L + at) * ESIZE;
#pragma unroll 1
                for (int r = 0; r < rows; ++r, og += out_row_bytes) {
                    const uint32_t bit = dw_row_bit<SPLIT>(rem, r, LB, pitch) + c_bit;
                    float v = 0.0f;
#pragma unroll
                    for (int i = 0; i < ND; ++i) v = __fmaf_rn(code(stage + (uint32_t)i * pp.dev_bytes, bit), c_s[i], v);
                    if (HAS_BIAS) v = __fadd_rn(v, c_b);
                    ds_store_one<FP32OUT>(og, 0, v);
                }
            }
            for (int h = at + DW_AUX; h < k; h += DW_AUX) {  // (more columns than threads)
                const int slot = __ldg(pp.pos + L + h);
                if (slot < 0 || !mine(slot)) continue;
                for (int r = 0; r < rows; ++r) {
                    float v = 0.0f;
                    for (int i = 0; i < N; ++i)
                        v = __fmaf_rn(code(stage + (uint32_t)i * pp.dev_bytes, dw_row_bit<SPLIT>(rem, r, LB, pitch) + (uint32_t)slot * B - bit0),
                                      __ldg(pp.s_k + (size_t)i * E + L + h), v);
                    if (HAS_BIAS) v = __fadd_rn(v, p.bias[L + h]);
                    ds_store_one<FP32OUT>(out0 + r * out_row_bytes, L + h, v);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&empty[st]));
            if (++st == nstage) {
                st = 0;
                parity ^= 1u;
            }
        }
        return;
    }
    // ---------------- main warps
    const int g = g0 + tid - 32 - DW_AUX;
    const int lanes = g >= g1 ? 0 : L - 8 * g < 8 ? L - 8 * g : 8;  // slots of the group (the last one may be short, idle threads have none)
    float2 sc[ND][4], b[4];
    uint32_t mask = 0;
    int hb = 0;
#pragma unroll
    for (int i = 0; i < ND; ++i)
#pragma unroll
        for (int h = 0; h < 4; ++h) sc[i][h] = make_float2(0.0f, 0.0f);
    if (lanes > 0) {
        const uint32_t gd = __ldg(p.grp + g);
        mask = gd & 0xFFu;
        if (lanes < 8) mask &= (1u << lanes) - 1u;
        hb = (int)(gd >> 8);
#pragma unroll
        for (int i = 0; i < ND; ++i)
            if (i < N) {
                const float4 u = __ldg(reinterpret_cast<const float4 *>(pp.s_k + (size_t)i * E + 8 * g));
                const float4 w = __ldg(reinterpret_cast<const float4 *>(pp.s_k + (size_t)i * E + 8 * g + 4));
                const float s8[8] = {u.x, u.y, u.z, u.w, w.x, w.y, w.z, w.w};
#pragma unroll
                for (int h = 0; h < 4; ++h)
                    sc[i][h] = make_float2(s8[2 * h] * (1.0f / (float)(1u << ds_pos(B, 2 * h))),
                                           s8[2 * h + 1] * (1.0f / (float)(1u << ds_pos(B, 2 * h + 1))));
            }
    }
    if (HAS_BIAS) tpq_grid_dep_wait();  // (the kernel ahead may be writing it)
#pragma unroll
    for (int h = 0; h < 4; ++h)
        b[h] = HAS_BIAS && lanes > 0 ? make_float2(p.bias[8 * g + 2 * h], p.bias[8 * g + 2 * h + 1]) : make_float2(0.0f, 0.0f);
    // (opaque: the compiler, short of registers, would otherwise load the steps again at every use)
#pragma unroll
    for (int i = 0; i < ND; ++i)
#pragma unroll
        for (int h = 0; h < 4; ++h) asm volatile("" : "+f"(sc[i][h].x), "+f"(sc[i][h].y));
    asm volatile("bar.sync 1, %0;" ::"r"(blockDim.x) : "memory");
    DSConsts<B> dc;
    dc.template init<true>();
    constexpr int ESIZE = FP32OUT ? 4 : 2;
    const int64_t out_row_bytes = p.out_stride * ESIZE;
    uint8_t *out = static_cast<uint8_t *>(p.out) + t_begin * out_row_bytes + (lanes > 0 ? g : 0) * (8 * ESIZE);
    const uint32_t g_bit = (uint32_t)(lanes > 0 ? g - g0 : 0) * (8 * B);
    const bool warp_holes = __any_sync(0xffffffffu, mask != 0);
    for (int it = 0, r0 = 0; r0 < rows_mine; r0 = dw_stage_row(++it, pp.first)) {
        const int cap = it == 0 ? pp.first : DW_ROWS, rows = rows_mine - r0 < cap ? rows_mine - r0 : cap;
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&full[st]), parity))) {
            atomicExch(pp.status, (int)TPQ_ERR_TIMEOUT);
            break;
        }
        const uint8_t *const stage = dw_smem + (size_t)st * stage_bytes;
        const uint32_t rem = (uint32_t)(((t_begin + r0) * (int64_t)LB + bit0) & 127);
        if (rows == DW_ROWS) {
            dw_rows<B, ND, SPLIT, DW_ROWS, FP32OUT, HAS_BIAS>(stage, pp.dev_bytes, rem, 0, LB, pitch, g_bit, sc, b, dc, out, out_row_bytes, lanes);
        } else {
#pragma unroll 1
            for (int r = 0; r < rows; ++r)
                dw_rows<B, ND, SPLIT, 1, FP32OUT, HAS_BIAS>(stage, pp.dev_bytes, rem, r, LB, pitch, g_bit, sc, b, dc, out + r * out_row_bytes, out_row_bytes, lanes);
        }
        if (warp_holes) {  // the selected features' lanes
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&sums_ready[st]), parity))) {
                atomicExch(pp.status, (int)TPQ_ERR_TIMEOUT);
                break;
            }
            uint32_t m = mask;
            for (int h = hb; m; ++h) {
                const int n = __ffs(m) - 1;
                m &= m - 1;
                const uint32_t *sum = sums + (size_t)st * DW_ROWS * k + h;
                uint8_t *at = out + n * ESIZE;
                for (int r = 0; r < rows; ++r, sum += k, at += out_row_bytes) {
                    if (FP32OUT)
                        *reinterpret_cast<uint32_t *>(at) = *sum;
                    else
                        *reinterpret_cast<uint16_t *>(at) = (uint16_t)*sum;
                }
            }
        }
        out += rows * out_row_bytes;
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&empty[st]));
        if (++st == nstage) {
            st = 0;
            parity ^= 1u;
        }
    }
}

// (Three as four: 1000 x 2048 to 5120, 4 bits, 5.0 to 7.8 us, as three 4.7 to 6.6; 8192 x 2048 31 and 26.  Five as eight: 4000 x
// 2560 22 us, as six 18; 8192 x 2048 32 and 26.)
int dw_nd(int N) { return N <= 2 ? 2 : N <= 4 ? N : N <= 6 ? 6 : 8; }

// two blocks to a run of rows
bool dw_split(const tpq_ctx *c) { return (c->E - c->k + 7) / 8 > dw_main(dw_nd(c->N)); }
// a device's code words in a stage
uint32_t dw_part_bytes(const tpq_ctx *c)
{
    const int L = c->E - c->k, G = (L + 7) / 8;
    return dw_split(c) ? DW_ROWS * dw_pitch((G + 1) / 2, c->bits) : dw_dev_bytes(L, c->bits);
}

// Whether this kernel is ahead of the panel kernel, six to eight devices and two blocks to a run of rows.  Both sides in ns, fitted
// to 1200 launches of each (64 to 1184 rows of 2624 to 5120 features, every width; 4 % off on average, 28 % at worst).  Here a row
// takes a copy per device and half, so its time hardly depends on the width.  The panel kernel takes steps: blocks of 16 rows,
// one to an SM, two, or two with several chunks each; it is at its best where they fill one wave (8 x 740 x 2624, 3 bits, 7.1 us
// against 9.1 here; 888 rows 11.3 and 10.1).  What this picks took 1.005 times as long as the faster of the two on average, 1.18 at
// worst.
bool dw_split_ahead(const tpq_ctx *c, int64_t T)
{
    struct { double one, one_dev, one_load, more, chunk, chunk_dev, load; } const fit[3] = {
        {2690, 212, 65, 1680, 1640, 172, 147},   // 2 bits
        {3470, 129, 62, 1590, 2050, 169, 171},   // 3 and 4 bits
        {1850, 454, 75, 2310, 576, 473, 179}};   // more: two devices to a step instead of four
    const auto &f = fit[c->bits == 2 ? 0 : c->bits <= 4 ? 1 : 2];
    constexpr int RC = DS_THREADS / DS_CG * DS_R;  // rows of a chunk there
    const int N = c->N, sm = c->sm_count, G = (c->E - c->k + 7) / 8, nd = dw_nd(N), warps = ((G + 1) / 2 + 31) / 32;
    const int panels = (G + DS_CG - 1) / DS_CG;
    const int64_t chunks = (T + RC - 1) / RC, room = 2 * sm / panels, deep = room < chunks ? room : chunks, runs = sm / 2;
    const double load = (double)(panels * chunks) / sm, per_block = (double)((chunks + deep - 1) / deep);
    const double panel = panels * deep <= sm ? f.one + (f.one_dev + f.one_load * load) * N
                                             : f.more + per_block * (f.chunk + f.chunk_dev * N) + f.load * load * N;
    return 1620.0 + 119.0 * nd + (double)((T + runs - 1) / runs) * (200.0 + nd * (16.4 + 5.9 * warps)) < panel;
}

// Ring depth; 0: the shape is the panel kernel's.  Up to four devices: this one.  Five to eight: from 160 groups on (below, 1024
// features, 0.5 to 0.9 times the panel kernel's time up to 444 rows, 1.0 to 1.5 beyond).  Rows of 160 to 199 groups leave a
// block five to seven warps: up to 16 rows an SM 0.6 to 1.05, beyond 0.95 to 1.2 at 2 to 4 bits, where the panel kernel's third
// panel is nearly full, 0.9 to 1.05 at more and 0.65 to 0.95 at 8.  From 200 groups on 0.55 to 1.0 times.  Above 320, two blocks
// to a run of rows: six devices or more, up to 8 rows an SM.
int dw_stages(const tpq_ctx *c, int64_t T, int64_t out_stride)
{
    const int L = c->E - c->k, G = (L + 7) / 8;
    if (c->N > 8 || c->E % 8 || out_stride % 8 || G > 640 || c->k > DW_MAX_K || (c->N > 4 && G < 160)) return 0;
    if (c->N > 4 && G < 200 && T > 16 * c->sm_count && c->bits < (c->N > 5 ? 5 : 8)) return 0;
    if (dw_split(c) && (c->N < 6 || T > 8 * c->sm_count || !dw_split_ahead(c, T))) return 0;
    int n = 4;
    while (n > 1 && dw_smem_bytes(dw_nd(c->N), dw_part_bytes(c), c->k, n) > (size_t)c->smem_optin) --n;
    return n > 1 ? n : 0;
}

template <int B, int ND, bool SPLIT>
cudaError_t launch_dequant_rows_nd(const DWParams &pp, int fp32_out, unsigned grid, int threads, size_t smem, cudaStream_t st)
{
    auto kern = pp.d.bias ? (fp32_out ? dequant_stream_rows<B, ND, SPLIT, true, true> : dequant_stream_rows<B, ND, SPLIT, false, true>)
                          : (fp32_out ? dequant_stream_rows<B, ND, SPLIT, true, false> : dequant_stream_rows<B, ND, SPLIT, false, false>);
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return tpq_launch_pdl(kern, dim3(grid), dim3(threads), smem, st, pp);
}

template <int B>
cudaError_t launch_dequant_rows(const DWParams &pp, int fp32_out, unsigned grid, int threads, size_t smem, cudaStream_t st)
{
    switch (dw_nd(pp.d.N)) {
    case 2: return launch_dequant_rows_nd<B, 2, false>(pp, fp32_out, grid, threads, smem, st);
    case 3: return launch_dequant_rows_nd<B, 3, false>(pp, fp32_out, grid, threads, smem, st);
    case 4: return launch_dequant_rows_nd<B, 4, false>(pp, fp32_out, grid, threads, smem, st);
    case 6: return pp.half_groups ? launch_dequant_rows_nd<B, 6, true>(pp, fp32_out, grid, threads, smem, st)
                                  : launch_dequant_rows_nd<B, 6, false>(pp, fp32_out, grid, threads, smem, st);
    default: break;
    }
    return pp.half_groups ? launch_dequant_rows_nd<B, 8, true>(pp, fp32_out, grid, threads, smem, st)
                          : launch_dequant_rows_nd<B, 8, false>(pp, fp32_out, grid, threads, smem, st);
}

}  // namespace

// Rows of at least 32 bits (a word of the stream spans two rows at most), bit strings that fit in shared memory,
// bit offsets inside a tile or chunk that fit 32 bits.
bool tpq_stream_ok(const tpq_ctx *c, int64_t T)
{
    const int64_t L = c->E - c->k;
    return T > 0 && T < (int64_t)QS_ROWS * 0x7FFFFFFF && L * c->bits >= 32 && c->E <= (1 << 18) && qt_smem_bytes((int)L, c->bits) <= (size_t)c->smem_optin &&
           ds_smem_bytes(c->bits, c->N) <= (size_t)c->smem_optin;
}

static cudaError_t launch_stream(const tpq_ctx *c, int shard0, int n, const void *const *ys, int64_t T, int64_t stride,
                                 void *const *payloads, int n_dst, uint32_t *const *arrived, uint32_t epoch, cudaStream_t st,
                                 int64_t *launches)
{
    const int E = c->E, k = c->k, L = E - k, G = (L + 7) / 8;
    int gpt = 0, warps = 0, nstage = 0;
    const bool pipe = qs_pipe_plan(c, stride, &gpt, &warps, &nstage);
    QPipeParams pp;
    QSParams &p = pp.q;
    p.T = T; p.stride = stride; p.lp_bytes = tpq_lp_bytes_i(T, E, k, c->bits);
    p.n_tiles = (T + QS_ROWS - 1) / QS_ROWS;
    p.E = E; p.k = k; p.L = L; p.n_holes = c->n_holes;
    p.row_words = qs_row_words(L, c->bits);
    p.grp = c->t.grp; p.hp_idx = c->t.hp_idx; p.hole = c->t.hole; p.filler = c->t.filler;
    for (int b0 = 0; b0 < n; b0 += QS_MAX_BATCH) {
        const int nb = n - b0 < QS_MAX_BATCH ? n - b0 : QS_MAX_BATCH;
        for (int b = 0; b < nb; ++b) {
            p.y[b] = static_cast<const uint16_t *>(ys[b0 + b]);
            p.payload[b] = static_cast<uint8_t *>(payloads[b0 + b]);
        }
        p.inv_s = c->t.inv_s + (size_t)(shard0 + b0) * E;
        cudaError_t e;
        if (pipe) {
            // the SMs are divided among the shards; no block has more than a row above the mean
            pp.nstage = nstage; pp.status = c->t.status; pp.done = c->t.push_done;
            pp.n_dst = n_dst; pp.epoch = epoch;
            for (int d = 0; d < n_dst; ++d) {
                p.payload[d] = static_cast<uint8_t *>(payloads[d]);
                pp.arrived[d] = arrived[d];
            }
            int64_t bps = c->sm_count / nb > 0 ? c->sm_count / nb : 1;
            if (bps > T) bps = T;
            pp.rows_per_block = (T + bps - 1) / bps;
            bps = (T + pp.rows_per_block - 1) / pp.rows_per_block;
            pp.bps = (int)bps;
            const int threads = warps * 32 + 64;
            const size_t smem = qs_pipe_bytes(E, c->bits, warps, gpt, nstage);
            const unsigned grid = (unsigned)(bps * nb);
            const bool push = n_dst > 0;
            switch (c->bits) {
            case 2: e = launch_quantize_pipe<2>(pp, push, gpt, threads, grid, smem, st); break;
            case 3: e = launch_quantize_pipe<3>(pp, push, gpt, threads, grid, smem, st); break;
            case 4: e = launch_quantize_pipe<4>(pp, push, gpt, threads, grid, smem, st); break;
            case 5: e = launch_quantize_pipe<5>(pp, push, gpt, threads, grid, smem, st); break;
            case 6: e = launch_quantize_pipe<6>(pp, push, gpt, threads, grid, smem, st); break;
            case 7: e = launch_quantize_pipe<7>(pp, push, gpt, threads, grid, smem, st); break;
            default: e = launch_quantize_pipe<8>(pp, push, gpt, threads, grid, smem, st); break;
            }
        } else {
            const bool vec = E % 8 == 0 && stride % 8 == 0;
            const int per = (G + QS_THREADS - 1) / QS_THREADS;  // an even share of the row's groups per thread
            int threads = ((G + per - 1) / per + 31) / 32 * 32;
            if (threads < 128) threads = 128;
            const dim3 grid((unsigned)p.n_tiles, (unsigned)nb);
            switch (c->bits) {
            case 2: e = launch_quantize_tile<2>(p, vec, threads, grid, st); break;
            case 3: e = launch_quantize_tile<3>(p, vec, threads, grid, st); break;
            case 4: e = launch_quantize_tile<4>(p, vec, threads, grid, st); break;
            case 5: e = launch_quantize_tile<5>(p, vec, threads, grid, st); break;
            case 6: e = launch_quantize_tile<6>(p, vec, threads, grid, st); break;
            case 7: e = launch_quantize_tile<7>(p, vec, threads, grid, st); break;
            default: e = launch_quantize_tile<8>(p, vec, threads, grid, st); break;
            }
        }
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    return cudaSuccess;
}

cudaError_t tpq_launch_quantize_stream(const tpq_ctx *c, int shard0, int n, const void *const *ys, int64_t T, int64_t stride,
                                       void *const *payloads, cudaStream_t st, int64_t *launches)
{
    return launch_stream(c, shard0, n, ys, T, stride, payloads, 0, nullptr, 0u, st, launches);
}

bool tpq_stream_pipe_ok(const tpq_ctx *c, int64_t T, int64_t stride)
{
    int gpt, warps, nstage;
    return tpq_stream_ok(c, T) && qs_pipe_plan(c, stride, &gpt, &warps, &nstage);
}

// One block per SM has a warp for 31 or 62 groups.  Rows of up to 256 groups leave it so few warps that the copies'
// latency shows once a block has several rows: 512 features (3 warps an SM against the group kernel's 8 and more) level at
// 1000 rows of a launch, 1.5 times as long at 2000, 2.4 at 32768; 2048 features 0.8 at 512 rows, 1.05 at 1000, 1.2 to 1.5
// beyond; 2112 features level at 5000 rows, 1.1 at 9600; from 2304 on 0.5 to 1.0.  Two groups a lane: up to three tokens (a
// thread of the group kernel takes four) 1.0 to 1.4 times as long; 0.7 to 0.9 at 30 rows, 0.9 to 1.1 at 100 to 300 and 0.7 to
// 1.0 at 9600 of 5376 to 8256 features (1.2 at 600 or 1200 rows of 6144, whose last stage of four holds one row); above
// 8704 features only up to 3 bits and from 500 rows on less (0.8 to 0.95).  Rows too long for the ring are the tile
// kernel's, a block to 8 rows: 0.8 to 0.9 times as long with 4000 rows at 2 and 3 bits, 1.0 to 2.2 at more, 1.1 to 5.8 with fewer.
bool tpq_stream_ahead(const tpq_ctx *c, int n, int64_t T, int64_t stride)
{
    int gpt, warps, nstage;
    const int G = (c->E - c->k + 7) / 8, sm = c->sm_count;
    const int64_t rows = (n < QS_MAX_BATCH ? n : QS_MAX_BATCH) * T;  // of a launch
    if (!tpq_stream_ok(c, T)) return false;
    if (!qs_pipe_plan(c, stride, &gpt, &warps, &nstage)) return c->bits <= 3 && rows >= 24 * sm;
    if (gpt > 1) return T >= 4 && (c->E <= 8704 || (c->bits <= 3 && rows >= 3 * sm));
    return G > 280 || rows < (G > 256 ? 32 : 7) * sm;
}

// The tile kernel against n launches of the shape-generic one.  A block takes 8 rows from end to end, 320 groups at a
// time, so however few rows there are the launch takes as long as a block: 3.6 us + 1.1 ns a feature (1.3 ns from 5 bits
// on), 2 us + 0.85 ns up to 4 rows, 0.5 ns for one.  The generic kernel takes 3.4 us a launch (6 at 2 bits, 5 at 3) and from
// about 400 000 values on 3 us + 2.5 ps a value (4.7 at 2 bits, 3.6 at 3).  Measured at 4 bits, generic against tile: one shard of 5121
// features 4.4 and 9.4 us at 64 rows, 6.3 and 9.5 at 256, 15.8 and 12.8 at 1024; of 16385 4.4 and 22.7 at 16, 23.7 and 25.4 at 512; two
// shards 8.4 and 22.8, 46 and 33; 16 of 1033 features 58 and 4.5 at 16 rows.
bool tpq_stream_tile_ahead(const tpq_ctx *c, int n, int64_t T)
{
    const int b = c->bits;
    const double E = c->E, values = (double)T * E;
    const double tile = T > 4 ? 3600.0 + (b > 4 ? 1.3 : 1.1) * E : 2000.0 + (T > 1 ? 0.85 : 0.5) * E;
    const double least = b == 2 ? 6000.0 : b == 3 ? 5000.0 : 3400.0;
    const double generic = (b <= 3 ? 3500.0 : 3000.0) + (b == 2 ? 4.7e-3 : b == 3 ? 3.6e-3 : 2.5e-3) * values;
    return tile < n * (generic > least ? generic : least);
}

// The copies and the publishing kernel cost the other way about 4 us and 1 us more per destination (16 destinations of few
// rows 25 us against 5 to 10), the push mode stores every word n_dst times.  Narrow rows: one destination 0.8 times as
// long at 256 rows, 1.2 at 1000, 1.5 to 1.8 at 2048; two 0.75, 1.1, 1.4; four 0.55, 0.8, 1.1.  Two groups a lane: one
// destination 0.8 to 1.1 at up to 256 rows, 1.2 at 1000, 1.4 at 2048 (1.2 at one row above 8704 features); two 0.9 and 1.2;
// sixteen 0.4 and 1.1.
bool tpq_stream_push_ahead(const tpq_ctx *c, int n_dst, int64_t T, int64_t stride)
{
    int gpt, warps, nstage;
    if (!qs_pipe_plan(c, stride, &gpt, &warps, &nstage)) return false;
    const int sm = c->sm_count;
    if (gpt > 1) return n_dst > 1 ? T < 10 * sm : T < 3 * sm && (c->E <= 8704 || T >= 24);
    return (c->E - c->k + 7) / 8 > 256 || T < 3 * sm * n_dst;
}

cudaError_t tpq_launch_quantize_stream_push(const tpq_ctx *c, int shard, const void *y, int64_t T, int64_t stride, void *const *dst,
                                            uint32_t *const *arrived, int n_dst, uint32_t epoch, cudaStream_t st, int64_t *launches)
{
    return launch_stream(c, shard, 1, &y, T, stride, dst, n_dst, arrived, epoch, st, launches);
}

cudaError_t tpq_launch_dequant_stream(const tpq_ctx *c, const void *const *payloads, int64_t T, void *out, int fp32_out,
                                      int64_t out_stride, cudaStream_t st, int64_t *launches)
{
    const int E = c->E, k = c->k, L = E - k, G = (L + 7) / 8;
    DSParams p;
    for (int i = 0; i < c->N; ++i) p.pl[i] = static_cast<const uint8_t *>(payloads[i]);
    p.N = c->N; p.E = E; p.k = k; p.L = L; p.T = T;
    p.lp_bytes = tpq_lp_bytes_i(T, E, k, c->bits);
    p.out_stride = out_stride;
    p.s_slot = c->t.s_slot; p.grp = c->t.grp; p.lp_idx = c->t.lp_idx; p.hp_idx = c->t.hp_idx;
    p.filler = c->t.filler; p.n_holes = c->n_holes;
    p.vec = E % 8 == 0 && out_stride % 8 == 0;
    p.out = out; p.bias = c->call_bias; p.arr = c->call_arr;
    cudaError_t e;
    if (const int nstage = dw_stages(c, T, out_stride)) {
        DWParams pp;
        pp.d = p;
        pp.s_k = c->t.s_k; pp.pos = c->t.pos; pp.nstage = nstage; pp.status = c->t.status;
        pp.dev_bytes = dw_part_bytes(c);
        pp.hp_bytes = dw_hp_bytes(k);
        pp.half_groups = dw_split(c) ? (G + 1) / 2 : 0;
        const int per_run = pp.half_groups ? 2 : 1;
        const int64_t runs = c->sm_count / per_run;
        pp.rows_per_block = (T + runs - 1) / runs;
        // A short first stage lands sooner: it takes the rows that do not fill a stage, at least two, so that there are no more
        // stages for it.  (Always two: 1000 rows of 1280 to 5120 features, 2 + 4 + 1 a block, 3.9 to 8.3 us, so 3.5 to 7.5 for one
        // to four devices.)  A block of one
        // stage has no ring: fewer barriers to set up, and shared memory left to the next launch's (148 x 3072 at 8 bits 2.2 to 3.0
        // and 2.1 to 2.7 us).  (A ring of two stages where there are two is no gain: 1000 x 2048 at 8 bits 5.0 to 5.5 us, 5.6 to 5.9
        // so, blocks of the next launch sharing an SM.)
        const int odd = (int)((pp.rows_per_block - 1) % DW_ROWS) + 1;
        pp.first = pp.rows_per_block <= DW_ROWS ? DW_ROWS : odd < 2 ? 2 : odd;
        if (pp.rows_per_block <= DW_ROWS) pp.nstage = 1;
        const unsigned grid = (unsigned)((T + pp.rows_per_block - 1) / pp.rows_per_block * per_run);
        const int threads = 32 + DW_AUX + ((pp.half_groups ? pp.half_groups : G) + 31) / 32 * 32;
        size_t smem = dw_smem_bytes(dw_nd(c->N), pp.dev_bytes, k, pp.nstage);
        // Where there are fewer blocks than SMs each gets one to itself: if two fit (narrow rows, or a device count that needs few
        // registers) the next launch's blocks start two to an SM on the SMs that are free first, and the launch waits for those.
        // (One to four devices of 512 to 3072 features, back to back, the time without this 1: 500 rows 0.96, 1500 rows of 1024
        // features 0.83, 3 x 3000 x 2304 0.74.  With a block for every SM two to one are no loss, and their prologues overlap: 740
        // rows 0.97 of the time with one, 1184 rows 0.98.)
        constexpr size_t ONE_PER_SM = 116 * 1024;
        if ((int)grid < c->sm_count && smem < ONE_PER_SM) smem = ONE_PER_SM;
        switch (c->bits) {
        case 2: e = launch_dequant_rows<2>(pp, fp32_out, grid, threads, smem, st); break;
        case 3: e = launch_dequant_rows<3>(pp, fp32_out, grid, threads, smem, st); break;
        case 4: e = launch_dequant_rows<4>(pp, fp32_out, grid, threads, smem, st); break;
        case 5: e = launch_dequant_rows<5>(pp, fp32_out, grid, threads, smem, st); break;
        case 6: e = launch_dequant_rows<6>(pp, fp32_out, grid, threads, smem, st); break;
        case 7: e = launch_dequant_rows<7>(pp, fp32_out, grid, threads, smem, st); break;
        default: e = launch_dequant_rows<8>(pp, fp32_out, grid, threads, smem, st); break;
        }
        if (e == cudaSuccess) ++*launches;
        return e;
    }
    constexpr int RC = DS_THREADS / DS_CG * DS_R;
    p.panels = (G + DS_CG - 1) / DS_CG;
    p.n_chunks = (T + RC - 1) / RC;
    const int per_sm = 2 * (ds_smem_bytes(c->bits, c->N) + 1024) <= 228 * 1024 ? 2 : 1;
    int64_t gy = (int64_t)c->sm_count * per_sm / p.panels;
    if (gy > p.n_chunks) gy = p.n_chunks;
    if (gy < 1) gy = 1;
    p.gy = (int)gy;
    switch (c->bits) {
    case 2: e = launch_dequant_stream<2>(p, fp32_out, st); break;
    case 3: e = launch_dequant_stream<3>(p, fp32_out, st); break;
    case 4: e = launch_dequant_stream<4>(p, fp32_out, st); break;
    case 5: e = launch_dequant_stream<5>(p, fp32_out, st); break;
    case 6: e = launch_dequant_stream<6>(p, fp32_out, st); break;
    case 7: e = launch_dequant_stream<7>(p, fp32_out, st); break;
    default: e = launch_dequant_stream<8>(p, fp32_out, st); break;
    }
    if (e == cudaSuccess) ++*launches;
    return e;
}
