// The pre-synchronisation linear layer fused with the compressor (Section 2: f^(i)(x^(i)) = x^(i) W^(i),
// then C^(i) of Section 3 on the result): one kernel computes the device's partial sums on the tensor cores
// and writes the payload; the [T][E] BF16 partial sums never go to memory.
//
// The weight matrix is static, so its rows are put into the payload's SLOT order once (tpq_permute_weight):
// output column c < L = E - k is then the feature that slot c carries (holes already filled with their
// fillers) and columns L .. E-1 are the selected features in rank order.  The epilogue therefore has no hole
// logic: a group of 8 columns is either one 32-bit word of codes or 8 BF16 values of the BF16 block.
//
// Kernel: tcgen05 (5th-generation tensor cores), persistent: one block per SM walks 128 x BN tiles of the
// output, or a PAIR of blocks (a cluster of two SMs, tcgen05 cta_group::2) walks 256 x BN tiles.  What bounds a
// block (from K of about 1000 on; below, the epilogue) is its shared memory's bandwidth, which the copies that write the operands and the MMAs that read them share: a
// 64-wide k-block of a 128 x 256 tile is 48 KB each way, 385 ns, against 260 ns of MMA.  In a pair each block fetches its
// own 128 rows of x and HALF of the weight tile, and the tensor cores of both read the halves from either's shared
// memory: 32 KB in and 48 KB out per block and k-block.
// Operands are staged by TMA (128-byte swizzle) in a ring of shared-memory stages that runs on
// across tiles; one thread issues tcgen05.mma (M = 128, N = BN, K = 16, BF16 x BF16 -> FP32) into one of TWO
// accumulators in tensor memory; four epilogue warps read the other one back (tcgen05.ld), round to BF16
// (the layer's output type), quantise and store, while the tensor cores work on the next tile.
//   warp 0    TMA producer (one lane)
//   warp 1    tensor-memory allocation (whole warp), MMA issue (one lane), de-allocation
//   warps 2-5 epilogue; warp w reads the 32 accumulator rows of lane quadrant w % 4
// Every wait is bounded: on expiry the block records TPQ_ERR_TIMEOUT, skips its stores, frees its tensor
// memory and returns.
#include "tpq_internal.h"

#include <cuda.h>
#include <cuda_bf16.h>

namespace {

constexpr int LQ_BM = 128, LQ_BK = 64, LQ_THREADS = 192;
constexpr int LQ_WAIT_LIMIT = 1 << 24;  // try_wait attempts (each suspends for a hardware time slice) ...
constexpr unsigned long long LQ_WAIT_NS = 1000000000ull;  // ... and one second, whichever ends first
constexpr uint32_t LQ_A_BYTES = LQ_BM * LQ_BK * 2;  // the x tile of a 64-wide k-block
constexpr uint32_t LQ_SMEM_MAX = 227u * 1024u;

// CG: blocks that share a tile (1, or 2: a pair, each with half of the weight tile)
// KB: 64-wide k-blocks of a stage
__host__ __device__ constexpr uint32_t lq_b_bytes(int BN, int CG) { return (uint32_t)(BN / CG) * LQ_BK * 2; }
__host__ __device__ constexpr uint32_t lq_stage_bytes(int BN, int CG, int KB) { return KB * (LQ_A_BYTES + lq_b_bytes(BN, CG)); }
__host__ __device__ constexpr int lq_stages(int BN, int CG, int KB)
{
    const int n = (int)((LQ_SMEM_MAX - 1024u - 176u - 8u * BN) / lq_stage_bytes(BN, CG, KB));
    return n > 8 ? 8 : n;
}
// two accumulators (the epilogue drains one while the tensor cores fill the other), a power of two of columns
__host__ __device__ constexpr uint32_t lq_tmem_cols(int BN) { return 2 * BN <= 64 ? 64 : 2 * BN <= 128 ? 128 : 2 * BN <= 256 ? 256 : 512; }
__host__ __device__ constexpr size_t lq_smem_bytes(int BN, int CG, int KB)
{
    // 1024 B of slack for the manual alignment; stages; 176 B: barriers (full[8], empty[8], accumulators 2 x 2)
    // and the tensor-memory address; the reciprocal steps of two tiles
    return 1024 + (size_t)lq_stages(BN, CG, KB) * lq_stage_bytes(BN, CG, KB) + 176 + 2 * (size_t)BN * 4;
}

struct LQParams {
    int64_t T;
    int E, k, K;
    int64_t lp_bytes;       // code section size (the BF16 block starts here)
    const float *inv_s;     // [E] of this device, feature order
    const int32_t *lp_idx;  // [L] slot -> feature
    uint8_t *payload;
    int x_rows;             // rows of an x box: 128, or where T is below that, T rounded up to 8 (the tile's other rows hold
                            // whatever was in shared memory; a row of the sum depends on its own row of x only)
    uint16_t *y_slots;      // optional [T][E] BF16 partial sums in slot order (NULL: not written)
    int *status;
};

__device__ __forceinline__ bool lq_mbar_wait(uint32_t bar, uint32_t parity)
{
    unsigned long long t0 = 0;
    for (int i = 0; i < LQ_WAIT_LIMIT; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((i & 63) == 63) {  // and a limit in time as well as in attempts
            unsigned long long t;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            if (t0 == 0) t0 = t;
            else if (t - t0 > LQ_WAIT_NS) return false;
        }
    }
    return false;
}

// ---- tcgen05; CG = 2: the instruction spans the pair of blocks
template <int CG>
__device__ __forceinline__ void tc_alloc(uint32_t smem_dst, uint32_t cols)
{
    if (CG == 2) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
}
template <int CG>
__device__ __forceinline__ void tc_dealloc(uint32_t taddr, uint32_t cols)
{
    if (CG == 2)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
    else
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// arrives at the barrier (of a pair: at the barrier at that offset in both blocks) when the MMAs so far are done
template <int CG>
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    if (CG == 2)
        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
                     "h"((uint16_t)3)
                     : "memory");
    else
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]; BF16 inputs, FP32 accumulation
template <int CG>
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    if (CG == 2)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
            : "memory");
}
// the same place in the shared memory of block `rank` of the cluster
__device__ __forceinline__ uint32_t lq_peer(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void lq_cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Stage kb of a tile's operand: rows y .. of KB 64-wide k-blocks, one behind the other.  KB = 1: a box of the 2-D map;
// more: one box of the 3-D map (64 values, rows, k-blocks).  CG = 2: `bar` is a cluster address in the pair's first block.
template <int CG, int KB>
__device__ __forceinline__ void lq_load(uint32_t dst, const void *map, int kb, int y, uint32_t bar)
{
    if (KB == 1 && CG == 2)
        asm volatile(
            "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
                dst),
            "l"(map), "r"(kb * LQ_BK), "r"(y), "r"(bar)
            : "memory");
    else if (KB == 1)
        tma_load_2d(dst, map, kb * LQ_BK, y, bar);
    else if (CG == 2)
        asm volatile(
            "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
                dst),
            "l"(map), "r"(0), "r"(y), "r"(kb * KB), "r"(bar)
            : "memory");
    else
        asm volatile(
            "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
            "l"(map), "r"(0), "r"(y), "r"(kb * KB), "r"(bar)
            : "memory");
}
// true in one lane of a converged warp, known to the compiler as a single active thread
__device__ __forceinline__ bool lq_elect()
{
    uint32_t one;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xFFFFFFFF;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(one));
    return one != 0;
}
// 32 lanes x 32 consecutive 32-bit columns: thread <-> its lane's row
__device__ __forceinline__ void tc_ld_32x32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Shared-memory operand descriptor: K-major tile of 128-byte rows written by TMA with the 128-byte swizzle
// (8-row groups of 1024 bytes); `addr` may be advanced by 32 bytes per K = 16 inside the swizzle atom.
__device__ __forceinline__ uint64_t lq_smem_desc(uint32_t addr)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4)   // start address
           | ((uint64_t)1 << 16)                // leading byte offset (unused with this layout): 16 B
           | ((uint64_t)(1024 >> 4) << 32)      // stride byte offset between 8-row groups
           | ((uint64_t)1 << 46)                // descriptor version of this architecture
           | ((uint64_t)2 << 61);               // 128-byte swizzle
}
// Instruction descriptor: FP32 accumulator, BF16 A and B, both K-major, M = 128 (of a pair 256), N = BN.
__host__ __device__ constexpr uint32_t lq_instr_desc(int BN, int CG)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(CG * LQ_BM >> 4) << 24);
}

// C^(i) of one value (Section 3): two binary32 roundings, clamp, round half to even; the low 4 bits of
// fl(u + 1.5 * 2^23) are the code's two's-complement nibble.
__device__ __forceinline__ uint32_t lq_code(float x, float inv)
{
    float u = __fmul_rn(x, inv);
    u = fminf(fmaxf(u, -8.0f), 7.0f);
    return __float_as_uint(__fadd_rn(u, 12582912.0f)) & 0xFu;
}

// Tile order: bands of LQ_GROUP_M row tiles; inside a band column tile by column tile, the band's row tiles
// innermost.  Blocks that run together share a weight tile, and a band's rows of x (LQ_GROUP_M x 128 x K
// values) stay in L2 while every column tile passes over them, whatever T is.
constexpr int LQ_GROUP_M = 16;
template <int CG>  // (a pair's tile is 256 rows: half as many make a band)
__device__ __forceinline__ void lq_tile_origin(int tile, int mt, int nt, int BN, int &m0, int &n0)
{
    constexpr int GM = LQ_GROUP_M / CG;
    const int per_band = GM * nt;
    const int band = tile / per_band, in_band = tile - band * per_band;
    const int rows = (mt - band * GM < GM) ? mt - band * GM : GM;  // the last band may be short
    const int n = in_band / rows, m = band * GM + (in_band - n * rows);
    m0 = m * (CG * LQ_BM);
    n0 = n * BN;
}

template <int BN, int CG, int KB>
__global__ void __launch_bounds__(LQ_THREADS, 1)
linear_quantize(const LQParams p, const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w)
{
    extern __shared__ uint8_t lq_raw[];
    constexpr int NS = lq_stages(BN, CG, KB);
    constexpr uint32_t STAGE = lq_stage_bytes(BN, CG, KB);
    constexpr uint32_t TCOLS = lq_tmem_cols(BN);
    const uint32_t base = (smem_u32(lq_raw) + 1023u) & ~1023u;  // swizzled tiles want 1024-byte alignment
    uint8_t *const gen = lq_raw + (base - smem_u32(lq_raw));
    // after the stages: full[8], empty[8], acc_full[2], acc_empty[2] (8 bytes each), the tensor-memory address,
    // then the reciprocal steps of two tiles
    const uint32_t bars = base + NS * STAGE;
    uint32_t *const tmem_slot = reinterpret_cast<uint32_t *>(gen + NS * STAGE + 160);
    float *const inv_tiles = reinterpret_cast<float *>(gen + NS * STAGE + 176);
    auto full = [&](int s) { return bars + 8u * s; };
    auto empty = [&](int s) { return bars + 8u * (8 + s); };
    auto acc_full = [&](int b) { return bars + 8u * (16 + b); };
    auto acc_empty = [&](int b) { return bars + 8u * (18 + b); };

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int L = p.E - p.k, L8 = L >> 3;
    const int nkb = (p.K + KB * LQ_BK - 1) / (KB * LQ_BK);  // stages per tile
    const int mt = (int)((p.T + CG * LQ_BM - 1) / (CG * LQ_BM)), nt = (p.E + BN - 1) / BN;
    const int tiles = mt * nt;
    // a pair: block `rank` owns rows rank * 128 .. of the tile and fetches half `rank` of the weight tile; the first
    // block's barriers count both blocks' copies and its MMA warp works for both
    const uint32_t rank = CG == 2 ? blockIdx.x & 1u : 0u;
    const int first_tile = blockIdx.x / CG, tile_step = gridDim.x / CG;

    if (tid == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(acc_full(b), 1);
            mbar_init(acc_empty(b), 4 * CG);  // one arrival per epilogue warp
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tc_alloc<CG>(smem_u32(tmem_slot), TCOLS);
    tc_fence_before();
    tpq_grid_dep_wait();  // the operands and the payload buffer may still be in use by the kernel ahead
    __syncthreads();
    if (CG == 2) lq_cluster_sync();  // the other block's barriers exist
    tpq_grid_dep_launch();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    bool ok = true;

    if (warp == 0) {
        if (lane == 0) {
            int it = 0;  // k-blocks issued so far, over all of this block's tiles
            for (int tile = first_tile; tile < tiles && ok; tile += tile_step) {
                int m0, n0;
                lq_tile_origin<CG>(tile, mt, nt, BN, m0, n0);
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = it % NS;
                    if (it >= NS && !lq_mbar_wait(empty(s), ((it / NS) - 1) & 1)) {
                        ok = false;
                        break;
                    }
                    if (CG == 2) {
                        if (rank == 0) mbar_expect_tx(full(s), 2 * STAGE);
                        const uint32_t bar = lq_peer(full(s), 0);
                        lq_load<2, KB>(base + s * STAGE, &map_x, kb, m0 + (int)rank * LQ_BM, bar);
                        lq_load<2, KB>(base + s * STAGE + KB * LQ_A_BYTES, &map_w, kb, n0 + (int)rank * (BN / 2), bar);
                    } else {
                        mbar_expect_tx(full(s), (uint32_t)(KB * p.x_rows) * (LQ_BK * 2) + KB * lq_b_bytes(BN, CG));
                        lq_load<1, KB>(base + s * STAGE, &map_x, kb, m0, full(s));
                        lq_load<1, KB>(base + s * STAGE + KB * LQ_A_BYTES, &map_w, kb, n0, full(s));
                    }
                }
            }
            const int last = it > NS ? it - NS : 0;
            if (!ok && rank == 0)  // giving up: let the copies already issued (a pair's: both blocks') land before the shared memory is released
                for (int j = last; j < it; ++j) (void)lq_mbar_wait(full(j % NS), (j / NS) & 1);
            if (CG == 2 && ok)  // the first block's MMA warp still arrives at the other's barriers: neither may end before
                for (int j = last; j < it; ++j) ok = ok && lq_mbar_wait(empty(j % NS), (j / NS) & 1);
        }
        __syncwarp();
    } else if (warp == 1) {
        // The whole warp walks the loop and one elected lane issues: with the issuing lane picked by a comparison of
        // its index the compiler cannot know that a single thread is active, and every MMA's operands (which the
        // instruction takes from uniform registers) cost a loop over the lanes.
        constexpr uint32_t idesc = lq_instr_desc(BN, CG);
        const uint64_t desc0 = lq_smem_desc(base);
        const uint32_t x_kb = CG == 2 ? LQ_A_BYTES >> 4 : (uint32_t)p.x_rows * (LQ_BK * 2 >> 4);  // from one k-block of x to the next
        int it = 0, n_tile = 0;
        for (int tile = rank == 0 ? first_tile : tiles; tile < tiles && ok; tile += tile_step, ++n_tile) {
            const int b = n_tile & 1;
            // the epilogue must have drained this accumulator (used two tiles ago)
            if (n_tile >= 2) ok = __all_sync(0xffffffffu, lq_mbar_wait(acc_empty(b), ((n_tile >> 1) - 1) & 1));
            if (!ok) break;
            tc_fence_after();
            const uint32_t d = tmem + (uint32_t)(b * BN);
            for (int kb = 0; kb < nkb; ++kb, ++it) {
                const int s = it % NS;
                ok = __all_sync(0xffffffffu, lq_mbar_wait(full(s), (it / NS) & 1));
                if (!ok) break;
                tc_fence_after();
                if (lq_elect()) {
                    const uint64_t a = desc0 + (uint64_t)((uint32_t)s * (STAGE >> 4));
#pragma unroll
                    for (int k4 = 0; k4 < KB * (LQ_BK / 16); ++k4) {
                        const uint64_t ka = (uint64_t)((k4 / 4) * x_kb + 2 * (k4 % 4));
                        const uint64_t kw = (uint64_t)((KB * LQ_A_BYTES + (k4 / 4) * lq_b_bytes(BN, CG)) >> 4) + 2 * (k4 % 4);
                        tc_mma_bf16<CG>(d, a + ka, a + kw, idesc, (kb | k4) != 0);
                    }
                    tc_commit<CG>(empty(s));  // arrives when the MMAs above have read the stage
                    if (kb == nkb - 1) tc_commit<CG>(acc_full(b));  // arrives when the tile's accumulator is complete
                }
                __syncwarp();
            }
        }
    } else {
        // ---------------- epilogue: tile i is drained while the tensor cores work on tile i + 1
        const int q = warp & 3, et = tid - 64;
        uint32_t *const lp_out = reinterpret_cast<uint32_t *>(p.payload);
        uint16_t *const hp_out = reinterpret_cast<uint16_t *>(p.payload + p.lp_bytes);
        int n_tile = 0;
        for (int tile = first_tile; tile < tiles; tile += tile_step, ++n_tile) {
            const int b = n_tile & 1;
            int m0, n0;
            lq_tile_origin<CG>(tile, mt, nt, BN, m0, n0);
            m0 += (int)rank * LQ_BM;
            float *const inv_tile = inv_tiles + b * BN;
            for (int c = et; c < BN; c += 128) {  // the tile's reciprocal steps in slot order
                const int col = n0 + c;
                inv_tile[c] = (col < L) ? __ldg(p.inv_s + __ldg(p.lp_idx + col)) : 0.0f;
            }
            // barrier of the four epilogue warps (the steps above are in place) that also tells every thread
            // whether ANY of them has given up: they leave the loop together, none is left waiting here
            uint32_t any_bad;
            asm volatile(
                "{\n\t.reg .pred p, q;\n\t"
                "setp.ne.u32 q, %1, 0;\n\t"
                "bar.red.or.pred p, 1, 128, q;\n\t"
                "selp.u32 %0, 1, 0, p;\n\t}"
                : "=r"(any_bad)
                : "r"((uint32_t)!ok)
                : "memory");
            if (any_bad) {
                ok = false;
                break;
            }
            if (!lq_mbar_wait(acc_full(b), (n_tile >> 1) & 1)) ok = false;
            ok = __all_sync(0xffffffffu, ok);  // the tensor-memory loads below are warp-wide
            if (!ok) continue;                 // (reported at the next barrier above; no tile follows a lost one)
            tc_fence_after();
            const int64_t row = (int64_t)m0 + q * 32 + lane;
            const bool row_on = row < p.T;
            for (int c0 = 0; c0 < BN; c0 += 32) {
                if (n0 + c0 >= p.E) break;  // uniform
                uint32_t r[32];
                tc_ld_32x32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * BN + c0), r);
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const int col = n0 + c0 + 8 * g;
                    if (col >= p.E || c0 + 8 * g >= BN) break;
                    uint32_t h[4];  // the 8 sums rounded to BF16 (the layer's output type), packed in pairs
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const __nv_bfloat162 v = __floats2bfloat162_rn(__uint_as_float(r[8 * g + 2 * j]),
                                                                       __uint_as_float(r[8 * g + 2 * j + 1]));
                        h[j] = *reinterpret_cast<const uint32_t *>(&v);
                    }
                    if (!row_on) continue;
                    if (p.y_slots) *reinterpret_cast<uint4 *>(p.y_slots + row * p.E + col) = make_uint4(h[0], h[1], h[2], h[3]);
                    if (col < L) {
                        const float4 i0 = *reinterpret_cast<const float4 *>(inv_tile + c0 + 8 * g);
                        const float4 i1 = *reinterpret_cast<const float4 *>(inv_tile + c0 + 8 * g + 4);
                        const float iv[8] = {i0.x, i0.y, i0.z, i0.w, i1.x, i1.y, i1.z, i1.w};
                        uint32_t word = 0;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint32_t c_lo = lq_code(__uint_as_float(h[j] << 16), iv[2 * j]);
                            const uint32_t c_hi = lq_code(__uint_as_float(h[j] & 0xFFFF0000u), iv[2 * j + 1]);
                            word |= (c_lo << (8 * j)) | (c_hi << (8 * j + 4));
                        }
                        lp_out[row * L8 + (col >> 3)] = word;
                    } else {
                        *reinterpret_cast<uint4 *>(hp_out + row * p.k + (col - L)) = make_uint4(h[0], h[1], h[2], h[3]);
                    }
                }
            }
            // this warp has read its quadrant of the accumulator: hand it back to the MMA thread
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (CG == 2)
                    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(lq_peer(acc_empty(b), 0)) : "memory");
                else
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(acc_empty(b)) : "memory");
            }
        }
        // zero padding of the code section (its size is rounded up to 16 bytes)
        if (blockIdx.x == 0 && warp == 2) {
            const int64_t valid = p.T * L8, words = p.lp_bytes / 4;
            for (int64_t w = valid + lane; w < words; w += 32) lp_out[w] = 0u;
        }
    }
    if (!ok) atomicExch(p.status, (int)TPQ_ERR_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if (CG == 2) lq_cluster_sync();  // neither block's shared or tensor memory is in use by the other any more
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tc_dealloc<CG>(tmem, TCOLS);
    }
}

// rows of a [E][K] weight matrix gathered into slot order: row c < L from feature lp_idx[c], row L + h from hp_idx[h]
__global__ void __launch_bounds__(256) permute_weight(const uint16_t *__restrict__ w, uint16_t *__restrict__ out, int E, int k,
                                                      int64_t K, const int32_t *__restrict__ lp_idx,
                                                      const int32_t *__restrict__ hp_idx)
{
    const int r = blockIdx.x, L = E - k;
    const int src = r < L ? __ldg(lp_idx + r) : __ldg(hp_idx + (r - L));
    const uint16_t *in = w + (int64_t)src * K;
    uint16_t *o = out + (int64_t)r * K;
    if ((K & 7) == 0) {
        for (int64_t c = threadIdx.x; c < K / 8; c += blockDim.x)
            reinterpret_cast<uint4 *>(o)[c] = __ldg(reinterpret_cast<const uint4 *>(in) + c);
    } else {
        for (int64_t c = threadIdx.x; c < K; c += blockDim.x) o[c] = in[c];
    }
}


// [rows][K] BF16, row-major -> boxes of box_rows rows x kb k-blocks of 64 elements with the 128-byte swizzle;
// out-of-range reads give 0.  Several k-blocks per box (K a multiple of 64): the row is cut into 64-value pieces, a third dimension.
bool lq_map(const void *ptr, int64_t rows, int64_t K, int box_rows, int kb, CUtensorMap *out)
{
    tpq_encode_tiled_fn fn = tpq_tensor_map_encoder();
    if (!fn) return false;
    const cuuint64_t dims2[2] = {(cuuint64_t)K, (cuuint64_t)rows}, dims3[3] = {LQ_BK, (cuuint64_t)rows, (cuuint64_t)(K / LQ_BK)};
    const cuuint64_t strides[2] = {(cuuint64_t)K * 2, LQ_BK * 2};
    const cuuint32_t box[3] = {(cuuint32_t)LQ_BK, (cuuint32_t)box_rows, (cuuint32_t)kb};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, kb > 1 ? 3 : 2, const_cast<void *>(ptr), kb > 1 ? dims3 : dims2, strides, box,
              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BN, int CG, int KB>
cudaError_t lq_launch(LQParams p, const void *x, const void *w, int sm_count, cudaStream_t st)
{
    p.x_rows = CG == 1 && p.T < LQ_BM ? (int)(p.T + 7) / 8 * 8 : LQ_BM;
    CUtensorMap mx, mw;
    if (!lq_map(x, p.T, p.K, p.x_rows, KB, &mx) || !lq_map(w, p.E, p.K, BN / CG, KB, &mw)) return cudaErrorNotSupported;
    const size_t smem = lq_smem_bytes(BN, CG, KB);
    cudaError_t e = cudaFuncSetAttribute(linear_quantize<BN, CG, KB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t tiles = ((p.T + CG * LQ_BM - 1) / (CG * LQ_BM)) * ((p.E + BN - 1) / BN);
    const int64_t places = sm_count / CG;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(CG * (tiles < places ? tiles : places)));  // persistent: a block (pair) walks tiles b, b + places, ...
    cfg.blockDim = dim3(LQ_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = CG;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = CG == 2 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, linear_quantize<BN, CG, KB>, p, mx, mw);
}

}  // namespace

bool tpq_linear_ok(const tpq_ctx *c, int64_t T, int64_t K)
{
    if (c->bits != 4) return false;
    if (c->E % 8 || c->k % 8 || c->E - c->k < 8) return false;
    if (T < 1 || K < 8 || K % 8) return false;  // 16-byte row pitch for the tensor maps
    if (T > (int64_t)1 << 31 || K > (int64_t)1 << 31) return false;
    return lq_smem_bytes(192, 2, 2) <= (size_t)c->smem_optin;
}

cudaError_t tpq_launch_permute_weight(const tpq_ctx *c, const void *w, void *out, int64_t K, cudaStream_t st, int64_t *launches)
{
    permute_weight<<<c->E, 256, 0, st>>>(static_cast<const uint16_t *>(w), static_cast<uint16_t *>(out), c->E, c->k, K,
                                         c->t.lp_idx, c->t.hp_idx);
    ++*launches;
    return cudaGetLastError();
}

cudaError_t tpq_launch_linear_quantize(const tpq_ctx *c, int shard, const void *x, const void *w_slots, int64_t T, int64_t K,
                                       void *payload, void *y_slots, cudaStream_t st, int64_t *launches)
{
    LQParams p;
    p.T = T; p.E = c->E; p.k = c->k; p.K = (int)K;
    p.lp_bytes = tpq_lp_bytes_i(T, c->E, c->k);
    p.inv_s = c->t.inv_s + (size_t)shard * c->E;
    p.lp_idx = c->t.lp_idx;
    p.payload = static_cast<uint8_t *>(payload);
    p.y_slots = static_cast<uint16_t *>(y_slots);
    p.status = c->t.status;
    // Tile shape: the least estimated time.  A tile's MMAs overlap the epilogue of the tile before it, so a place takes
    // start-up + one tile's k-blocks + (tiles - 1) x the longer of k-blocks and epilogue + one epilogue.
    // A 64-wide k-block is bound by shared memory, 128 bytes a clock for the copies that write the operands and the MMAs
    // that read them: a single block writes and reads 16 KB of x and BN / 8 KB of weights, one of a pair writes 16 + BN / 16 KB
    // and reads 16 + BN / 8 KB (the MMAs alone would take 260 ns at 256 columns).  The epilogue takes 15 ns a column (four
    // warps) and a hand-over of 0.8 us, between two blocks 1.8 us: below K = 1000 or so it is what bounds a tile, and pairs,
    // which save k-blocks' time, only cost theirs.  The constants (ns) are fitted to all ten shapes at K = 64 to 3456, E = 512 to
    // 8192, T = 1 to 4096: the choice is within 0.5 % of the fastest one on average, 12 % at worst.  2048 x 3456 x 5120: 59.9 us
    // with single blocks of 192 columns, 51.0 us with pairs of 192 (256: 55.8, 160: 55.0); 8192 tokens 208 -> 180 us (pairs of
    // 256); 300 x 256 x 8192: pairs of 256 8.4 us, single blocks of 192 6.5; 64 x 1280 x 5120 9.2 -> 6.6 us (single blocks of 48:
    // 107 of them instead of 40); 1 x 1280 x 5120 11.9 -> 6.6 us (x boxes of 8 rows instead of 128); 128 x 8192 x 8192 42.5 -> 29.7 us.
    struct Shape { int bn, cg, kb; };
    constexpr Shape shapes[] = {{256, 2, 307}, {192, 2, 265}, {160, 2, 236}, {128, 2, 230}, {256, 1, 385},
                                {192, 1, 376}, {128, 1, 260}, {64, 1, 207},  {48, 1, 186},  {32, 1, 180}};
    int best = 0;
    int64_t best_cost = 0;
    for (int j = 0; j < (int)(sizeof shapes / sizeof *shapes); ++j) {
        const int bn = shapes[j].bn, cg = shapes[j].cg;
        const int64_t tiles = ((T + cg * LQ_BM - 1) / (cg * LQ_BM)) * ((c->E + bn - 1) / bn), places = c->sm_count / cg;
        const int64_t waves = (tiles + places - 1) / places;
        const int64_t main = (K + LQ_BK - 1) / LQ_BK * shapes[j].kb, epilogue = (cg == 2 ? 1800 : 800) + 15 * bn;
        const int64_t cost = (cg == 2 ? 1000 : 1400) + main + (waves - 1) * (main > epilogue ? main : epilogue) + epilogue;
        if (j == 0 || cost < best_cost) {
            best_cost = cost;
            best = j;
        }
    }
    // Stages of 128 values of K where its 64-value pieces are whole: half as many copies and barrier rounds (48-column
    // blocks 186 against 250 ns per k-block), except where such a stage leaves room for three at most (256 columns).
    const bool k2 = K % LQ_BK == 0 && K >= 2 * LQ_BK;
    cudaError_t e;
#define LQ_GO(BN, CG) e = k2 ? lq_launch<BN, CG, 2>(p, x, w_slots, c->sm_count, st) : lq_launch<BN, CG, 1>(p, x, w_slots, c->sm_count, st)
    switch (best) {
    case 0: e = lq_launch<256, 2, 1>(p, x, w_slots, c->sm_count, st); break;
    case 1: LQ_GO(192, 2); break;
    case 2: LQ_GO(160, 2); break;
    case 3: LQ_GO(128, 2); break;
    case 4: e = lq_launch<256, 1, 1>(p, x, w_slots, c->sm_count, st); break;
    case 5: LQ_GO(192, 1); break;
    case 6: LQ_GO(128, 1); break;
    case 7: LQ_GO(64, 1); break;
    case 8: LQ_GO(48, 1); break;
    default: LQ_GO(32, 1); break;
    }
#undef LQ_GO
    if (e == cudaSuccess) ++*launches;
    return e;
}
