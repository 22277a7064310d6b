// Range aggregation, top-k feature selection and table construction
// (paper Section 3 "Selecting High Precision Features"; k = floor(E/64) in Section 4).
#include "tpq_internal.h"

namespace {

// R^(i)_j = 2 max(-m, M); Rbar_j = sum_i R^(i)_j (binary32, devices ascending);
// step s = R/(2^bits - 1) (R/15 for Int4) floored at 2^-23 and its reciprocal (IEEE division, no fast-math).
// (Dependent launch: no pointer is __restrict__, the calibration ahead may still be writing m and M.  A thread's loads of
// RG_N devices are in flight together, and blocks of 64 features spread them over the GPU.)
constexpr int RG_THREADS = 64, RG_N = 8;

// The order of aggregated ranges as integers: -0 and +0 are equal, and a NaN (calibrated on or restored) has a place, ahead of
// the infinities, so that exactly k features are selected whatever the ranges are; the tables rely on that.
__device__ __forceinline__ int order_key(float x)
{
    const int i = __float_as_int(__fadd_rn(x, 0.0f));  // (-0 -> +0, any NaN -> the positive one)
    return i ^ ((i >> 31) & 0x7FFFFFFF);
}

__global__ void __launch_bounds__(RG_THREADS) ranges_kernel(const float *m, const float *M, int N, int E, float levels, float *R,
                                                            float *Rbar, int32_t *key, float *s, float *inv_s)
{
    tpq_grid_dep_launch();
    tpq_grid_dep_wait();
    const int j = blockIdx.x * RG_THREADS + threadIdx.x;
    if (j >= E) return;
    float acc = 0.0f;
    for (int i0 = 0; i0 < N; i0 += RG_N) {
        float lo[RG_N], hi[RG_N];
#pragma unroll
        for (int u = 0; u < RG_N; ++u)
            if (i0 + u < N) {
                lo[u] = m[(size_t)(i0 + u) * E + j];
                hi[u] = M[(size_t)(i0 + u) * E + j];
            }
#pragma unroll
        for (int u = 0; u < RG_N; ++u)
            if (i0 + u < N) {
                const size_t o = (size_t)(i0 + u) * E + j;
                const float a = -lo[u], b = hi[u];
                const float A = (a > b) ? a : b;
                const float r = __fmul_rn(2.0f, A);
                R[o] = r;
                acc = (i0 + u == 0) ? r : __fadd_rn(acc, r);
                float sv = __fdiv_rn(r, levels);
                if (!(sv >= 1.1920928955078125e-07f)) sv = 1.1920928955078125e-07f;
                s[o] = sv;
                inv_s[o] = __fdiv_rn(1.0f, sv);
            }
    }
    Rbar[j] = acc;
    key[j] = order_key(acc);
}

// Feature j is selected iff fewer than k features beat it, where a beats j when
// Rbar_a > Rbar_j, or Rbar_a == Rbar_j and a < j.  O(E^2) comparisons, a warp per feature: its lanes compare side by
// side, four values per load (a few tens of KB, so the loads hit L1).  (One thread per feature, the values
// through shared memory, left all but 18 SMs idle: 68 us at E = 4608.)
// The keys are made once, by the kernel ahead, and lie in the array of the prefix counts, which the kernels behind this one fill and
// no step's kernel reads.  Those ahead of j's own four are compared with one less: a comparison and an addition each.  (With the key
// made anew at every comparison, us per call: 2 x 32768 380 and now 203, 2 x 131072 5250 and 2460; as comparisons of the values
// and their places 310 and 4100.)
constexpr int TK_WARPS = 8;

__global__ void __launch_bounds__(32 * TK_WARPS) topk_flags_kernel(const int32_t *key, int E, int k, uint8_t *flag)
{
    tpq_grid_dep_launch();
    tpq_grid_dep_wait();  // (the keys are the kernel ahead's)
    const int j = blockIdx.x * TK_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (j >= E) return;
    const int mine = key[j], least = mine - 1;  // (no key is the least integer)
    int beats = 0;
    const int E4 = E >> 2, jq = j >> 2;
#pragma unroll 4
    for (int q = lane; q < E4; q += 32) {
        const int4 v = reinterpret_cast<const int4 *>(key)[q];
        const int than = q < jq ? least : mine;
        beats += (v.x > than) + (v.y > than) + (v.z > than) + (v.w > than);
    }
    if (lane < (E & 3)) beats += key[4 * E4 + lane] > mine;
    if (lane < (j & 3)) beats += key[4 * jq + lane] == mine;  // j's own four
    beats = __reduce_add_sync(0xffffffffu, beats);
    if (lane == 0) flag[j] = beats < k ? 1 : 0;
}

// One block: exclusive scan of the flags -> selected list, hole / filler lists.  A warp takes an even share of adjacent
// features, 32 at a time (its lanes' loads and stores are adjacent), first to count, then to place; one block-wide scan
// of the warps' counts lies between, whatever E is.  (An even share per thread, strided loads and stores: tpq_set_features
// of 131072 features 366 us, so 102; 1048576: 2565 and 478; 4608 of 8 devices 57 and 55.)
__global__ void __launch_bounds__(1024) scan_kernel(tpq_tables t, int E, int k)
{
    __shared__ int2 warp_sums[32];  // a warp's selected features, those of them below L
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int L = E - k;
    const int per = ((E + 31) / 32 + 31) / 32 * 32;  // features of a warp
    const int j0 = wid * per < E ? wid * per : E, j1 = j0 + per < E ? j0 + per : E;
    int all = 0, below = 0;
#pragma unroll 4
    for (int j = j0 + lane; j < j1; j += 32) {
        const int f = t.flag[j];
        all += f;
        below += j < L ? f : 0;
    }
    all = __reduce_add_sync(0xffffffffu, all);
    below = __reduce_add_sync(0xffffffffu, below);
    if (lane == 0) warp_sums[wid] = make_int2(all, below);
    __syncthreads();
    const int2 w = warp_sums[lane];
    const int m = __reduce_add_sync(0xffffffffu, w.y);                       // selected features below L
    int run = __reduce_add_sync(0xffffffffu, lane < wid ? w.x : 0);          // selected features before the warp's next 32
#pragma unroll 4
    for (int base = j0; base < j1; base += 32) {
        const int j = base + lane;
        const int f = j < j1 ? t.flag[j] : 0;
        const uint32_t set = __ballot_sync(0xffffffffu, f != 0);
        const int before = run + __popc(set & ((1u << lane) - 1u));
        run += __popc(set);
        if (j < j1) {
            t.hpre[j] = before;
            // holes: selected features below L; fillers: unselected features at or above L (equally many)
            if (f) {
                t.hp_idx[before] = j;
                if (j < L) t.hole[before] = j;
            } else if (j >= L) {
                t.filler[(j - L) - (before - m)] = j;
            }
        }
    }
}

// One feature's entries of the tables: slot order, per-feature slots, the dequantiser's zeroed-step and slot-order step
// copies and, every 8 features, a group descriptor.  f: selected; pre: selected features before j; src: the feature held
// by slot j (< 0: there is no slot j); slot: the slot of an unselected feature; mask: flags of features j .. j + 7.
__device__ __forceinline__ void put_feature(const tpq_tables &t, int N, int E, int j, int f, int pre, int src, int slot, uint32_t mask)
{
    if (src >= 0) t.lp_idx[j] = src;
    for (int i0 = 0; i0 < N; i0 += RG_N) {  // (the loads of RG_N devices in flight together)
        float own[RG_N], at[RG_N];
#pragma unroll
        for (int u = 0; u < RG_N; ++u)
            if (i0 + u < N) {
                const size_t row = (size_t)(i0 + u) * E;
                own[u] = t.s[row + j];
                at[u] = src >= 0 && src != j ? t.s[row + src] : 0.0f;
            }
#pragma unroll
        for (int u = 0; u < RG_N; ++u)
            if (i0 + u < N) {
                const size_t row = (size_t)(i0 + u) * E;
                t.s_k[row + j] = f ? 0.0f : own[u];
                t.s_slot[row + j] = src < 0 ? 0.0f : src == j ? own[u] : at[u];
            }
    }
    t.pos[j] = f ? -(pre + 1) : slot;
    if ((j & 7) == 0) t.grp[j >> 3] = ((uint32_t)pre << 8) | mask;
}

// Behind scan_kernel, a thread per feature over the whole GPU.  (As loops of the scan's one block these N*E-long copies took
// most of its 35 us at 8 x 4608.)
__global__ void __launch_bounds__(256) tables_kernel(tpq_tables t, int N, int E, int k)
{
    const int j = blockIdx.x * 256 + threadIdx.x;
    if (j >= E) return;
    const int L = E - k, f = t.flag[j], pre = t.hpre[j];
    const int m = L < E ? t.hpre[L] : 0;
    uint32_t mask = 0;
    if ((j & 7) == 0)
        for (int n = 0; n < 8; ++n)
            if (j + n < E && t.flag[j + n]) mask |= 1u << n;
    put_feature(t, N, E, j, f, pre, j < L ? (f ? t.filler[pre] : j) : -1, f || j < L ? j : t.hole[(j - L) - (pre - m)], mask);
}

// Scan and tables in one launch, for up to ST_MAX_E features: a block needs no more of the other features than their flags,
// which it packs into bits and counts by itself (E bytes out of L2 for each block of 64 features).  A feature's rank is
// a count of bits below it, the r-th hole or filler a search for the word that holds it.  (With dependent launches, three
// instead of four, and the feature list copied once: the selection call 60.3 -> 38.5 us at 8 x 4608, 51.5 -> 28.7 at
// 2 x 1024, 79.5 -> 63 at 16 x 8192.  Above 32 768 features the flags are scanned once, by one block.)
constexpr int ST_THREADS = 64, ST_MAX_E = 1 << 15, ST_WORDS = ST_MAX_E / 32;

__global__ void __launch_bounds__(ST_THREADS) scan_tables_kernel(tpq_tables t, int N, int E, int k)
{
    __shared__ uint32_t bits[ST_WORDS + 1];  // flags, a bit per feature
    __shared__ int before[ST_WORDS + 1];     // flags before a word
    __shared__ int warp_sums[ST_THREADS / 32];
    tpq_grid_dep_launch();
    tpq_grid_dep_wait();  // (the flags and the steps are the kernel ahead's)
    const int tid = threadIdx.x, lane = tid & 31, L = E - k;
    const int words = (E + 31) / 32, per = (words + ST_THREADS - 1) / ST_THREADS;
    int sum = 0;
    for (int w = tid * per; w < (tid + 1) * per && w < words; ++w) {
        uint32_t v = 0;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (32 * w + 16 * q >= E) break;  // (the array is padded to a multiple of 16 bytes)
            const uint4 u = reinterpret_cast<const uint4 *>(t.flag)[2 * w + q];
            const uint32_t x[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int b = 0; b < 4; ++b)  // four bytes of 0 or 1 -> four bits
                v |= (((x[b] & 0x01010101u) * 0x10204080u) >> 28) << (16 * q + 4 * b);
        }
        if (32 * w + 32 > E) v &= (1u << (E & 31)) - 1u;
        bits[w] = v;
        sum += __popc(v);
    }
    int incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
    }
    if (lane == 31) warp_sums[tid >> 5] = incl;
    __syncthreads();
    int run = incl - sum;
    for (int w = 0; w < (tid >> 5); ++w) run += warp_sums[w];
    for (int w = tid * per; w < (tid + 1) * per && w < words; ++w) {
        before[w] = run;
        run += __popc(bits[w]);
    }
    __syncthreads();
    const int j = blockIdx.x * ST_THREADS + tid;
    if (j >= E) return;
    auto selected_before = [&](int x) { return before[x >> 5] + __popc(bits[x >> 5] & ((1u << (x & 31)) - 1u)); };
    const int f = bits[j >> 5] >> (j & 31) & 1u, pre = selected_before(j);
    const int m = L < E ? selected_before(L) : 0;  // selected features below L
    // the r-th (from 0) selected feature, or the r-th unselected one: the last word with at most r before it, then its bits
    auto find = [&](int r, bool sel) {
        int lo = 0, hi = words - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if ((sel ? before[mid] : 32 * mid - before[mid]) <= r) lo = mid;
            else hi = mid - 1;
        }
        uint32_t v = sel ? bits[lo] : ~bits[lo];
        for (int n = r - (sel ? before[lo] : 32 * lo - before[lo]); n > 0; --n) v &= v - 1;
        return 32 * lo + __ffs(v) - 1;
    };
    t.hpre[j] = pre;
    int src = j, slot = j;
    if (f) {
        t.hp_idx[pre] = j;
        if (j < L) {
            t.hole[pre] = j;
            src = find(L - m + pre, false);  // the pre-th filler: L - m unselected features lie below L
        }
    } else if (j >= L) {
        const int r = (j - L) - (pre - m);
        t.filler[r] = j;
        slot = find(r, true);  // the r-th hole is the r-th selected feature
    }
    put_feature(t, N, E, j, f, pre, j < L ? src : -1, slot, (bits[j >> 5] >> (j & 31)) & 0xFFu);
}

}  // namespace

cudaError_t tpq_launch_ranges(const tpq_tables &t, int N, int E, int bits, cudaStream_t st, int64_t *launches)
{
    ++*launches;
    return tpq_launch_pdl(ranges_kernel, dim3((E + RG_THREADS - 1) / RG_THREADS), dim3(RG_THREADS), 0, st, t.m, t.M, N, E,
                          (float)((1 << bits) - 1), t.R, t.Rbar, t.hpre, t.s, t.inv_s);
}

cudaError_t tpq_launch_topk_flags(const tpq_tables &t, int E, int k, cudaStream_t st, int64_t *launches)
{
    ++*launches;
    return tpq_launch_pdl(topk_flags_kernel, dim3((E + TK_WARPS - 1) / TK_WARPS), dim3(32 * TK_WARPS), 0, st, t.hpre, E, k, t.flag);
}

cudaError_t tpq_launch_tables(const tpq_tables &t, int N, int E, int k, cudaStream_t st, int64_t *launches)
{
    if (E <= ST_MAX_E) {
        ++*launches;
        return tpq_launch_pdl(scan_tables_kernel, dim3((E + ST_THREADS - 1) / ST_THREADS), dim3(ST_THREADS), 0, st, t, N, E, k);
    }
    scan_kernel<<<1, 1024, 0, st>>>(t, E, k);
    ++*launches;
    tables_kernel<<<(E + 255) / 256, 256, 0, st>>>(t, N, E, k);
    ++*launches;
    return cudaGetLastError();
}
