// Range aggregation, top-k feature selection and table construction
// (paper Section 3 "Selecting High Precision Features"; k = floor(E/64) in Section 4).
#include "tpq_internal.h"

namespace {

// R^(i)_j = 2 max(-m, M); Rbar_j = sum_i R^(i)_j (binary32, devices ascending);
// step s = R/(2^bits - 1) (R/15 for Int4) floored at 2^-23 and its reciprocal (IEEE division, no fast-math).
__global__ void __launch_bounds__(256) ranges_kernel(const float *__restrict__ m, const float *__restrict__ M, int N,
                                                     int E, float levels, float *__restrict__ R,
                                                     float *__restrict__ Rbar, float *__restrict__ s,
                                                     float *__restrict__ inv_s)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= E) return;
    float acc = 0.0f;
    for (int i = 0; i < N; ++i) {
        const size_t o = (size_t)i * E + j;
        const float a = -m[o], b = M[o];
        const float A = (a > b) ? a : b;
        const float r = __fmul_rn(2.0f, A);
        R[o] = r;
        acc = (i == 0) ? r : __fadd_rn(acc, r);
        float sv = __fdiv_rn(r, levels);
        if (!(sv >= 1.1920928955078125e-07f)) sv = 1.1920928955078125e-07f;
        s[o] = sv;
        inv_s[o] = __fdiv_rn(1.0f, sv);
    }
    Rbar[j] = acc;
}

// Feature j is selected iff fewer than k features beat it, where a beats j when
// Rbar_a > Rbar_j, or Rbar_a == Rbar_j and a < j.  O(E^2) comparisons, a warp per feature: its lanes compare side by
// side, four values per load (Rbar is a few tens of KB, so the loads hit L1).  (One thread per feature, the values
// through shared memory, left all but 18 SMs idle: 68 us at E = 4608.  With this kernel and the two below
// the whole selection call takes 61 instead of 135 us at 8 x 4608, 82 instead of 227 us at 16 x 8192.)
constexpr int TK_WARPS = 8;

__global__ void __launch_bounds__(32 * TK_WARPS) topk_flags_kernel(const float *__restrict__ Rbar, int E, int k,
                                                                   uint8_t *__restrict__ flag)
{
    const int j = blockIdx.x * TK_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (j >= E) return;
    const float mine = __ldg(Rbar + j);
    int beats = 0;
    const int E4 = E >> 2;
#pragma unroll 4
    for (int q = lane; q < E4; q += 32) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(Rbar) + q);
        const int a = 4 * q;
        beats += (v.x > mine || (v.x == mine && a < j)) + (v.y > mine || (v.y == mine && a + 1 < j)) +
                 (v.z > mine || (v.z == mine && a + 2 < j)) + (v.w > mine || (v.w == mine && a + 3 < j));
    }
    if (lane < (E & 3)) {
        const int a = 4 * E4 + lane;
        const float v = __ldg(Rbar + a);
        beats += v > mine || (v == mine && a < j);
    }
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

// Per feature, over the whole GPU: slot order, per-feature slots, the dequantiser's zeroed-step and slot-order step
// copies and the per-8-feature group descriptors.  (As loops of the scan's one block these N*E-long copies took most of
// its 35 us at 8 x 4608.)
__global__ void __launch_bounds__(256) tables_kernel(tpq_tables t, int N, int E, int k)
{
    const int j = blockIdx.x * 256 + threadIdx.x;
    if (j >= E) return;
    const int L = E - k, f = t.flag[j], pre = t.hpre[j];
    const int m = L < E ? t.hpre[L] : 0;
    const int src = j < L ? (f ? t.filler[pre] : j) : -1;  // feature held by slot j
    if (j < L) t.lp_idx[j] = src;
#pragma unroll 4
    for (int i = 0; i < N; ++i) {
        const size_t row = (size_t)i * E;
        t.s_k[row + j] = f ? 0.0f : t.s[row + j];
        t.s_slot[row + j] = src >= 0 ? t.s[row + src] : 0.0f;
    }
    t.pos[j] = f ? -(pre + 1) : j < L ? j : t.hole[(j - L) - (pre - m)];
    if ((j & 7) == 0) {
        uint32_t mask = 0;
        for (int n = 0; n < 8; ++n)
            if (j + n < E && t.flag[j + n]) mask |= 1u << n;
        t.grp[j >> 3] = ((uint32_t)pre << 8) | mask;
    }
}

}  // namespace

cudaError_t tpq_launch_ranges(const tpq_tables &t, int N, int E, int bits, cudaStream_t st, int64_t *launches)
{
    ranges_kernel<<<(E + 255) / 256, 256, 0, st>>>(t.m, t.M, N, E, (float)((1 << bits) - 1), t.R, t.Rbar, t.s, t.inv_s);
    ++*launches;
    return cudaGetLastError();
}

cudaError_t tpq_launch_topk_flags(const tpq_tables &t, int E, int k, cudaStream_t st, int64_t *launches)
{
    topk_flags_kernel<<<(E + TK_WARPS - 1) / TK_WARPS, 32 * TK_WARPS, 0, st>>>(t.Rbar, E, k, t.flag);
    ++*launches;
    return cudaGetLastError();
}

cudaError_t tpq_launch_tables(const tpq_tables &t, int N, int E, int k, cudaStream_t st, int64_t *launches)
{
    scan_kernel<<<1, 1024, 0, st>>>(t, E, k);
    ++*launches;
    tables_kernel<<<(E + 255) / 256, 256, 0, st>>>(t, N, E, k);
    ++*launches;
    return cudaGetLastError();
}
