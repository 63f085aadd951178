// CQ encode of a few vectors per head: the device code of encode_few_kernel and of the append of a decode step.
#pragma once

#include "cq_common.cuh"

namespace cq {

namespace {

// Few vectors per head and 256 centroids.  A warp holds the centroids of one (head, group), eight per lane, in registers and
// takes its share of the vectors past them.  Distances are the direct form sum (x - C)^2 in fp32 in the order of the
// generic kernel, lowest index on ties.  Issue slots are what it takes (c multiply-adds and subtractions per centroid);
// with a centroid per thread and the argmin over the eight warps of a CTA the reductions were a third of them: 30 vectors x
// 40 heads of CQ-4c8b, key and value, 18.1 -> 14.2 us (where the CTA is the better form all the same: few_by_cta).
constexpr int kFewThreads = 256;
constexpr int kFewVecs = 16;              // vectors a warp takes at most

// Vectors a warp takes: as few as one wave of CTAs allows (sixteen warps an SM; key and value counted): 16 vectors of one
// head, CQ-4c8b: 3.1 us, 4.8 with 16 to a warp.  Units of work: head, group, share of the vectors; one per warp.
constexpr int kFewWarpsPerSm = 16;
inline int few_share(const Shape& sh, int n_vec, int warps_per_sm = kFewWarpsPerSm)
{
    int share = 1;
    while (share < kFewVecs && 2 * (int64_t)sh.n_kv_heads * sh.G * ((n_vec + share - 1) / share) > warps_per_sm * (int64_t)device_sm_count()) ++share;
    return share;
}
inline int64_t few_ctas(const Shape& sh, int n_vec, int share)
{
    return ((int64_t)sh.n_kv_heads * sh.G * ((n_vec + share - 1) / share) + kFewThreads / 32 - 1) / (kFewThreads / 32);
}

template <int kC>
__device__ __forceinline__ void encode_few(const __half* __restrict__ x, const float* __restrict__ cb, const int32_t* __restrict__ seq_offsets,
                                           const Shape& sh, int cta, int n_vec, int share, int n_tokens, int64_t token_offset,
                                           uint8_t* __restrict__ codes, bool clamp_offsets)
{
    const int lane = threadIdx.x & 31;
    const int shares = (n_vec + share - 1) / share, n_heads = sh.n_kv_heads;
    const int64_t unit = (int64_t)cta * (kFewThreads / 32) + (threadIdx.x >> 5);
    const int64_t hg = unit / shares;
    const int h = (int)(hg / sh.G), g = (int)(hg % sh.G);
    if (h >= n_heads) return;
    const int v0 = (int)(unit % shares) * share;
    const int nv = n_vec - v0 < share ? n_vec - v0 : share;          // (share <= 32: lane v keeps the result of vector v)
    int mine = 0;                              // lane v keeps the code of vector v
    float cv[8][kC];
    const float* src = cb + (hg * 256 + lane) * kC;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        if (kC == 2) {
            const float2 a = *reinterpret_cast<const float2*>(src + t * 32 * kC);
            cv[t][0] = a.x; cv[t][1 % kC] = a.y;
        } else {
#pragma unroll
            for (int w = 0; w < kC; w += 4) {
                const float4 a = *reinterpret_cast<const float4*>(src + t * 32 * kC + w);
                cv[t][w] = a.x; cv[t][(w + 1) % kC] = a.y; cv[t][(w + 2) % kC] = a.z; cv[t][(w + 3) % kC] = a.w;
            }
        }
    }
    const __half* xp = x + ((int64_t)v0 * n_heads + h) * sh.head_dim + g * kC;
    const int64_t step = (int64_t)n_heads * sh.head_dim;
    __half next[kC];
#pragma unroll
    for (int e = 0; e < kC; ++e) next[e] = nv > 0 ? xp[e] : __float2half(0.f);
    for (int v = 0; v < nv; ++v) {
        float xv[kC];
#pragma unroll
        for (int e = 0; e < kC; ++e) xv[e] = __half2float(next[e]);
        if (v + 1 < nv)
#pragma unroll
            for (int e = 0; e < kC; ++e) next[e] = xp[(v + 1) * step + e];
        float best = __builtin_huge_valf();
        int arg = 0;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            float d = 0.f;
#pragma unroll
            for (int e = 0; e < kC; ++e) {
                const float diff = xv[e] - cv[t][e];
                d = fmaf(diff, diff, d);
            }
            if (d < best) { best = d; arg = t * 32 + lane; }      // ascending: strict < keeps the lowest index
        }
        // (distances are not negative: their bits order as they do)
        const unsigned db = __float_as_uint(best), dm = __reduce_min_sync(0xffffffffu, db);
        const unsigned am = __reduce_min_sync(0xffffffffu, db == dm ? (unsigned)arg : 0xffffffffu);
        if (lane == v) mine = (int)am;
    }
    if (lane >= nv) return;
    const int v = v0 + lane, s = v / n_tokens, i = v - s * n_tokens;
    int off = seq_offsets ? seq_offsets[s] : 0;
    if (clamp_offsets && off < 0) off = 0;
    const int64_t pos = token_offset + off + i;
    if (pos < 0 || pos >= sh.max_tokens) return;
    codes[code_word_offset(sh, n_heads, s, h, pos / kTokenBlock, g) + pos % kTokenBlock] = (uint8_t)mine;
}

}  // namespace

}  // namespace cq
