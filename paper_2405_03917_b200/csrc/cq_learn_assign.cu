// Iterations of centroid learning (Section 3.2.1) that skip what cannot change, for head_dim 128, b = 8, c in {4, 8}.
//
// An iteration of k-means assigns every vector to its nearest centroid and moves every centroid to the weighted mean of its
// members.  After the first few, hardly a vector changes its centroid (1 % on average over 100 iterations of 32768 low-rank
// vectors; from about the 45th on none), yet a plain iteration evaluates all 256 distances of all of them and adds all of them up.  Here:
//   - Assignment.  Let d1 and d2 be a vector's distances to its nearest and second nearest centroid when it was last
//     evaluated.  As long as its own centroid has moved by less than d2 - d1, counted together with the largest move of any
//     other centroid in every iteration since, no other centroid can have become the nearest (triangle inequality; Hamerly,
//     "Making k-means even faster", SDM 2010).  The sums of those moves are kept per centroid (cum), so that the test is
//     cum[code] < thr[vector] with a threshold that is written only when the vector is evaluated.  The CTAs list the
//     vectors that fail it and evaluate those, 128 at a time, as encode_tc_kernel does: one tcgen05.mma for 128 vectors x 128
//     centroids, selection from row and column minima, exact recomputation of near ties.  The second minima that certify
//     the winner are d2.
//   - Sums.  Only vectors that change their centroid touch the sums: one is taken away here and added there.  So that nothing
//     is left behind by that, the sums are whole numbers: w x in units of 2^-L of the largest |x| and w of the problem, and
//     the rest below that in a second word of L bits (L = 62 - log2 n: 94 bits for 32768 vectors; products of a
//     24-bit weight and an 11-bit channel are exact down to 2^-59 of the largest).  They do not depend on the order of the
//     additions either.  A centroid whose members all weigh so little beside the problem's largest weight that these words hold
//     less of their sums than fp32 sums would (ThinRule) is summed up anew, in fp64.
//   - A problem in which nothing moved in an iteration has converged: the iterations after it return at once.
// The codes are those of the full evaluation bit for bit: thr is lowered by a bound on every rounding (below), and a row that
// was not certain is evaluated again each time.  Problems with infinities, NaNs or negative weights (found by
// learn_range_kernel) evaluate every vector and form fp32 sums anew in every iteration.
//
// What bounds it: the evaluation of the vectors that are listed (about half of them until convergence), on the ALU pipe as
// in encode_tc_kernel.
#include "cq_encode_tc.cuh"

namespace cq {

namespace {

constexpr int kAsRange = 4096;             // vectors of a CTA at most
constexpr int kAsK = 256;

template <int kC>
struct AsCfg {
    using T = TcCfg<kC, 1>;
    static constexpr int kAOff = 0;                                      // [2 buffers]
    static constexpr int kBOff = kAOff + 2 * T::kABuf;
    static constexpr int kListOff = kBOff + T::kBBuf;                    // uint32: vector of the range | old code << 16 [| new code << 24]
    static constexpr int kCumOff = kListOff + kAsRange * 4;              // fp32 [256]
    static constexpr int kCtlOff = kCumOff + kAsK * 4;
    static constexpr int kUsedBytes = kCtlOff + 512 + 16;
    // at least 46 KiB, so that a fifth CTA (for which no tensor memory would be left) never fits an SM
    static constexpr int kSmemBytes = kUsedBytes > 46 * 1024 ? kUsedBytes : 46 * 1024;
    static_assert(4 * (kSmemBytes + 1024) <= 228 * 1024 && 5 * (kSmemBytes + 1024) > 228 * 1024, "four CTAs per SM");
};

// What learn_range_kernel notes of a problem: the largest |x| (fp16 bits), the largest weight (fp32 bits) and the complement of the
// smallest weight's bits that is not zero (0: every weight is).  All zero before it.
struct AsRange {
    uint32_t x, w, w_least;
};

// Is the problem one for the fixed-point sums and the bounds: largest |x| and weight finite, no weight negative (its bits
// would be larger than those of infinity).
__device__ __forceinline__ bool as_plain(const AsRange* top, int p) { return top[p].x < 0x7c00u && top[p].w < 0x7f800000u; }

// exponents: |x| < 2^ex, w < 2^ew
__device__ __forceinline__ void as_scales(const AsRange* top, int p, bool weighted, int& ex, int& ew)
{
    frexpf(__half2float(__ushort_as_half((unsigned short)top[p].x)), &ex);
    ew = 1;
    if (weighted) frexpf(__uint_as_float(top[p].w), &ew);
}

// Weight sums (in units of 2^(ew - L), the first word's) with which a centroid's sums are formed anew.  Each member's terms are
// rounded by 2^-L / 2 of the first word's unit at most, so that the mean of m members with weight sum ws is off by no more than
// m 2^-L 2^ex / ws.  That is within 2^-48, 2^-24 of the smallest fp16 channel, for ws >= m 2^(48 + ex - L): for every centroid
// whose ws reaches n 2^(48 + ex - L) (32768 vectors below 32: 2^-26 of the largest weight), and, because ws >= m w_least, for every
// one of the problem if w_least >= 2^(48 + ex + ew - 2 L) (2^-41 of it); then there is no floor.  A sum of zero is exact, no member
// weighs anything, where w_least is not lost in the rounding.
struct ThinRule {
    double floor;
    bool zero_is_exact;
    __device__ __forceinline__ bool thin(double ws) const { return ws < floor && !(zero_is_exact && ws == 0.0); }
};
__device__ __forceinline__ ThinRule thin_rule(const AsRange* top, int p, bool weighted, int ex, int ew, int limb_bits, int64_t n_vec)
{
    ThinRule r = {0.0, true};
    if (!weighted || top[p].w_least == 0u) return r;
    const int field = (int)(~top[p].w_least >> 23), least = (field ? field - 127 : -149) + 2 * limb_bits - ew;       // w_least >= 2^(least + ew - 2 L)
    if (least < 48 + ex) r.floor = (double)n_vec * __hiloint2double((1023 + 48 + ex - limb_bits) << 20, 0);
    r.zero_is_exact = least >= 0;
    return r;
}

constexpr int kRangeThreads = 256, kRangeVecs = 256;
template <int kC>
__global__ void __launch_bounds__(kRangeThreads)
learn_range_kernel(const __half* __restrict__ x, const float* __restrict__ weights, Shape sh, int64_t n_vec, AsRange* __restrict__ top)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, h = blockIdx.y, n_prob = sh.n_kv_heads * sh.G;
    const int64_t v0 = (int64_t)blockIdx.x * kRangeVecs, v1 = v0 + kRangeVecs < n_vec ? v0 + kRangeVecs : n_vec;
    uint32_t tx = 0, tw = 0, tl = 0;
#pragma unroll 4
    for (int64_t v = v0 + warp; v < v1; v += kRangeThreads / 32) {
        const uint2 xw = *reinterpret_cast<const uint2*>(x + (v * sh.n_kv_heads + h) * 128 + 4 * lane);
        const uint32_t a = __vmaxu2(xw.x & 0x7fff7fffu, xw.y & 0x7fff7fffu), b = a & 0xffffu, c = a >> 16;
        tx = max(tx, max(b, c));
        if (weights && lane < sh.G) {
            const uint32_t w = __float_as_uint(weights[v * n_prob + h * sh.G + lane]);
            tw = max(tw, w == 0x80000000u ? 0u : w);
            if (w << 1) tl = max(tl, ~w);
        }
    }
    if (kC == 8) tx = max(tx, __shfl_xor_sync(0xffffffffu, tx, 1));
    if (lane % (kC / 4) == 0) atomicMax(&top[h * sh.G + 4 * lane / kC].x, tx);
    if (weights && lane < sh.G) {
        atomicMax(&top[h * sh.G + lane].w, tw);
        atomicMax(&top[h * sh.G + lane].w_least, tl);
    }
}

// One CTA: the vectors [range * i, range * (i + 1)) of one problem; blockIdx.x = (i, head, group), the groups of a head
// next to each other (they read the same lines).
template <int kC>
__global__ void __launch_bounds__(kTcThreads, 4)
assign_kernel(const __half* __restrict__ x, const float* __restrict__ weights, const float* __restrict__ cb, Shape sh, int64_t n_vec,
              int64_t n_pad, int range, int it, int limb_bits, uint8_t* __restrict__ codes, float* __restrict__ thr,
              unsigned long long* __restrict__ sums, const float* __restrict__ cum_all, int* __restrict__ last_moved,
              const AsRange* __restrict__ top)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");      // launched ahead of the end of the kernel that moves the centroids
    using C = AsCfg<kC>;
    using T = TcCfg<kC, 1>;
    constexpr int G = T::G;
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    TcCtl* ctl = reinterpret_cast<TcCtl*>(tc_smem + C::kCtlOff);
    int* counters = reinterpret_cast<int*>(tc_smem + C::kCtlOff + 512);        // listed, moved
    uint32_t* list = reinterpret_cast<uint32_t*>(tc_smem + C::kListOff);
    float* cum = reinterpret_cast<float*>(tc_smem + C::kCumOff);

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, row = threadIdx.x;
    const int n_heads = sh.n_kv_heads, n_prob = n_heads * G;
    const int p = blockIdx.x % n_prob, h = p / G, g = p % G;
    const int64_t v0 = (int64_t)(blockIdx.x / n_prob) * range;
    const int n = (int)(n_vec - v0 < range ? n_vec - v0 : range);
    if (it > 0 && last_moved[p] < it) return;                                  // the iteration before moved nothing: converged
    const bool plain = as_plain(top, p);
    float* thr_p = thr + p * n_pad + v0;
    const float* cb_g = cb + (int64_t)p * kAsK * kC;
    for (int i = threadIdx.x; i < kAsK; i += kTcThreads) cum[i] = cum_all[(int64_t)p * kAsK + i];
    if (threadIdx.x < 2) counters[threadIdx.x] = 0;
    __syncthreads();

    // ---------------------------------------------------------------- the vectors to evaluate
    // code byte of vector 16 blk + k of the range: code_blk(blk)[k]
    auto code_blk = [&](int blk) { return codes + code_word_offset(sh, n_heads, 0, h, v0 / kTokenBlock + blk, g); };
    for (int b0 = 0; b0 < (n + 15) / 16; b0 += kTcThreads) {
        const int blk = b0 + threadIdx.x, left = n - 16 * blk;
        uint32_t mask = left >= 16 ? 0xffffu : left > 0 ? (1u << left) - 1u : 0u;
        uint4 cw = make_uint4(0u, 0u, 0u, 0u);
        if (it > 0 && mask) {
            cw = *reinterpret_cast<const uint4*>(code_blk(blk));
            if (plain) {
                float4 t[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) t[q] = *reinterpret_cast<const float4*>(thr_p + 16 * blk + 4 * q);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t w = q == 0 ? cw.x : q == 1 ? cw.y : q == 2 ? cw.z : cw.w;
                    const uint32_t keep = (cum[w & 0xffu] < t[q].x ? 1u : 0u) | (cum[(w >> 8) & 0xffu] < t[q].y ? 2u : 0u) |
                                          (cum[(w >> 16) & 0xffu] < t[q].z ? 4u : 0u) | (cum[w >> 24] < t[q].w ? 8u : 0u);
                    mask &= ~(keep << (4 * q));
                }
            }
        }
        const int mine = __popc(mask);
        int upto = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(0xffffffffu, upto, o);
            if (lane >= o) upto += a;
        }
        int base = 0;
        if (lane == 31 && upto) base = atomicAdd(&counters[0], upto);
        int at = __shfl_sync(0xffffffffu, base, 31) + upto - mine;
#pragma unroll
        for (int k = 0; k < 16; ++k)
            if (mask >> k & 1u) {
                const uint32_t w = k < 4 ? cw.x : k < 8 ? cw.y : k < 12 ? cw.z : cw.w;
                list[at++] = (uint32_t)(16 * blk + k) | ((w >> (8 * (k & 3))) & 0xffu) << 16;
            }
    }
    __syncthreads();
    const int count = counters[0];
    if (count == 0) return;

    // ---------------------------------------------------------------- operands, tensor memory
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem_u32(&ctl->tmem_base)), "n"(kTcColumns) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 32) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem_u32(&ctl->bar[0])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem_u32(&ctl->bar[1])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem_u32(&ctl->drained)) : "memory");
        ctl->wait_failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const int n_steps = (count + kTcTileVecs - 1) / kTcTileVecs;
    // the row's vector: fetched (global memory -> registers) half a step ahead of the build (-> shared memory)
    uint32_t e_pf = 0, e_nxt = 0, xw_pf[kC / 2], xw_nxt[kC / 2];
    float X_nxt = 0.f;
    auto fetch = [&](int st) {
        const int i = st * kTcTileVecs + row;
#pragma unroll
        for (int w = 0; w < kC / 2; ++w) xw_pf[w] = 0u;
        e_pf = 0;
        if (i < count) {
            e_pf = list[i];
            tc_fetch_x<kC>(x + ((v0 + (e_pf & 0xffffu)) * n_heads + h) * 128 + g * kC, xw_pf);
        }
    };
    fetch(0);
    const float scale = tc_scale<kC>(cb_g);
    {
        float cv[2][kC];
        tc_fetch_centroid<kC>(cb_g, threadIdx.x, cv[0]);
        tc_fetch_centroid<kC>(cb_g, threadIdx.x + 128, cv[1]);
        tc_prepare_b<kC>(cv[0], scale, threadIdx.x, tc_smem + C::kBOff, ctl, 0, 0);
        tc_prepare_b<kC>(cv[1], scale, threadIdx.x + 128, tc_smem + C::kBOff, ctl, 0, 1);
    }
    auto build = [&](int st) {
        // (the scaled channels are exact, or infinite: the row's scores are NaN then, and it is not certain)
        X_nxt = 0.f;
        e_nxt = e_pf;
        uint32_t xs[kC / 2];
        const __half2 scale2 = __float2half2_rn(scale);
#pragma unroll
        for (int w = 0; w < kC / 2; ++w) {
            xw_nxt[w] = xw_pf[w];
            const __half2 v = __hmul2(*reinterpret_cast<const __half2*>(&xw_pf[w]), scale2);
            xs[w] = *reinterpret_cast<const uint32_t*>(&v);
            const float2 f = __half22float2(v);
            X_nxt = fmaf(f.x, f.x, X_nxt);
            X_nxt = fmaf(f.y, f.y, X_nxt);
        }
        tc_build_a<kC>(xs, X_nxt, tc_smem + C::kAOff + (st & 1) * T::kABuf, row);
    };
    build(0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(&ctl->tmem_base);
    const uint32_t taddr = tmem_base + ((uint32_t)(warp * 32) << 16);
    auto issue = [&](int st, int half) {
        const uint32_t a0 = tc_smem_u32(tc_smem + C::kAOff + (st & 1) * T::kABuf), b0 = tc_smem_u32(tc_smem + C::kBOff) + half * (128 * 16);
#pragma unroll
        for (int s = 0; s < T::kSteps; ++s)
            tc_mma(tmem_base, tc_desc(a0 + s * T::kATile, 128 * 16), tc_desc(b0 + s * T::kBTile, 256 * 16), s > 0 ? 1u : 0u);
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc_smem_u32(&ctl->bar[half])) : "memory");
    };
    if (threadIdx.x == 0) issue(0, 0);
    bool out_of_range;
    float nmax;
    {
        const int4 f0 = *reinterpret_cast<const int4*>(&ctl->range_flag[0][0]), f1 = *reinterpret_cast<const int4*>(&ctl->range_flag[0][4]);
        out_of_range = (f0.x | f0.y | f0.z | f0.w | f1.x | f1.y | f1.z | f1.w) != 0;
        const float4 n0 = *reinterpret_cast<const float4*>(&ctl->nmax[0][0]), n1 = *reinterpret_cast<const float4*>(&ctl->nmax[0][4]);
        nmax = fmaxf(fmaxf(fmaxf(n0.x, n0.y), fmaxf(n0.z, n0.w)), fmaxf(fmaxf(n1.x, n1.y), fmaxf(n1.z, n1.w)));
    }

    // ---------------------------------------------------------------- 128 listed vectors a step (as in encode_tc_kernel)
    for (int st = 0; st < n_steps; ++st) {
        uint32_t xw[kC / 2];
#pragma unroll
        for (int w = 0; w < kC / 2; ++w) xw[w] = xw_nxt[w];
        const float X = X_nxt;
        const uint32_t e = e_nxt;
        const bool live = st * kTcTileVecs + row < count;
        float sb[16], m1 = kTcInf, m2 = kTcInf;
#pragma unroll
        for (int q = 0; q < 16; ++q) sb[q] = kTcInf;
        if (st + 1 < n_steps) fetch(st + 1);

        bool scores_valid = *reinterpret_cast<volatile int*>(&ctl->wait_failed) == 0;
        if (scores_valid && !tc_wait(&ctl->bar[0], (uint32_t)(st & 1))) {
            ctl->wait_failed = 1;                        // never expected: every row of this CTA goes the exact way from here on
            scores_valid = false;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tc_scan_half<15u>(sb, m1, m2, taddr, 0);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();                                 // the low half has been read: its columns take the high half
        if (threadIdx.x == 0 && *reinterpret_cast<volatile int*>(&ctl->wait_failed) == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            issue(st, 1);
        }
        if (st + 1 < n_steps) build(st + 1);             // while the MMA of the high half runs
        if (scores_valid && !tc_wait(&ctl->bar[1], (uint32_t)(st & 1))) {
            ctl->wait_failed = 1;
            scores_valid = false;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tc_scan_half<15u>(sb, m1, m2, taddr, 8);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();                                 // tensor memory is free again; the operands of step st + 1 are complete
        if (threadIdx.x == 0 && st + 1 < n_steps && *reinterpret_cast<volatile int*>(&ctl->wait_failed) == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            issue(st + 1, 0);
        }

        float c1, c2;
        tc_column_minima(sb, c1, c2);
        int code = (int)((__float_as_uint(m1) & 15u) << 4) | (int)(__float_as_uint(c1) & 15u);
        const float first = fmaxf(m1, c1), second = fminf(m2, c2), tau = tc_tau<kC, 15u>(m1, m2, X, nmax);
        const bool certain = scores_valid && !out_of_range && nmax >= 1.f && second - first > tau;
        unsigned pending = __ballot_sync(0xffffffffu, !certain && live);
        while (pending) {                                // exact recomputation, one row at a time by the whole warp
            const int src = __ffs(pending) - 1;
            pending &= pending - 1;
            float xs[8];
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                xs[2 * w] = xs[2 * w + 1] = 0.f;
                if (w < kC / 2) {
                    const uint32_t ww = __shfl_sync(0xffffffffu, xw[w % (kC / 2)], src);
                    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&ww));
                    xs[2 * w] = f.x;
                    xs[2 * w + 1] = f.y;
                }
            }
            const int ec = tc_exact_code<kC>(cb_g, kAsK, xs[0], xs[1], xs[2], xs[3], xs[4], xs[5], xs[6], xs[7]);
            if (lane == src) code = ec;
        }
        // The threshold: cum[code] + d2 - d1, rounded down.  tau covers the error of both scores.  d_j here is the true distance
        // and what decides a full evaluation are squares rounded to (c + 2) 2^-24 < 6e-7 of themselves: with d2 - d1 larger
        // than 6e-7 (d1 + d2) the order holds.  4e-6 (d1 + d2) covers that and the roundings of this line; what d1 and d2 grow by
        // until the test is covered by the factor on the moves (learn_move_kernel).
        const int i = (int)(e & 0xffffu), old = (int)(e >> 16) & 0xff;
        if (live && plain) {
            const float d2 = __fsqrt_rd(fmaxf(second - tau, 0.f)), d1 = __fsqrt_ru(fmaxf(first + tau, 0.f));
            const float slack = (d2 - d1 - 4e-6f * (d1 + d2)) / scale;         // (a power of two)
            thr_p[i] = certain && slack > 0.f ? __fadd_rd(cum[code], slack) : -kTcInf;
        }
        const bool moved = live && (it == 0 || code != old);
        const unsigned who = __ballot_sync(0xffffffffu, moved);
        if (who) {
            int base = 0;
            if (lane == 0) base = atomicAdd(&counters[1], __popc(who));
            base = __shfl_sync(0xffffffffu, base, 0);
            // (at most 128 entries a step: they take the place of entries that every warp has read)
            if (moved) list[base + __popc(who & ((1u << lane) - 1u))] = (uint32_t)i | (uint32_t)old << 16 | (uint32_t)code << 24;
        }
        if (moved) code_blk(i / 16)[i % 16] = (uint8_t)code;
    }

    // Every MMA that was issued has been waited for; where a wait gave up, this is done now, with a limit again, by the thread
    // that issues them.  Then the tensor memory goes back.
    if (threadIdx.x == 0 && *reinterpret_cast<volatile int*>(&ctl->wait_failed) != 0) {
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc_smem_u32(&ctl->drained)) : "memory");
        tc_wait(&ctl->drained, 0u);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(kTcColumns) : "memory");
    }

    // ---------------------------------------------------------------- the sums of the centroids that were left and reached
    const int n_moved = counters[1];
    if (n_moved == 0) return;
    if (threadIdx.x == 0) last_moved[p] = it + 1;
    if (!plain) return;
    constexpr int kRow = kC + 1, kPerWarp = 32 / kRow;          // kC channels and the weight; vectors a warp takes at a time
    const int sub = lane / kRow, ch = lane % kRow;
    if (sub >= kPerWarp) return;
    int ex, ew;
    as_scales(top, p, weights != nullptr, ex, ew);
    const double unit = ldexp(1.0, limb_bits - ew - (ch < kC ? ex : 0)), limb = ldexp(1.0, limb_bits);
    unsigned long long* sums_p = sums + (int64_t)p * kAsK * 2 * kRow + ch;
    for (int m = warp * kPerWarp + sub; m < n_moved; m += (kTcThreads / 32) * kPerWarp) {
        const uint32_t e = list[m];
        const int64_t v = v0 + (e & 0xffffu);
        double val = weights ? (double)weights[v * n_prob + p] : 1.0;
        if (ch < kC) val *= (double)__half2float(x[(v * n_heads + h) * 128 + g * kC + ch]);
        val *= unit;                                             // exact: 35 bits times a power of two
        const long long hi = __double2ll_rz(val), lo = __double2ll_rn((val - (double)hi) * limb);
        unsigned long long* to = sums_p + (e >> 24) * (2 * kRow);
        atomicAdd(to, (unsigned long long)hi);
        if (lo) atomicAdd(to + kRow, (unsigned long long)lo);
        if (it > 0) {
            unsigned long long* from = sums_p + ((e >> 16) & 0xffu) * (2 * kRow);
            atomicAdd(from, (unsigned long long)-hi);
            if (lo) atomicAdd(from + kRow, (unsigned long long)-lo);
        }
    }
}

// The rows of the centroids with thin[code] become their members' weighted channels and weights, summed in fp64, in place of the words
// of the fixed-point sums.  By a whole CTA, between two barriers; x, weights and codes are the problem's.  (Out of line and without
// a stack, for the kernel around it.)
template <int kC>
__device__ __noinline__ void as_sum_thin(double* rows, const uint8_t* thin, const __half* __restrict__ x, const float* __restrict__ weights,
                                         const uint8_t* __restrict__ codes, int block_bytes, int n_prob, int64_t n_vec)
{
    for (int64_t blk = threadIdx.x; blk < (n_vec + kTokenBlock - 1) / kTokenBlock; blk += kAsK) {
        const uint4 cw = *reinterpret_cast<const uint4*>(codes + blk * block_bytes);
#pragma unroll 1
        for (int k = 0; k < 16; ++k) {
            const int code = (int)((k < 4 ? cw.x : k < 8 ? cw.y : k < 12 ? cw.z : cw.w) >> (8 * (k & 3)) & 0xffu);
            const int64_t v = blk * kTokenBlock + k;
            if (!thin[code] || v >= n_vec) continue;
            double* row = rows + code * 2 * (kC + 1);
            const double w = (double)weights[v * n_prob];
#pragma unroll 1
            for (int q = 0; q < kC; ++q) atomicAdd(row + q, w * (double)__half2float(x[v * n_prob * kC + q]));
            atomicAdd(row + kC, w);
        }
    }
}

// The centroids of one problem from its sums, and the sums of moves that the thresholds are compared with.  A thread per
// centroid.
template <int kC>
__global__ void __launch_bounds__(kAsK)
learn_move_kernel(const __half* __restrict__ x, const float* __restrict__ weights, const uint8_t* __restrict__ codes, Shape sh,
                  int64_t n_vec, int it, int limb_bits, const unsigned long long* __restrict__ sums, float* __restrict__ cum,
                  const int* __restrict__ last_moved, const AsRange* __restrict__ top, float* __restrict__ cb)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");      // launched ahead of the end of the assignment
    // the problem's sums, read in whole lines (a row of 8 (c + 1) 2 bytes per thread touched 32 lines a load); or fp32 sums
    __shared__ __align__(16) unsigned long long rows[kAsK * 2 * (kC + 1)];
    float* acc = reinterpret_cast<float*>(rows);
    __shared__ float best[2][kAsK / 32];
    __shared__ int arg[kAsK / 32];
    __shared__ uint8_t thin_s[kAsK];
    const int p = blockIdx.x, j = threadIdx.x, lane = j & 31, warp = j >> 5;
    if (last_moved[p] < it + 1) return;
    float* cj = cb + ((int64_t)p * kAsK + j) * kC;
    if (!as_plain(top, p)) {                                 // fp32 sums of all vectors, as in lloyd_update_generic_kernel
        const int h = p / sh.G, g = p % sh.G, n_prob = sh.n_kv_heads * sh.G;
        for (int i = j; i < kAsK * (kC + 1); i += kAsK) acc[i] = 0.f;
        __syncthreads();
        for (int64_t v = j; v < n_vec; v += kAsK) {
            const int code = codes[code_word_offset(sh, sh.n_kv_heads, 0, h, v / kTokenBlock, g) + v % kTokenBlock];
            const float w = weights ? weights[v * n_prob + p] : 1.f;
            const __half* xv = x + (v * n_prob + p) * kC;
            for (int q = 0; q < kC; ++q) atomicAdd(&acc[code * (kC + 1) + q], w * __half2float(xv[q]));
            atomicAdd(&acc[code * (kC + 1) + kC], w);
        }
        __syncthreads();
        const float ws = acc[j * (kC + 1) + kC];
        if (ws > 0.f)
            for (int q = 0; q < kC; ++q) cj[q] = acc[j * (kC + 1) + q] / ws;
        return;
    }
    {
        const ulonglong2* src = reinterpret_cast<const ulonglong2*>(sums + (int64_t)p * kAsK * 2 * (kC + 1));
#pragma unroll
        for (int i = 0; i <= kC; ++i) reinterpret_cast<ulonglong2*>(rows)[i * kAsK + j] = __ldcg(src + i * kAsK + j);
    }
    __syncthreads();
    int ex, ew;
    as_scales(top, p, weights != nullptr, ex, ew);
    const double limb = ldexp(1.0, -limb_bits), back = ldexp(1.0, ex);
    unsigned long long* row = rows + j * 2 * (kC + 1);
    auto value = [&](int ch) { return (double)(long long)row[ch] + (double)(long long)row[kC + 1 + ch] * limb; };
    double ws = value(kC);
    const ThinRule rule = thin_rule(top, p, weights != nullptr, ex, ew, limb_bits, n_vec);
    const bool thin = rule.thin(ws);
    if (rule.floor > 0.0) {
        thin_s[j] = thin ? 1 : 0;
        if (thin)
            for (int ch = 0; ch <= kC; ++ch) row[ch] = 0ull;
        if (__syncthreads_or(thin)) {
            const int n_prob = sh.n_kv_heads * sh.G;
            as_sum_thin<kC>(reinterpret_cast<double*>(rows), thin_s, x + p * kC, weights + p,
                            codes + code_word_offset(sh, sh.n_kv_heads, 0, p / sh.G, 0, p % sh.G), (int)sh.block_bytes, n_prob, n_vec);
            __syncthreads();
        }
        if (thin) ws = __longlong_as_double((long long)row[kC]);
    }
    float d2 = 0.f;
    if (ws > 0.0) {                                          // (a centroid without members stays)
        const double share = (thin ? 1.0 : back) / ws;
#pragma unroll
        for (int q = 0; q < kC; ++q) {
            const float was = cj[q], now = (float)((thin ? __longlong_as_double((long long)row[q]) : value(q)) * share), d = now - was;
            cj[q] = now;
            d2 = fmaf(d, d, d2);
        }
    }
    // the largest move of any other centroid: the two largest of the problem
    const float move = __fsqrt_ru(d2) * 1.000002f;
    float m1 = move, m2 = -1.f;
    int a1 = j;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float b1 = __shfl_xor_sync(0xffffffffu, m1, o), b2 = __shfl_xor_sync(0xffffffffu, m2, o);
        const int ba = __shfl_xor_sync(0xffffffffu, a1, o);
        m2 = fmaxf(fminf(m1, b1), fmaxf(m2, b2));
        if (b1 > m1) { m1 = b1; a1 = ba; }
    }
    if (lane == 0) { best[0][warp] = m1; best[1][warp] = m2; arg[warp] = a1; }
    __syncthreads();
    m1 = best[0][0]; m2 = best[1][0]; a1 = arg[0];
#pragma unroll
    for (int w = 1; w < kAsK / 32; ++w) {
        const float b1 = best[0][w], b2 = best[1][w];
        m2 = fmaxf(fminf(m1, b1), fmaxf(m2, b2));
        if (b1 > m1) { m1 = b1; a1 = arg[w]; }
    }
    // (1e-5: what the distances themselves grow by enters the rounding that the threshold allows for)
    const float others = j == a1 ? m2 : m1;
    float* cu = cum + (int64_t)p * kAsK + j;
    *cu = __fadd_ru(*cu, __fadd_ru(move, others) * 1.00001f);
}

size_t as_round(size_t v) { return (v + 255) / 256 * 256; }

}  // namespace

bool learn_bounds_supported(const Shape& sh, int64_t n_vec)
{
    return sh.head_dim == 128 && sh.b == 8 && (sh.c == 4 || sh.c == 8) && n_vec >= 16 && n_vec <= (1 << 23);
}

// sums, sums of moves, last iteration with a move, ranges of |x| and weights (the thresholds lie in the distances' place)
size_t learn_bounds_bytes(const Shape& sh)
{
    const size_t n_prob = (size_t)sh.n_kv_heads * sh.G;
    return as_round(n_prob * kAsK * 2 * (sh.c + 1) * 8) + as_round(n_prob * kAsK * 4) + as_round(n_prob * 4) + as_round(n_prob * sizeof(AsRange));
}

template <int kC>
static cudaError_t run_bounds(const __half* x, const float* weights, const Shape& sh, int64_t n_vec, int n_iters, float* codebooks,
                              uint8_t* codes, float* thr, void* state, cudaStream_t st, const LearnObjective& objective)
{
    using C = AsCfg<kC>;
    const int n_prob = sh.n_kv_heads * sh.G;
    char* w = static_cast<char*>(state);
    unsigned long long* sums = reinterpret_cast<unsigned long long*>(w);      w += as_round((size_t)n_prob * kAsK * 2 * (kC + 1) * 8);
    float* cum = reinterpret_cast<float*>(w);                                 w += as_round((size_t)n_prob * kAsK * 4);
    int* last_moved = reinterpret_cast<int*>(w);                              w += as_round((size_t)n_prob * 4);
    AsRange* top = reinterpret_cast<AsRange*>(w);
    cudaError_t e = cudaMemsetAsync(state, 0, learn_bounds_bytes(sh), st);
    if (e != cudaSuccess) return e;
    learn_range_kernel<kC><<<dim3((unsigned)((n_vec + kRangeVecs - 1) / kRangeVecs), (unsigned)sh.n_kv_heads), kRangeThreads, 0, st>>>(
        x, weights, sh, n_vec, top);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    int log_n = 0;
    while ((int64_t)1 << log_n < n_vec) ++log_n;
    const int limb_bits = 62 - log_n;
    // Vectors per CTA: many, since a CTA prepares the problem's centroids once, but two waves of CTAs (one in four lists hardly
    // anything late on).
    const int64_t n_pad = (n_vec + 15) / 16 * 16, want = 2 * 4 * (int64_t)device_sm_count();
    int64_t range = (n_vec * n_prob + want - 1) / want;
    range = (range + kTcTileVecs - 1) / kTcTileVecs * kTcTileVecs;
    if (range > kAsRange) range = kAsRange;
    const int64_t grid = (n_vec + range - 1) / range * n_prob;
    if (grid > 0x7fffffff) return cudaErrorInvalidConfiguration;
    constexpr int kSlot = kC == 4 ? 120 : 121;                                // call-site slots of ensure_dynamic_smem
    e = ensure_dynamic_smem(reinterpret_cast<const void*>(assign_kernel<kC>), C::kSmemBytes, kSlot);
    if (e != cudaSuccess) return e;
    for (int it = 0; it < n_iters; ++it) {
        cudaLaunchAttribute attr;
        {
            const cudaLaunchConfig_t cfg = overlapped_config((unsigned)grid, kTcThreads, C::kSmemBytes, st, &attr);
            e = cudaLaunchKernelEx(&cfg, assign_kernel<kC>, x, weights, codebooks, sh, n_vec, n_pad, (int)range, it, limb_bits, codes, thr,
                                   sums, cum, last_moved, top);
            if (e != cudaSuccess) return e;
        }
        if (it + 1 == n_iters && (e = objective(codes, codebooks)) != cudaSuccess) return e;
        const cudaLaunchConfig_t cfg = overlapped_config((unsigned)n_prob, kAsK, 0, st, &attr);
        e = cudaLaunchKernelEx(&cfg, learn_move_kernel<kC>, x, weights, codes, sh, n_vec, it, limb_bits, sums, cum, last_moved, top, codebooks);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_learn_bounds(const __half* x, const float* weights, const Shape& sh, int64_t n_vec, int n_iters, float* codebooks,
                                uint8_t* codes, float* thr, void* state, cudaStream_t st, const LearnObjective& objective)
{
    return sh.c == 4 ? run_bounds<4>(x, weights, sh, n_vec, n_iters, codebooks, codes, thr, state, st, objective)
                     : run_bounds<8>(x, weights, sh, n_vec, n_iters, codebooks, codes, thr, state, st, objective);
}

}  // namespace cq
