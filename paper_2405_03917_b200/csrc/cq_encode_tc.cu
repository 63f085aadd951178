// Bulk encode on the fifth-generation tensor cores (tcgen05, accumulators in tensor memory) for
// head_dim 128, b in {8, 9, 10}, c in {2, 4, 8}.
//
// CQ encode (Section 3.2 of the paper, the map CQ(.) of Eq. 5): every group of c contiguous
// channels of a vector is replaced by the index of its nearest centroid in L2 distance, lowest
// index on exact ties.
//
// Arithmetic: that of encode_tuned_kernel.  For 128 vectors x 128 centroids of one group ONE
// tcgen05.mma (M = 128, N = 128, K = 16; two of them, accumulating, for c = 8) evaluates
//     d_j ~ ||x_g||^2 - 2 <x_g, C_j> + ||C_j||^2
// with the fp32 centroids and norms carried as sums of three fp16 terms, so that every product is
// exact and only the fp32 accumulation rounds.  fp16 ends at 2^-24: vectors and centroids of a group
// are first scaled by a power of two (tc_scale), so that the terms are as good for channels of
// standard deviation 0.001 as for channels of standard deviation 1.  K slots, in pairs:
//     c = 2   A: x | x | x | (1,1) | (X_hi,X_lo) | (1,0) | 0 | 0
//             B: t0 | t1 | t2 | (N_hi,N_lo) | (1,1) | (N_lo2,0) | 0 | 0        (-2C = t0 + t1 + t2)
//     c = 4   A: x x | x x | x x | (1,1) | (X_hi,X_lo)      B: t0 t0 | t1 t1 | t2 t2 | (N_hi,N_lo) | (1,1)
//     c = 8   two K steps: (x x x x | x x x x) against (t0 | t1), then (x x x x | (1,1), X, (1,0), 0)
//             against (t2 | N, (1,1), (N_lo2,0), 0)
// What differs is where the scores go.  The accumulator tile lives in tensor memory, row i in
// lane i, and a thread reads the scores of ITS row with tcgen05.ld: no accumulator registers to
// clear, no B fragments to fetch in the selecting warps, no quad to merge.  The 256 scores of a
// (vector, group) are a 16 x 16 grid, and a thread keeps the minimum of every row and of every
// column: 1.25 operations per score, no index packed into it.  The row and the column with the smallest minima name
// the winner, and whatever else there is lies in another row or in another column, so the second
// smallest minima bound it from below.  The winner is accepted if that bound is farther away than a
// bound on the evaluation error; otherwise (near-ties, ties, codebooks fp16 cannot carry) the warp
// recomputes that row over all centroids exactly: sum (x - C)^2 in fp32, lowest index on ties.
// (Before, the winning column's 16 centroids were evaluated exactly from shared memory: at c = 8 the bank
// conflicts of those reads kept the shared-memory pipe 74 % busy.  8192 vectors x 32 heads: c = 8
// 350 -> 215 us.)  More than 256 centroids (b = 9, 10) come in chunks of 256 whose operands all
// stay in shared memory while a row tile passes them; the grid then has 32 or 64 rows.  (CQ-8c10b,
// 32768 vectors x 8 heads: 3.1 -> 1.13 ms against the mma.sync kernel.)
//
// A CTA is one tile of 128 vectors of one head: 4 warps, warp w owning the tensor memory lanes
// 32 w ... 32 w + 31, and 128 tensor-memory columns, so that four CTAs (fewer for wide codes, whose
// operands take more shared memory) live on an SM and fill each other's waits.  The accumulator is
// therefore 128 x 128: the scores of a step arrive in two halves (centroids 0-127, then 128-255)
// through the same columns, and the operand preparation and the row finishing are placed behind
// the MMA issues.  A CTA takes up to eight row tiles through every group before it moves to the
// next group, so a group's centroids are prepared once per up to 1024 vectors.
#include "cq_encode_tc.cuh"

namespace cq {

namespace {

// One step = one row tile (128 vectors) against one chunk of 256 centroids of a group.  A CTA takes 2^log_rt row tiles
// through its groups, all chunks of a group per row tile; blockIdx.x = (block of row tiles, head, group split).
template <int kC, int kChunks>
__global__ void __launch_bounds__(kTcThreads, TcCfg<kC, kChunks>::kCtasPerSm)
encode_tc_kernel(const __half* __restrict__ x1, const float* __restrict__ cb1, const int32_t* __restrict__ seq_offsets,
                 Shape sh, int64_t n_tokens, int64_t token_offset, uint8_t* __restrict__ codes1, int groups_per_cta, int log_rt,
                 const __half* __restrict__ x2, const float* __restrict__ cb2, uint8_t* __restrict__ codes2)
{
    // Launched ahead of the end of the kernel before it.  It lets nothing go ahead itself: what follows gains nothing from waiting on the
    // SMs, and an attention whose CTAs come in beside these loses.  us, let ahead / not: step of 64 x 80 tokens, 40 heads of CQ-8c10b
    // 346.8 / 340.4, of 40 x 2000, 32 heads 211.1 / 209.4; encode of 512 tokens, 8 heads of CQ-8c8b, and prefill 68.5 / 64.5; encodes back to
    // back level.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const __half* x = blockIdx.y ? x2 : x1;
    const float* cb = blockIdx.y ? cb2 : cb1;
    uint8_t* codes = blockIdx.y ? codes2 : codes1;
    using C = TcCfg<kC, kChunks>;
    constexpr int G = C::G;
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    TcCtl* ctl = reinterpret_cast<TcCtl*>(tc_smem + C::kCtlOff);

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row = threadIdx.x;                         // row within the tile = tensor memory lane
    const int n_heads = sh.n_kv_heads;
    const int64_t n_vec = sh.n_seq * n_tokens;

    const int n_gsplit = (G + groups_per_cta - 1) / groups_per_cta;
    const int gs = blockIdx.x % n_gsplit;
    const int h = (blockIdx.x / n_gsplit) % n_heads;
    const int64_t tile_block = blockIdx.x / (n_gsplit * n_heads);
    const int g_begin = gs * groups_per_cta;
    const int g_end = g_begin + groups_per_cta < G ? g_begin + groups_per_cta : G;
    const int rt_mask = (1 << log_rt) - 1;
    // step st: row step st / kChunks (group g_begin + (rs >> log_rt), row tile rs & rt_mask), chunk st % kChunks
    const int n_steps = ((g_end - g_begin) << log_rt) * kChunks;

    // tensor memory (warp 0 allocates the CTA's columns and frees them at the end), the MMA barriers
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
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(&ctl->tmem_base);
    const uint32_t taddr = tmem_base + ((uint32_t)(warp * 32) << 16);

    auto a_buf = [&](int rs) { return tc_smem + C::kAOff + (rs & 1) * C::kABuf; };
    auto slot_of = [&](int st) { return kChunks == 1 ? (st >> log_rt) & 1 : st % kChunks; };
    auto b_buf = [&](int slot) { return tc_smem + C::kBOff + slot * C::kBBuf; };
    // Where the code of group 0 of this thread's row of row tile r goes (the low byte of group g follows kTokenBlock * g
    // bytes on): offsets[r * kTcThreads], worked out once; -1: no position in the cache, -2: no such vector.
    int64_t* offsets = reinterpret_cast<int64_t*>(tc_smem + C::kRowOff) + threadIdx.x;
    const int64_t v_first = tile_block * (rt_mask + 1) * kTcTileVecs + row;
    for (int r = 0; r <= rt_mask; ++r) {
        const int64_t v = v_first + r * kTcTileVecs;
        int64_t off = -2;
        if (v < n_vec) {
            const int64_t s = v / n_tokens, i = v % n_tokens;
            const int64_t pos = token_offset + (seq_offsets ? seq_offsets[s] : 0) + i;
            off = pos >= 0 && pos < sh.max_tokens ? code_word_offset(sh, n_heads, s, h, pos / kTokenBlock, 0) + pos % kTokenBlock : -1;
        }
        offsets[r * kTcThreads] = off;                   // read back by this thread only
    }

    // The vector's words travel global memory -> registers (fetch, half a step ahead) -> shared memory (build).
    uint32_t xw_pf[kC / 2];
    auto fetch = [&](int rs) {
        const int64_t v = v_first + (rs & rt_mask) * kTcTileVecs;
#pragma unroll
        for (int w = 0; w < kC / 2; ++w) xw_pf[w] = 0u;
        if (v < n_vec) tc_fetch_x<kC>(x + (v * n_heads + h) * 128 + (g_begin + (rs >> log_rt)) * kC, xw_pf);
    };
    uint32_t xw_nxt[kC / 2];
    float X_nxt = 0.f, scale = 1.f;                      // squared norm of the scaled vector; scale of the group built last
    // what step st needs and its predecessor has not left: the chunk's centroids (first row tile of a group), the row
    // tile's vectors (first chunk)
    auto build = [&](int st) {
        const int rs = st / kChunks, ch = st % kChunks, slot = slot_of(st);
        if ((rs & rt_mask) == 0) {                       // centroids threadIdx.x and threadIdx.x + 128 of the chunk
            const float* cb_g = cb + (((int64_t)h * G + g_begin + (rs >> log_rt)) * kChunks + ch) * 256 * kC;
            if (ch == 0) scale = tc_scale<kC>(cb_g);
            float cv[2][kC];
            tc_fetch_centroid<kC>(cb_g, threadIdx.x, cv[0]);
            tc_fetch_centroid<kC>(cb_g, threadIdx.x + 128, cv[1]);
            tc_prepare_b<kC>(cv[0], scale, threadIdx.x, b_buf(slot), ctl, slot, 0);
            tc_prepare_b<kC>(cv[1], scale, threadIdx.x + 128, b_buf(slot), ctl, slot, 1);
        }
        if (ch != 0) return;
        // (the scaled channels are exact, or infinite: the row's scores are NaN then, and it is not certain)
        X_nxt = 0.f;
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
        tc_build_a<kC>(xs, X_nxt, a_buf(rs), row);
    };
    // the MMA of one half of step st (half 1 = centroids 128 ... 255), then the commit that arrives on that half's
    // barrier when it is done
    auto issue = [&](int st, int half) {
        const uint32_t a0 = tc_smem_u32(a_buf(st / kChunks)), b0 = tc_smem_u32(b_buf(slot_of(st))) + half * (128 * 16);
#pragma unroll
        for (int s = 0; s < C::kSteps; ++s)
            tc_mma(tmem_base, tc_desc(a0 + s * C::kATile, 128 * 16), tc_desc(b0 + s * C::kBTile, 256 * 16), s > 0 ? 1u : 0u);
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc_smem_u32(&ctl->bar[half])) : "memory");
    };

    // Selection state of this thread's row: minima over the columns of the 16-wide grid of scores (centroid index mod
    // 16), and the smallest and second smallest minimum over its rows (index / 16, carried in the low mantissa bits)
    constexpr uint32_t kRowBits = kChunks == 1 ? 15u : 63u;
    float sb[16], m1 = kTcInf, m2 = kTcInf, nmax = 0.f;
    bool out_of_range = false, scores_valid = true;
    auto scan_half = [&](int row0) { tc_scan_half<kRowBits>(sb, m1, m2, taddr, row0); };

    fetch(0);
    build(0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        issue(0, 0);
    }

    uint32_t xw[kC / 2];
    float X = 0.f;
    for (int st = 0; st < n_steps; ++st) {
        const int rs = st / kChunks, ch = st % kChunks, slot = slot_of(st);
        const int g = g_begin + (rs >> log_rt);
        if (ch == 0) {
#pragma unroll
            for (int w = 0; w < kC / 2; ++w) xw[w] = xw_nxt[w];
            X = X_nxt;
#pragma unroll
            for (int q = 0; q < 16; ++q) sb[q] = kTcInf;
            m1 = m2 = kTcInf;
            nmax = 0.f;
            out_of_range = false;
            scores_valid = true;
        }
        if (ch == kChunks - 1 && st + 1 < n_steps) fetch(rs + 1);

        scores_valid = scores_valid && *reinterpret_cast<volatile int*>(&ctl->wait_failed) == 0;
        if (scores_valid && !tc_wait(&ctl->bar[0], (uint32_t)(st & 1))) {
            ctl->wait_failed = 1;                        // never expected: every row of this CTA goes the exact way from here on
            scores_valid = false;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        scan_half(ch * 16);
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
        scan_half(ch * 16 + 8);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();                                 // tensor memory is free again; the operands of step st + 1 are complete
        if (threadIdx.x == 0 && st + 1 < n_steps && *reinterpret_cast<volatile int*>(&ctl->wait_failed) == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            issue(st + 1, 0);
        }

        // control words of this step's chunk
        {
            const int4 f0 = *reinterpret_cast<const int4*>(&ctl->range_flag[slot][0]);
            const int4 f1 = *reinterpret_cast<const int4*>(&ctl->range_flag[slot][4]);
            out_of_range = out_of_range || (f0.x | f0.y | f0.z | f0.w | f1.x | f1.y | f1.z | f1.w) != 0;
            const float4 n0 = *reinterpret_cast<const float4*>(&ctl->nmax[slot][0]);
            const float4 n1 = *reinterpret_cast<const float4*>(&ctl->nmax[slot][4]);
            nmax = fmaxf(nmax, fmaxf(fmaxf(fmaxf(n0.x, n0.y), fmaxf(n0.z, n0.w)), fmaxf(fmaxf(n1.x, n1.y), fmaxf(n1.z, n1.w))));
        }
        if (ch != kChunks - 1) continue;

        float c1, c2;
        tc_column_minima(sb, c1, c2);
        int code = (int)((__float_as_uint(m1) & kRowBits) << 4) | (int)(__float_as_uint(c1) & 15u);
        const float gap = fminf(m2, c2) - fmaxf(m1, c1), tau = tc_tau<kC, kRowBits>(m1, m2, X, nmax);
        const bool certain = scores_valid && !out_of_range && nmax >= 1.f && gap > tau;
        const int64_t off = offsets[(rs & rt_mask) * kTcThreads];
        // exact recomputation of the uncertain rows, one row at a time by the whole warp
        unsigned pending = __ballot_sync(0xffffffffu, !certain && off != -2);
        while (pending) {
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
            const int ec = tc_exact_code<kC>(cb + ((int64_t)h * G + g) * (kChunks * 256) * kC, kChunks * 256, xs[0], xs[1], xs[2],
                                             xs[3], xs[4], xs[5], xs[6], xs[7]);
            if (lane == src) code = ec;
        }
        if (off >= 0) codes[off + g * kTokenBlock] = (uint8_t)code;
        if (kChunks > 1) {
            // Upper bits: 16 tokens share a word of 2 hb bytes.  Where a half warp holds the 16 tokens of one block it
            // writes the word; otherwise the bits are replaced in the aligned 32-bit word that other tokens share.
            constexpr int kHb = kChunks == 2 ? 1 : 2;
            const int64_t block = off >= 0 ? off & ~(int64_t)15 : -1;
            const int64_t block0 = __shfl_sync(0xffffffffu, block, lane & 16);
            const unsigned whole = __ballot_sync(0xffffffffu, off >= 0 && block == block0 && (int)(off & 15) == (lane & 15));
            const unsigned half_mask = 0xffffu << (lane & 16);
            if ((whole & half_mask) == half_mask) {
                const uint32_t word = __reduce_or_sync(half_mask, ((uint32_t)code >> 8) << (kHb * (lane & 15)));
                unsigned char* dst = codes + block + G * kTokenBlock + g * 2 * kHb;
                if ((lane & 15) == 0) {
                    if (kHb == 2) *reinterpret_cast<uint32_t*>(dst) = word;
                    else *reinterpret_cast<uint16_t*>(dst) = (uint16_t)word;
                }
            } else if (off >= 0) {
                const int bit = (int)(off & 15) * kHb;
                const uintptr_t a = reinterpret_cast<uintptr_t>(codes) + (uintptr_t)(block + G * kTokenBlock + g * 2 * kHb + (bit >> 3));
                unsigned int* w = reinterpret_cast<unsigned int*>(a & ~(uintptr_t)3);
                const int shift = (int)(a & 3) * 8 + (bit & 7);
                atomicAnd(w, ~((unsigned int)((1 << kHb) - 1) << shift));
                atomicOr(w, (unsigned int)(code >> 8) << shift);
            }
        }
    }

    // Every MMA that was issued has been waited for; where a wait gave up (the rows since went the exact way), this is
    // done now, with a limit again, by the thread that issues them.  Then the tensor memory goes back.
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
}

template <int kC, int kChunks>
cudaError_t launch_enc_tc(const __half* x, const float* cb, const int32_t* seq_offsets, const Shape& sh, int64_t n_tokens,
                          int64_t token_offset, uint8_t* codes, cudaStream_t st, const __half* x2, const float* cb2, uint8_t* codes2)
{
    using C = TcCfg<kC, kChunks>;
    const int64_t n_vec = sh.n_seq * n_tokens;
    const int64_t tiles = (n_vec + kTcTileVecs - 1) / kTcTileVecs;
    const int64_t slots = C::kCtasPerSm * (int64_t)device_sm_count();          // CTAs in flight
    // Row tiles per CTA.  A group's centroids are prepared once per CTA, which costs `prepare` of a row tile's step (from the times
    // below), and the tiles past the last vector are stepped through as well; the least of both together, as long as the
    // groups can be split into three waves of CTAs (with four asked for, 1665 x 8 of CQ-8c8b 30.2 instead of 27.8 us, with two
    // 2500 x 8 37.8 instead of 35.8).  Against one tile per CTA wherever whole rows of groups do not fill four waves, key and
    // value: 40000 vectors x 8 heads of CQ-8c8b 481 -> 401 us, 4000 x 40 259 -> 210, 1665 x 8 30.2 -> 27.8; CQ-4c8b 14688 x 8
    // 306 -> 279; CQ-2c8b 4000 x 40 860 -> 762; CQ-8c10b 4000 x 8 304 -> 235.
    constexpr double prepare = kChunks > 1 ? 0.44 : kC == 8 ? 0.3 : kC == 4 ? 0.2 : 0.15;
    int log_rt = 0;
    double least = 1e30;
    for (int l = 0; l <= C::kMaxLogRt; ++l) {
        const int64_t n = (tiles + (1 << l) - 1) >> l;
        const double cost = (double)n * ((1 << l) + prepare);
        if ((l == 0 || n * sh.n_kv_heads * C::G * (x2 ? 2 : 1) >= 3 * slots) && cost < least) {
            log_rt = l;
            least = cost;
        }
    }
    const int64_t blocks = (tiles + (1 << log_rt) - 1) >> log_rt;
    // Split the groups over CTAs: to one wave per tensor where the input is small, and up to four waves, both tensors
    // counted, while a CTA keeps two groups: a last wave that is nearly empty then costs a quarter of what it does with
    // one wave, and a CTA's own start is about one group's work (64 x 32 heads, c = 4, one group each: 17.3 -> 19.5 us).  (Key and value, against
    // one wave per tensor: 1000 vectors x 4 sequences x 8 heads of CQ-8c8b 62.3 -> 58.8 us, 1665 vectors 31.3 -> 30.5,
    // 1200 of CQ-8c10b 115.6 -> 104.0; 4000 x 32 heads, four waves without a split, unchanged.)
    const int64_t units = blocks * sh.n_kv_heads * (x2 ? 2 : 1);
    const int64_t four_waves = (4 * slots + units - 1) / units;
    int64_t n_gsplit = (slots + blocks * sh.n_kv_heads - 1) / (blocks * sh.n_kv_heads);
    if (n_gsplit < C::G / 2 && n_gsplit < four_waves) n_gsplit = four_waves < C::G / 2 ? four_waves : C::G / 2;
    if (n_gsplit > C::G) n_gsplit = C::G;
    if (n_gsplit < 1) n_gsplit = 1;
    const int groups_per_cta = (int)((C::G + n_gsplit - 1) / n_gsplit);
    n_gsplit = (C::G + groups_per_cta - 1) / groups_per_cta;
    const int64_t grid = blocks * sh.n_kv_heads * n_gsplit;
    if (grid > 0x7fffffff) return cudaErrorInvalidConfiguration;
    // call-site slots 38, 39, 43 ... 47, 62, 63 of ensure_dynamic_smem
    constexpr int kSlots[9] = {38, 39, 43, 44, 45, 46, 47, 62, 63};
    constexpr int kSlot = kSlots[3 * (kC == 2 ? 0 : kC == 4 ? 1 : 2) + (kChunks == 1 ? 0 : kChunks == 2 ? 1 : 2)];
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(encode_tc_kernel<kC, kChunks>), C::kSmemBytes, kSlot);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr;
    cudaLaunchConfig_t cfg = overlapped_config((unsigned)grid, kTcThreads, C::kSmemBytes, st, &attr);
    cfg.gridDim.y = x2 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, encode_tc_kernel<kC, kChunks>, x, cb, seq_offsets, sh, n_tokens, token_offset, codes, groups_per_cta,
                              log_rt, x2, cb2, codes2);
}

}  // namespace

bool encode_tc_supported(const Shape& sh)
{
    return sh.head_dim == 128 && (sh.b == 8 || sh.b == 9 || sh.b == 10) && (sh.c == 2 || sh.c == 4 || sh.c == 8);
}

cudaError_t launch_encode_tc(const __half* x, const float* cb, const int32_t* seq_offsets, const Shape& sh, int64_t n_tokens,
                             int64_t token_offset, uint8_t* codes, cudaStream_t st, const __half* x2, const float* cb2, uint8_t* codes2)
{
    if (sh.n_seq * n_tokens == 0) return cudaSuccess;
#define CQ_TC(C_)                                                                                                              \
    return sh.b == 8   ? launch_enc_tc<C_, 1>(x, cb, seq_offsets, sh, n_tokens, token_offset, codes, st, x2, cb2, codes2)    \
           : sh.b == 9 ? launch_enc_tc<C_, 2>(x, cb, seq_offsets, sh, n_tokens, token_offset, codes, st, x2, cb2, codes2)    \
                       : launch_enc_tc<C_, 4>(x, cb, seq_offsets, sh, n_tokens, token_offset, codes, st, x2, cb2, codes2)
    switch (sh.c) {
        case 2: CQ_TC(2);
        case 4: CQ_TC(4);
        case 8: CQ_TC(8);
        default: return cudaErrorNotSupported;
    }
#undef CQ_TC
}

}  // namespace cq
