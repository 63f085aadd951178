// Tuned decode attention over codes of keys that were quantised BEFORE the rotary position embedding
// (last sentence of Section 3.2), for head_dim 128, b = 8, c in {4, 8} and the pairing (i, i + 64).
//
// The key of Eq. 1 is the reconstruction rotated by its position, K_a = k_a cos - k_b sin,
// K_b = k_b cos + k_a sin for the channel pair (a, b) = (i, i + 64), so a score is a dot product of
// the query with a dequantised, rotated key: there is no table of per-code score terms.  What the
// kernel does instead:
//   - A CTA serves up to 8 query heads of one KV head (what the bins leave room for) over a range of
//     the context; the KV head's key centroids sit in shared memory as fp16 (64 KiB), code-major
//     ([code][group][channel]), so that the 32 lanes of a gather - each in its own group's columns -
//     touch 32 different banks whatever the codes are.  The bins are code-major for the same reason.
//   - Lane l of a warp owns the pairs i = 2l, 2l + 1.  For a batch of 32 / heads consecutive tokens it
//     gathers the two half2 words of its channels per token, rotates them and multiplies by its slice
//     of every head's query: 32 partial scores per lane, which a five-stage exchange between the
//     lanes sums so that lane (head, token) ends up with that score.
//   - The cosines and sines of a batch are read from the tables once, for its first token; the next
//     tokens' values follow by the angle-addition rule with the step (cos, sin) taken from the
//     tables' first two rows.  At the end of the batch the result is compared with the table row of
//     the token after the batch; if it differs (tables that are not of the form cos / sin of
//     position x frequency + phase) the batch is done again with every row read from the tables, and
//     so are the warp's later batches.
//   - Scores of a chunk of the range are kept in shared memory; their largest one and the sum of
//     the weights so far fix the unit in which the bins per (head, group, value code) count: whole
//     numbers, the total just below 2^31 (the bins are shifted when the unit grows).  Lane = group
//     adds the weights in that unit, and bins x value centroids closes the partial.  Adds to shared
//     memory run at 32 lanes per clock for whole numbers and at 4 to 8 for fp32.  Partials and their merge are those of the other
//     decode kernels.
// What bounds it: scores (42 of a CTA's 75 thousand cycles at 4096 tokens, one head) and values (16); neither the issue slots nor
// a pipe is full.  Rotation, dot and address in packed and permuting instructions (28 -> 21 a token and head) took 153.4 to
// 151.7 us only; four blocks of value codes in flight instead of one, or their prefetch to L2, nothing or less (spills).  16 sequences of 4096 tokens, 32
// heads, c = 4: 273 us with fp32 bins, 206 with whole numbers, 188 with 32 warps for one head, 164 with
// set-up and end that read the codebooks in whole lines; 32 sequences, 32 heads on 8, c = 8: 308 -> 176.
#include "cq_common.cuh"
#include "cq_decode_util.cuh"
#include <type_traits>

namespace cq {

namespace {

constexpr int kRtMostWarps = 32;
constexpr int kRtScoreBytes = 32 * 1024;

struct RtCtl {
    float m_run[8];                    // per head: whole number not below the largest score (log2 domain)
    float factor[8];                   // per head: 2^(old m_run - new m_run) of the current chunk
    float e_run[8];                    // per head: the bins count in units of 2^e_run
    float unit[8];                     // per head: 2^(m_run - e_run)
    int shift[8];                      // per head: by how much e_run rose with the current chunk (32: more than the bins hold)
    float warp_max[kRtMostWarps][8];       // per warp and head: largest score of the current chunk
    float l_part[kRtMostWarps][8];         // per warp and head: sum of weights (final reduction)
};

template <int kC, int kHeads>
struct RtCfg {
    static constexpr int G = 128 / kC;
    static constexpr int kT = 32 / kHeads;                        // tokens of a warp's batch
    static constexpr int kChunk = kRtScoreBytes / 4 / kHeads;     // tokens whose scores are kept at a time
    static constexpr int kBookOff = 0;                            // fp16 [256][G][kC]
    static constexpr int kBinsOff = 128 * 256 * 2;                // uint32 [kHeads][256][G]
    static constexpr int kScoreOff = kBinsOff + kHeads * G * 256 * 4;      // fp32 [kHeads][kChunk]
    static constexpr int kCtlOff = kScoreOff + kRtScoreBytes;
    static constexpr int kSmemBytes = kCtlOff + 2560;
    static constexpr int kThreads = kHeads == 1 ? 1024 : 512;
    static_assert(sizeof(RtCtl) <= 2560, "control block");
    static_assert(kSmemBytes <= 227 * 1024, "shared memory");
    static_assert(kChunk % 32 == 0 && kT >= 4, "batches of whole words");
};

// byte j of a run of code bytes held in 32-bit words (little endian)
template <int kWords>
__device__ __forceinline__ uint32_t rt_code(const uint32_t (&w)[kWords], int j)
{
    return (w[j >> 2] >> (8 * (j & 3))) & 0xffu;
}

// Two fp32 values in a register pair: one instruction multiplies and adds both.
typedef unsigned long long rt_pair;
__device__ __forceinline__ rt_pair rt_pack(float x, float y)
{
    rt_pair d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ float2 rt_unpack(rt_pair a)
{
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(a));
    return d;
}
__device__ __forceinline__ rt_pair rt_mul(rt_pair a, rt_pair b)
{
    rt_pair d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ rt_pair rt_fma(rt_pair a, rt_pair b, rt_pair c)
{
    rt_pair d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

template <int kC, int kHeads>
__global__ void __launch_bounds__(RtCfg<kC, kHeads>::kThreads, 1)
decode_rope_tuned_kernel(const __half* __restrict__ q, const uint8_t* __restrict__ kc, const uint8_t* __restrict__ vc,
                         const float* __restrict__ kcb, const float* __restrict__ vcb, const int32_t* __restrict__ seq_lens,
                         const float* __restrict__ rope_cos, const float* __restrict__ rope_sin, float scale_log2e, Shape sh,
                         int n_splits, int split_tokens, float* __restrict__ partials, float* __restrict__ out)
{
    // Launched ahead of the end of the kernel before it.  It lets nothing go ahead itself: a CTA fills an SM, so that what follows finds
    // room only where a CTA has ended, and its CTAs then share SMs while others idle.  Calls back to back, us, let ahead at the
    // start / not: 2 x 10183 tokens, 32 heads on 8 of CQ-4c8b 39.5 / 37.6, 8 x 2480 of CQ-8c8b 47.1 / 46.0, 16 x 4096, 32 heads of CQ-4c8b 150.1 / 150.1.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    using C = RtCfg<kC, kHeads>;
    constexpr int G = C::G, kT = C::kT, kWords = kT / 4, kRtThreads = C::kThreads, kRtWarps = kRtThreads / 32;
    extern __shared__ __align__(16) unsigned char rt_smem[];
    uint32_t* bins = reinterpret_cast<uint32_t*>(rt_smem + C::kBinsOff);
    float* scores = reinterpret_cast<float*>(rt_smem + C::kScoreOff);
    RtCtl* ctl = reinterpret_cast<RtCtl*>(rt_smem + C::kCtlOff);

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n_hgroups = sh.n_q_heads / kHeads;
    const int split = blockIdx.x % n_splits;
    const int hg = (blockIdx.x / n_splits) % n_hgroups;
    const int64_t s = seq_by_rank(seq_lens, (int)sh.n_seq, sh.max_tokens, (int)(blockIdx.x / (n_splits * n_hgroups)));   // longest first
    const int hq0 = hg * kHeads, hkv = hq0 / sh.R;
    const int stride = partial_stride(128);

    int64_t n = seq_lens[s];
    n = n < 0 ? 0 : (n > sh.max_tokens ? sh.max_tokens : n);
    const int64_t t_begin = (int64_t)split * split_tokens;
    const int64_t t_end = t_begin + split_tokens < n ? t_begin + split_tokens : n;
    float* part0 = partials + ((s * sh.n_q_heads + hq0) * n_splits + split) * (int64_t)stride;      // head h: + h * n_splits * stride
    float* o0 = out + (s * sh.n_q_heads + hq0) * 128;
    if (t_end <= t_begin) {          // empty range: neutral element of the merge, or a zero row where there is none
        if (n_splits == 1) {
            for (int i = threadIdx.x; i < kHeads * 128; i += kRtThreads) o0[i] = 0.f;
            return;
        }
        for (int i = threadIdx.x; i < kHeads * stride; i += kRtThreads) {
            const int h = i / stride, d = i % stride;
            part0[(int64_t)h * n_splits * stride + d] = d == 0 ? -INFINITY : 0.f;
        }
        return;
    }

    // ------------------------------------------------------------------ set-up
    // this lane's channels: a = 2 lane, 2 lane + 1 and b = a + 64; its slice of every head's query
    float qa[kHeads][2], qb[kHeads][2];
#pragma unroll
    for (int h = 0; h < kHeads; ++h) {
        const __half* qh = q + (s * sh.n_q_heads + hq0 + h) * 128;
        qa[h][0] = __half2float(qh[2 * lane]) * scale_log2e;
        qa[h][1] = __half2float(qh[2 * lane + 1]) * scale_log2e;
        qb[h][0] = __half2float(qh[64 + 2 * lane]) * scale_log2e;
        qb[h][1] = __half2float(qh[64 + 2 * lane + 1]) * scale_log2e;
    }
    // rotation from one position to the next, from the tables' first two rows: row1 x conj(row0) / |row0|^2
    float2 st_re = make_float2(1.f, 1.f), st_im = make_float2(0.f, 0.f);
    bool exact = sh.max_tokens < 2;              // true: every token's row is read from the tables
    if (!exact) {
        const float2 c0 = *reinterpret_cast<const float2*>(rope_cos + 2 * lane), s0 = *reinterpret_cast<const float2*>(rope_sin + 2 * lane);
        const float2 c1 = *reinterpret_cast<const float2*>(rope_cos + 64 + 2 * lane), s1 = *reinterpret_cast<const float2*>(rope_sin + 64 + 2 * lane);
        const float nx = c0.x * c0.x + s0.x * s0.x, ny = c0.y * c0.y + s0.y * s0.y;
        if (!(nx > 1e-12f) || !(ny > 1e-12f)) exact = true;
        st_re.x = (c1.x * c0.x + s1.x * s0.x) / nx;
        st_im.x = (s1.x * c0.x - c1.x * s0.x) / nx;
        st_re.y = (c1.y * c0.y + s1.y * s0.y) / ny;
        st_im.y = (s1.y * c0.y - c1.y * s0.y) / ny;
        exact = __any_sync(0xffffffffu, exact);
    }
    // key centroids of the KV head as fp16, bins at zero
    {
        // A warp takes 64 bytes of eight groups at a time, a quarter of it two groups: two lines of memory per quarter of a
        // load, and at most four lanes that meet in a bank of a store.  (In the order of the codebook all 32 met.)
        const float4* src = reinterpret_cast<const float4*>(kcb + (int64_t)hkv * 128 * 256);
        constexpr int kTasks = 256, kBatch = 8;
        static_assert(kTasks % (kRtWarps * kBatch) == 0, "whole batches");
        const int gl = lane >> 2, j = lane & 3;
#pragma unroll 1
        for (int i0 = warp; i0 < kTasks; i0 += kBatch * kRtWarps) {
            float4 x[kBatch];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const int i = i0 + u * kRtWarps, g = 8 * (i % (G / 8)) + gl;
                x[u] = ldg_f4(reinterpret_cast<const float*>(src + (g * 16 * kC + i / (G / 8)) * 4 + j));
            }
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const int i = i0 + u * kRtWarps, g = 8 * (i % (G / 8)) + gl, seg = i / (G / 8);
                const __half2 lo = __floats2half2_rn(x[u].x, x[u].y), hi = __floats2half2_rn(x[u].z, x[u].w);
                const int at = kC == 8 ? (seg * 2 + (j >> 1)) * 256 + g * 16 + (j & 1) * 8 : (seg * 4 + j) * 256 + g * 8;
                *reinterpret_cast<uint2*>(rt_smem + C::kBookOff + at) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
            }
        }
        for (int i = threadIdx.x; i < kHeads * G * 256 / 4; i += kRtThreads)
            reinterpret_cast<float4*>(bins)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (threadIdx.x < 8) ctl->m_run[threadIdx.x] = ctl->e_run[threadIdx.x] = -INFINITY;
    }
    // words of the lane's two channels inside a centroid, and its two groups
    const int gA = (2 * lane) / kC, gB = gA + G / 2;
    // word of the lane's channels a in the centroid row of a code: code * (64 words) + colA; channels b: + 32 words
    // (in bytes: a row is 256 of them, so that one byte permutation puts a code byte and a column together)
    const uint32_t colA = (uint32_t)(gA * kC + (2 * lane) % kC) * 2u, colB = colA + 128u;
    static_assert(128 * 2 == 256, "bytes of a code's row");
    const rt_pair re2 = rt_pack(st_re.x, st_re.y), im2 = rt_pack(st_im.x, st_im.y), nim2 = rt_pack(-st_im.x, -st_im.y);
    const uint8_t* kseq = kc + code_word_offset(sh, sh.n_kv_heads, s, hkv, 0, 0);
    const uint8_t* vseq = vc + code_word_offset(sh, sh.n_kv_heads, s, hkv, 0, 0);
    float l_thr[kHeads];
#pragma unroll
    for (int h = 0; h < kHeads; ++h) l_thr[h] = 0.f;
    __syncthreads();

    for (int64_t chunk_begin = t_begin; chunk_begin < t_end; chunk_begin += C::kChunk) {
        const int chunk_len = (int)(t_end - chunk_begin < C::kChunk ? t_end - chunk_begin : C::kChunk);

        // -------------------------------------------------------------- scores of the chunk
        float lane_max = -INFINITY;                  // over the scores of this lane's head
        // a batch's key codes of the lane's two groups and the table rows of its first token
        auto load_batch = [&](int64_t t0, uint32_t (&ca)[kWords], uint32_t (&cbw)[kWords], float2& cs0, float2& sn0) {
            const uint8_t* pa = kseq + (t0 / kTokenBlock) * sh.block_bytes + (t0 % kTokenBlock);
            if (kT == 32) {
                const bool two = t0 + 16 < t_end;
                const uint4 a0 = *reinterpret_cast<const uint4*>(pa + gA * kTokenBlock), b0w = *reinterpret_cast<const uint4*>(pa + gB * kTokenBlock);
                const uint4 a1 = two ? *reinterpret_cast<const uint4*>(pa + sh.block_bytes + gA * kTokenBlock) : make_uint4(0u, 0u, 0u, 0u);
                const uint4 b1 = two ? *reinterpret_cast<const uint4*>(pa + sh.block_bytes + gB * kTokenBlock) : make_uint4(0u, 0u, 0u, 0u);
                ca[0] = a0.x; ca[1 % kWords] = a0.y; ca[2 % kWords] = a0.z; ca[3 % kWords] = a0.w;
                ca[4 % kWords] = a1.x; ca[5 % kWords] = a1.y; ca[6 % kWords] = a1.z; ca[7 % kWords] = a1.w;
                cbw[0] = b0w.x; cbw[1 % kWords] = b0w.y; cbw[2 % kWords] = b0w.z; cbw[3 % kWords] = b0w.w;
                cbw[4 % kWords] = b1.x; cbw[5 % kWords] = b1.y; cbw[6 % kWords] = b1.z; cbw[7 % kWords] = b1.w;
            } else if (kT == 16) {
                const uint4 a0 = *reinterpret_cast<const uint4*>(pa + gA * kTokenBlock), b0w = *reinterpret_cast<const uint4*>(pa + gB * kTokenBlock);
                ca[0] = a0.x; ca[1 % kWords] = a0.y; ca[2 % kWords] = a0.z; ca[3 % kWords] = a0.w;
                cbw[0] = b0w.x; cbw[1 % kWords] = b0w.y; cbw[2 % kWords] = b0w.z; cbw[3 % kWords] = b0w.w;
            } else if (kT == 8) {
                const uint2 a0 = *reinterpret_cast<const uint2*>(pa + gA * kTokenBlock), b0w = *reinterpret_cast<const uint2*>(pa + gB * kTokenBlock);
                ca[0] = a0.x; ca[1 % kWords] = a0.y;
                cbw[0] = b0w.x; cbw[1 % kWords] = b0w.y;
            } else {
                ca[0] = *reinterpret_cast<const uint32_t*>(pa + gA * kTokenBlock);
                cbw[0] = *reinterpret_cast<const uint32_t*>(pa + gB * kTokenBlock);
            }
            cs0 = *reinterpret_cast<const float2*>(rope_cos + t0 * 64 + 2 * lane);
            sn0 = *reinterpret_cast<const float2*>(rope_sin + t0 * 64 + 2 * lane);
        };
        uint32_t ca[kWords], cbw[kWords];
        float2 cs0 = make_float2(1.f, 1.f), sn0 = make_float2(0.f, 0.f);
        if (warp * kT < chunk_len) load_batch(chunk_begin + warp * kT, ca, cbw, cs0, sn0);
        for (int b0 = warp * kT; b0 < chunk_len; b0 += kRtWarps * kT) {
            const int64_t t0 = chunk_begin + b0;
            constexpr int kSlots = kHeads == 1 ? 1 : 32;
            float p[kSlots];
            // The scores of the batch, summed over the lanes as they come; from_tables: every token's row is read from the tables, else the rows
            // after the first follow by the step rotation.  Returns false when the stepped rows leave the tables.
            // With one head per CTA the query is rotated instead of the key (by the opposite angle): the rotated
            // query u = q_a cos + q_b sin, v = q_b cos - q_a sin steps like the angle does, and the score term of a
            // pair is k_a u + k_b v.
            auto batch = [&](auto from_tables) -> bool {
                constexpr bool kFromTables = decltype(from_tables)::value;
                float2 cs = cs0, sn = sn0;
                // Sum over the lanes, two values at a time: a lane keeps the one whose slot has the bit of the offset like its
                // own lane number, the other lane's share of it added; slot = (head, token of the batch).  At the end lane L
                // holds slot L = (head L / kT, token L % kT).  With one head tokens 2i and 2i + 1 are joined at once, then
                // pairs, ...: few values wait in registers, so that 32 warps fit the SM, and the exchanges pass between the
                // gathers (16 sequences of 4096 tokens, 32 heads, c = 4: 206 -> 187 us).  With several heads the 16 warps'
                // multiply-adds hide the exchange better when it comes in one piece (four heads, c = 4: 173 against 181 us).
                auto join = [&](float lower, float upper, int o) {
                    const bool up = (lane & o) != 0;
                    return (up ? upper : lower) + __shfl_xor_sync(0xffffffffu, up ? lower : upper, o);
                };
                float waiting[5];
                // (one head: the rotated query; several: cosines and sines)
                rt_pair u2 = rt_pack(cs.x, cs.y), v2 = rt_pack(sn.x, sn.y);
                auto rotated_query = [&]() {
                    u2 = rt_pack(fmaf(qa[0][0], cs.x, qb[0][0] * sn.x), fmaf(qa[0][1], cs.y, qb[0][1] * sn.y));
                    v2 = rt_pack(fmaf(qb[0][0], cs.x, -qa[0][0] * sn.x), fmaf(qb[0][1], cs.y, -qa[0][1] * sn.y));
                };
                if (kHeads == 1) rotated_query();
#pragma unroll
                for (int j = 0; j < kT; ++j) {
                    const uint32_t wa = *reinterpret_cast<const uint32_t*>(rt_smem + C::kBookOff + __byte_perm(ca[j >> 2], colA, 0x5504u | (j & 3) << 4));
                    const uint32_t wb = *reinterpret_cast<const uint32_t*>(rt_smem + C::kBookOff + __byte_perm(cbw[j >> 2], colB, 0x5504u | (j & 3) << 4));
                    const float2 fa = __half22float2(*reinterpret_cast<const __half2*>(&wa));
                    const float2 fb = __half22float2(*reinterpret_cast<const __half2*>(&wb));
                    const rt_pair ka = rt_pack(fa.x, fa.y), kb = rt_pack(fb.x, fb.y);
                    float x[kHeads];
                    if (kHeads == 1) {
                        const float2 t = rt_unpack(rt_fma(ka, u2, rt_mul(kb, v2)));
                        x[0] = t.x + t.y;
                    } else {
                        // the rotated key of the lane's four channels
                        const rt_pair ra = rt_fma(ka, u2, rt_mul(kb, v2 ^ 0x8000000080000000ull)), rb = rt_fma(kb, u2, rt_mul(ka, v2));
#pragma unroll
                        for (int h = 0; h < kHeads; ++h) {
                            const float2 t = rt_unpack(rt_fma(rt_pack(qa[h][0], qa[h][1]), ra, rt_mul(rt_pack(qb[h][0], qb[h][1]), rb)));
                            x[h] = t.x + t.y;
                        }
                    }
                    if (kHeads == 1) {
#pragma unroll
                        for (int b = 0; b < 5; ++b) {
                            if ((j & ((1 << b) - 1)) != (1 << b) - 1) break;     // some lower bit is clear: it waits already
                            if ((j >> b) & 1) x[0] = join(waiting[b], x[0], 1 << b);
                            else waiting[b] = x[0];
                        }
                        p[0] = x[0];
                    } else {
#pragma unroll
                        for (int h = 0; h < kHeads; ++h) p[(h * kT + j) % kSlots] = x[h];
                    }
                    // the next position
                    if (kFromTables) {
                        if (j + 1 < kT) {
                            const int64_t tn = t0 + j + 1 < sh.max_tokens ? t0 + j + 1 : t0 + j;
                            cs = *reinterpret_cast<const float2*>(rope_cos + tn * 64 + 2 * lane);
                            sn = *reinterpret_cast<const float2*>(rope_sin + tn * 64 + 2 * lane);
                            if (kHeads == 1) rotated_query();
                            else { u2 = rt_pack(cs.x, cs.y); v2 = rt_pack(sn.x, sn.y); }
                        }
                    } else if (kHeads == 1) {
                        const rt_pair un = rt_fma(u2, re2, rt_mul(v2, im2)), vn = rt_fma(v2, re2, rt_mul(u2, nim2));
                        u2 = un;
                        v2 = vn;
                    } else {
                        const rt_pair cn = rt_fma(u2, re2, rt_mul(v2, nim2)), sn2 = rt_fma(v2, re2, rt_mul(u2, im2));
                        u2 = cn;
                        v2 = sn2;
                    }
                }
                if (kFromTables) return true;
                const float2 u = rt_unpack(u2), v = rt_unpack(v2);
                // what was stepped to is the prediction for position t0 + kT: it must be what the tables hold there
                bool off = false;
                if (t0 + kT < sh.max_tokens) {
                    const float2 ct = *reinterpret_cast<const float2*>(rope_cos + (t0 + kT) * 64 + 2 * lane);
                    const float2 stt = *reinterpret_cast<const float2*>(rope_sin + (t0 + kT) * 64 + 2 * lane);
                    const float tol = 2e-5f;
                    if (kHeads == 1) {
                        const float ux = fmaf(qa[0][0], ct.x, qb[0][0] * stt.x), uy = fmaf(qa[0][1], ct.y, qb[0][1] * stt.y);
                        const float vx = fmaf(qb[0][0], ct.x, -qa[0][0] * stt.x), vy = fmaf(qb[0][1], ct.y, -qa[0][1] * stt.y);
                        const float bx = tol * (fabsf(qa[0][0]) + fabsf(qb[0][0])) * (1.f + fabsf(ct.x) + fabsf(stt.x));
                        const float by = tol * (fabsf(qa[0][1]) + fabsf(qb[0][1])) * (1.f + fabsf(ct.y) + fabsf(stt.y));
                        off = !(fabsf(ux - u.x) <= bx) || !(fabsf(vx - v.x) <= bx) || !(fabsf(uy - u.y) <= by) || !(fabsf(vy - v.y) <= by);
                    } else {
                        off = !(fabsf(ct.x - u.x) <= tol * (1.f + fabsf(ct.x))) || !(fabsf(ct.y - u.y) <= tol * (1.f + fabsf(ct.y))) ||
                              !(fabsf(stt.x - v.x) <= tol * (1.f + fabsf(stt.x))) || !(fabsf(stt.y - v.y) <= tol * (1.f + fabsf(stt.y)));
                    }
                }
                return !__any_sync(0xffffffffu, off);
            };
            if (exact || !batch(std::false_type())) {
                exact = true;                            // this batch, and every later one of the warp, from the tables
                batch(std::true_type());
            }
            // the next batch's words travel during the exchange
            {
                const int nb = b0 + kRtWarps * kT;
                if (nb < chunk_len) load_batch(chunk_begin + nb, ca, cbw, cs0, sn0);
            }
            if (kHeads > 1) {
#pragma unroll
                for (int o = 16; o >= 1; o >>= 1) {
                    const bool upper = (lane & o) != 0;
#pragma unroll
                    for (int i = 0; i < o; ++i) {
                        const float send = upper ? p[i % kSlots] : p[(i + o) % kSlots];
                        const float keep = upper ? p[(i + o) % kSlots] : p[i % kSlots];
                        p[i % kSlots] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                    }
                }
            }
            const int h = lane / kT, j = lane % kT;
            const bool valid = t0 + j < t_end;
            const float sc = valid ? p[0] : -INFINITY;
            scores[h * C::kChunk + b0 + j] = sc;
            lane_max = fmaxf(lane_max, sc);
        }
        // largest score per head: over the lanes of a head, then over the warps
#pragma unroll
        for (int o = 1; o < kT; o <<= 1) lane_max = fmaxf(lane_max, __shfl_xor_sync(0xffffffffu, lane_max, o));
        if (lane % kT == 0) ctl->warp_max[warp][lane / kT] = lane_max;
        __syncthreads();
        // (warp h takes head h, a lane per warp: one thread that walked the warps' values cost a thousand cycles each time)
        if (warp < kHeads) {
            float m = lane < kRtWarps ? ceilf(ctl->warp_max[lane][warp]) : -INFINITY;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
            if (lane == 0) {
                const float old = ctl->m_run[warp];
                m = fmaxf(m, old);
                ctl->factor[warp] = old == m ? 1.f : exp2f(old - m);      // 0 when there was no reference yet
                ctl->m_run[warp] = m;
            }
        }
        __syncthreads();
        // weights of the chunk, relative to m_run, and the total so far
#pragma unroll
        for (int h = 0; h < kHeads; ++h) {
            const float m = ctl->m_run[h];
            float l = l_thr[h] * ctl->factor[h];
            for (int i = threadIdx.x; i < chunk_len; i += kRtThreads) {
                const float w = exp2f(scores[h * C::kChunk + i] - m);
                scores[h * C::kChunk + i] = w;
                l += w;
            }
            l_thr[h] = l;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
            if (lane == 0) ctl->l_part[warp][h] = l;
        }
        __syncthreads();
        // The unit that lets the total fill 31 bits: no bin can run over, and a weight keeps as many bits as fp32 gives it
        // down to 2^-8 of the total.
        if (warp < kHeads) {
            float total = lane < kRtWarps ? ctl->l_part[lane][warp] : 0.f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
            if (lane == 0) {
                const float m = ctl->m_run[warp], old = ctl->e_run[warp];
                const float wanted = m + (ceilf(log2f(total)) - 31.f), e = wanted < old ? old : wanted;
                const float rise = e - old;                                   // (infinite when there was no unit yet: bins are zero)
                ctl->shift[warp] = rise < 32.f ? (int)rise : 32;
                ctl->e_run[warp] = e;
                ctl->unit[warp] = exp2f(m - e);
            }
        }
        __syncthreads();
#pragma unroll
        for (int h = 0; h < kHeads; ++h) {
            const int shift = chunk_begin > t_begin ? ctl->shift[h] : 0;
            if (shift > 0)
                for (int i = threadIdx.x; i < G * 256; i += kRtThreads) {
                    const uint32_t v = bins[h * G * 256 + i];
                    bins[h * G * 256 + i] = shift < 32 ? (v >> shift) + ((v >> (shift - 1)) & 1u) : 0u;
                }
            const float unit = ctl->unit[h];
            const int padded = (chunk_len + kTokenBlock - 1) / kTokenBlock * kTokenBlock;
            for (int i = threadIdx.x; i < padded; i += kRtThreads)
                reinterpret_cast<uint32_t*>(scores)[h * C::kChunk + i] = i < chunk_len ? __float2uint_rn(scores[h * C::kChunk + i] * unit) : 0u;
        }
        __syncthreads();
        // -------------------------------------------------------------- value side: weights into the bins
        // a warp per block of 16 tokens; lane = (group, run of tokens of the block)
        {
            constexpr int kLanesPerGroup = 32 / G;                  // 2 for c = 8, 1 for c = 4
            constexpr int kRun = 16 / kLanesPerGroup;               // tokens of the block per lane
            const int g = lane % G, run = lane / G;
            const int n_blk = (chunk_len + kTokenBlock - 1) / kTokenBlock;
            // (the next block's codes travel during the adds of this one)
            auto load_codes = [&](int blk, uint32_t (&cw)[kRun / 4]) {
                const uint8_t* pv = vseq + ((chunk_begin / kTokenBlock) + blk) * sh.block_bytes + g * kTokenBlock + run * kRun;
                if (kRun == 16) {
                    const uint4 v4 = *reinterpret_cast<const uint4*>(pv);
                    cw[0] = v4.x; cw[1 % (kRun / 4)] = v4.y; cw[2 % (kRun / 4)] = v4.z; cw[3 % (kRun / 4)] = v4.w;
                } else {
                    const uint2 v2 = *reinterpret_cast<const uint2*>(pv);
                    cw[0] = v2.x; cw[1 % (kRun / 4)] = v2.y;
                }
            };
            const uint32_t bin0 = (uint32_t)__cvta_generic_to_shared(bins + g);
            uint32_t cw[kRun / 4], next[kRun / 4];
            if (warp < n_blk) load_codes(warp, next);
            for (int blk = warp; blk < n_blk; blk += kRtWarps) {
#pragma unroll
                for (int i = 0; i < kRun / 4; ++i) cw[i] = next[i];
                if (blk + kRtWarps < n_blk) load_codes(blk + kRtWarps, next);
#pragma unroll
                for (int k = 0; k < kRun; k += 4) {
                    uint4 w[kHeads];                            // (the weights behind the end of the chunk are zero)
#pragma unroll
                    for (int h = 0; h < kHeads; ++h)
                        w[h] = *reinterpret_cast<const uint4*>(scores + h * C::kChunk + blk * kTokenBlock + run * kRun + k);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint32_t bin = bin0 + rt_code<kRun / 4>(cw, k + j) * (G * 4);
#pragma unroll
                        for (int h = 0; h < kHeads; ++h)
                            asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(bin + h * (256 * G * 4)),
                                         "r"(j == 0 ? w[h].x : j == 1 ? w[h].y : j == 2 ? w[h].z : w[h].w) : "memory");
                    }
                }
            }
        }
        __syncthreads();
    }

    // ------------------------------------------------------------------ partial: reference, normaliser, bins x value centroids
#pragma unroll
    for (int h = 0; h < kHeads; ++h) {
        float l = l_thr[h];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) ctl->l_part[warp][h] = l;
    }
    __syncthreads();
    if (warp < kHeads) {
        float l = lane < kRtWarps ? ctl->l_part[lane][warp] : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) {
            l *= ctl->unit[warp];
            ctl->factor[warp] = l;
            if (n_splits > 1) {
                part0[(int64_t)warp * n_splits * stride + 0] = ctl->e_run[warp];
                part0[(int64_t)warp * n_splits * stride + 1] = l;
            }
        }
    }
    // Bins x value centroids: a warp takes 64 bytes of eight groups at a time, as in the set-up, for all heads together
    // (one group per lane touched 32 lines of memory per load and read the codebook once per head: 11 thousand cycles per
    // head); the warps' sums are added through shared memory (the score area is free now).
    {
        constexpr int kOct = G / 8, kTasks = 256 / kRtWarps, kBatch = kTasks < 4 ? kTasks : 4;
        static_assert(kRtWarps % kOct == 0, "a warp stays with its eight groups");
        const int gl = lane >> 2, j = lane & 3;
        const int g = 8 * (warp % kOct) + gl;
        const float4* src = reinterpret_cast<const float4*>(vcb + (int64_t)hkv * 128 * 256) + g * 64 * kC + j;
        float acc[kHeads][4];
#pragma unroll
        for (int h = 0; h < kHeads; ++h) acc[h][0] = acc[h][1] = acc[h][2] = acc[h][3] = 0.f;
#pragma unroll 1
        for (int i0 = 0; i0 < kTasks; i0 += kBatch) {
            float4 x[kBatch];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) x[u] = ldg_f4(reinterpret_cast<const float*>(src + (warp + (i0 + u) * kRtWarps) / kOct * 4));
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const int seg = (warp + (i0 + u) * kRtWarps) / kOct, code = kC == 8 ? seg * 2 + (j >> 1) : seg * 4 + j;
#pragma unroll
                for (int h = 0; h < kHeads; ++h) {
                    const float w = (float)bins[(h * 256 + code) * G + g];
                    acc[h][0] = fmaf(w, x[u].x, acc[h][0]);
                    acc[h][1] = fmaf(w, x[u].y, acc[h][1]);
                    acc[h][2] = fmaf(w, x[u].z, acc[h][2]);
                    acc[h][3] = fmaf(w, x[u].w, acc[h][3]);
                }
            }
        }
        float* red = scores;                                     // [heads][warps][8 groups][kC]
        constexpr int kRow = 8 * kC;
        static_assert(kHeads * kRtWarps * kRow * 4 <= kRtScoreBytes, "room");
#pragma unroll
        for (int h = 0; h < kHeads; ++h) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                acc[h][k] += __shfl_xor_sync(0xffffffffu, acc[h][k], 2);
                if (kC == 4) acc[h][k] += __shfl_xor_sync(0xffffffffu, acc[h][k], 1);
            }
            if (j < kC / 4)
                *reinterpret_cast<float4*>(red + (h * kRtWarps + warp) * kRow + gl * kC + (kC == 8 ? 4 * (j & 1) : 0)) =
                    make_float4(acc[h][0], acc[h][1], acc[h][2], acc[h][3]);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < kHeads * 128; i += kRtThreads) {
            const int h = i >> 7, d = i & 127;
            float v = 0.f;
#pragma unroll
            for (int w = 0; w < kRtWarps / kOct; ++w) v += red[(h * kRtWarps + w * kOct + d / kRow) * kRow + d % kRow];
            if (n_splits == 1) o0[h * 128 + d] = v / ctl->factor[h];       // a range is the whole context: no merge
            else part0[(int64_t)h * n_splits * stride + 2 + d] = v;
        }
    }
}

template <int kC, int kHeads>
cudaError_t launch_rt(const __half* q, const uint8_t* kc, const uint8_t* vc, const float* kcb, const float* vcb,
                      const int32_t* seq_lens, const float* rope_cos, const float* rope_sin, float scale, const Shape& sh,
                      int n_splits, int split_tokens, float* partials, float* out, cudaStream_t st)
{
    using C = RtCfg<kC, kHeads>;
    constexpr int kSlot = 48 + (kC == 8 ? 0 : 4) + (kHeads == 1 ? 0 : kHeads == 2 ? 1 : kHeads == 4 ? 2 : 3);    // 48 ... 55
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(decode_rope_tuned_kernel<kC, kHeads>), C::kSmemBytes, kSlot);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)(sh.n_seq * (sh.n_q_heads / kHeads) * n_splits);
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = overlapped_config(grid, C::kThreads, C::kSmemBytes, st, &attr);
    return cudaLaunchKernelEx(&cfg, decode_rope_tuned_kernel<kC, kHeads>, q, kc, vc, kcb, vcb, seq_lens, rope_cos, rope_sin,
                              scale * kLog2e, sh, n_splits, split_tokens, partials, out);
}

int rope_heads_per_cta(const Shape& sh)
{
    const int most = sh.c == 8 ? 8 : 4;              // what the bins leave room for
    int h = 1;
    while (h * 2 <= most && sh.R % (h * 2) == 0) h *= 2;
    return h;
}

}  // namespace

bool decode_rope_tuned_supported(const Shape& sh, int pairing)
{
    return pairing == 0 && sh.head_dim == 128 && sh.b == 8 && (sh.c == 4 || sh.c == 8);
}

cudaError_t launch_decode_rope_tuned(const __half* q, const uint8_t* kc, const uint8_t* vc, const float* kcb,
                                     const float* vcb, const int32_t* seq_lens, const float* rope_cos, const float* rope_sin,
                                     float scale, const Shape& sh, float* out, float* partials, cudaStream_t st)
{
    const int heads = rope_heads_per_cta(sh);
    // ranges of the context: enough CTAs for two per SM... one CTA fills an SM, so two waves; never more partial slots
    // than the workspace holds (those of decode_generic_splits), ranges of whole 256 tokens
    const int64_t items = sh.n_seq * (sh.n_q_heads / heads);
    int64_t want = (2 * (int64_t)device_sm_count() + items - 1) / items;
    const int64_t cap = (sh.max_tokens + 1023) / 1024;
    if (want > cap) want = cap;
    const int most = decode_generic_splits(sh);
    if (want > most) want = most;
    if (want < 1) want = 1;
    int64_t split_tokens = (sh.max_tokens + want - 1) / want;
    split_tokens = (split_tokens + 255) / 256 * 256;
    const int n_splits = (int)((sh.max_tokens + split_tokens - 1) / split_tokens);
    cudaError_t e = cudaErrorNotSupported;
#define CQ_RT(C_, H_) e = launch_rt<C_, H_>(q, kc, vc, kcb, vcb, seq_lens, rope_cos, rope_sin, scale, sh, n_splits, (int)split_tokens, partials, out, st)
    if (sh.c == 8) {
        switch (heads) { case 1: CQ_RT(8, 1); break; case 2: CQ_RT(8, 2); break; case 4: CQ_RT(8, 4); break; case 8: CQ_RT(8, 8); break; default: break; }
    } else {
        switch (heads) { case 1: CQ_RT(4, 1); break; case 2: CQ_RT(4, 2); break; case 4: CQ_RT(4, 4); break; default: break; }
    }
#undef CQ_RT
    if (e != cudaSuccess || n_splits == 1) return e;
    return launch_merge(partials, n_splits, sh, out, st);
}

}  // namespace cq
