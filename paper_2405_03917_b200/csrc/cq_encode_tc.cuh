// Nearest centroids on the fifth-generation tensor cores: the device code that encode_tc_kernel (cq_encode_tc.cu, where the
// method is described) and assign_kernel (cq_learn_assign.cu) share.
#pragma once

#include "cq_common.cuh"

namespace cq {

namespace {

constexpr int kTcThreads = 128;
constexpr int kTcTileVecs = 128;          // vectors of a row tile
constexpr float kTcInf = __builtin_huge_valf();

// kChunks: 256-centroid chunks per group (b = 8, 9, 10: 1, 2, 4)
template <int kC, int kChunks>
struct TcCfg {
    static constexpr int G = 128 / kC;
    static constexpr int kSteps = (kC == 8) ? 2 : 1;              // K steps (16 fp16 slots each)
    static constexpr int kATile = 128 * 32;                       // bytes of one A tile of one K step
    static constexpr int kBTile = 256 * 32;
    static constexpr int kABuf = kSteps * kATile;
    static constexpr int kBBuf = kSteps * kBTile;
    static constexpr int kBSlots = kChunks == 1 ? 2 : kChunks;    // prepared chunks: this group's and the next one's, or all of a group's
    static constexpr int kMaxLogRt = (kC == 8 || kChunks > 1) ? 2 : 3;    // up to 2^kMaxLogRt row tiles per CTA
    static constexpr int kCtasPerSm = (kC == 8 && kChunks == 4) ? 2 : (kC == 8 && kChunks == 2) ? 3 : 4;
    static constexpr int kAOff = 0;                               // [2 buffers]
    static constexpr int kBOff = kAOff + 2 * kABuf;               // [kBSlots]
    static constexpr int kRowOff = kBOff + kBSlots * kBBuf;       // [row tiles][128 threads] code offset of the row
    static constexpr int kCtlOff = kRowOff + (1 << kMaxLogRt) * kTcThreads * 8;
    static constexpr int kUsedBytes = kCtlOff + 512;
    // at least 46 KiB, so that a fifth CTA (for which no tensor memory would be left) never fits an SM
    static constexpr int kSmemBytes = kUsedBytes > 46 * 1024 ? kUsedBytes : 46 * 1024;
    static_assert(kCtasPerSm * (kSmemBytes + 1024) <= 228 * 1024, "shared memory of an SM");
    static_assert(5 * (kSmemBytes + 1024) > 228 * 1024, "one CTA too many would fit");
};

constexpr int kTcColumns = 128;            // tensor-memory columns of a CTA

struct TcCtl {
    int range_flag[4][8];      // per slot, warp and pass, non-zero: those centroids of the prepared chunk hold values fp16 cannot carry
    float nmax[4][8];          // per slot, warp and pass, the largest ||C_j||^2 among those centroids (scaled)
    uint32_t tmem_base;
    int wait_failed;           // a wait on an MMA barrier gave up
    uint64_t bar[2];           // completion of the MMA of the low / high half of a step
    uint64_t drained;          // completion of everything issued, after a wait gave up
};

__device__ __forceinline__ uint32_t tc_smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t tc_pack_half2(float lo, float hi)
{
    return (uint32_t)__half_as_ushort(__float2half_rn(lo)) | ((uint32_t)__half_as_ushort(__float2half_rn(hi)) << 16);
}

// v = t0 + t1 + t2 with fp16 terms (t2 absorbs what two terms leave, about 2^-33 |v| remains)
__device__ __forceinline__ void tc_split3(float v, float& t0, float& t1, float& t2)
{
    t0 = __half2float(__float2half_rn(v));
    const float r1 = v - t0;
    t1 = __half2float(__float2half_rn(r1));
    t2 = __half2float(__float2half_rn(r1 - t1));
}

__device__ __forceinline__ float tc_min3(float a, float b, float c)
{
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Shared-memory matrix descriptor of a K-major operand tile without swizzle: the 16-byte chunk kc (8 fp16 K slots)
// of row r sits at kc * rows * 16 + r * 16 bytes, so a core matrix (8 rows x 16 bytes) is 128 contiguous bytes, the
// next 8 rows follow 128 bytes on (stride byte offset) and the next K chunk rows * 16 bytes on (leading byte offset).
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr, uint32_t chunk_stride_bytes)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3fffu);
    d |= (uint64_t)((chunk_stride_bytes >> 4) & 0x3fffu) << 16;
    d |= (uint64_t)((128u >> 4) & 0x3fffu) << 32;
    d |= (uint64_t)1 << 46;                      // descriptor version of sm_100
    return d;
}

// D[128 x 128] (+)= A[128 x 16] * B[128 x 16]^T, fp16 operands from shared memory, fp32 accumulator in tensor memory
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t accumulate)
{
    // instruction descriptor: D fp32, A and B fp16, both K-major, N = 128, M = 128
    const uint32_t idesc = (1u << 4) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5}, p;\n\t}"
                 ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(0) : "memory");
}

// Starts the load of 32 consecutive accumulator columns of this thread's row; the values are there after tc_ld_wait.
__device__ __forceinline__ void tc_ld32_issue(float (&v)[32], uint32_t taddr)
{
    uint32_t* u = reinterpret_cast<uint32_t*>(v);
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15]), "=r"(u[16]), "=r"(u[17]), "=r"(u[18]), "=r"(u[19]), "=r"(u[20]), "=r"(u[21]), "=r"(u[22]), "=r"(u[23]), "=r"(u[24]), "=r"(u[25]), "=r"(u[26]), "=r"(u[27]), "=r"(u[28]), "=r"(u[29]), "=r"(u[30]), "=r"(u[31])
                 : "r"(taddr) : "memory");
}
// Waits for the loads issued so far.  The registers pass through the statement, so that nothing that uses them is
// scheduled ahead of the wait.
__device__ __forceinline__ void tc_ld_wait(float (&v)[32])
{
    uint32_t* u = reinterpret_cast<uint32_t*>(v);
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(u[0]), "+r"(u[1]), "+r"(u[2]), "+r"(u[3]), "+r"(u[4]), "+r"(u[5]), "+r"(u[6]), "+r"(u[7]), "+r"(u[8]), "+r"(u[9]), "+r"(u[10]), "+r"(u[11]), "+r"(u[12]), "+r"(u[13]), "+r"(u[14]), "+r"(u[15]), "+r"(u[16]), "+r"(u[17]), "+r"(u[18]), "+r"(u[19]), "+r"(u[20]), "+r"(u[21]), "+r"(u[22]), "+r"(u[23]), "+r"(u[24]), "+r"(u[25]), "+r"(u[26]), "+r"(u[27]), "+r"(u[28]), "+r"(u[29]), "+r"(u[30]), "+r"(u[31])
                 :: "memory");
}

// Waits for the phase with the given parity; gives up after a bounded number of polls (returns false).
__device__ __forceinline__ bool tc_wait(uint64_t* bar, uint32_t parity)
{
    for (int poll = 0; poll < (1 << 22); ++poll) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(tc_smem_u32(bar)), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}

// Centroid j of a group, from global memory into registers.
template <int kC>
__device__ __forceinline__ void tc_fetch_centroid(const float* __restrict__ cb_g, int j, float (&cv)[kC])
{
    if (kC == 2) {
        const float2 a = *reinterpret_cast<const float2*>(cb_g + j * 2);
        cv[0] = a.x; cv[1] = a.y;
    } else {
        const float4 a = *reinterpret_cast<const float4*>(cb_g + j * kC);
        cv[0] = a.x; cv[1] = a.y; cv[2 % kC] = a.z; cv[3 % kC] = a.w;
        if (kC == 8) {
            const float4 b = *reinterpret_cast<const float4*>(cb_g + j * kC + 4);
            cv[4 % kC] = b.x; cv[5 % kC] = b.y; cv[6 % kC] = b.z; cv[7 % kC] = b.w;
        }
    }
}

// Exact nearest centroid of one group of one vector, computed by the whole warp:
// d_j = sum_i (x_i - C_ji)^2 in fp32 (same operation order as the generic kernel), centroids from
// global memory (rare, and in L1 after the first), lowest j on ties.
template <int kC>
__device__ __noinline__ int tc_exact_code(const float* __restrict__ cb_g, int n_centroids, float x0, float x1, float x2, float x3,
                                          float x4, float x5, float x6, float x7)
{
    const float xs[8] = {x0, x1, x2, x3, x4, x5, x6, x7};
    const int lane = threadIdx.x & 31;
    float best = kTcInf;
    int arg = 0;
#pragma unroll 4
    for (int j = lane; j < n_centroids; j += 32) {
        float cv[kC];
        tc_fetch_centroid<kC>(cb_g, j, cv);
        float d = 0.f;
#pragma unroll
        for (int i = 0; i < kC; ++i) {
            const float diff = xs[i] - cv[i];
            d = fmaf(diff, diff, d);
        }
        if (d < best) { best = d; arg = j; }        // j increases: strict < keeps the lowest index
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oa = __shfl_xor_sync(0xffffffffu, arg, o);
        if (ob < best || (ob == best && oa < arg)) { best = ob; arg = oa; }
    }
    return arg;
}

// The scale of a group: the power of two s >= 1 that brings the largest of 32 channels spread over the centroids of a
// chunk (the same ones in every warp: no exchange between warps, and no load that waits for another) to [1, 2).  Larger
// ones stay: fp16 carries them, and a vector's channels would lose their last bits to a scale below one.  Whatever the
// other channels are, the largest squared norm N of the scaled centroids is then at least 1, and what three fp16 terms
// leave of a channel or a norm is 2^-25 at most.  Where s would have to exceed 2^15, N stays below 1 and no row is
// certain; where another centroid is so much larger (a hundred times) that fp16 does not carry its norm, neither.
// (The largest norm of all centroids instead took a barrier more: 8192 vectors x 32 heads, c = 8, 227 against 215 us,
// 211 without any scale and with wrong codes below a standard deviation of 0.03.)
template <int kC>
__device__ __forceinline__ float tc_scale(const float* __restrict__ cb_g)
{
    const int lane = threadIdx.x & 31;
    const uint32_t top = __reduce_max_sync(0xffffffffu, __float_as_uint(cb_g[lane * (8 * kC) + lane % kC]) & 0x7fffffffu);
    const int k = 127 - (int)(top >> 23);
    return __uint_as_float((uint32_t)(127 + (k < 0 ? 0 : (k > 15 ? 15 : k))) << 23);
}

// B operand of one chunk, one centroid (scaled): K slots as in the header comment; every warp leaves its largest squared
// norm and its range flag of this pass in the control block.
template <int kC>
__device__ __forceinline__ void tc_prepare_b(const float (&cv)[kC], float scale, int j, unsigned char* bbuf, TcCtl* ctl, int slot, int pass)
{
    using C = TcCfg<kC, 1>;
    float nrm = 0.f;
    float t0[kC], t1[kC], t2[kC];
#pragma unroll
    for (int i = 0; i < kC; ++i) {
        nrm = fmaf(cv[i], cv[i], nrm);
        tc_split3(-2.f * scale * cv[i], t0[i], t1[i], t2[i]);
    }
    nrm *= scale * scale;
    float n0, n1, n2;
    tc_split3(nrm, n0, n1, n2);
    const bool bad = !(nrm < 60000.f);
    const unsigned any_bad = __ballot_sync(0xffffffffu, bad);
    const float wmax = __uint_as_float(__reduce_max_sync(0xffffffffu, bad ? 0u : __float_as_uint(nrm)));   // nrm >= 0: bits order as values
    if ((threadIdx.x & 31) == 0) {
        ctl->range_flag[slot][pass * 4 + (threadIdx.x >> 5)] = any_bad != 0;
        ctl->nmax[slot][pass * 4 + (threadIdx.x >> 5)] = wmax;
    }
    const uint32_t ones = 0x3c003c00u;               // half2(1, 1)
    uint32_t pr[C::kSteps][8];
    if (kC == 2) {
        pr[0][0] = tc_pack_half2(t0[0], t0[1]);
        pr[0][1] = tc_pack_half2(t1[0], t1[1]);
        pr[0][2] = tc_pack_half2(t2[0], t2[1]);
        pr[0][3] = tc_pack_half2(n0, n1);
        pr[0][4] = ones;
        pr[0][5] = tc_pack_half2(n2, 0.f);
        pr[0][6] = 0u;
        pr[0][7] = 0u;
    } else if (kC == 4) {
        pr[0][0] = tc_pack_half2(t0[0], t0[1]);
        pr[0][1] = tc_pack_half2(t0[2 % kC], t0[3 % kC]);
        pr[0][2] = tc_pack_half2(t1[0], t1[1]);
        pr[0][3] = tc_pack_half2(t1[2 % kC], t1[3 % kC]);
        pr[0][4] = tc_pack_half2(t2[0], t2[1]);
        pr[0][5] = tc_pack_half2(t2[2 % kC], t2[3 % kC]);
        pr[0][6] = tc_pack_half2(n0, n1);
        pr[0][7] = ones;
    } else {
        constexpr int kLast = C::kSteps - 1;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            pr[0][w] = tc_pack_half2(t0[(2 * w) % kC], t0[(2 * w + 1) % kC]);
            pr[0][4 + w] = tc_pack_half2(t1[(2 * w) % kC], t1[(2 * w + 1) % kC]);
            pr[kLast][w] = tc_pack_half2(t2[(2 * w) % kC], t2[(2 * w + 1) % kC]);
        }
        pr[kLast][4] = tc_pack_half2(n0, n1);
        pr[kLast][5] = ones;
        pr[kLast][6] = tc_pack_half2(n2, 0.f);
        pr[kLast][7] = 0u;
    }
#pragma unroll
    for (int s = 0; s < C::kSteps; ++s) {
        unsigned char* dst = bbuf + s * C::kBTile + j * 16;
        *reinterpret_cast<uint4*>(dst) = make_uint4(pr[s][0], pr[s][1], pr[s][2], pr[s][3]);              // K slots 0 ... 7
        *reinterpret_cast<uint4*>(dst + 256 * 16) = make_uint4(pr[s][4], pr[s][5], pr[s][6], pr[s][7]);   // K slots 8 ... 15
    }
}

// The kC / 2 words (two fp16 channels each) of one group of one vector, from global memory.
template <int kC>
__device__ __forceinline__ void tc_fetch_x(const __half* gp, uint32_t (&xw)[kC / 2])
{
    if (kC == 2) {
        xw[0] = *reinterpret_cast<const uint32_t*>(gp);
    } else if (kC == 4) {
        const uint2 t = *reinterpret_cast<const uint2*>(gp);
        xw[0] = t.x; xw[1 % (kC / 2)] = t.y;
    } else {
        const uint4 t = *reinterpret_cast<const uint4*>(gp);
        xw[0] = t.x; xw[1 % (kC / 2)] = t.y; xw[2 % (kC / 2)] = t.z; xw[3 % (kC / 2)] = t.w;
    }
}

// A operand row of one vector for one group.  xw: the group's words, X its squared norm; atile: the row tile's first K step.
template <int kC>
__device__ __forceinline__ void tc_build_a(const uint32_t (&xw)[kC / 2], float X, unsigned char* atile, int row)
{
    using C = TcCfg<kC, 1>;
    const uint32_t ones = 0x3c003c00u, one_zero = 0x00003c00u;   // half2(1, 1), half2(1, 0)
    const float x0 = __half2float(__float2half_rn(X));
    const uint32_t xn = tc_pack_half2(x0, X - x0);
    uint4 lo[C::kSteps], hi[C::kSteps];
    if (kC == 2) {
        lo[0] = make_uint4(xw[0], xw[0], xw[0], ones);
        hi[0] = make_uint4(xn, one_zero, 0u, 0u);
    } else if (kC == 4) {
        lo[0] = make_uint4(xw[0], xw[1 % (kC / 2)], xw[0], xw[1 % (kC / 2)]);
        hi[0] = make_uint4(xw[0], xw[1 % (kC / 2)], ones, xn);
    } else {
        constexpr int kLast = C::kSteps - 1;
        const uint4 xs = make_uint4(xw[0], xw[1 % (kC / 2)], xw[2 % (kC / 2)], xw[3 % (kC / 2)]);
        lo[0] = xs;
        hi[0] = xs;
        lo[kLast] = xs;
        hi[kLast] = make_uint4(ones, xn, one_zero, 0u);
    }
#pragma unroll
    for (int s = 0; s < C::kSteps; ++s) {
        unsigned char* dst = atile + s * C::kATile + row * 16;
        *reinterpret_cast<uint4*>(dst) = lo[s];
        *reinterpret_cast<uint4*>(dst + 128 * 16) = hi[s];
    }
}

static_assert(sizeof(TcCtl) <= 512, "control block");

// The scores of half a step (128 columns of tensor memory, this thread's row) into the minima of the grid's columns (sb) and
// the smallest and second smallest minimum of its rows (m1, m2; the row's index rides in the low mantissa bits).  row0: the
// first grid row of the half.
template <uint32_t kRowBits>
__device__ __forceinline__ void tc_scan_half(float (&sb)[16], float& m1, float& m2, uint32_t taddr, int row0)
{
    float va[32], vb[32];
    auto consume = [&](const float (&v)[32], int first) {
#pragma unroll
        for (int q = 0; q < 16; ++q) sb[q] = tc_min3(sb[q], v[q], v[q + 16]);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            float t[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) t[k] = tc_min3(v[16 * e + 3 * k], v[16 * e + 3 * k + 1], v[16 * e + 3 * k + 2]);
            const float r = fminf(tc_min3(t[0], t[1], t[2]), tc_min3(t[3], t[4], v[16 * e + 15]));
            const float rt = __uint_as_float((__float_as_uint(r) & ~kRowBits) | (uint32_t)(first + e));
            m2 = fminf(m2, fmaxf(m1, rt));
            m1 = fminf(m1, rt);
        }
    };
    tc_ld32_issue(va, taddr);
    tc_ld_wait(va);
    tc_ld32_issue(vb, taddr + 32);
    consume(va, row0);
    tc_ld_wait(vb);
    tc_ld32_issue(va, taddr + 64);
    consume(vb, row0 + 2);
    tc_ld_wait(va);
    tc_ld32_issue(vb, taddr + 96);
    consume(va, row0 + 4);
    tc_ld_wait(vb);
    consume(vb, row0 + 6);
}

// Smallest and second smallest column minimum (a tournament of (smallest, second) pairs); the column rides in the low four
// mantissa bits, which also makes the 16 values differ.
__device__ __forceinline__ void tc_column_minima(const float (&sb)[16], float& c1, float& c2)
{
    float lo[8], hi[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float ta = __uint_as_float((__float_as_uint(sb[2 * i]) & ~15u) | (uint32_t)(2 * i));
        const float tb = __uint_as_float((__float_as_uint(sb[2 * i + 1]) & ~15u) | (uint32_t)(2 * i + 1));
        lo[i] = fminf(ta, tb);
        hi[i] = fmaxf(ta, tb);
    }
#pragma unroll
    for (int n = 4; n >= 1; n >>= 1)
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float m = fminf(lo[i], lo[i + n]);
            hi[i] = tc_min3(fmaxf(lo[i], lo[i + n]), hi[i], hi[i + n]);
            lo[i] = m;
        }
    c1 = lo[0];
    c2 = hi[0];
}

// Every centroid but the named one lies in another row or another column of the grid, so its score is at least
// the smaller of the two second minima.  tau bounds, for two scores and in units of X + N (of the scaled values,
// N = nmax): the sums of an MMA, exact terms of at most X + N each, aligned to the largest and cut below its last
// fp32 bit (11, 16 and, in two MMAs, 30 of them: 2.7e-6, 3.9e-6, 7.2e-6 for c = 2, 4, 8); the rounding of the exact
// distances that decide elsewhere, (c + 2) 2^-24 of at most 2 (X + N) each, and of the norms, c 2^-24 (1.3e-6,
// 2.0e-6, 3.4e-6); what the fp16 terms leave (0.2e-6; 0.4e-6 for c = 4, whose norms have two); and, on top, the
// mantissa bits given to the indexes.
template <int kC, uint32_t kRowBits>
__device__ __forceinline__ float tc_tau(float m1, float m2, float X, float nmax)
{
    return (kC == 8 ? 1.2e-5f : kC == 4 ? 6.5e-6f : 4.5e-6f) * (X + nmax) + (kRowBits == 15u ? 2.1e-6f : 8e-6f) * (fabsf(m2) + fabsf(m1));
}

}  // namespace

}  // namespace cq
