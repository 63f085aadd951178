// Causal attention of a run of new tokens over the CQ-coded cache (a prompt, or a chunk of one).
//
// Section 2.1 of the paper: Eq. 1 gives the output of "the current token" from the keys and values
// of all tokens up to and including it; here it is applied to each of the n_q newest cached tokens,
// with K and V replaced by their CQ reconstructions (Section 3.2).  Query i of sequence s sits at
// position seq_lens[s] - n_q + i and attends the cached tokens 0 ... that position.
//
// With many queries per cached token the per-query lookup tables of the decode kernels no longer
// pay (one table per query); the codes are turned back into vectors instead and the two
// contractions run on the tensor cores:
//   prefill_tc_kernel (head_dim 128, one byte per code, c = 2, 4 or 8): one CTA per (sequence, KV
//     head, 256 (query, head of the KV head's group) rows), as two row tiles of 128, one row per lane
//     of tensor memory.  Both codebooks are kept in shared memory as fp16, code-major, so that the
//     lanes of a gather (one group each) meet in no bank whatever the codes are.  Four producer warps
//     gather the codes of 64 cached tokens into swizzled fp16 tiles (three stages); S = Q Khat^T and
//     O += P Vhat are tcgen05 MMAs with fp32 accumulators, Q and P read from tensor memory, issued by
//     a warp each; eight softmax warps take a row per thread (running maximum, log2 domain).
//     What bounds it: per 64 tokens and 256 rows the MMAs take 1024 cycles and the exponentials 1024
//     (two per clock and SM quarter); each waits for the other in turn through the two row tiles.
//     4 x 2048 queries over 8192 tokens, 32 heads on 8, CQ-8c8b: 3.20 ms with m16n8k16 MMAs and the
//     tiles' fragments in registers, 1.36 ms with one MMA-issuing thread that did scores and sums in
//     turn, 0.95 ms now, 0.57 ms being the contractions at the measured GEMM rate.
//   prefill_generic_kernel: any supported shape, one CTA per (sequence, query, head), plain loops.
#include "cq_common.cuh"

#include <type_traits>

namespace cq {

namespace {

// ------------------------------------------------------------------------------------------
// generic kernel
// ------------------------------------------------------------------------------------------
constexpr int kGenWarps = 4;
constexpr int kMaxLaneCh = 8;          // head_dim <= 256: up to 8 channels per lane

__global__ void __launch_bounds__(kGenWarps * 32)
prefill_generic_kernel(const __half* __restrict__ q, const uint8_t* __restrict__ kc, const uint8_t* __restrict__ vc,
                       const float* __restrict__ kcb, const float* __restrict__ vcb,
                       const int32_t* __restrict__ seq_lens, float scale_log2e, Shape sh, int n_q, float* __restrict__ out)
{
    __shared__ float red_m[kGenWarps], red_l[kGenWarps];
    __shared__ float red_acc[kGenWarps][256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int hq = blockIdx.x % sh.n_q_heads;
    const int qi = (blockIdx.x / sh.n_q_heads) % n_q;
    const int64_t s = blockIdx.x / ((int64_t)sh.n_q_heads * n_q);
    const int hkv = hq / sh.R;
    int64_t n = seq_lens[s];
    n = n < 0 ? 0 : (n > sh.max_tokens ? sh.max_tokens : n);
    const int64_t n_att = n - n_q + qi + 1;                              // tokens 0 .. position of the query
    const int64_t row = (s * n_q + qi) * sh.n_q_heads + hq;
    float* o = out + row * sh.head_dim;
    if (n_att <= 0) {
        for (int d = threadIdx.x; d < sh.head_dim; d += blockDim.x) o[d] = 0.f;
        return;
    }
    float qd[kMaxLaneCh], acc[kMaxLaneCh];
#pragma unroll
    for (int j = 0; j < kMaxLaneCh; ++j) {
        const int d = lane + 32 * j;
        qd[j] = d < sh.head_dim ? __half2float(q[row * sh.head_dim + d]) * scale_log2e : 0.f;
        acc[j] = 0.f;
    }
    float m = -INFINITY, l = 0.f;
    for (int64_t t = warp; t < n_att; t += kGenWarps) {
        const uint8_t* kblk = kc + code_word_offset(sh, sh.n_kv_heads, s, hkv, t / kTokenBlock, 0);
        const uint8_t* vblk = vc + code_word_offset(sh, sh.n_kv_heads, s, hkv, t / kTokenBlock, 0);
        const int k = (int)(t % kTokenBlock);
        float dot = 0.f, vv[kMaxLaneCh];
#pragma unroll
        for (int j = 0; j < kMaxLaneCh; ++j) {
            const int d = lane + 32 * j;
            vv[j] = 0.f;
            if (d < sh.head_dim) {
                const int g = d / sh.c, i = d % sh.c;
                dot = fmaf(qd[j], kcb[(((int64_t)hkv * sh.G + g) * sh.K + read_code(kblk, sh, g, k)) * sh.c + i], dot);
                vv[j] = vcb[(((int64_t)hkv * sh.G + g) * sh.K + read_code(vblk, sh, g, k)) * sh.c + i];
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
        const float m_new = fmaxf(m, dot);
        const float corr = exp2f(m - m_new), p = exp2f(dot - m_new);
        l = l * corr + p;
#pragma unroll
        for (int j = 0; j < kMaxLaneCh; ++j) acc[j] = fmaf(p, vv[j], acc[j] * corr);
        m = m_new;
    }
    if (lane == 0) { red_m[warp] = m; red_l[warp] = l; }
#pragma unroll
    for (int j = 0; j < kMaxLaneCh; ++j) red_acc[warp][lane + 32 * j] = acc[j];
    __syncthreads();
    float M = -INFINITY;
    for (int w = 0; w < kGenWarps; ++w) M = fmaxf(M, red_m[w]);
    float L = 0.f;
    for (int w = 0; w < kGenWarps; ++w) L += red_m[w] == -INFINITY ? 0.f : exp2f(red_m[w] - M) * red_l[w];
    for (int d = threadIdx.x; d < sh.head_dim; d += blockDim.x) {
        float a = 0.f;
        for (int w = 0; w < kGenWarps; ++w)
            if (red_m[w] != -INFINITY) a = fmaf(exp2f(red_m[w] - M), red_acc[w][d], a);
        o[d] = a / L;
    }
}

// ------------------------------------------------------------------------------------------
// tensor-core kernel
// ------------------------------------------------------------------------------------------
struct PfCfg {
    static constexpr int kRows = 256;             // (query, head) rows per CTA: two tiles of 128, one tensor-memory lane each
    static constexpr int kMmaWarp = 8;            // one thread issues the MMAs; the warps before it: softmax, four per row tile, a thread per row
    static constexpr int kProducerWarp0 = 9, kProducerWarps = 4;       // dequantise the tiles
    static constexpr int kSumWarp = kProducerWarp0 + kProducerWarps;
    static constexpr int kThreads = (kSumWarp + 1) * 32;
    static constexpr int kTile = 64;              // cached tokens per step
    static constexpr int kStages = 3;
    static constexpr int kCbBytes = 128 * 256 * 2;                     // one codebook as fp16, code-major
    static constexpr int kKcbOffset = 0, kVcbOffset = kCbBytes;
    static constexpr int kHalfBytes = kTile * 128;                     // 64 channels of a tile: rows of 128 bytes, one per token
    static constexpr int kTileBytes = 2 * kHalfBytes;
    static constexpr int kVtOffset = 2 * kCbBytes;                     // [stages]
    static constexpr int kKtOffset = kVtOffset + kStages * kTileBytes; // [stages]
    static constexpr int kCtlOffset = kKtOffset + kStages * kTileBytes;
    static constexpr int kSmemBytes = kCtlOffset + 256;                // 224.25 KiB
    // tensor-memory columns: output accumulators (fp32) and queries (fp16, two per column) of both row tiles, ONE tile of
    // scores (fp32) that the row tiles use in turn, weights (fp16) of both row tiles
    static constexpr int kOCol = 0, kQCol = 256, kSCol = 384, kPCol = 448;
    // where the set-up leaves the queries: behind stage 0, which the producers fill while they are read
    static constexpr int kOutStride = 144;        // bytes between the rows of a warp's 32 x 32 block of results (in the codebooks' place)
    __host__ __device__ static constexpr int q_offset(int rho) { return (rho < 128 ? kVtOffset : kKtOffset) + kTileBytes + (rho & 127) * 256; }
    static_assert(kStages >= 3 && 8 * 32 * kOutStride <= 2 * kCbBytes, "room");
    static_assert(kKtOffset % 1024 == 0 && kTileBytes % 1024 == 0, "swizzled tiles");
    static_assert(kSmemBytes <= 227 * 1024, "shared memory");
};

struct PfCtl {
    uint64_t full[PfCfg::kStages];        // K and V tile of the stage are written (one arrival per producer warp)
    uint64_t empty[PfCfg::kStages];       // the MMAs that read the stage are done
    uint64_t s_full[2];                   // scores of the row tile are in tensor memory
    uint64_t s_free[2];                   // they have been read (one arrival per warp): their columns take the other row tile's
    uint64_t q_full[2];                   // queries of the row tile are in tensor memory (one arrival per warp)
    uint64_t p_full[2];                   // its weights are (one arrival per warp)
    uint64_t pv_done[2];                  // the sums with those weights are done
    uint64_t drained[2];                  // every MMA of the warp that issues the scores / the sums is done
    uint32_t tmem_base;
    int failed;                           // a wait gave up
};
static_assert(sizeof(PfCtl) <= 256, "control block");

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi)
{
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// 2^x by the special-function unit (two units in the last place; P is rounded to fp16 afterwards)
__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float max3(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

__device__ __forceinline__ void pf_init(uint64_t* bar, int arrivals)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(arrivals) : "memory");
}
__device__ __forceinline__ void pf_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Waits for the phase with the given parity; gives up after a bounded number of polls, or when another wait has, and then
// returns false: the other roles leave their loops (by a vote: the lanes of a warp can come out of it with different
// answers), the softmax warps run through theirs, in step and for nothing, and their rows become NaN.
#ifndef CQ_PREFILL_POLLS
#define CQ_PREFILL_POLLS (1 << 17)
#endif
__device__ __forceinline__ bool pf_wait(PfCtl* ctl, uint64_t* bar, uint32_t parity)
{
    for (int poll = 0; poll < CQ_PREFILL_POLLS; ++poll) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(smem_u32(bar)), "r"(parity) : "memory");
        if (done) return true;
        if ((poll & 63) == 63 && *reinterpret_cast<volatile int*>(&ctl->failed)) return false;
    }
    ctl->failed = 1;
    return false;
}

// Shared-memory matrix descriptor of a tile of 128-byte rows with the 128-byte swizzle (16-byte chunk index XOR row mod 8).
// Rows = tokens.  As keys (contraction along the row) eight rows are one core matrix group of 1024 bytes; as values (the
// row is the N dimension) the next 64 channels are kHalfBytes on and the next eight tokens 1024 bytes.  Low word: start
// address and leading offset in 16-byte units; high word: stride offset, descriptor version of sm_100, swizzle.
__device__ __forceinline__ uint32_t pf_desc_lo(uint32_t saddr, uint32_t leading_bytes) { return (saddr >> 4) | ((leading_bytes >> 4) << 16); }
constexpr uint32_t kPfDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
// D[128 x N] (+)= A[128 x 16] * B, A (fp16) from tensor memory, B (fp16) from shared memory, fp32 accumulator
__device__ __forceinline__ void pf_mma(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t idesc, bool accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 d;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b64 d, {%2, %3};\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], d, %4, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(kPfDescHi), "r"(idesc), "r"(accumulate ? 1u : 0u) : "memory");
}
// One lane of the warp, the same one every time.  (A branch on this, unlike one on the lane number, lets the compiler keep
// the operands of the MMAs in uniform registers: an issue costs some ten cycles instead of seventy.)
__device__ __forceinline__ bool pf_elect()
{
    uint32_t is;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(is));
    return is != 0;
}
__device__ __forceinline__ void pf_commit(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Waits, also after another wait has given up, until the MMAs that this warp has issued are done with shared memory and
// tensor memory: the CTA gives both back next.
__device__ __forceinline__ void pf_drain(uint64_t* bar)
{
    if (pf_elect()) pf_commit(bar);
    for (int poll = 0; poll < (1 << 20); ++poll) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(smem_u32(bar)) : "memory");
        if (done) break;
    }
    __syncwarp();
}

#define CQ_R32(u) "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15]), "=r"(u[16]), "=r"(u[17]), "=r"(u[18]), "=r"(u[19]), "=r"(u[20]), "=r"(u[21]), "=r"(u[22]), "=r"(u[23]), "=r"(u[24]), "=r"(u[25]), "=r"(u[26]), "=r"(u[27]), "=r"(u[28]), "=r"(u[29]), "=r"(u[30]), "=r"(u[31])
#define CQ_RW32(u) "+r"(u[0]), "+r"(u[1]), "+r"(u[2]), "+r"(u[3]), "+r"(u[4]), "+r"(u[5]), "+r"(u[6]), "+r"(u[7]), "+r"(u[8]), "+r"(u[9]), "+r"(u[10]), "+r"(u[11]), "+r"(u[12]), "+r"(u[13]), "+r"(u[14]), "+r"(u[15]), "+r"(u[16]), "+r"(u[17]), "+r"(u[18]), "+r"(u[19]), "+r"(u[20]), "+r"(u[21]), "+r"(u[22]), "+r"(u[23]), "+r"(u[24]), "+r"(u[25]), "+r"(u[26]), "+r"(u[27]), "+r"(u[28]), "+r"(u[29]), "+r"(u[30]), "+r"(u[31])
#define CQ_IN32(u) "r"(u[0]), "r"(u[1]), "r"(u[2]), "r"(u[3]), "r"(u[4]), "r"(u[5]), "r"(u[6]), "r"(u[7]), "r"(u[8]), "r"(u[9]), "r"(u[10]), "r"(u[11]), "r"(u[12]), "r"(u[13]), "r"(u[14]), "r"(u[15]), "r"(u[16]), "r"(u[17]), "r"(u[18]), "r"(u[19]), "r"(u[20]), "r"(u[21]), "r"(u[22]), "r"(u[23]), "r"(u[24]), "r"(u[25]), "r"(u[26]), "r"(u[27]), "r"(u[28]), "r"(u[29]), "r"(u[30]), "r"(u[31])
// 32 consecutive columns of this thread's row (the values are there after pf_ld_wait, whose registers pass through it)
__device__ __forceinline__ void pf_ld32(uint32_t (&u)[32], uint32_t taddr)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : CQ_R32(u) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void pf_ld_wait(uint32_t (&u)[32]) { asm volatile("tcgen05.wait::ld.sync.aligned;" : CQ_RW32(u)::"memory"); }
__device__ __forceinline__ void pf_st32(uint32_t taddr, const uint32_t (&u)[32])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
                 ::"r"(taddr), CQ_IN32(u) : "memory");
}
__device__ __forceinline__ void pf_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void pf_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void pf_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

template <int kC>
__global__ void __launch_bounds__(PfCfg::kThreads, 1)
prefill_tc_kernel(const __half* __restrict__ q, const uint8_t* __restrict__ kc, const uint8_t* __restrict__ vc,
                  const float* __restrict__ kcb, const float* __restrict__ vcb,
                  const int32_t* __restrict__ seq_lens, float scale_log2e, Shape sh, int n_q, int row_tiles,
                  float* __restrict__ out)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");      // launched ahead of the end of the kernel before it, and
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");       // the kernel behind it ahead of its own
    using C = PfCfg;
    constexpr int G = 128 / kC;
    extern __shared__ __align__(1024) uint8_t smem[];
    PfCtl* ctl = reinterpret_cast<PfCtl*>(smem + C::kCtlOffset);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int R = sh.R;
    const int q_per_tile = C::kRows / R;                                   // query tokens of one row tile

    const int tile = row_tiles - 1 - blockIdx.x % row_tiles;               // later queries attend more tokens: they start first
    const int hkv = (blockIdx.x / row_tiles) % sh.n_kv_heads;
    const int64_t s = blockIdx.x / ((int64_t)row_tiles * sh.n_kv_heads);
    int64_t n = seq_lens[s];
    n = n < 0 ? 0 : (n > sh.max_tokens ? sh.max_tokens : n);
    const int qi0 = tile * q_per_tile;
    // row rho of the CTA: query qi0 + rho / R, head hkv * R + rho % R, position n - n_q + query
    const int64_t pos0 = n - n_q + qi0;                                    // position of the tile's first query (may be negative)
    int q_last = qi0 + q_per_tile - 1;
    if (q_last > n_q - 1) q_last = n_q - 1;
    const int64_t pos_last = n - n_q + q_last;                             // largest position of the tile
    const int n_tiles = pos_last < 0 ? 0 : (int)(pos_last / C::kTile + 1);
    const int n_halves = (q_last - qi0 + 1) * R > 128 ? 2 : 1;             // row tiles of 128 in use
    // (a negative scale: the queries change sign instead; a zero one: they become zero; both are exact)
    const uint32_t q_sign = scale_log2e < 0.f ? 0x80008000u : 0u, q_keep = scale_log2e == 0.f ? 0u : 0xffffffffu;
    const float scale = scale_log2e == 0.f ? 1.f : fabsf(scale_log2e);

    // ---- barriers, tensor memory
    if (threadIdx.x == 0) {
        for (int i = 0; i < C::kStages; ++i) {
            pf_init(&ctl->full[i], C::kProducerWarps);
            pf_init(&ctl->empty[i], 1);
        }
        for (int t = 0; t < 2; ++t) {
            pf_init(&ctl->s_full[t], 1);
            pf_init(&ctl->s_free[t], 4);
            pf_init(&ctl->q_full[t], 4);
            pf_init(&ctl->p_full[t], 4);
            pf_init(&ctl->pv_done[t], 1);
            pf_init(&ctl->drained[t], 1);
        }
        ctl->failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == C::kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&ctl->tmem_base)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // ---- queries, coalesced, into the tile buffers of stages 1 and 2 (row tile 0: the values', 1: the keys'); 16-byte chunk
    // i of row rho goes to chunk i XOR (rho mod 8) of its 256 bytes, so that a thread per row can read them without conflicts
#pragma unroll 4
    for (int i = threadIdx.x; i < n_halves * 128 * 16; i += C::kThreads) {
        const int rho = i >> 4, qi = qi0 + rho / R;
        uint4 x = make_uint4(0u, 0u, 0u, 0u);
        if (qi < n_q) x = reinterpret_cast<const uint4*>(q + ((s * n_q + qi) * sh.n_q_heads + hkv * R + rho % R) * 128)[i & 15];
        *reinterpret_cast<uint4*>(smem + C::q_offset(rho) + (((i & 15) ^ (rho & 7)) << 4)) = x;
    }
    // ---- codebooks as fp16, code-major ([code][group][channel]): the lanes of a gather take different groups, so they
    // meet in no bank whatever the codes are.  For c = 2 (one word per centroid) group g sits in column
    // 16 (g mod 4) + g / 4.  A warp takes 64 bytes of eight groups at a time, a quarter of it two groups: two lines of
    // memory per quarter of a load, and at most four lanes that meet in a bank of a store.  (Straight copies, whose stores
    // met eight at a time, took 12.7 thousand cycles per CTA; 4 thousand are what the L2 takes to deliver 256 KB.)
    {
        constexpr int kTasks = 2 * 256, kBatch = 6, kWarps = C::kThreads / 32;
        const int gl = lane >> 2, j = lane & 3;
#pragma unroll 1
        for (int i0 = warp; i0 < kTasks; i0 += kBatch * kWarps) {
            float4 x[kBatch];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const int i = i0 + u * kWarps, o = (i & 255) % (G / 8), seg = (i & 255) / (G / 8);
                const int g = kC == 2 ? 4 * (8 * (o >> 2) + gl) + (o & 3) : 8 * o + gl;
                if (i < kTasks)
                    x[u] = reinterpret_cast<const float4*>((i < 256 ? kcb : vcb) + (int64_t)hkv * 128 * 256)[(g * 16 * kC + seg) * 4 + j];
            }
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const int i = i0 + u * kWarps, o = (i & 255) % (G / 8), seg = (i & 255) / (G / 8);
                if (i >= kTasks) break;
                uint8_t* book = smem + (i < 256 ? C::kKcbOffset : C::kVcbOffset);
                const uint32_t lo = pack_half2(x[u].x, x[u].y), hi = pack_half2(x[u].z, x[u].w);
                if (kC == 8) *reinterpret_cast<uint2*>(book + (seg * 2 + (j >> 1)) * 256 + (8 * o + gl) * 16 + (j & 1) * 8) = make_uint2(lo, hi);
                if (kC == 4) *reinterpret_cast<uint2*>(book + (seg * 4 + j) * 256 + (8 * o + gl) * 8) = make_uint2(lo, hi);
                if (kC == 2) {
                    uint8_t* dst = book + (seg * 8 + 2 * j) * 256 + (16 * (o & 3) + 8 * (o >> 2) + gl) * 4;
                    *reinterpret_cast<uint32_t*>(dst) = lo;
                    *reinterpret_cast<uint32_t*>(dst + 256) = hi;
                }
            }
        }
    }
    pf_fence_before();
    __syncthreads();
    pf_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&ctl->tmem_base);

    if (warp >= C::kProducerWarp0 && warp < C::kSumWarp) {
        // ---------------------------------------------------------------- producers: codes -> fp16 tiles of 64 tokens
        // A warp takes one 16-token block of the tile.  16-byte chunk `ch` (channels 8 ch ... + 7) of token t goes to byte
        // (ch / 8) * kHalfBytes + t * 128 + ((ch % 8) ^ (t % 8)) * 16: eight lanes of a store hold the chunks of one token,
        // so they meet in no bank either.
        const int pw = warp - C::kProducerWarp0;
        const uint8_t* kbase = kc + code_word_offset(sh, sh.n_kv_heads, s, hkv, 0, 0);
        const uint8_t* vbase = vc + code_word_offset(sh, sh.n_kv_heads, s, hkv, 0, 0);
        constexpr int kW = kC == 8 ? 2 : kC == 4 ? 4 : 8;                   // code words a lane takes of a block, per tensor
        uint32_t kw[kW], vw[kW], kn[kW], vn[kW];        // this tile's and the next one's, loaded a whole tile ahead of their use
        auto load_codes = [&](int jt, uint32_t (&kw)[kW], uint32_t (&vw)[kW]) {
            const int64_t blk = (int64_t)jt * (C::kTile / kTokenBlock) + pw;
#pragma unroll
            for (int i = 0; i < kW; ++i) kw[i] = vw[i] = 0u;
            if (jt >= n_tiles || blk >= sh.n_blocks) return;
            const uint8_t* kp = kbase + blk * (G * kTokenBlock);
            const uint8_t* vp = vbase + blk * (G * kTokenBlock);
            if (kC == 8) {                              // lane = (token half, group)
                const int off = (lane & 15) * kTokenBlock + 8 * (lane >> 4);
                const uint2 a = *reinterpret_cast<const uint2*>(kp + off), b = *reinterpret_cast<const uint2*>(vp + off);
                kw[0] = a.x; kw[1] = a.y; vw[0] = b.x; vw[1] = b.y;
            } else if (kC == 4) {                       // lane = group
                const uint4 a = *reinterpret_cast<const uint4*>(kp + lane * kTokenBlock), b = *reinterpret_cast<const uint4*>(vp + lane * kTokenBlock);
                kw[0] = a.x; kw[1] = a.y; kw[2 % kW] = a.z; kw[3 % kW] = a.w;
                vw[0] = b.x; vw[1] = b.y; vw[2 % kW] = b.z; vw[3 % kW] = b.w;
            } else {                                    // lane = (token half, chunk of four groups, taken in another order by the other half)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int off = (4 * (lane & 15) + (i ^ (lane >> 4))) * kTokenBlock + 8 * (lane >> 4);
                    const uint2 a = *reinterpret_cast<const uint2*>(kp + off), b = *reinterpret_cast<const uint2*>(vp + off);
                    kw[(2 * i) % kW] = a.x; kw[(2 * i + 1) % kW] = a.y; vw[(2 * i) % kW] = b.x; vw[(2 * i + 1) % kW] = b.y;
                }
            }
        };
        auto fill = [&](const uint32_t (&w)[kW], int book, int tile_off) {
            if (kC == 4) {
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const uint32_t code = (w[(k >> 2) % kW] >> (8 * (k & 3))) & 0xffu;
                    const int tok = 16 * pw + k;
                    const uint32_t dst = (uint32_t)((lane >> 4) * C::kHalfBytes + tok * 128 + ((((lane >> 1) & 7) ^ (k & 7)) << 4) + 8 * (lane & 1));
                    *reinterpret_cast<uint2*>(smem + tile_off + dst) = *reinterpret_cast<const uint2*>(smem + book + (code * G + lane) * 8);
                }
            } else {
                const int ch = lane & 15;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int tok = 16 * pw + 8 * (lane >> 4) + k;
                    const uint32_t dst = (uint32_t)((ch >> 3) * C::kHalfBytes + tok * 128 + (((ch & 7) ^ k) << 4));
                    uint4 v;
                    if (kC == 8) {
                        const uint32_t code = (w[(k >> 2) % kW] >> (8 * (k & 3))) & 0xffu;
                        v = *reinterpret_cast<const uint4*>(smem + book + (code * G + ch) * 16);
                    } else {
                        // (the halves' gathers fall into different halves of the banks)
                        const int hb = lane >> 4;
                        uint32_t e[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const uint32_t code = (w[(2 * i + (k >> 2)) % kW] >> (8 * (k & 3))) & 0xffu;
                            e[i] = *reinterpret_cast<const uint32_t*>(smem + book + (code * G + 16 * (i ^ hb) + ch) * 4);
                        }
                        v = hb ? make_uint4(e[1], e[0], e[3], e[2]) : make_uint4(e[0], e[1], e[2], e[3]);
                    }
                    *reinterpret_cast<uint4*>(smem + tile_off + dst) = v;
                }
            }
        };
        load_codes(0, kn, vn);
        for (int jt = 0; jt < n_tiles; ++jt) {
            const int stage = jt % C::kStages;
#pragma unroll
            for (int i = 0; i < kW; ++i) { kw[i] = kn[i]; vw[i] = vn[i]; }
            load_codes(jt + 1, kn, vn);
            bool ok = jt < C::kStages || pf_wait(ctl, &ctl->empty[stage], (uint32_t)(jt / C::kStages - 1) & 1u);
            if (jt == 1) ok = ok && pf_wait(ctl, &ctl->q_full[lane % n_halves], 0u);      // the queries lay there
            if (!__all_sync(0xffffffffu, ok)) break;
            fill(kw, C::kKcbOffset, C::kKtOffset + stage * C::kTileBytes);
            fill(vw, C::kVcbOffset, C::kVtOffset + stage * C::kTileBytes);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) pf_arrive(&ctl->full[stage]);
        }
    } else if (warp == C::kMmaWarp) {
        // ---------------------------------------------------------------- scores: Q Khat^T of (tile, row tile) 0, 1, 2, ...
        // (All lanes of the warp go round the loop, a turn of which goes once round the stages, and different lanes wait for
        // different barriers: with everything in a one-thread branch an MMA took some 60 cycles to issue and a wait, behind
        // the exponentials in the queue that it shares with them, 200.)
        constexpr uint32_t kScores = (1u << 4) | ((64u >> 3) << 17) | ((128u >> 4) << 24);       // D fp32, A and B fp16, M = 128, N = 64
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0), kdesc = pf_desc_lo(smem_u32(smem + C::kKtOffset), 16);
        const int n_work = __shfl_sync(0xffffffffu, n_tiles * n_halves, 0);
        auto go = [&](auto halves_in_use) {
            constexpr int kHalves = decltype(halves_in_use)::value, kTurn = kHalves * C::kStages;
            if (!__all_sync(0xffffffffu, pf_wait(ctl, &ctl->q_full[lane % kHalves], 0u))) return;                // the queries
            for (int o = 0; o * kTurn < n_work; ++o) {
#pragma unroll
                for (int u = 0; u < kTurn; ++u) {
                    if (o * kTurn + u >= n_work) break;
                    const int t = u % kHalves, stage = u / kHalves, jt = o * C::kStages + stage;
                    // even lanes: the scores of the work before have been read; odd lanes: the tile is there
                    const bool first = o == 0 && u == 0;
                    uint64_t* bar = (lane & 1) || first ? &ctl->full[stage] : &ctl->s_free[t == 0 ? kHalves - 1 : 0];
                    const uint32_t parity = (lane & 1) || first ? (uint32_t)o & 1u : (uint32_t)(t == 0 ? jt - 1 : jt) & 1u;
                    if (!__all_sync(0xffffffffu, pf_wait(ctl, bar, parity))) return;
                    pf_fence_after();
                    if (pf_elect()) {
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)               // 16 channels = 32 bytes of the 128-byte rows
                            pf_mma(tm + C::kSCol, tm + C::kQCol + 64 * t + 8 * ks,
                                   kdesc + (stage * C::kTileBytes + (ks >> 2) * C::kHalfBytes + (ks & 3) * 32) / 16, kScores, ks > 0);
                        pf_commit(&ctl->s_full[t]);
                    }
                }
            }
        };
        if (n_work > 0) {
            if (n_halves == 2) go(std::integral_constant<int, 2>());
            else go(std::integral_constant<int, 1>());
            __syncwarp();
            pf_drain(&ctl->drained[0]);
        }
    } else if (warp == C::kSumWarp) {
        // ---------------------------------------------------------------- sums: P Vhat, in the same order
        constexpr uint32_t kSums = (1u << 4) | (1u << 16) | ((128u >> 3) << 17) | ((128u >> 4) << 24);   // N = 128, B's rows along N
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0), vdesc = pf_desc_lo(smem_u32(smem + C::kVtOffset), C::kHalfBytes);
        const int n_work = __shfl_sync(0xffffffffu, n_tiles * n_halves, 0);
        auto go = [&](auto halves_in_use) {
            constexpr int kHalves = decltype(halves_in_use)::value, kTurn = kHalves * C::kStages;
            for (int o = 0; o * kTurn < n_work; ++o) {
#pragma unroll
                for (int u = 0; u < kTurn; ++u) {
                    if (o * kTurn + u >= n_work) break;
                    const int t = u % kHalves, stage = u / kHalves, jt = o * C::kStages + stage;
                    uint64_t* bar = lane & 1 ? &ctl->full[stage] : &ctl->p_full[t];
                    const uint32_t parity = lane & 1 ? (uint32_t)o & 1u : (uint32_t)jt & 1u;
                    if (!__all_sync(0xffffffffu, pf_wait(ctl, bar, parity))) return;
                    pf_fence_after();
                    const bool more = jt > 0;
                    if (pf_elect()) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)               // 16 tokens = 2048 bytes
                            pf_mma(tm + C::kOCol + 128 * t, tm + C::kPCol + 32 * t + 8 * ks,
                                   vdesc + (stage * C::kTileBytes + ks * 2048) / 16, kSums, more || ks > 0);
                        pf_commit(&ctl->pv_done[t]);
                        if (t == kHalves - 1) pf_commit(&ctl->empty[stage]);
                    }
                }
            }
        };
        if (n_work > 0) {
            if (n_halves == 2) go(std::integral_constant<int, 2>());
            else go(std::integral_constant<int, 1>());
            __syncwarp();
            pf_drain(&ctl->drained[1]);
        }
    } else if (warp < 4 * n_halves) {
        // ---------------------------------------------------------------- softmax: a thread per row
        const int t = warp >> 2, rho = threadIdx.x;
        const uint32_t lanes = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const uint32_t s_addr = lanes + C::kSCol, p_addr = lanes + C::kPCol + 32 * t, o_addr = lanes + C::kOCol + 128 * t;
        const int qi = qi0 + rho / R;
        const bool live = qi < n_q;
        const int64_t pos = live ? pos0 + rho / R : -1;
        const int64_t pos_warp = pos0 + (warp * 32) / R;                   // smallest position among the warp's rows
        {
            uint32_t u[32];
#pragma unroll
            for (int half = 0; half < 2; ++half) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint4 v = *reinterpret_cast<const uint4*>(smem + C::q_offset(rho) + (((8 * half + i) ^ (rho & 7)) << 4));
                    u[4 * i] = (v.x ^ q_sign) & q_keep; u[4 * i + 1] = (v.y ^ q_sign) & q_keep;
                    u[4 * i + 2] = (v.z ^ q_sign) & q_keep; u[4 * i + 3] = (v.w ^ q_sign) & q_keep;
                }
                pf_st32(lanes + C::kQCol + 64 * t + 32 * half, u);
            }
            pf_st_wait();
            pf_fence_before();
            __syncwarp();
            if (lane == 0) pf_arrive(&ctl->q_full[t]);
        }
        float m = -INFINITY, l = 0.f;                                       // reference of the weights (log2 domain), their sum
        bool ok = true;
        for (int jt = 0; jt < n_tiles; ++jt) {
            ok &= pf_wait(ctl, &ctl->s_full[t], (uint32_t)jt & 1u);
            pf_fence_after();
            uint32_t a[32], b[32];
            pf_ld32(a, s_addr);
            pf_ld32(b, s_addr + 32);
            pf_ld_wait(a);
            pf_ld_wait(b);
            pf_fence_before();
            __syncwarp();
            if (lane == 0) pf_arrive(&ctl->s_free[t]);
            float* sa = reinterpret_cast<float*>(a);
            float* sb = reinterpret_cast<float*>(b);
            const int64_t j0 = (int64_t)jt * C::kTile;
            if (j0 + C::kTile - 1 > pos_warp) {                             // some row's causal limit lies in the tile
                const int64_t left = pos - j0;                              // columns 0 ... left are attended
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    if (i > left) sa[i] = -INFINITY;
                    if (i + 32 > left) sb[i] = -INFINITY;
                }
            }
            float mx[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) mx[i] = max3(sa[i], sb[i], sa[i + 4]);
#pragma unroll
            for (int i = 8; i < 32; i += 8)
#pragma unroll
                for (int k = 0; k < 4; ++k) mx[k] = max3(mx[k], sa[i + k], sa[i + 4 + k]);
#pragma unroll
            for (int i = 4; i < 28; i += 8)
#pragma unroll
                for (int k = 0; k < 4; ++k) mx[k] = max3(mx[k], sb[i + k], sb[i + 4 + k]);
#pragma unroll
            for (int k = 0; k < 4; ++k) mx[k] = fmaxf(mx[k], sb[28 + k]);
            const float top = max3(fmaxf(mx[0], mx[1]), mx[2], mx[3]);
            const float m_tile = top * scale;                               // (-inf: the row attends nothing of the tile)
            // The weights' reference follows the maximum only when it is more than 8 (a factor of 256) behind: the sums
            // rarely have to be rescaled, and fp16 weights up to 256 are as precise as weights up to 1.
            const bool move = m_tile > m + 8.f || (m == -INFINITY && m_tile > -INFINITY);
            const bool rescale = __any_sync(0xffffffffu, move);
            float f = 1.f;
            if (rescale) {
                const float m_new = fmaxf(m, m_tile);
                f = m == -INFINITY ? 0.f : exp2f(m - m_new);
                m = m_new;
                l *= f;
            }
            const float mm = m == -INFINITY ? 0.f : m;
            uint32_t p[32];
            float l0 = 0.f, l1 = 0.f;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float x0 = ex2_approx(fmaf(sa[2 * i], scale, -mm)), x1 = ex2_approx(fmaf(sa[2 * i + 1], scale, -mm));
                l0 += x0;
                l1 += x1;
                p[i] = pack_half2(x0, x1);
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float x0 = ex2_approx(fmaf(sb[2 * i], scale, -mm)), x1 = ex2_approx(fmaf(sb[2 * i + 1], scale, -mm));
                l0 += x0;
                l1 += x1;
                p[16 + i] = pack_half2(x0, x1);
            }
            l += l0 + l1;
            if (jt > 0) {                                                   // the last sums are done with the weights' columns
                ok &= pf_wait(ctl, &ctl->pv_done[t], (uint32_t)(jt - 1) & 1u);
                pf_fence_after();
                if (rescale) {
#pragma unroll 1
                    for (int c0 = 0; c0 < 128; c0 += 32) {
                        uint32_t o[32];
                        pf_ld32(o, o_addr + c0);
                        pf_ld_wait(o);
#pragma unroll
                        for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
                        pf_st32(o_addr + c0, o);
                    }
                }
            }
            pf_st32(p_addr, p);
            pf_st_wait();
            pf_fence_before();
            __syncwarp();
            if (lane == 0) pf_arrive(&ctl->p_full[t]);
        }
        // ---- normalise and write: through shared memory (the codebooks are done with when the last sums are), so that the
        // stores take whole lines; a thread per row wrote 32 lines at a time (10.8 thousand cycles per CTA)
        if (n_tiles > 0) ok &= pf_wait(ctl, &ctl->pv_done[t], (uint32_t)(n_tiles - 1) & 1u);
        ok = __all_sync(0xffffffffu, ok);
        pf_fence_after();
        // no position: zero row; a wait gave up: NaN rows, so that nothing takes them for a result
        const float inv = !ok ? __int_as_float(0x7fffffff) : l > 0.f ? 1.f / l : 0.f;
        uint8_t* block = smem + warp * 32 * C::kOutStride;
#pragma unroll 1
        for (int c0 = 0; c0 < 128; c0 += 32) {
            uint32_t o[32];
            if (n_tiles > 0) {
                pf_ld32(o, o_addr + c0);
                pf_ld_wait(o);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i)
                *reinterpret_cast<float4*>(block + lane * C::kOutStride + 16 * i) =
                    inv == 0.f ? make_float4(0.f, 0.f, 0.f, 0.f)
                               : make_float4(__uint_as_float(o[4 * i]) * inv, __uint_as_float(o[4 * i + 1]) * inv,
                                             __uint_as_float(o[4 * i + 2]) * inv, __uint_as_float(o[4 * i + 3]) * inv);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int rw = 4 * i + (lane >> 3), rr = warp * 32 + rw, qr = qi0 + rr / R;
                if (qr < n_q)
                    *reinterpret_cast<float4*>(out + ((s * n_q + qr) * sh.n_q_heads + hkv * R + rr % R) * 128 + c0 + 4 * (lane & 7)) =
                        *reinterpret_cast<const float4*>(block + rw * C::kOutStride + 16 * (lane & 7));
            }
            __syncwarp();
        }
        pf_fence_before();
    }
    // every MMA that was issued has been waited for; hand the tensor memory back
    __syncthreads();
    if (warp == C::kMmaWarp) {
        pf_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

}  // namespace

bool prefill_mma_supported(const Shape& sh)
{
    return sh.head_dim == 128 && sh.b == 8 && (sh.c == 2 || sh.c == 4 || sh.c == 8) && sh.R <= 64 && PfCfg::kRows % sh.R == 0;
}

cudaError_t launch_prefill(const __half* q, const uint8_t* kc, const uint8_t* vc, const float* kcb, const float* vcb,
                           const int32_t* seq_lens, float scale, const Shape& sh, int n_q, float* out, bool generic,
                           cudaStream_t st)
{
    if (!generic && prefill_mma_supported(sh)) {
        using C = PfCfg;
        const int q_per_tile = C::kRows / sh.R;
        const int row_tiles = (n_q + q_per_tile - 1) / q_per_tile;
        const int64_t grid = sh.n_seq * sh.n_kv_heads * row_tiles;
        if (grid > 0x7fffffff) return cudaErrorInvalidConfiguration;
        cudaLaunchAttribute attr;
        const cudaLaunchConfig_t cfg = overlapped_config((unsigned)grid, C::kThreads, C::kSmemBytes, st, &attr);
        auto go = [&](auto kernel, int slot) {
            const cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), C::kSmemBytes, slot);
            if (e != cudaSuccess) return e;
            return cudaLaunchKernelEx(&cfg, kernel, q, kc, vc, kcb, vcb, seq_lens, scale * kLog2e, sh, n_q, row_tiles, out);
        };
        return sh.c == 8 ? go(prefill_tc_kernel<8>, 40) : sh.c == 4 ? go(prefill_tc_kernel<4>, 41) : go(prefill_tc_kernel<2>, 42);
    }
    const int64_t grid = sh.n_seq * (int64_t)n_q * sh.n_q_heads;
    if (grid > 0x7fffffff) return cudaErrorInvalidConfiguration;
    prefill_generic_kernel<<<(unsigned)grid, kGenWarps * 32, 0, st>>>(q, kc, vc, kcb, vcb, seq_lens, scale * kLog2e, sh, n_q, out);
    return cudaGetLastError();
}

}  // namespace cq
