// The kernel ahead of the attention of a decode step: the append of the new tokens and, for few queries, the attention's
// tables.
//
// Append.  A CTA of the attention that works the new token's codes out itself reads the value centroids (128 KiB) once more
// than it otherwise would, per sequence; here they are read once per 16 sequences (encode_few).  16 x 4096 tokens, 32 heads
// of CQ-4c8b: step 72.9 -> 66.2 us (attention alone 59.4); 15 x 10 k, 40 heads of CQ-2c8b: 281 -> 264.
//
// Tables.  The attention (cq_decode.cu) looks the scores up in scale * log2(e) * <q_g, C_j> per (query head, group, code value).
// With few queries its few CTAs read the key centroids one after the other while most SMs idle; here a warp takes 4 kU code
// values of eight groups past all queries, so that the table is ready in the time of one load.  One sequence of 1024
// tokens, one head of CQ-8c8b, calls back to back on the same buffers: 14.3 -> 9.3 to 9.8 us (append alone: 11); a first call on
// buffers that the GPU has not seen 24.
#include "cq_encode_few.cuh"

namespace cq {

namespace {

constexpr int kTabThreads = 256;
constexpr int kTabRows = 32;              // queries of a KV head that a CTA takes at most
// Entries up to which tables ahead pay (step, us, tables by the attention's CTAs before this kernel appended > tables ahead; the
// append ahead alone takes attention + 3): 32 heads of CQ-8c8b, 128 tokens, 1 sequence (2^17 entries) 14.5 > 10.7, 2 (2^18)
// 14.5 > 13.3, 4 (2^19) 14.5 > 14.2; 32 heads of CQ-4c8b, 1 sequence of 1063 tokens (2^18) 18.4 > 19.0; 32 heads on 8, 4
// sequences (2^20) 18.6 > 19.8.
// With many queries the attention's CTAs overlap their builds with each other's loops, and the tables only cost a
// trip through L2: 64 sequences of 1024 tokens, 32 heads on 8, CQ-2c8b: attention 180 > 216.
constexpr int64_t kMostEntries = 1 << 17;

// A warp: eight neighbouring groups x four neighbouring code values at a time (whole sectors of the codebook and of the
// tables), kU such steps of centroids in registers.
template <int kC, int kPer>
__global__ void __launch_bounds__(kTabThreads)
decode_ahead_kernel(const __half* __restrict__ q, const float* __restrict__ kcb, const float* __restrict__ vcb,
                     const int32_t* __restrict__ seq_lens, float scale_log2e, Shape sh, int rows_per_cta, int n_append_ctas, int append_share, int next_at_start,
                     float* __restrict__ tables, AppendArgs app)
{
    // launched ahead of the end of whatever lies before it; next_at_start: the attention behind it may be launched from here on, and
    // waits (see the launch)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (next_at_start) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    constexpr int kRows = 256 * kPer, kU = kC == 8 ? 4 : 8;
    constexpr int kPerCta = kTabThreads / 32 * 4 * kU;             // code values of a CTA
    static_assert(kRows % kPerCta == 0, "whole CTAs");
    if ((int)blockIdx.x < n_append_ctas) {                         // (key and value; the longer CTAs first)
        const int e = blockIdx.x, each = n_append_ctas / 2;
        const bool value = e >= each;
        if constexpr (kPer == 1)
            encode_few<kC>(value ? app.v_new : app.k_new, value ? vcb : kcb, seq_lens, sh, value ? e - each : e, (int)sh.n_seq, append_share, 1, 0,
                           value ? app.vc_w : app.kc_w, true);
        return;
    }
    __shared__ __align__(16) float qs[kTabRows][8 * kC];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int octets = sh.G / 8, n_rows = (int)sh.n_seq * sh.R;
    int e = blockIdx.x - n_append_ctas;
    const int jr = e % (kRows / kPerCta);          e /= kRows / kPerCta;
    const int oct = e % octets;                    e /= octets;
    const int hkv = e % sh.n_kv_heads, row0 = e / sh.n_kv_heads * rows_per_cta;
    const int nr = n_rows - row0 < rows_per_cta ? n_rows - row0 : rows_per_cta;
    const int gl = lane & 7, g = oct * 8 + gl, j0 = jr * kPerCta + warp * 4 * kU + (lane >> 3);
    float cv[kU][kC];
    const float* src = kcb + (((int64_t)hkv * sh.G + g) * kRows + j0) * kC;
#pragma unroll
    for (int u = 0; u < kU; ++u) {
        if (kC == 2) {
            const float2 a = *reinterpret_cast<const float2*>(src + u * 4 * kC);
            cv[u][0] = a.x; cv[u][1] = a.y;
        } else {
#pragma unroll
            for (int w = 0; w < kC; w += 4) {
                const float4 a = *reinterpret_cast<const float4*>(src + u * 4 * kC + w);
                cv[u][w] = a.x; cv[u][(w + 1) % kC] = a.y; cv[u][(w + 2) % kC] = a.z; cv[u][(w + 3) % kC] = a.w;
            }
        }
    }
    for (int i = threadIdx.x; i < nr * 8 * kC; i += kTabThreads) {
        const int row = i / (8 * kC), d = i % (8 * kC);
        const int64_t at = (int64_t)((row0 + row) / sh.R) * sh.n_q_heads + hkv * sh.R + (row0 + row) % sh.R;
        qs[row][d] = __half2float(q[at * sh.head_dim + oct * 8 * kC + d]) * scale_log2e;
    }
    __syncthreads();
    for (int row = 0; row < nr; ++row) {
        float qv[kC];
#pragma unroll
        for (int i = 0; i < kC; ++i) qv[i] = qs[row][gl * kC + i];
        const int64_t at = (int64_t)((row0 + row) / sh.R) * sh.n_q_heads + hkv * sh.R + (row0 + row) % sh.R;
        float* dst = tables + (at * kRows + j0) * sh.G + g;
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            float dot = 0.f;                       // (the order of the attention kernels' own build)
#pragma unroll
            for (int i = 0; i < kC; ++i) dot = fmaf(qv[i], cv[u][i], dot);
            dst[u * 4 * sh.G] = dot;
        }
    }
}

template <int kC, int kPer>
cudaError_t launch_ahead(const __half* q, const float* kcb, const float* vcb, const int32_t* seq_lens, float scale, const Shape& sh,
                          float* tables, const AppendArgs& app, cudaStream_t st)
{
    constexpr int kPerCta = kTabThreads / 32 * 4 * (kC == 8 ? 4 : 8);
    const int64_t base = (int64_t)sh.n_kv_heads * (sh.G / 8) * (256 * kPer / kPerCta), rows = sh.n_seq * sh.R;
    if (app.k_new && kPer != 1) return cudaErrorNotSupported;
    // one wave: two CTAs an SM, of at least four queries each
    int64_t per = (rows * base + 2 * (int64_t)device_sm_count() - 1) / (2 * (int64_t)device_sm_count());
    per = per < 4 ? 4 : (per > kTabRows ? kTabRows : per);
    const int64_t table_ctas = tables ? base * ((rows + per - 1) / per) : 0;
    const DecodeCtas next = decode_tuned_ctas(sh);
    // The append of CQ-2c8b takes half as many registers.  Before an attention that has nothing merged behind it, and so little of its own to
    // do, it spreads its vectors over twice the warps, unless that attention has a last wave that is nearly empty.  12 x 1000 tokens, 12
    // heads 20.2 -> 16.8 us, 37 x 1000, 8 heads 32.9 -> 30.9; but 8 x 5000, 8 heads, three CTAs to a context, 33.8 -> 34.4, 5 x 500, 32 on 16 (160
    // CTAs) 25.0 -> 25.5, and 12 x 1000, 12 heads of CQ-8c8b 12.6 -> 14.5.
    const int64_t sms = device_sm_count(), last = next.grid % sms;
    const bool wide = kC == 2 && next.parts == 1 && (next.grid <= sms || last == 0 || 2 * last >= sms);
    const int share = few_share(sh, (int)sh.n_seq, wide ? 2 * kFewWarpsPerSm : kFewWarpsPerSm);
    const int64_t append_ctas = app.k_new ? 2 * few_ctas(sh, (int)sh.n_seq, share) : 0, grid = table_ctas + append_ctas;
    if (grid > 0x7fffffff) return cudaErrorInvalidConfiguration;
    // An attention with an SM to each CTA, of which two would fit, is launched when this kernel ends, unless both together have an SM
    // for each of their CTAs: launched beside an append, its CTAs go where that has left most room, two to an SM, and stay there.  Steps
    // back to back, us, launched at the start / at the end: 12 x 1000 tokens, 12 heads of CQ-8c8b 15.4 / 12.6, of CQ-4c8b 16.9 / 13.4, 1 x 4500, 36
    // heads of CQ-4c8b 21.1 / 16.1, 64 x 1900, 2 heads on one of CQ-8c8b 26.3 / 20.3; 8 x 1900, 6 heads on 2 (64 + 48 CTAs) 12.0 / 12.2.  With more
    // CTAs than SMs (4 x 1000, 40 heads of CQ-8c8b 15.8 / 16.1, 8 x 5000, 8 heads of CQ-4c8b 22.0 / 22.8) or one that fills an SM (8 x 1000, 8 heads
    // of CQ-2c8b 16.3 / 16.7) the launch had better pass behind the append.
    const int next_at_start = tables || next.per_sm != 2 || next.grid > sms || next.grid + append_ctas <= sms ? 1 : 0;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = overlapped_config((unsigned)grid, kTabThreads, 0, st, &attr);
    auto go = [&](auto kernel) {
        return cudaLaunchKernelEx(&cfg, kernel, q, kcb, vcb, seq_lens, scale * kLog2e, sh, (int)per, (int)append_ctas, share, next_at_start, tables, app);
    };
    return go(decode_ahead_kernel<kC, kPer>);
}

// A step's inputs from pinned host memory: reads over the bus, a thread 16 bytes at a time, and no hand-over between the copy
// engine and the kernels behind.
constexpr int kFetchThreads = 256;
__global__ void __launch_bounds__(kFetchThreads) fetch_host_kernel(HostPieces p)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");      // whatever lies ahead may still read the staging area
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const size_t t = (size_t)blockIdx.x * kFetchThreads + threadIdx.x, step = (size_t)gridDim.x * kFetchThreads;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const char* src = static_cast<const char*>(p.src[i]);
        char* dst = static_cast<char*>(p.dst[i]);
        if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15u) == 0) {
            const size_t n = p.bytes[i] / 16;
            for (size_t k = t; k < n; k += step) reinterpret_cast<uint4*>(dst)[k] = reinterpret_cast<const uint4*>(src)[k];
            if (t < p.bytes[i] % 16) dst[n * 16 + t] = src[n * 16 + t];
        } else {
            for (size_t k = t; k < p.bytes[i]; k += step) dst[k] = src[k];
        }
    }
}

}  // namespace

cudaError_t launch_fetch_host(const HostPieces& pieces, cudaStream_t st)
{
    const size_t total = pieces.bytes[0] + pieces.bytes[1] + pieces.bytes[2] + pieces.bytes[3];
    const size_t ctas = (total + 16 * kFetchThreads - 1) / (16 * kFetchThreads), most = 2 * (size_t)device_sm_count();
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = overlapped_config((unsigned)(ctas < most ? ctas : most), kFetchThreads, 0, st, &attr);
    return cudaLaunchKernelEx(&cfg, fetch_host_kernel, pieces);
}

bool decode_tables_pay(const Shape& sh)
{
    return decode_tuned_supported(sh) && sh.head_dim == 128 && !decode_pair_supported(sh) &&
           sh.n_seq * sh.n_q_heads * sh.G * sh.K <= kMostEntries;
}

size_t decode_tables_bytes(const Shape& sh) { return (size_t)sh.n_seq * sh.n_q_heads * sh.G * sh.K * sizeof(float); }

cudaError_t launch_decode_ahead(const __half* q, const float* kcb, const float* vcb, const int32_t* seq_lens, float scale,
                                 const Shape& sh, float* tables, const AppendArgs& app, cudaStream_t st)
{
    if (sh.K == 1024 && sh.c == 8) return launch_ahead<8, 4>(q, kcb, vcb, seq_lens, scale, sh, tables, app, st);
    if (sh.K != 256) return cudaErrorNotSupported;
    switch (sh.c) {
        case 2: return launch_ahead<2, 1>(q, kcb, vcb, seq_lens, scale, sh, tables, app, st);
        case 4: return launch_ahead<4, 1>(q, kcb, vcb, seq_lens, scale, sh, tables, app, st);
        case 8: return launch_ahead<8, 1>(q, kcb, vcb, seq_lens, scale, sh, tables, app, st);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace cq
