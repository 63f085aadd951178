// Centroid learning (Section 3.2.1 of the paper): k-means++ initialisation and k-means
// iterations, uniform (Eq. 5) or weighted per group vector (Eq. 6), for every (head, group)
// problem of a key or value tensor at once.  The assignment step of an iteration is cq_encode.
//
// k-means++ decides integers (which vector becomes the next centre) from sums of squared
// distances.  By definition those sums are formed in fp64, in index order, with one multiply and one
// add per term and no fused multiply-add, so that the decision does not depend on the machine.
// pp_cluster_kernel draws the same vectors from sums in another order, with a proof per draw that the
// order does not matter (and the ordered sum where it might); pp_pick_kernel and pp_dist_kernel are
// the plain form for shapes it does not take.
#include "cq_bulk_copy.cuh"
#include "cq_common.cuh"

namespace cq {

namespace {

// problem p = h * G + g; vector i.  dist[p][i]: squared distance of vector i to its nearest centre
// so far; contrib[p][i] = w_i * dist[p][i], the term of the k-means++ draw.

// One CTA per problem.  The CTA stages tiles of contributions in shared memory (coalesced loads, the next
// tile while the current one is summed); thread 0 adds them up in index order, so the fp64 running sum is
// the sequential one.  The running sum at the end of every tile is kept: it never decreases (the
// contributions are not negative), so the walk that looks for the drawn vector starts at the first tile
// whose end reaches the target, from the sum before that tile - the same additions in the same order as a
// walk from the first vector, without repeating them.
constexpr int kPickThreads = 128;
constexpr int kPickTile = 2048;
constexpr int kPickPrefixes = 1024;              // tile ends that are kept (later tiles are walked one by one)

// sum += v[0] + ... in order, sixteen loads in flight ahead of the chain of additions
__device__ __forceinline__ double pick_sum_tile(const double* tile, int m, double sum)
{
    int e = 0;
    for (; e + 16 <= m; e += 16) {
        double v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = tile[e + j];
#pragma unroll
        for (int j = 0; j < 16; ++j) sum = __dadd_rn(sum, v[j]);
    }
    for (; e < m; ++e) sum = __dadd_rn(sum, tile[e]);
    return sum;
}

__global__ void __launch_bounds__(kPickThreads)
pp_pick_kernel(const __half* __restrict__ x, const double* __restrict__ uniforms, const double* __restrict__ contrib,
               int64_t n_vec, int n_prob, int c, int K, int k, float* __restrict__ codebooks)
{
    __shared__ double tile[2][kPickTile];
    __shared__ double s_prefix[kPickPrefixes];
    __shared__ double s_total;
    __shared__ long long s_pick;
    const int p = blockIdx.x;
    const double u = uniforms[(int64_t)p * K + k];
    const double* cp = contrib + (int64_t)p * n_vec;
    const int64_t n_tiles = (n_vec + kPickTile - 1) / kPickTile;
    auto stage = [&](int64_t t, int buf) {
        const int64_t t0 = t * kPickTile;
        const int m = (int)(n_vec - t0 < kPickTile ? n_vec - t0 : kPickTile);
        // warp 0 does not stage: its first thread is busy with the chain of additions
        for (int e = (int)threadIdx.x - 32; e >= 0 && e < m; e += kPickThreads - 32) tile[buf][e] = cp[t0 + e];
    };
    if (threadIdx.x == 0) s_pick = -1;
    if (k > 0) {
        double total = 0.0;
        stage(0, 0);
        for (int64_t t = 0; t < n_tiles; ++t) {
            __syncthreads();                                  // tile t is staged, the other buffer is free
            if (t + 1 < n_tiles) stage(t + 1, (int)((t + 1) & 1));
            if (threadIdx.x == 0) {
                const int64_t t0 = t * kPickTile;
                const int m = (int)(n_vec - t0 < kPickTile ? n_vec - t0 : kPickTile);
                total = pick_sum_tile(tile[t & 1], m, total);
                if (t < kPickPrefixes) s_prefix[t] = total;
            }
        }
        if (threadIdx.x == 0) s_total = total;
        __syncthreads();
        if (s_total > 0.0) {
            const double target = __dmul_rn(u, s_total);
            // first tile whose end reaches the target (every thread takes the same decision)
            int64_t first = 0;
            const int64_t kept = n_tiles < kPickPrefixes ? n_tiles : kPickPrefixes;
            while (first < kept && !(s_prefix[first] >= target)) ++first;
            if (first == n_tiles) first = n_tiles - 1;      // rounding put the target past the total: the last tile decides
            double run = first > 0 ? s_prefix[first - 1] : 0.0;
            for (int64_t t = first; t < n_tiles; ++t) {
                const int64_t t0 = t * kPickTile;
                const int m = (int)(n_vec - t0 < kPickTile ? n_vec - t0 : kPickTile);
                __syncthreads();
                if (s_pick >= 0) break;                     // same value in every thread: read after the barrier
                for (int e = threadIdx.x; e < m; e += kPickThreads) tile[0][e] = cp[t0 + e];
                __syncthreads();
                if (threadIdx.x == 0)
                    for (int e = 0; e < m; ++e) {
                        run = __dadd_rn(run, tile[0][e]);
                        if (run >= target && tile[0][e] > 0.0) { s_pick = t0 + e; break; }
                    }
            }
            __syncthreads();
            if (threadIdx.x == 0 && s_pick < 0) s_pick = n_vec - 1;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        long long pick = s_pick;
        if (pick < 0) pick = (long long)__dmul_rn(u, (double)n_vec);       // first centre, or no vector left to draw
        if (pick >= n_vec) pick = n_vec - 1;
        // x row of vector `pick`: all problems of a vector are contiguous (p * c = h * D + g * c)
        const __half* xv = x + pick * (int64_t)n_prob * c + (int64_t)p * c;
        float* cb = codebooks + ((int64_t)p * K + k) * c;
        for (int q = 0; q < c; ++q) cb[q] = __half2float(xv[q]);
    }
}

// k-means++ of a whole problem by one thread-block cluster.  The vectors of the problem are split over the CTAs of
// the cluster (kPpSlice each at most) and stay on chip for all the draws: the vectors and weights in shared memory,
// distances and contributions in registers.  One draw is two exchanges:
//   1. every thread brings the distances of its vectors up to date with the last centre (an fp32 bound with its
//      rounding error taken off rules out nearly all of them, the others are evaluated in fp64 as defined), the warps
//      sum their contributions and hand the sums to every CTA of the cluster;
//   2. every warp finds the warp whose range holds the target, that warp finds the vector and hands it to all.
// The definition asks for the running sum in index order, an n-long chain of dependent fp64 additions (0.8 ms a draw
// at 32768 vectors, which is what bounded this step).  The sums here are taken in another order, but a draw only
// depends on which vector's running sum first reaches the target: any order of n non-negative terms is within
// n 2^-53 of the total T, so where the target is farther than that from both ends of the vector's interval the two
// orders draw the same vector.  Otherwise (about one draw in a million) the cluster writes its contributions out and
// one thread adds them up in index order.  Measured (32768 vectors, 512 problems, 256 centres, c = 8, weighted):
// 213 -> 21.7 ms with a cluster barrier after each exchange and the drawn vector read from memory again, 19.9 as it is now.
// A draw takes 12.8 thousand cycles with two CTAs on an SM: 3.9 the distances (mostly those that go to fp64, where the
// conversions take the time; exact differences built from the bits instead of conversions: 28.8 ms), 2.8 the wait for the
// slowest warp's sum, 1.5 finding the warp, 1.6 the wait for the vector.
constexpr int kPpThreads = 512;
constexpr int kPpWarps = kPpThreads / 32;
constexpr int kPpPer = 8;                          // vectors per thread
constexpr int kPpSlice = kPpThreads * kPpPer;      // vectors per CTA
constexpr int kPpUniforms = 256;                   // of a problem, kept on chip
constexpr int kPpMaxCluster = 8;                   // portable cluster size

// Draw k uses the buffers k & 1.  A CTA sends what belongs to draw k + 2 only when it knows the centre of draw k + 1, which
// takes the sums of every warp of the cluster, so whatever belongs to draw k has been read by then.
struct PpCtl {
    double sums[2][kPpMaxCluster * kPpWarps];      // contributions per (CTA of the cluster, warp), in index order
    alignas(16) uint32_t centre[2][4];             // the drawn vector's channels, fp16
    long long pick[2];                             // the drawn vector; -1: too close to call
    uint64_t sums_here[2], pick_here[2];           // mbarriers: all of that has arrived
};

// Stores to another CTA's shared memory that count themselves at an mbarrier there.
__device__ __forceinline__ void pp_send64(uint32_t to, unsigned long long v, uint32_t bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(to), "l"(v), "r"(bar) : "memory");
}
template <int kWords>
__device__ __forceinline__ void pp_send32(uint32_t to, const uint32_t (&w)[kWords], uint32_t bar)
{
    if (kWords == 4)
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                     ::"r"(to), "r"(w[0]), "r"(w[1 % kWords]), "r"(w[2 % kWords]), "r"(w[3 % kWords]), "r"(bar) : "memory");
    else if (kWords == 2)
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];"
                     ::"r"(to), "r"(w[0]), "r"(w[1 % kWords]), "r"(bar) : "memory");
    else
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(to), "r"(w[0]), "r"(bar) : "memory");
}
// The next phase of an mbarrier (nothing is ordered by it: what it counts is sent later).
__device__ __forceinline__ void pp_arm(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.relaxed.cta.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
// Waits for the phase with the given parity; gives up after some seconds (returns false).  The limit is one of time, since a poll may
// suspend the thread for as long as the hardware likes; the clock is read every 256 polls (every poll: 51.4 -> 52.2 ms of the whole call).
constexpr long long kPpWaitCycles = 1ll << 33;
__device__ __forceinline__ bool pp_wait(uint64_t* bar, uint32_t parity)
{
    long long since = 0;
    for (;;) {
        for (int poll = 0; poll < 256; ++poll) {
            uint32_t done;
            asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                         : "=r"(done) : "r"(smem_addr(bar)), "r"(parity) : "memory");
            if (done) return true;
        }
        const long long now = clock64();
        if (since == 0) since = now;
        if (now - since > kPpWaitCycles) return false;
    }
}

__device__ __forceinline__ uint32_t pp_map_shared(const void* p, int rank)
{
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void pp_cluster_sync()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// squared distance as the definition has it: one subtraction, one multiplication and one addition per channel, fp64
template <int kC>
__device__ __forceinline__ double pp_exact(const uint32_t (&xw)[kC / 2], const uint32_t (&cw)[kC / 2])
{
    double d = 0.0;
#pragma unroll
    for (int q = 0; q < kC / 2; ++q) {
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&xw[q]));
        const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&cw[q]));
        const double dx = __dsub_rn((double)a.x, (double)b.x), dy = __dsub_rn((double)a.y, (double)b.y);
        d = __dadd_rn(d, __dmul_rn(dx, dx));
        d = __dadd_rn(d, __dmul_rn(dy, dy));
    }
    return d;
}

template <int kC>
__device__ __forceinline__ void pp_words(const unsigned char* p, uint32_t (&w)[kC / 2])
{
    if (kC == 8) {
        const uint4 v = *reinterpret_cast<const uint4*>(p);
        w[0] = v.x; w[1 % (kC / 2)] = v.y; w[2 % (kC / 2)] = v.z; w[3 % (kC / 2)] = v.w;
    } else if (kC == 4) {
        const uint2 v = *reinterpret_cast<const uint2*>(p);
        w[0] = v.x; w[1 % (kC / 2)] = v.y;
    } else {
        w[0] = *reinterpret_cast<const uint32_t*>(p);
    }
}

// The draw as defined, by one thread: the running sum in index order, then the first vector with a contribution whose
// running sum reaches u times the total.  (The total is known to be positive.)
__device__ __noinline__ long long pp_serial_pick(const double* cp, int64_t n_vec, double u)
{
    double total = 0.0;
    int64_t i = 0;
    for (; i + 16 <= n_vec; i += 16) {
        double v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = __ldcg(cp + i + j);
#pragma unroll
        for (int j = 0; j < 16; ++j) total = __dadd_rn(total, v[j]);
    }
    for (; i < n_vec; ++i) total = __dadd_rn(total, __ldcg(cp + i));
    const double target = __dmul_rn(u, total);
    double run = 0.0;
    for (i = 0; i < n_vec; ++i) {
        const double v = __ldcg(cp + i);
        run = __dadd_rn(run, v);
        if (run >= target && v > 0.0) return i;
    }
    return n_vec - 1;
}

template <int kC>
__global__ void __launch_bounds__(kPpThreads, 2)
pp_cluster_kernel(const __half* __restrict__ x, const float* __restrict__ weights, const double* __restrict__ uniforms,
                  int64_t n_vec, int n_prob, int K, int cluster, int slice, double* contrib, float* __restrict__ codebooks)
{
    extern __shared__ __align__(16) unsigned char pp_smem[];        // [slice][kC] fp16, then [slice] weights
    __shared__ PpCtl ctl;
    __shared__ double us[kPpUniforms];
    unsigned char* xs = pp_smem;
    float* ws = reinterpret_cast<float*>(pp_smem + (size_t)slice * kC * 2);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rank = blockIdx.x % cluster, p = blockIdx.x / cluster;
    const int64_t base = (int64_t)rank * slice;
    const int64_t left = n_vec - base;
    const int m = left <= 0 ? 0 : (left < slice ? (int)left : slice);      // vectors of this CTA
    for (int i = threadIdx.x; i < m; i += kPpThreads) {
        uint32_t w[kC / 2];
        pp_words<kC>(reinterpret_cast<const unsigned char*>(x + ((base + i) * n_prob + p) * kC), w);
#pragma unroll
        for (int q = 0; q < kC / 2; ++q) reinterpret_cast<uint32_t*>(xs + (size_t)i * kC * 2)[q] = w[q];
        if (weights) ws[i] = weights[(base + i) * n_prob + p];
    }
    // a warp holds a run of 32 * per vectors of the slice, 32 consecutive ones per step j < per
    const int per = (slice + kPpThreads - 1) / kPpThreads;
    const int first = warp * (32 * per) + lane;
    double dist[kPpPer], part[kPpPer];
#pragma unroll
    for (int j = 0; j < kPpPer; ++j) {
        dist[j] = j < per && first + 32 * j < m ? (double)INFINITY : 0.0;
        part[j] = 0.0;
    }
    const double* up = uniforms + (int64_t)p * K;
    for (int i = threadIdx.x; i < kPpMaxCluster * kPpWarps; i += kPpThreads) ctl.sums[0][i] = ctl.sums[1][i] = 0.0;
    constexpr uint32_t kPickBytes = kC * 2 + 8;
    const uint32_t sums_bytes = (uint32_t)cluster * kPpWarps * 8;
    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(&ctl.sums_here[b], 1);
            mbar_init(&ctl.pick_here[b], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int b = 0; b < 2; ++b) {
            pp_arm(&ctl.sums_here[b], sums_bytes);
            pp_arm(&ctl.pick_here[b], kPickBytes);
        }
    }
    __syncthreads();
    pp_cluster_sync();                                              // every CTA of the cluster has started: its memory may be written

    // The vector `pick` (index within the problem, its words w) becomes centre k: one whole warp hands it to every CTA.  plain:
    // between two cluster barriers, for a draw that was undecided; otherwise counted at the CTAs' mbarriers.
    auto publish = [&](int64_t pick, int k, const uint32_t (&w)[kC / 2], bool plain) {
        const int b = k & 1;
        if (lane < cluster) {
            if (plain) {
#pragma unroll
                for (int q = 0; q < kC / 2; ++q)
                    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(pp_map_shared(&ctl.centre[b][q], lane)), "r"(w[q]) : "memory");
                asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(pp_map_shared(&ctl.pick[b], lane)), "l"((long long)pick) : "memory");
            } else {
                const uint32_t bar = pp_map_shared(&ctl.pick_here[b], lane);
                pp_send32<kC / 2>(pp_map_shared(&ctl.centre[b][0], lane), w, bar);
                pp_send64(pp_map_shared(&ctl.pick[b], lane), (unsigned long long)pick, bar);
            }
        }
        if (pick < 0) return;
        if (lane == 0) {
            float* cb = codebooks + ((int64_t)p * K + k) * kC;
#pragma unroll
            for (int q = 0; q < kC / 2; ++q) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[q]));
                cb[2 * q] = f.x;
                cb[2 * q + 1] = f.y;
            }
        }
    };
    auto publish_any = [&](int64_t pick, int k, bool plain) {        // (a vector that may lie in another CTA's slice)
        uint32_t w[kC / 2];
        pp_words<kC>(reinterpret_cast<const unsigned char*>(x + (pick * n_prob + p) * kC), w);
        publish(pick, k, w, plain);
    };
    // no running sum decides: the first centre, or every vector already is a centre
    auto plain_pick = [&](double u) {
        int64_t pick = (int64_t)__dmul_rn(u, (double)n_vec);
        return pick >= n_vec ? n_vec - 1 : pick;
    };

    bool ok = true;                      // false: a wait gave up (never expected); the problem's centroids become NaN
    for (int k = 0; k < K; ++k) {
        if (k % kPpUniforms == 0) {      // (from memory, each would be a trip of a tenth of a draw)
            __syncthreads();
            if (threadIdx.x < kPpUniforms && k + (int)threadIdx.x < K) us[threadIdx.x] = up[k + threadIdx.x];
            __syncthreads();
        }
        const double u = us[k % kPpUniforms];
        if (k == 0) {
            if (rank == 0 && warp == 0) publish_any(plain_pick(u), 0, false);
            if (!(ok = pp_wait(&ctl.pick_here[0], 0u))) break;
            if (threadIdx.x == 0) pp_arm(&ctl.pick_here[0], kPickBytes);
            continue;
        }
        const int b = k & 1;
        // ---- distances to the centre drawn last; sum of the contributions of this warp's vectors
        uint32_t cw[kC / 2];
        float cf[kC];
#pragma unroll
        for (int q = 0; q < kC / 2; ++q) {
            cw[q] = ctl.centre[b ^ 1][q];
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&cw[q]));
            cf[2 * q] = f.x;
            cf[2 * q + 1] = f.y;
        }
        double sum = 0.0;
#pragma unroll
        for (int j = 0; j < kPpPer; ++j) {
            const int i = first + 32 * j;
            if (j < per && i < m) {
                uint32_t xw[kC / 2];
                pp_words<kC>(xs + (size_t)i * kC * 2, xw);
                float d32 = 0.f;
#pragma unroll
                for (int q = 0; q < kC / 2; ++q) {
                    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&xw[q]));
                    const float dx = f.x - cf[2 * q], dy = f.y - cf[2 * q + 1];
                    d32 = fmaf(dx, dx, d32);
                    d32 = fmaf(dy, dy, d32);
                }
                // d32 is within 2e-6 of the distance (differences of fp16 values rounded once, sums of squares).  The comparison
                // is one of the upper words of doubles, which a float's bits give without a conversion (d32 is zero, normal
                // or not finite: squares of fp16 differences are 2^-48 at least): never false for a smaller distance.
                if ((int)((__float_as_uint(d32 * 0.999996f) >> 3) + (896u << 20)) <= __double2hiint(dist[j])) {
                    const double d = pp_exact<kC>(xw, cw);
                    if (d < dist[j]) {
                        dist[j] = d;
                        part[j] = __dmul_rn(weights ? (double)ws[i] : 1.0, d);
                    }
                }
            }
            sum += part[j];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane < cluster)
            pp_send64(pp_map_shared(&ctl.sums[b][rank * kPpWarps + warp], lane), (unsigned long long)__double_as_longlong(sum),
                      pp_map_shared(&ctl.sums_here[b], lane));
        if (!(ok = pp_wait(&ctl.sums_here[b], (uint32_t)((k - 1) >> 1) & 1u))) break;
        if (threadIdx.x == 0) pp_arm(&ctl.sums_here[b], sums_bytes);         // for draw k + 2

        // ---- which warp's range holds the target (the same answer in every warp of the cluster)
        constexpr int kPerLane = kPpMaxCluster * kPpWarps / 32;
        double s[kPerLane], run = 0.0;
#pragma unroll
        for (int e = 0; e < kPerLane; ++e) {
            s[e] = ctl.sums[b][lane * kPerLane + e];
            run += s[e];
        }
        double upto = run;                                          // inclusive over the lanes
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double t = __shfl_up_sync(0xffffffffu, upto, o);
            if (lane >= o) upto += t;
        }
        const double total = __shfl_sync(0xffffffffu, upto, 31);
        const double target = __dmul_rn(u, total);
        if (!(total > 0.0) || target != target) {
            // (zero times an infinite total is not a number: no running sum reaches it, and as defined the last vector is drawn)
            if (rank == 0 && warp == 0) publish_any(total > 0.0 ? n_vec - 1 : plain_pick(u), k, false);
        } else {
            const double slack = total * ((double)n_vec + 64.0) * 4.5e-16;
            const unsigned hit = __ballot_sync(0xffffffffu, upto >= target);
            // (the lanes' order of the sums is the vectors' order; no hit: the target is within rounding of the total)
            const int at = hit ? __ffs(hit) - 1 : 31;
            double before = __shfl_sync(0xffffffffu, upto - run, at);
            int unit = at * kPerLane + kPerLane - 1;
#pragma unroll
            for (int e = 0; e < kPerLane - 1; ++e) {
                const double se = __shfl_sync(0xffffffffu, s[e], at);
                if (unit == at * kPerLane + kPerLane - 1) {
                    if (before + se >= target) unit = at * kPerLane + e;
                    else before += se;
                }
            }
            if (unit == rank * kPpWarps + warp) {
                int64_t pick = -1;
                // sums of the steps j: after the exchanges with lane masks 16, 8, 4 a lane holds step lane / 4
                static_assert(kPpPer == 8, "the exchange folds eight sums");
                double f4[4], f2[2], rows;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const double keep = (lane & 16) ? part[e + 4] : part[e], send = (lane & 16) ? part[e] : part[e + 4];
                    f4[e] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
                }
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const double keep = (lane & 8) ? f4[e + 2] : f4[e], send = (lane & 8) ? f4[e] : f4[e + 2];
                    f2[e] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
                }
                {
                    const double keep = (lane & 4) ? f2[1] : f2[0], send = (lane & 4) ? f2[0] : f2[1];
                    rows = keep + __shfl_xor_sync(0xffffffffu, send, 4);
                }
                rows += __shfl_xor_sync(0xffffffffu, rows, 2);
                rows += __shfl_xor_sync(0xffffffffu, rows, 1);
                double inc = rows;
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) {
                    const double t = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += t;
                }
                const unsigned in = __ballot_sync(0xffffffffu, before + inc >= target);
                if (in) {
                    const int src = (__ffs(in) - 1) & ~3, j = src >> 2;
                    before += __shfl_sync(0xffffffffu, inc - rows, src);
                    double v = part[0];
#pragma unroll
                    for (int t = 1; t < kPpPer; ++t) v = j == t ? part[t] : v;
                    inc = v;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const double t = __shfl_up_sync(0xffffffffu, inc, o);
                        if (lane >= o) inc += t;
                    }
                    // (rounding may leave the target above this step's last sum: then it is too close to call)
                    const unsigned hit_in = __ballot_sync(0xffffffffu, before + inc >= target);
                    const int l = hit_in ? __ffs(hit_in) - 1 : 0;
                    const bool clear = target - (before + (inc - v)) > slack && (before + inc) - target > slack;
                    if (__shfl_sync(0xffffffffu, clear ? 1 : 0, l) && hit_in) pick = base + warp * (32 * per) + 32 * j + l;
                }
                if (pick < 0 || pick >= n_vec) pick = -1;
                uint32_t w[kC / 2];                                  // (this CTA's slice holds it)
                pp_words<kC>(xs + (size_t)(pick < 0 ? 0 : pick - base) * kC * 2, w);
                publish(pick, k, w, false);
            }
        }
        if (!(ok = pp_wait(&ctl.pick_here[b], (uint32_t)(k >> 1) & 1u))) break;
        if (threadIdx.x == 0) pp_arm(&ctl.pick_here[b], kPickBytes);

        if (*reinterpret_cast<volatile long long*>(&ctl.pick[b]) < 0) {         // the same value in every CTA of the cluster
            double* cp = contrib + (int64_t)p * n_vec;
#pragma unroll
            for (int j = 0; j < kPpPer; ++j)
                if (j < per && first + 32 * j < m) cp[base + first + 32 * j] = part[j];
            __threadfence();
            pp_cluster_sync();
            if (rank == 0 && warp == 0) {
                long long pick = 0;
                if (lane == 0) pick = pp_serial_pick(cp, n_vec, u);
                pick = __shfl_sync(0xffffffffu, pick, 0);
                publish_any(pick, k, true);
            }
            pp_cluster_sync();
        }
    }
    pp_cluster_sync();                                              // no CTA leaves while another may write to its memory
    if (!ok && lane == 0)
        for (int i = 0; i < K * kC; ++i) codebooks[(int64_t)p * K * kC + i] = __int_as_float(0x7fc00000);
}

// Distances to the nearest chosen centre and the contributions w * D, for tiles of 32 vectors x 32 problems.
// x and the weights are vector-major, the distances and contributions problem-major (a draw reads one
// problem's run): the tile is turned in shared memory so that every global access runs along the
// contiguous index.  Thread (tx, ty): tx is the vector when the problem-major arrays are touched and the
// problem when x is read.
constexpr int kDistTile = 32;
__global__ void __launch_bounds__(256)
pp_dist_kernel(const __half* __restrict__ x, const float* __restrict__ weights, const float* __restrict__ codebooks,
               int64_t n_vec, int n_prob, int c, int K, int k, double* __restrict__ dist, double* __restrict__ contrib)
{
    __shared__ double d_s[kDistTile][kDistTile + 1];          // [problem][vector]
    __shared__ double c_s[kDistTile][kDistTile + 1];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t tiles_i = (n_vec + kDistTile - 1) / kDistTile;
    const int64_t tiles_p = (n_prob + kDistTile - 1) / kDistTile;
    for (int64_t tile = blockIdx.x; tile < tiles_i * tiles_p; tile += gridDim.x) {
        const int64_t i0 = (tile % tiles_i) * kDistTile;
        const int p0 = (int)(tile / tiles_i) * kDistTile;
        if (k > 0) {
            for (int pp = ty; pp < kDistTile; pp += 8)
                if (p0 + pp < n_prob && i0 + tx < n_vec) d_s[pp][tx] = dist[(int64_t)(p0 + pp) * n_vec + i0 + tx];
        }
        __syncthreads();
        for (int ii = ty; ii < kDistTile; ii += 8) {
            const int64_t i = i0 + ii;
            const int p = p0 + tx;
            if (i < n_vec && p < n_prob) {
                const __half* xv = x + (i * n_prob + p) * c;
                const float* cb = codebooks + ((int64_t)p * K + k) * c;
                double d = 0.0;
                for (int q = 0; q < c; ++q) {
                    const double diff = __dsub_rn((double)__half2float(xv[q]), (double)cb[q]);
                    d = __dadd_rn(d, __dmul_rn(diff, diff));
                }
                if (k > 0 && !(d < d_s[tx][ii])) d = d_s[tx][ii];
                const double w = weights ? (double)weights[i * n_prob + p] : 1.0;
                d_s[tx][ii] = d;
                c_s[tx][ii] = __dmul_rn(w, d);
            }
        }
        __syncthreads();
        for (int pp = ty; pp < kDistTile; pp += 8)
            if (p0 + pp < n_prob && i0 + tx < n_vec) {
                const int64_t idx = (int64_t)(p0 + pp) * n_vec + i0 + tx;
                dist[idx] = d_s[pp][tx];
                contrib[idx] = c_s[pp][tx];
            }
        __syncthreads();
    }
}

// New centroids and objective for two neighbouring groups of a head (kPair = 2: their channels of a vector share a
// 32-byte sector at c = 8, their weights and codes lie side by side) or for one.  The vectors are taken in tiles: the tile
// is staged in shared memory and counting-sorted by code (one integer atomic per vector), then every kC / 2
// lanes walk an equal run of the sorted members and add up one centroid after the other.  The form before this added every channel of every vector
// with an fp32 shared-memory atomic, a compare-and-swap loop that kept the shared-memory pipe 85 % busy.
// A cluster of CTAs shares the tiles of a problem (few problems) and adds its accumulators up at the end.
// The objective is formed only where it is asked for.  Measured (32768 vectors, 512 problems, c = 8, weighted):
// 1.42 -> 0.41 ms; the staging's loads (every lane another row) and the sort take most of that.
constexpr int kUpdThreads = 512;
constexpr int kUpdWarps = kUpdThreads / 32;
constexpr int kUpdTile = 2048;
constexpr int kUpdPer = kUpdTile / kUpdThreads;
constexpr int kUpdMaxK = 256;

template <int kC, int kPair>
struct UpdCfg {
    static constexpr int kXBytes = kUpdTile * kC * 2;                            // one problem's vectors
    static constexpr int kXOff = 0;
    static constexpr int kWOff = kXOff + kPair * kXBytes;                        // fp32 weights
    static constexpr int kIdxOff = kWOff + kPair * kUpdTile * 4;                 // uint16 vectors of the tile, sorted by code
    static constexpr int kCodeOff = kIdxOff + kPair * kUpdTile * 2;              // and their codes, one byte each
    static constexpr int kAccOff = kCodeOff + kPair * kUpdTile;                  // fp32 [kMaxK][kC + 1] sums, weight sum last
    static constexpr int kCountOff = kAccOff + kPair * kUpdMaxK * (kC + 1) * 4;  // members per code, then run starts
    static constexpr int kSmemBytes = kCountOff + kPair * (kUpdMaxK + 1) * 4;
    static_assert(kXOff % 16 == 0 && kWOff % 16 == 0 && kIdxOff % 4 == 0 && kAccOff % 4 == 0, "alignment");
    static_assert(kSmemBytes <= 113 * 1024, "two CTAs per SM");
};

// kN fp16 channels of a vector in one load (32 bytes where x is aligned to them: every lane reads another row, so each
// load instruction costs 32 tag look-ups, and their number is what the staging takes)
template <int kN>
__device__ __forceinline__ void upd_load_x(const __half* p, bool aligned32, uint32_t (&w)[kN / 2])
{
    if (kN == 16 && aligned32) {
        asm volatile("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(w[0]), "=r"(w[1 % (kN / 2)]), "=r"(w[2 % (kN / 2)]), "=r"(w[3 % (kN / 2)]), "=r"(w[4 % (kN / 2)]),
                       "=r"(w[5 % (kN / 2)]), "=r"(w[6 % (kN / 2)]), "=r"(w[7 % (kN / 2)])
                     : "l"(p));
        return;
    }
    if (kN >= 8) {
#pragma unroll
        for (int e = 0; e < kN / 8; ++e) {
            const uint4 v = *reinterpret_cast<const uint4*>(p + 8 * e);
            w[(4 * e) % (kN / 2)] = v.x; w[(4 * e + 1) % (kN / 2)] = v.y; w[(4 * e + 2) % (kN / 2)] = v.z; w[(4 * e + 3) % (kN / 2)] = v.w;
        }
    } else if (kN == 4) {
        const uint2 v = *reinterpret_cast<const uint2*>(p);
        w[0] = v.x; w[1 % (kN / 2)] = v.y;
    } else {
        w[0] = *reinterpret_cast<const uint32_t*>(p);
    }
}

template <int kC, int kPair>
__global__ void __launch_bounds__(kUpdThreads, 2)
lloyd_update_kernel(const __half* __restrict__ x, const float* __restrict__ weights, const uint8_t* __restrict__ codes,
                    const float* __restrict__ cb_in, Shape sh, int64_t n_vec, int cluster, int x_aligned32,
                    int w_aligned8, float* __restrict__ cb_out, double* __restrict__ objective)
{
    using C = UpdCfg<kC, kPair>;
    extern __shared__ __align__(16) unsigned char upd_smem[];
    __shared__ double obj_sum[kPair];
    __shared__ double obj_warp[kUpdWarps][kPair];
    float* acc = reinterpret_cast<float*>(upd_smem + C::kAccOff);
    int* count = reinterpret_cast<int*>(upd_smem + C::kCountOff);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rank = blockIdx.x % cluster;
    const int p0 = (int)(blockIdx.x / cluster) * kPair, h = p0 / sh.G, g0 = p0 % sh.G, K = sh.K;      // problems p0 ... p0 + kPair - 1
    const int n_prob = sh.n_kv_heads * sh.G;
    for (int e = threadIdx.x; e < kPair * kUpdMaxK * (kC + 1); e += kUpdThreads) acc[e] = 0.f;
    double obj[kPair];
#pragma unroll
    for (int s = 0; s < kPair; ++s) obj[s] = 0.0;

    const int64_t n_tiles = (n_vec + kUpdTile - 1) / kUpdTile;
    for (int64_t t = rank; t < n_tiles; t += cluster) {
        const int64_t i0 = t * kUpdTile;
        for (int e = threadIdx.x; e < kPair * (kUpdMaxK + 1); e += kUpdThreads) count[e] = 0;
        __syncthreads();                                    // (also: the previous tile has been summed)
        int code[kUpdPer][kPair], place[kUpdPer][kPair];
        constexpr int kAhead = 2;                           // vectors whose loads are in flight together
#pragma unroll
        for (int u0 = 0; u0 < kUpdPer; u0 += kAhead) {
            uint32_t xw[kAhead][kPair * kC / 2];
            float w[kAhead][kPair];
#pragma unroll
            for (int a = 0; a < kAhead; ++a) {
                const int64_t i = i0 + (u0 + a) * kUpdThreads + threadIdx.x;
                const bool live = i < n_vec;
                const int64_t is = live ? i : 0;
                const uint8_t* cp = codes + code_word_offset(sh, sh.n_kv_heads, 0, h, is / kTokenBlock, g0) + is % kTokenBlock;
                upd_load_x<kPair * kC>(x + (is * n_prob + p0) * kC, x_aligned32 != 0, xw[a]);
#pragma unroll
                for (int s = 0; s < kPair; ++s) {
                    code[u0 + a][s] = live ? (int)cp[s * kTokenBlock] : -1;
                    w[a][s] = 1.f;
                }
                if (weights) {
                    const float* wp = weights + is * n_prob + p0;
                    if (kPair == 2 && w_aligned8) {
                        const float2 w2 = *reinterpret_cast<const float2*>(wp);
                        w[a][0] = w2.x;
                        w[a][kPair - 1] = w2.y;
                    } else {
#pragma unroll
                        for (int s = 0; s < kPair; ++s) w[a][s] = wp[s];
                    }
                }
            }
#pragma unroll
            for (int a = 0; a < kAhead; ++a) {
                const int li = (u0 + a) * kUpdThreads + threadIdx.x;
#pragma unroll
                for (int s = 0; s < kPair; ++s) {
                    const int cs = code[u0 + a][s];
                    if (cs < 0) continue;
                    uint32_t* dst = reinterpret_cast<uint32_t*>(upd_smem + C::kXOff + s * C::kXBytes) + li * (kC / 2);
                    if (kC == 8) *reinterpret_cast<uint4*>(dst) = make_uint4(xw[a][s * (kC / 2)], xw[a][s * (kC / 2) + 1 % (kC / 2)], xw[a][s * (kC / 2) + 2 % (kC / 2)], xw[a][s * (kC / 2) + 3 % (kC / 2)]);
                    else if (kC == 4) *reinterpret_cast<uint2*>(dst) = make_uint2(xw[a][s * (kC / 2)], xw[a][s * (kC / 2) + 1 % (kC / 2)]);
                    else *dst = xw[a][s * (kC / 2)];
                    reinterpret_cast<float*>(upd_smem + C::kWOff)[s * kUpdTile + li] = w[a][s];
                    place[u0 + a][s] = atomicAdd(&count[s * (kUpdMaxK + 1) + cs], 1);
                    if (objective) {
                        const float* cc = cb_in + ((int64_t)(p0 + s) * K + cs) * kC;
                        double d = 0.0;
#pragma unroll
                        for (int q = 0; q < kC / 2; ++q) {
                            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&xw[a][s * (kC / 2) + q]));
                            const double dx = (double)f.x - (double)cc[2 * q], dy = (double)f.y - (double)cc[2 * q + 1];
                            d += dx * dx;
                            d += dy * dy;
                        }
                        obj[s] += (double)w[a][s] * d;
                    }
                }
            }
        }
        __syncthreads();
        // members per code -> first member of every code (warp s: problem s)
        if (warp < kPair) {
            int* cs = count + warp * (kUpdMaxK + 1);
            constexpr int kPerLane = kUpdMaxK / 32;
            int v[kPerLane], sum = 0;
#pragma unroll
            for (int e = 0; e < kPerLane; ++e) { v[e] = cs[lane * kPerLane + e]; sum += v[e]; }
            int upto = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int a = __shfl_up_sync(0xffffffffu, upto, o);
                if (lane >= o) upto += a;
            }
            int at = upto - sum;
#pragma unroll
            for (int e = 0; e < kPerLane; ++e) { cs[lane * kPerLane + e] = at; at += v[e]; }
            if (lane == 31) cs[kUpdMaxK] = at;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kUpdPer; ++u)
#pragma unroll
            for (int s = 0; s < kPair; ++s)
                if (code[u][s] >= 0) {
                    const int at = s * kUpdTile + count[s * (kUpdMaxK + 1) + code[u][s]] + place[u][s];
                    reinterpret_cast<uint16_t*>(upd_smem + C::kIdxOff)[at] = (uint16_t)(u * kUpdThreads + threadIdx.x);
                    (upd_smem + C::kCodeOff)[at] = (uint8_t)code[u][s];
                }
        __syncthreads();
        // kC / 2 lanes take an equal run of the sorted members, whatever the centroids' shares are, and add a
        // centroid's sum up when the code changes (its other members may be a neighbour's: hence the atomic)
        {
            constexpr int kLanes = kC / 2, kSubs = 32 / kLanes;
            constexpr int kRun = kUpdTile / (kUpdWarps / kPair * kSubs);
            static_assert(kRun % 4 == 0, "members are taken four at a time");
            const int q = lane % kLanes, sub = lane / kLanes;
            const int s = kPair == 2 ? warp & 1 : 0;
            const uint32_t* xt = reinterpret_cast<const uint32_t*>(upd_smem + C::kXOff + s * C::kXBytes) + q;
            const float* wt = reinterpret_cast<const float*>(upd_smem + C::kWOff) + s * kUpdTile;
            const int begin = (warp / kPair * kSubs + sub) * kRun;
            const uint16_t* it = reinterpret_cast<const uint16_t*>(upd_smem + C::kIdxOff) + s * kUpdTile + begin;
            const uint8_t* ct = upd_smem + C::kCodeOff + s * kUpdTile + begin;
            const int total = count[s * (kUpdMaxK + 1) + kUpdMaxK];
            const int left = total - begin < kRun ? total - begin : kRun;
            float a0 = 0.f, a1 = 0.f, aw = 0.f;
            int cur = -1;
            auto flush = [&]() {
                float* aj = acc + (s * kUpdMaxK + cur) * (kC + 1);
                atomicAdd(aj + 2 * q, a0);
                atomicAdd(aj + 2 * q + 1, a1);
                if (q == 0) atomicAdd(aj + kC, aw);
            };
            for (int e = 0; e < left; e += 4) {
                const uint2 i4 = *reinterpret_cast<const uint2*>(it + e);
                const uint32_t c4 = *reinterpret_cast<const uint32_t*>(ct + e);
                float w[4];
                uint32_t xw[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t i = ((k < 2 ? i4.x : i4.y) >> (16 * (k & 1))) & (kUpdTile - 1);
                    w[k] = e + k < left ? wt[i] : 0.f;
                    xw[k] = e + k < left ? xt[i * kLanes] : 0u;
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int code = (int)((c4 >> (8 * k)) & 0xffu);
                    if (e + k < left && code != cur) {
                        if (cur >= 0) flush();
                        cur = code;
                        a0 = a1 = aw = 0.f;
                    }
                    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&xw[k]));
                    a0 = fmaf(w[k], f.x, a0);
                    a1 = fmaf(w[k], f.y, a1);
                    aw += w[k];
                }
            }
            if (cur >= 0) flush();
        }
    }
    // objective of this CTA's tiles
    if (objective) {
#pragma unroll
        for (int s = 0; s < kPair; ++s) {
            double o = obj[s];
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) o += __shfl_xor_sync(0xffffffffu, o, d);
            if (lane == 0) obj_warp[warp][s] = o;
        }
        __syncthreads();
        if (threadIdx.x < kPair) {
            double o = 0.0;
            for (int w = 0; w < kUpdWarps; ++w) o += obj_warp[w][threadIdx.x];
            obj_sum[threadIdx.x] = o;
        }
    }
    pp_cluster_sync();
    auto remote_f32 = [](const float* p, int r) {
        float v;
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(pp_map_shared(p, r)) : "memory");
        return v;
    };
    // this CTA's share of the centroids, summed over the cluster
    for (int e = rank * kUpdThreads + threadIdx.x; e < kPair * K * kC; e += cluster * kUpdThreads) {
        const int s = e / (K * kC), j = e / kC % K, q = e % kC;
        const float* aj = acc + (s * kUpdMaxK + j) * (kC + 1);
        float v = 0.f, ws = 0.f;
        for (int r = 0; r < cluster; ++r) {
            v += remote_f32(aj + q, r);
            ws += remote_f32(aj + kC, r);
        }
        const int64_t at = ((int64_t)(p0 + s) * K + j) * kC + q;
        cb_out[at] = ws > 0.f ? v / ws : cb_in[at];
    }
    if (objective && rank == 0 && threadIdx.x < kPair) {
        double o = 0.0;
        for (int r = 0; r < cluster; ++r) {
            double v;
            asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(pp_map_shared(&obj_sum[threadIdx.x], r)) : "memory");
            o += v;
        }
        objective[p0 + threadIdx.x] = o;
    }
    pp_cluster_sync();                                      // no CTA leaves while another reads its memory
}

// Every other shape (more than 256 centroids, other group sizes): one CTA per problem, weighted sums by fp32 atomics
// in shared memory.
constexpr int kUpdGenericThreads = 256;
__global__ void __launch_bounds__(kUpdGenericThreads)
lloyd_update_generic_kernel(const __half* __restrict__ x, const float* __restrict__ weights, const uint8_t* __restrict__ codes,
                    const float* __restrict__ cb_in, Shape sh, int64_t n_vec, float* __restrict__ cb_out,
                    double* __restrict__ objective)
{
    extern __shared__ float upd_gen_smem[];            // [K][c] sums, [K] weight sums, [K][c] input centroids
    const int p = blockIdx.x, h = p / sh.G, g = p % sh.G, c = sh.c, K = sh.K;
    const int n_prob = sh.n_kv_heads * sh.G;
    float* sums = upd_gen_smem;
    float* wsum = sums + K * c;
    float* cin = wsum + K;
    for (int e = threadIdx.x; e < K * c; e += kUpdGenericThreads) { sums[e] = 0.f; cin[e] = cb_in[(int64_t)p * K * c + e]; }
    for (int e = threadIdx.x; e < K; e += kUpdGenericThreads) wsum[e] = 0.f;
    __syncthreads();
    double obj = 0.0;
    for (int64_t i = threadIdx.x; i < n_vec; i += kUpdGenericThreads) {
        const int code = read_code(codes + code_word_offset(sh, sh.n_kv_heads, 0, h, i / kTokenBlock, 0), sh, g,
                                   (int)(i % kTokenBlock));
        const float w = weights ? weights[i * n_prob + p] : 1.f;
        const __half* xv = x + (i * n_prob + p) * (int64_t)c;
        double d = 0.0;
        for (int q = 0; q < c; ++q) {
            const float xf = __half2float(xv[q]);
            const double diff = (double)xf - (double)cin[code * c + q];
            d += diff * diff;
            atomicAdd(&sums[code * c + q], w * xf);
        }
        atomicAdd(&wsum[code], w);
        obj += (double)w * d;
    }
    // objective: block reduction in fp64
    __shared__ double red[kUpdGenericThreads / 32];
    for (int o = 16; o > 0; o >>= 1) obj += __shfl_xor_sync(0xffffffffu, obj, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = obj;
    __syncthreads();
    if (threadIdx.x == 0 && objective) {
        double t = 0.0;
        for (int wv = 0; wv < kUpdGenericThreads / 32; ++wv) t += red[wv];
        objective[p] = t;
    }
    for (int e = threadIdx.x; e < K * c; e += kUpdGenericThreads) {
        const float ws = wsum[e / c];
        cb_out[(int64_t)p * K * c + e] = ws > 0.f ? sums[e] / ws : cin[e];
    }
}

// `attr` belongs to the caller and must outlive the launch
cudaLaunchConfig_t cluster_config(int grid, int threads, size_t smem, int cluster, cudaStream_t st, cudaLaunchAttribute* attr)
{
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)cluster;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// Cluster size of pp_cluster_kernel: what the vectors need, and more CTAs per problem while the device has room for
// all of them at once (few problems: a draw is then shorter).  0: more vectors than a cluster of portable size holds
// (kPpMaxCluster * kPpSlice = 32768); the draws then take two launches each.
int pp_cluster_size(int64_t n_vec, int n_prob)
{
    int c = 1;
    while (c < kPpMaxCluster && n_vec > (int64_t)c * kPpSlice) c *= 2;
    if (n_vec > (int64_t)c * kPpSlice) return 0;
    while (c < kPpMaxCluster && 2 * c * (int64_t)n_prob <= 2 * (int64_t)device_sm_count() && n_vec > (int64_t)c * 512) c *= 2;
    return c;
}

template <int kC>
cudaError_t launch_pp_cluster(const __half* x, const float* weights, const double* uniforms, const Shape& sh, int64_t n_vec,
                              int cluster, double* contrib, float* codebooks, cudaStream_t st)
{
    const int n_prob = sh.n_kv_heads * sh.G;
    const int slice = (int)(((n_vec + cluster - 1) / cluster + 31) / 32 * 32);
    const size_t smem = (size_t)slice * (kC * 2 + (weights ? 4 : 0));
    constexpr int kSlot = kC == 2 ? 35 : kC == 4 ? 36 : 37;           // call-site slots of ensure_dynamic_smem
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(pp_cluster_kernel<kC>), kPpSlice * (kC * 2 + 4), kSlot);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = cluster_config(n_prob * cluster, kPpThreads, smem, cluster, st, &attr);
    return cudaLaunchKernelEx(&cfg, pp_cluster_kernel<kC>, x, weights, uniforms, n_vec, n_prob, sh.K, cluster, slice, contrib, codebooks);
}

template <int kC, int kPair>
cudaError_t launch_update(const __half* x, const float* weights, const uint8_t* codes, const float* cb_in, const Shape& sh,
                          int64_t n_vec, float* cb_out, double* objective, cudaStream_t st)
{
    using C = UpdCfg<kC, kPair>;
    const int units = sh.n_kv_heads * sh.G / kPair;
    const int64_t tiles = (n_vec + kUpdTile - 1) / kUpdTile;
    // CTAs per unit: as many as the device has room for at once, and no more than there are tiles
    int cluster = 1;
    while (cluster < kPpMaxCluster && 2 * cluster * (int64_t)units <= 2 * (int64_t)device_sm_count() && 2 * cluster <= tiles) cluster *= 2;
    constexpr int kSlot = 56 + 2 * (kC == 2 ? 0 : kC == 4 ? 1 : 2) + (kPair - 1);     // call-site slots 56 ... 61 of ensure_dynamic_smem
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(lloyd_update_kernel<kC, kPair>), C::kSmemBytes, kSlot);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = cluster_config(units * cluster, kUpdThreads, C::kSmemBytes, cluster, st, &attr);
    return cudaLaunchKernelEx(&cfg, lloyd_update_kernel<kC, kPair>, x, weights, codes, cb_in, sh, n_vec, cluster,
                              (reinterpret_cast<uintptr_t>(x) & 31u) == 0 ? 1 : 0, (reinterpret_cast<uintptr_t>(weights) & 7u) == 0 ? 1 : 0,
                              cb_out, objective);
}

cudaError_t update_dispatch(const __half* x, const float* weights, const uint8_t* codes, const float* cb_in, const Shape& sh,
                            int64_t n_vec, float* cb_out, double* objective, cudaStream_t st)
{
#define CQ_UPD(C_) return sh.G % 2 == 0 ? launch_update<C_, 2>(x, weights, codes, cb_in, sh, n_vec, cb_out, objective, st)   \
                                        : launch_update<C_, 1>(x, weights, codes, cb_in, sh, n_vec, cb_out, objective, st)
    switch (sh.c) {
        case 2: CQ_UPD(2);
        case 4: CQ_UPD(4);
        default: CQ_UPD(8);
    }
#undef CQ_UPD
}

size_t round256(size_t v) { return (v + 255) / 256 * 256; }

struct LearnLayout {
    size_t codes, dist, tmp_cb, total;
};

LearnLayout learn_layout(const Shape& sh, int64_t n_vec)
{
    LearnLayout l;
    const size_t n_prob = (size_t)sh.n_kv_heads * sh.G;
    l.codes = round256((size_t)sh.n_kv_heads * ((n_vec + kTokenBlock - 1) / kTokenBlock) * sh.block_bytes);
    l.dist = round256((size_t)n_vec * n_prob * sizeof(double));
    l.tmp_cb = round256(n_prob * sh.K * sh.c * sizeof(float));
    l.total = l.codes + 2 * l.dist + l.tmp_cb;      // dist and contrib
    return l;
}

}  // namespace

size_t learn_least_bytes(const Shape& sh, int64_t n_vec) { return learn_layout(sh, n_vec).total; }
size_t learn_workspace_bytes(const Shape& sh, int64_t n_vec)
{
    return learn_least_bytes(sh, n_vec) + (learn_bounds_supported(sh, n_vec) ? learn_bounds_bytes(sh) : 0);
}

cudaError_t launch_kmeanspp_init(const __half* x, const float* weights, const double* uniforms, const Shape& sh,
                                 int64_t n_vec, float* codebooks, void* workspace, cudaStream_t st)
{
    const LearnLayout l = learn_layout(sh, n_vec);
    double* dist = reinterpret_cast<double*>(static_cast<char*>(workspace) + l.codes);
    const int n_prob = sh.n_kv_heads * sh.G;
    const int64_t dist_tiles = ((n_vec + kDistTile - 1) / kDistTile) * ((n_prob + kDistTile - 1) / kDistTile);
    const int64_t dist_cap = (int64_t)device_sm_count() * 64;
    const int dist_grid = (int)(dist_tiles < dist_cap ? dist_tiles : dist_cap);
    double* contrib = reinterpret_cast<double*>(static_cast<char*>(workspace) + l.codes + l.dist);
    const int cluster = pp_cluster_size(n_vec, n_prob);
    if (cluster && (sh.c == 2 || sh.c == 4 || sh.c == 8)) {
        switch (sh.c) {
            case 2: return launch_pp_cluster<2>(x, weights, uniforms, sh, n_vec, cluster, contrib, codebooks, st);
            case 4: return launch_pp_cluster<4>(x, weights, uniforms, sh, n_vec, cluster, contrib, codebooks, st);
            default: return launch_pp_cluster<8>(x, weights, uniforms, sh, n_vec, cluster, contrib, codebooks, st);
        }
    }
    // other group sizes, and more vectors than a cluster holds: one launch per draw and distance update
    for (int k = 0; k < sh.K; ++k) {
        pp_pick_kernel<<<n_prob, kPickThreads, 0, st>>>(x, uniforms, contrib, n_vec, n_prob, sh.c, sh.K, k, codebooks);
        pp_dist_kernel<<<dist_grid, 256, 0, st>>>(x, weights, codebooks, n_vec, n_prob, sh.c, sh.K, k, dist, contrib);
    }
    return cudaGetLastError();
}

cudaError_t launch_lloyd_step(const __half* x, const float* weights, const float* cb_in, const Shape& sh, int64_t n_vec,
                              float* cb_out, double* objective, void* workspace, cudaStream_t st)
{
    uint8_t* codes = static_cast<uint8_t*>(workspace);
    // assignment: the vectors are one sequence of n_vec tokens
    Shape es = sh;
    es.n_seq = 1;
    es.max_tokens = n_vec;
    es.n_blocks = (n_vec + kTokenBlock - 1) / kTokenBlock;
    cudaError_t e = encode_tuned_supported(es) ? launch_encode_tuned(x, cb_in, nullptr, es, n_vec, 0, codes, st)
                                               : launch_encode_generic(x, cb_in, nullptr, es, n_vec, 0, codes, st);
    if (e != cudaSuccess) return e;
    if (sh.K <= kUpdMaxK && (sh.c == 2 || sh.c == 4 || sh.c == 8)) return update_dispatch(x, weights, codes, cb_in, es, n_vec, cb_out, objective, st);
    const size_t smem = (size_t)(2 * sh.K * sh.c + sh.K) * sizeof(float);
    e = ensure_dynamic_smem(reinterpret_cast<const void*>(lloyd_update_generic_kernel), (int)smem, 34);
    if (e != cudaSuccess) return e;
    lloyd_update_generic_kernel<<<sh.n_kv_heads * sh.G, kUpdGenericThreads, smem, st>>>(x, weights, codes, cb_in, es, n_vec, cb_out,
                                                                                        objective);
    return cudaGetLastError();
}

cudaError_t launch_learn(const __half* x, const float* weights, const double* uniforms, const Shape& sh, int64_t n_vec,
                         int n_iters, float* codebooks, double* objective, void* workspace, size_t workspace_bytes, cudaStream_t st)
{
    const LearnLayout l = learn_layout(sh, n_vec);
    float* tmp = reinterpret_cast<float*>(static_cast<char*>(workspace) + l.codes + 2 * l.dist);
    cudaError_t e = launch_kmeanspp_init(x, weights, uniforms, sh, n_vec, codebooks, workspace, st);
    if (e != cudaSuccess) return e;
    if (n_iters > 0 && learn_bounds_supported(sh, n_vec) && workspace_bytes >= l.total + learn_bounds_bytes(sh)) {
        Shape es = sh;                                      // the vectors are one sequence of n_vec tokens
        es.n_seq = 1;
        es.max_tokens = n_vec;
        es.n_blocks = (n_vec + kTokenBlock - 1) / kTokenBlock;
        // (the thresholds take the place of the distances of the initialisation: 4 bytes for 8)
        return launch_learn_bounds(x, weights, es, n_vec, n_iters, codebooks, static_cast<uint8_t*>(workspace),
                                   reinterpret_cast<float*>(static_cast<char*>(workspace) + l.codes), static_cast<char*>(workspace) + l.total, st,
                                   [&](const uint8_t* codes, const float* cb) {
                                       return objective ? update_dispatch(x, weights, codes, cb, es, n_vec, tmp, objective, st) : cudaSuccess;
                                   });
    }
    float* cur = codebooks;
    float* nxt = tmp;
    for (int it = 0; it < n_iters; ++it) {
        // (only the last assignment's objective is asked for)
        e = launch_lloyd_step(x, weights, cur, sh, n_vec, nxt, it + 1 == n_iters ? objective : nullptr, workspace, st);
        if (e != cudaSuccess) return e;
        float* t = cur; cur = nxt; nxt = t;
    }
    if (cur != codebooks)
        e = cudaMemcpyAsync(codebooks, cur, (size_t)sh.n_kv_heads * sh.G * sh.K * sh.c * sizeof(float),
                            cudaMemcpyDeviceToDevice, st);
    return e;
}

}  // namespace cq
