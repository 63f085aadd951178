// Bulk encode for groups of two channels (head_dim 128, c = 2, b = 8).
//
// CQ encode (Section 3.2 of the paper): every group of c channels of a vector is replaced by the index of its nearest
// centroid, lowest index on exact ties.  With c = 2 a group is a point of the plane, and a point's nearest centroid is
// one of the few whose Voronoi cells its neighbourhood meets.  The kernel cuts the plane of every group into 64 x 64
// boxes, lists for each box the centroids that can be nearest to a point of it (two on average, four fit the box's
// word), and evaluates only those per vector: sum (x - C)^2 in fp32 in the order of every other encode kernel, lowest
// index on ties, so the codes are theirs bit for bit.
//
// The boxes are narrow where centroids are dense: an axis is cut in t = z / sqrt(1 + z^2), z = (x - mean) / (1.2533
// standard deviation), which is close to the distribution function of a Gaussian.  A list leaves centroid j out when
// the centroid k nearest to the box's middle is nearer in all of the box: d_j - d_k is linear there, so its smallest
// value sits in a corner; it must exceed a bound on the rounding of both distances.  Lists are narrowed step by step, for
// blocks of 16 x 16, 8 x 8 and 4 x 4 boxes and then for each box.  Boxes with more than four centroids name a longer
// list; points outside the grid (6 standard deviations) and boxes with more than 12 go through all centroids.
//
// A CTA (one per SM) holds the tables of eight groups - 32 bytes of a vector, one sector - and takes an equal share of
// all (tensor, head, set of eight groups, vector); a thread takes a vector through the eight groups.
//
// Measured (8 x 8192 tokens, 32 heads, key and value): 8.25 ms on the tensor-memory kernel before, 2.33 ms here, of
// which the tables take 0.8 to 0.9 ms (what is left when the time is carried back to no vectors).  Bound: the issue
// slots, 69 to 72 % busy (142 warp instructions per 32 vectors of a group: the difference of two inputs' counts; 28 find
// the box, 40 evaluate a word's four centroids); the shared-memory pipe, where words and centroids are gathered (six
// wavefronts per centroid and warp), is 60 % busy.  A vector's row is fetched from DRAM once per set of eight groups and
// not once in all: a set reads 32 bytes of it, DRAM delivers more (4.3 GB read where the vectors are 1.07).
#include "cq_common.cuh"

namespace cq {

namespace {

constexpr int kGrThreads = 1024;
constexpr int kGrGroups = 8;                     // groups of a CTA
constexpr int kGrN = 64;                         // boxes per axis
constexpr int kGrLong = 2048;                    // longer lists of a CTA, 12 centroids each
constexpr float kGrEdge = 0.98f;                 // the grid covers |t| <= kGrEdge
constexpr uint32_t kGrAll = 0xffff00ffu;         // word of a box: all centroids; 0xiiii00ff: longer list i; else four ascending codes

struct GrAxis { float mean, inv; };              // z = (x - mean) * inv

struct GrSmem {
    static constexpr int kCellOff = 0;                                                   // uint32 [groups][64][64]
    static constexpr int kCentOff = kCellOff + kGrGroups * kGrN * kGrN * 4;              // float2 [groups][256]
    static constexpr int kLongOff = kCentOff + kGrGroups * 256 * 8;                      // [lists][words, -, -, -, up to 12 codes]
    static constexpr int kEightOff = kLongOff + kGrLong * 16;                            // [groups][64 blocks of 8 x 8][up to 63 codes, count]
    static constexpr int kAxisOff = kEightOff + kGrGroups * 64 * 64;                     // GrAxis [groups][2]
    static constexpr int kEdgeOff = kAxisOff + kGrGroups * 2 * 8;                        // float z edges [65]
    static constexpr int kEndOff = kEdgeOff + 272;                                       // float [groups][4][65] ends of the boxes
    static constexpr int kCountOff = kEndOff + kGrGroups * 4 * (kGrN + 1) * 4;                                     // number of longer lists
    static constexpr int kBytes = kCountOff + 16;
    static_assert(kBytes <= 227 * 1024, "shared memory");
};

__device__ __forceinline__ float gr_edge(int i)
{
    const float t = kGrEdge * ((float)i * (2.f / kGrN) - 1.f);
    return t * rsqrtf(1.f - t * t);
}

// box of a point along one axis; negative: outside the grid
__device__ __forceinline__ int gr_cell(float x, GrAxis a)
{
    const float z = fminf(fmaxf((x - a.mean) * a.inv, -1e15f), 1e15f);
    const float t = z * rsqrtf(fmaf(z, z, 1.f)) * (kGrN / 2 / kGrEdge) + kGrN / 2;
    const int i = (int)t;                        // (t > -1: truncation towards zero only for points outside)
    return t >= 0.f && i < kGrN ? i : -1;
}

// A box, and the centroids found nearest to its middle and corners (two opposite ones of three points, where that is enough): what the other centroids are tested against.
// Centroid q cannot be nearest to any point of the box when one of them, c, is nearer in all of it:
//   |q - p|^2 - |c - p|^2 - 2 max (x - p) . (q - c) > 0,   p the middle, the maximum |q - c|_x h_x + |q - c|_y h_y,
// with 3e-6 of the squares involved to spare for the rounding of this test and of the two distances at any point.
template <int kP>
struct GrNear {
    float2 p[kP];              // middle, then the corners
    float hx2, hy2;            // sides (twice the half sides)
    float d[kP];
    int at[kP];
    float2 c[kP];
    __device__ __forceinline__ GrNear(float2 lo, float2 hi)
    {
        p[0] = make_float2(0.5f * (lo.x + hi.x), 0.5f * (lo.y + hi.y));
        hx2 = 1.000001f * (hi.x - lo.x);
        hy2 = 1.000001f * (hi.y - lo.y);
#pragma unroll
        for (int i = 1; i < kP; ++i) p[i] = make_float2((i & 1) ? lo.x : hi.x, (i == 1 || i == 4) ? lo.y : hi.y);
#pragma unroll
        for (int i = 0; i < kP; ++i) { d[i] = INFINITY; at[i] = 0; }
    }
    __device__ __forceinline__ void see(float2 q, int j)
    {
#pragma unroll
        for (int i = 0; i < kP; ++i) {
            const float dx = q.x - p[i].x, dy = q.y - p[i].y, e = fmaf(dx, dx, dy * dy);
            at[i] = e < d[i] ? j : at[i];
            d[i] = fminf(e, d[i]);
        }
    }
    // after the last see(): d[i] becomes the constant of the test against c[i]
    __device__ __forceinline__ void done(const float2* cent)
    {
#pragma unroll
        for (int i = 0; i < kP; ++i) c[i] = cent[at[i]];
        const float r2 = 0.25f * fmaf(hx2, hx2, hy2 * hy2);
#pragma unroll
        for (int i = 0; i < kP; ++i) {
            const float kx = c[i].x - p[0].x, ky = c[i].y - p[0].y;
            d[i] = fmaf(1.000003f, fmaf(kx, kx, ky * ky), 8e-6f * r2 + 1e-30f);
        }
    }
    __device__ __forceinline__ bool keep(float2 q) const
    {
        const float dx = q.x - p[0].x, dy = q.y - p[0].y, e = 0.999997f * fmaf(dx, dx, dy * dy);
        bool out = false;
#pragma unroll
        for (int i = 0; i < kP; ++i) {
            const float t = fmaf(-hy2, fabsf(q.y - c[i].y), fmaf(-hx2, fabsf(q.x - c[i].x), e - d[i]));
            out = out || t > 0.f;
        }
        return !out;
    }
};

__global__ void __launch_bounds__(kGrThreads, 1)
encode_grid_kernel(const __half* __restrict__ x1, const float* __restrict__ cb1, const int32_t* __restrict__ seq_offsets, Shape sh,
                   uint32_t n_tokens, int64_t token_offset, uint8_t* __restrict__ codes1, const __half* __restrict__ x2,
                   const float* __restrict__ cb2, uint8_t* __restrict__ codes2, int n_units, uint32_t warps_per_unit)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");      // launched ahead of the end of the kernel before it, and
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");       // the kernel behind it ahead of its own
    constexpr int G = 64, kSets = G / kGrGroups;
    extern __shared__ __align__(16) unsigned char gr_smem[];
    uint32_t* cells = reinterpret_cast<uint32_t*>(gr_smem + GrSmem::kCellOff);
    float2* cents = reinterpret_cast<float2*>(gr_smem + GrSmem::kCentOff);
    uint8_t* longs = gr_smem + GrSmem::kLongOff;
    GrAxis* axes = reinterpret_cast<GrAxis*>(gr_smem + GrSmem::kAxisOff);
    float* edges = reinterpret_cast<float*>(gr_smem + GrSmem::kEdgeOff);
    int* long_count = reinterpret_cast<int*>(gr_smem + GrSmem::kCountOff);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n_heads = sh.n_kv_heads;
    const uint32_t n_vec = (uint32_t)sh.n_seq * n_tokens;
    if (threadIdx.x <= kGrN) edges[threadIdx.x] = gr_edge(threadIdx.x);

    // this CTA's share, in runs of 32 vectors of a unit (unit: tensor, head, set of eight groups)
    const uint64_t total = (uint64_t)n_units * warps_per_unit;
    uint64_t at = total * blockIdx.x / gridDim.x;
    const uint64_t share_end = total * (blockIdx.x + 1) / gridDim.x;
    while (at < share_end) {
        const int unit = (int)(at / warps_per_unit);
        const uint32_t first = (uint32_t)(at % warps_per_unit);
        const uint32_t last = (uint32_t)(share_end - at < warps_per_unit - first ? first + (share_end - at) : warps_per_unit);
        at += last - first;
        const int set = unit % kSets, h = unit / kSets % n_heads;
        const bool second = unit / (kSets * n_heads) != 0;
        const __half* x = second ? x2 : x1;
        uint8_t* codes = second ? codes2 : codes1;
        const float2* cb = reinterpret_cast<const float2*>(second ? cb2 : cb1) + ((int64_t)h * G + set * kGrGroups) * 256;

        // ---- tables of the eight groups
        __syncthreads();                                 // the previous unit's tables are no longer read
        for (int i = threadIdx.x; i < kGrGroups * 256; i += kGrThreads) cents[i] = cb[i];
        if (threadIdx.x == 0) *long_count = 0;
        __syncthreads();
        if (warp < kGrGroups) {
            float2 v[8], m = make_float2(0.f, 0.f), s = make_float2(0.f, 0.f);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                v[e] = cents[warp * 256 + e * 32 + lane];
                m.x += v[e].x;
                m.y += v[e].y;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                m.x += __shfl_xor_sync(0xffffffffu, m.x, o);
                m.y += __shfl_xor_sync(0xffffffffu, m.y, o);
            }
            m.x *= 1.f / 256.f;
            m.y *= 1.f / 256.f;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                s.x += (v[e].x - m.x) * (v[e].x - m.x);
                s.y += (v[e].y - m.y) * (v[e].y - m.y);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
                s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
            }
            // 1 / (1.2533 standard deviation); kept finite and positive, so that a box always has two ends
            if (lane == 0) {
                axes[warp * 2] = GrAxis{m.x, fminf(fmaxf(16.f / 1.2533f * rsqrtf(s.x), 1e-12f), 1e12f)};
                axes[warp * 2 + 1] = GrAxis{m.y, fminf(fmaxf(16.f / 1.2533f * rsqrtf(s.y), 1e-12f), 1e12f)};
            }
        }
        __syncthreads();
        {
            const int gl = threadIdx.x >> 7, t = threadIdx.x & 127;     // 128 threads per group
            const float2* cent = cents + gl * 256;
            const GrAxis ax = axes[gl * 2], ay = axes[gl * 2 + 1];
            // ends of the boxes, moved apart a little (the box of a point is computed with rounding)
            float* ends = reinterpret_cast<float*>(gr_smem + GrSmem::kEndOff) + gl * 4 * (kGrN + 1);      // [x lo, x hi, y lo, y hi][65]
            for (int i = t; i < 2 * (kGrN + 1); i += 128) {
                const int axis = i / (kGrN + 1), e = i % (kGrN + 1);
                const GrAxis a = axis ? ay : ax;
                const float z = edges[e], r = 1.f / a.inv;
                const float zl = edges[e > 0 ? e - 1 : 0], zr = edges[e < kGrN ? e + 1 : kGrN];
                const float w = (zr - zl) * 0.005f + 2e-5f * (fabsf(z) + 1.f), u = 2.4e-7f * fabsf(a.mean);
                ends[(2 * axis) * (kGrN + 1) + e] = fmaf(z - w, r, a.mean) - u;
                ends[(2 * axis + 1) * (kGrN + 1) + e] = fmaf(z + w, r, a.mean) + u;
            }
            __syncthreads();
            auto box_of = [&](int grp, int x0, int y0, int w, float2& lo, float2& hi) {
                const float* ends = reinterpret_cast<const float*>(gr_smem + GrSmem::kEndOff) + grp * 4 * (kGrN + 1);
                lo = make_float2(ends[x0], ends[2 * (kGrN + 1) + y0]);
                hi = make_float2(ends[(kGrN + 1) + x0 + w], ends[3 * (kGrN + 1) + y0 + w]);
            };
            // 16 quarters of 16 x 16 boxes: eight lanes each, from all centroids
            uint8_t* quarter = longs + (gl * 16 + (t >> 3)) * 128;              // [up to 127 codes, count]
            {
                float2 lo, hi;
                box_of(gl, (t >> 3) % 4 * 16, (t >> 5) * 16, 16, lo, hi);
                GrNear<5> near(lo, hi);
                for (int e = t & 7; e < 256; e += 8) near.see(cent[e], e);
#pragma unroll
                for (int o = 1; o < 8; o <<= 1)
#pragma unroll
                    for (int i = 0; i < 5; ++i) {
                        const float od = __shfl_xor_sync(0xffffffffu, near.d[i], o);
                        const int oa = __shfl_xor_sync(0xffffffffu, near.at[i], o);
                        if (od < near.d[i] || (od == near.d[i] && oa < near.at[i])) { near.d[i] = od; near.at[i] = oa; }
                    }
                near.done(cent);
                int n = 0;
                for (int e = t & 7; e < 256; e += 8) {
                    const bool keep = near.keep(cent[e]);
                    const unsigned in = (__ballot_sync(0xffffffffu, keep) >> (lane & 24)) & 0xffu;
                    const int at_ = n + __popc(in & ((1u << (lane & 7)) - 1u));
                    if (keep && at_ < 127) quarter[at_] = (uint8_t)e;
                    n += __popc(in);
                }
                if ((t & 7) == 0) quarter[127] = n <= 127 ? (uint8_t)n : 255;
            }
            __syncthreads();
            // 64 blocks of 8 x 8 boxes from their quarter's list, 256 of 4 x 4 boxes from theirs; the last one goes to the words of the block's boxes
            // (byte e of it: row e / 16 of the block, byte e % 16; the count in byte 63, 255: all centroids)
            auto block_byte = [&](int grp, int bx, int by, int e) {
                return reinterpret_cast<uint8_t*>(cells + grp * kGrN * kGrN + (by * 4 + (e >> 4)) * kGrN + bx * 4) + (e & 15);
            };
            // the list of a block of w x w boxes from a longer one that holds all it can need
            auto narrow = [&](int grp, int x0, int y0, int w, const uint8_t* list, int count, auto out) {
                const bool all = count == 255;
                const int ln = all ? 256 : count;
                float2 lo, hi;
                box_of(grp, x0, y0, w, lo, hi);
                const float2* cent = cents + grp * 256;
                GrNear<3> near(lo, hi);
                for (int e = 0; e < ln; ++e) {
                    const int j = all ? e : (int)list[e];
                    near.see(cent[j], j);
                }
                near.done(cent);
                int n = 0;
                for (int e = 0; e < ln; ++e) {
                    const int j = all ? e : (int)list[e];
                    if (near.keep(cent[j])) {
                        if (n < 63) *out(n) = (uint8_t)j;
                        ++n;
                    }
                }
                *out(63) = n <= 63 ? (uint8_t)n : 255;
            };
            // (from here on every group's blocks are spread over all warps: the lists of one group can be much longer)
            uint8_t* eights = gr_smem + GrSmem::kEightOff;
            if (threadIdx.x < kGrGroups * 64) {
                const int grp = threadIdx.x >> 6, c = threadIdx.x & 63, bx = c & 7, by = c >> 3;
                const uint8_t* list = longs + (grp * 16 + (by >> 1) * 4 + (bx >> 1)) * 128;
                narrow(grp, bx * 8, by * 8, 8, list, list[127], [&](int e) { return eights + (grp * 64 + c) * 64 + e; });
            }
            __syncthreads();
            for (int i = threadIdx.x; i < kGrGroups * 256; i += kGrThreads) {
                const int grp = i >> 8, bx = i & 15, by = (i >> 4) & 15;
                const uint8_t* list = eights + (grp * 64 + (by >> 1) * 8 + (bx >> 1)) * 64;
                narrow(grp, bx * 4, by * 4, 4, list, list[63], [&](int e) { return block_byte(grp, bx, by, e); });
            }
            __syncthreads();
            // the boxes: a thread takes four of them, 2 x 2 (four threads a block), which share the loads and most of the
            // arithmetic
            for (int i = threadIdx.x; i < kGrGroups * 1024; i += kGrThreads) {
                const int grp = i >> 10, bx = (i >> 2) & 15, by = (i >> 6) & 15, qx = bx * 4 + 2 * (i & 1), qy = by * 4 + (i & 2);
                const float2* cent = cents + grp * 256;
                const float* ends = reinterpret_cast<const float*>(gr_smem + GrSmem::kEndOff) + grp * 4 * (kGrN + 1);
                float mx[2], hx[2], my[2], hy[2];        // middles and sides of the two columns and the two rows
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float xl = ends[qx + e], xh = ends[(kGrN + 1) + qx + e + 1];
                    const float yl = ends[2 * (kGrN + 1) + qy + e], yh = ends[3 * (kGrN + 1) + qy + e + 1];
                    mx[e] = 0.5f * (xl + xh); hx[e] = 1.000001f * (xh - xl);
                    my[e] = 0.5f * (yl + yh); hy[e] = 1.000001f * (yh - yl);
                }
                const int ln = *block_byte(grp, bx, by, 63);
                uint32_t word[4];
                int n[4], slot[4];
#pragma unroll
                for (int b = 0; b < 4; ++b) { word[b] = kGrAll; n[b] = 0; slot[b] = kGrLong; }
                if (ln != 255) {
                    float dn[4] = {INFINITY, INFINITY, INFINITY, INFINITY};
                    int at_[4] = {0, 0, 0, 0};
                    for (int e0 = 0; e0 < ln; e0 += 4) {
                        const uint32_t c4 = *reinterpret_cast<const uint32_t*>(block_byte(grp, bx, by, e0));
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            if (e0 + k >= ln) break;
                            const int j = (int)((c4 >> (8 * k)) & 0xffu);
                            const float2 q = cent[j];
                            const float dx0 = q.x - mx[0], dx1 = q.x - mx[1], dy0 = q.y - my[0], dy1 = q.y - my[1];
                            const float xx[2] = {dx0 * dx0, dx1 * dx1}, yy[2] = {dy0 * dy0, dy1 * dy1};
#pragma unroll
                            for (int b = 0; b < 4; ++b) {
                                const float d = xx[b & 1] + yy[b >> 1];
                                at_[b] = d < dn[b] ? j : at_[b];
                                dn[b] = fminf(d, dn[b]);
                            }
                        }
                    }
                    float2 c[4];                         // nearest to the middle of each box
                    float kc[4];                         // the constants of GrNear's test
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        c[b] = cent[at_[b]];
                        const float kx = c[b].x - mx[b & 1], ky = c[b].y - my[b >> 1], wx = hx[b & 1], wy = hy[b >> 1];
                        kc[b] = fmaf(1.000003f, fmaf(kx, kx, ky * ky), fmaf(2e-6f, fmaf(wx, wx, wy * wy), 1e-30f));
                    }
                    for (int e0 = 0; e0 < ln; e0 += 4) {
                        const uint32_t c4 = *reinterpret_cast<const uint32_t*>(block_byte(grp, bx, by, e0));
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const uint32_t j = (c4 >> (8 * k)) & 0xffu;
                            const float2 q = cent[j];
                            const float dx0 = q.x - mx[0], dx1 = q.x - mx[1], dy0 = q.y - my[0], dy1 = q.y - my[1];
                            const float xx[2] = {0.999997f * dx0 * dx0, 0.999997f * dx1 * dx1}, yy[2] = {0.999997f * dy0 * dy0, 0.999997f * dy1 * dy1};
#pragma unroll
                            for (int b = 0; b < 4; ++b) {
                                const float t = fmaf(-hy[b >> 1], fabsf(q.y - c[b].y),
                                                     fmaf(-hx[b & 1], fabsf(q.x - c[b].x), (xx[b & 1] + yy[b >> 1]) - kc[b]));
                                if (e0 + k >= ln || t > 0.f) continue;
                                if (n[b] >= 4) {         // rare: the box gets a longer list
                                    if (n[b] == 4) {
                                        slot[b] = atomicAdd(long_count, 1);
                                        if (slot[b] < kGrLong) *reinterpret_cast<uint32_t*>(longs + slot[b] * 16 + 4) = word[b];
                                    }
                                    if (n[b] < 12 && slot[b] < kGrLong) longs[slot[b] * 16 + 4 + n[b]] = (uint8_t)j;
                                }
                                word[b] = (word[b] >> 8) | (j << 24);
                                ++n[b];
                            }
                        }
                    }
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        const uint32_t end = word[b] >> 24;                    // the last code, repeated to the end of its word
                        if (n[b] <= 4) {
                            for (int e = n[b]; e < 4; ++e) word[b] = (word[b] >> 8) | (end << 24);
                        } else if (n[b] <= 12 && slot[b] < kGrLong) {
                            for (int e = n[b]; e & 3; ++e) longs[slot[b] * 16 + 4 + e] = (uint8_t)end;
                            longs[slot[b] * 16] = (uint8_t)((n[b] + 3) >> 2);
                            word[b] = ((uint32_t)slot[b] << 16) | 0xffu;
                        } else {
                            word[b] = kGrAll;
                        }
                    }
                }
                __syncwarp();                            // the block's list has been read by its four threads
#pragma unroll
                for (int b = 0; b < 2; ++b)
                    *reinterpret_cast<uint2*>(cells + (grp * kGrN + qy + b) * kGrN + qx) = make_uint2(word[2 * b], word[2 * b + 1]);
            }
        }
        __syncthreads();

        // ---- the vectors
        const int row_step = n_heads * 128;
        for (uint32_t run = first + warp; run < last; run += kGrThreads / 32) {
            const uint32_t v = run * 32 + lane;
            if (v >= n_vec) break;
            const uint4* gp = reinterpret_cast<const uint4*>(x + (int64_t)v * row_step + h * 128 + set * kGrGroups * 2);
            const uint4 xa = gp[0], xb = gp[1];
            const uint32_t xw[kGrGroups] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
            const uint32_t s = v / n_tokens, i = v - s * n_tokens;
            const int64_t pos = token_offset + (seq_offsets ? seq_offsets[s] : 0) + i;
            uint8_t* dst = nullptr;
            if (pos >= 0 && pos < sh.max_tokens)
                dst = codes + code_word_offset(sh, n_heads, s, h, pos / kTokenBlock, set * kGrGroups) + pos % kTokenBlock;
            uint32_t word[kGrGroups];
#pragma unroll
            for (int g = 0; g < kGrGroups; ++g) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&xw[g]));
                const int cx = gr_cell(f.x, axes[g * 2]), cy = gr_cell(f.y, axes[g * 2 + 1]);
                word[g] = (cx | cy) < 0 ? kGrAll : cells[(g * kGrN + cy) * kGrN + cx];
            }
#pragma unroll
            for (int g = 0; g < kGrGroups; ++g) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&xw[g]));
                const float2* cent = cents + g * 256;
                float best = INFINITY;
                uint32_t arg = 0u;
                auto look = [&](uint32_t j) {
                    const float2 c = cent[j];
                    const float dx = f.x - c.x, dy = f.y - c.y;
                    const float d = fmaf(dy, dy, dx * dx);
                    if (d < best) { best = d; arg = j; }               // ascending codes: strict < keeps the lowest on ties
                };
                uint32_t w = word[g];
                int words = 1;
                uint4 l = make_uint4(0u, 0u, 0u, 0u);
                if ((w & 0xffffu) == 0x00ffu && w != kGrAll) {
                    l = *reinterpret_cast<const uint4*>(longs + (w >> 16) * 16);
                    words = (int)(l.x & 0xffu);
                    w = l.y;
                }
                if (w != kGrAll) {
                    look(w & 0xffu);
                    look((w >> 8) & 0xffu);
                    look((w >> 16) & 0xffu);
                    look(w >> 24);
                    if (words > 1) {
                        look(l.z & 0xffu);
                        look((l.z >> 8) & 0xffu);
                        look((l.z >> 16) & 0xffu);
                        look(l.z >> 24);
                        if (words > 2) {
                            look(l.w & 0xffu);
                            look((l.w >> 8) & 0xffu);
                            look((l.w >> 16) & 0xffu);
                            look(l.w >> 24);
                        }
                    }
                } else {
#pragma unroll 4
                    for (uint32_t j = 0; j < 256; ++j) look(j);
                }
                if (dst) dst[g * kTokenBlock] = (uint8_t)arg;
            }
        }
    }
}

}  // namespace

// Making the tables of eight groups takes a CTA about 140 us, and a CTA makes those of its share of the units and of
// one cut unit more; after that a vector of a head costs 1.8 ns less than on the tensor-memory kernel.  (32 heads, one
// tensor: 6636 vectors, the first that come here, 567 against 557 us, 7000 573 against 580, 8192 585 against 674, 65536
// 1212 against 4672.)
bool encode_grid_pays(const Shape& sh, int64_t n_tokens, int n_tensors)
{
    const int64_t n_vec = sh.n_seq * n_tokens;
    if (sh.head_dim != 128 || sh.c != 2 || sh.b != 8 || n_vec >= ((int64_t)1 << 31) - 64 || sh.n_kv_heads > 4096) return false;
    const double units = (double)n_tensors * sh.n_kv_heads * (64 / kGrGroups);
    return (units / device_sm_count() + 1.0) * 140e3 < 1.8 * (double)n_vec * sh.n_kv_heads * n_tensors;
}

cudaError_t launch_encode_grid(const __half* x, const float* cb, const int32_t* seq_offsets, const Shape& sh, int64_t n_tokens,
                               int64_t token_offset, uint8_t* codes, cudaStream_t st, const __half* x2, const float* cb2, uint8_t* codes2)
{
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(encode_grid_kernel), GrSmem::kBytes, 14);
    if (e != cudaSuccess) return e;
    const int n_units = (x2 ? 2 : 1) * sh.n_kv_heads * (64 / kGrGroups);
    const uint32_t per_unit = (uint32_t)((sh.n_seq * n_tokens + 31) / 32);
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = overlapped_config((unsigned)device_sm_count(), kGrThreads, GrSmem::kBytes, st, &attr);
    return cudaLaunchKernelEx(&cfg, encode_grid_kernel, x, cb, seq_offsets, sh, (uint32_t)n_tokens, token_offset, codes, x2, cb2, codes2,
                              n_units, per_unit);
}

}  // namespace cq
