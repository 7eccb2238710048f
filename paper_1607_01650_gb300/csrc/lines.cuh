// Line table: the system matrix of a fan-beam plan in the form in which A x of
// narrow batches streams it (dect_project up to 16 interleaved images, dect_adm_tv
// up to 8).
//
// A ray with |dx| <= |dy| ("class 0") crosses the image line by line along the
// rows: in row i it meets at most two pixels, (i, c) and (i, c + 1), and its
// length inside the row is the same in every row.  The table holds, per view,
// line and ray, which fraction of that length lies in pixel c and which in
// c + 1, 4 bytes per ray and line, and per ray the length L (two words):
//   y = L sum over the lines of q x[c] + p x[c + 1],  q + p = 1.
// Stored is the smaller fraction, with a minus sign if that is p, so that a piece of
// any size keeps its 24 bits (q itself, with p = 1 - q, held small p to 2^-25 of L).
// Rays with |dx| > |dy| ("class 1") are stored the same way with rows and columns
// exchanged, and gather from a transposed copy of the image.  Columns outside
// the image stand for the part of a line that a ray spends outside it.
//   Against the CSR form (8 bytes per element, 1.44 elements per ray and line)
// the table is 2.6 times smaller, 90 MB at 512^2, 60 views and 736 bins, and a
// warp whose lanes are adjacent rays gathers adjacent pixels, where a warp on
// one CSR row touches a line of the cache per element: A of two images takes
// 33 us instead of 74.  q lies in tiles of 32 lines x 32 rays, which a warp
// streams as 4 KB (line by line across all bins, each warp's 128 bytes of a line
// came from another DRAM page: 45 us).
//   The columns come from the same FP64 Siddon walk that fills the CSR tables.
// Plans where the form does not hold (rays that end inside the image, n < 4 or
// n > 4096) keep to the CSR kernels.  A pixel beside a ray's only column in a
// line carries the weight 0, which is no protection from a value there that is
// not finite: a sum that is not finite is formed again without such pixels.
//   A^T stays on the pixel-major CSR table: from this one it has to find each
// pixel's rays per view, and took 105 us against 72.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "dect_internal.cuh"
#include "kernels.cuh"

namespace dect {

// widest batch that takes the line table
constexpr int kLineMaxImages = 16;

// Walk word of a ray and a block of 32 lines: .x = column c of the block's
// first line + 1 (16 bits), bit 16: c falls along the lines (else rises), bit
// 17: some line of the block has a column outside the image or there are fewer
// than 32, bit 18: the ray is of class 1, bit 19: the ray meets the image in none
// of the block's lines; .y bit k: c changes by one from line k to line k + 1.
constexpr unsigned kWalkFalls = 1u << 16, kWalkEdge = 1u << 17, kWalkCls1 = 1u << 18, kWalkOut = 1u << 19;
// A block takes 32 adjacent rays of a view: LPE warps share the rays, and
// kLineParts such sets the line blocks.  The kernels give both launch bounds:
// with the block size alone ptxas trades the loads in flight for occupancy.
constexpr int kLineParts = 4;

// Lanes: LPE lanes share an element and take VW of its images each, so that the
// pieces a warp reads are contiguous (one lane holding all images of a pixel
// read 16 bytes every 64: 3.5 times the L1 wavefronts at 16 images).
template <int NB>
struct LineShape {
    static constexpr int VW = Batch<NB>::VW, LPE = NB / VW;
    static constexpr int PER = 32 / LPE;       // rays of a warp
    static constexpr int U = VW == 2 ? 8 : 4;  // lines whose loads are in flight together
    static constexpr int BLOCK = kLineParts * 32 * LPE;
    static constexpr int BLOCKS = (VW == 2 ? 7 : 8) / LPE;  // resident per SM
    static_assert(LPE <= 4, "narrow batches only");
};

// Brings `bytes` bytes (a multiple of 16, 16-byte aligned) into L2, without registers or a wait.
__device__ __forceinline__ void l2_prefetch(const void *p, unsigned bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// The fractions (q, p) of an entry of the table, and the entry of given fractions.
__device__ __forceinline__ void line_weights(float v, float &q, float &p)
{
    const float small = fabsf(v), large = 1.f - small;
    const bool neg = __float_as_int(v) < 0;
    q = neg ? large : small;
    p = neg ? small : large;
}
__device__ __forceinline__ float line_entry(double q, double p) { return q <= p ? (float)q : -(float)p; }

inline int line_groups(const LineTable &T) { return T.nv * T.ngb; }

// The 32 lines of a block, none of whose columns lies outside the image: sum of
// q x[c] + p x[c + 1].  qt: the ray's entry of the tile's first line.
template <int NB>
__device__ __forceinline__ void line_block(const float *__restrict__ x, const float *__restrict__ qt, int n, int s0,
                                           const uint2 &w, float (&acc)[LineShape<NB>::VW])
{
    constexpr int VW = LineShape<NB>::VW, U = LineShape<NB>::U;
    const float *xp = x + ((int64_t)s0 * n + (int)(w.x & 0xffffu) - 1) * NB;
    // floats from a line's column to the next line's, where c stays and where it changes
    const unsigned up0 = (unsigned)n * NB, up1 = (w.x & kWalkFalls) ? up0 - NB : up0 + NB;
    unsigned bits = w.y;
#pragma unroll 1
    for (int k0 = 0; k0 < 32; k0 += U) {
        float q[U];
        Vec<VW> lo[U], hi[U];
#pragma unroll
        for (int u = 0; u < U; ++u) q[u] = __ldg(qt + u * 32);
        qt += U * 32;
#pragma unroll
        for (int u = 0; u < U; ++u) {
#ifdef DECT_CHECKED
            if (!DECT_IDX_OK(xp - x, (int64_t)n * n * NB - NB, CHK_GATHER_A)) xp = x;
#endif
            lo[u] = ld_il<VW>(xp);
            hi[u] = ld_il<VW>(xp + NB);
            xp += (bits & (1u << u)) ? up1 : up0;
        }
        bits >>= U;
        // round, block and part sum up on their own: fewer roundings at the size of the ray's sum
        float sum[VW];
#pragma unroll
        for (int t = 0; t < VW; ++t) sum[t] = 0.f;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            float a, b;
            line_weights(q[u], a, b);
#pragma unroll
            for (int t = 0; t < VW; ++t) sum[t] = fmaf(a, lo[u].v[t], fmaf(b, hi[u].v[t], sum[t]));
        }
#pragma unroll
        for (int t = 0; t < VW; ++t) acc[t] += sum[t];
    }
}

// The same where some column (or line) lies outside: it is given the weight 0
// and a place inside the image.
template <int NB>
__device__ __forceinline__ void line_block_edge(const float *__restrict__ x, const float *__restrict__ qt, int n,
                                                int s0, const uint2 &w, float (&acc)[LineShape<NB>::VW])
{
    constexpr int VW = LineShape<NB>::VW, U = 4;
    int c = (int)(w.x & 0xffffu) - 1;
    const int dir = (w.x & kWalkFalls) ? -1 : 1, ns = min(32, n - s0);
    unsigned bits = w.y;
    const float *row = x + (int64_t)s0 * n * NB;
#pragma unroll 1
    for (int k0 = 0; k0 < ns; k0 += U) {
        float q[U], p[U];
        Vec<VW> lo[U], hi[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool on = k0 + u < ns;
            line_weights(on ? __ldg(qt + (k0 + u) * 32) : 0.f, q[u], p[u]);
            if (!on || c + 1 >= n) p[u] = 0.f;
            if (c < 0) q[u] = 0.f;
            const int c0 = max(c, 0), c1 = min(c + 1, n - 1);
            lo[u] = ld_il<VW>(row + (int64_t)c0 * NB);
            hi[u] = ld_il<VW>(row + (int64_t)c1 * NB);
            if (k0 + u + 1 < ns) row += (int64_t)n * NB;
            c += (bits & (1u << u)) ? dir : 0;
        }
        bits >>= U;
        float sum[VW];
#pragma unroll
        for (int t = 0; t < VW; ++t) sum[t] = 0.f;
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int t = 0; t < VW; ++t) sum[t] = fmaf(q[u], lo[u].v[t], fmaf(p[u], hi[u].v[t], sum[t]));
#pragma unroll
        for (int t = 0; t < VW; ++t) acc[t] += sum[t];
    }
}

// The same line by line, pixels of weight 0 left out.
template <int NB>
__device__ __noinline__ void line_block_careful(const float *x, const float *qt, int n, int s0, const uint2 w,
                                                float (&acc)[LineShape<NB>::VW])
{
    constexpr int VW = LineShape<NB>::VW;
    int c = (int)(w.x & 0xffffu) - 1;
    const int dir = (w.x & kWalkFalls) ? -1 : 1, ns = min(32, n - s0);
    for (int k = 0; k < ns; ++k) {
        float q, p;
        line_weights(__ldg(qt + k * 32), q, p);
        const float *row = x + (int64_t)(s0 + k) * n * NB;
        if (c >= 0 && c < n && q != 0.f) {
            const Vec<VW> v = ld_il<VW>(row + (int64_t)c * NB);
#pragma unroll
            for (int t = 0; t < VW; ++t) acc[t] = fmaf(q, v.v[t], acc[t]);
        }
        if (c + 1 >= 0 && c + 1 < n && p != 0.f) {
            const Vec<VW> v = ld_il<VW>(row + (int64_t)(c + 1) * NB);
#pragma unroll
            for (int t = 0; t < VW; ++t) acc[t] = fmaf(p, v.v[t], acc[t]);
        }
        c += ((w.y >> k) & 1u) ? dir : 0;
    }
}

// Sum over the warp's line blocks for the lane's ray of group (v, gb) and its
// images, x = src or, for rays of class 1, the transposed image srcT.
template <int NB>
__device__ __forceinline__ void line_ray_sums(const LineTable &T, int v, int gb, const float *__restrict__ src,
                                              const float *__restrict__ srcT, float (&acc)[LineShape<NB>::VW])
{
    using S = LineShape<NB>;
    constexpr int VW = S::VW, PARTS = kLineParts;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = T.n;
    const int part = warp / S::LPE, ray = (warp % S::LPE) * S::PER + lane / S::LPE;
    const int b = min(gb * 32 + ray, T.nb - 1);  // idle lanes repeat the last ray
    const uint2 *__restrict__ walk = T.walk + (int64_t)v * T.nblk * T.nbp + b;
    const float *__restrict__ q = T.q + T.at(v, 0, b);  // tiles of the next 32 lines: ngb * 1024 on
    const int64_t tile = (int64_t)T.ngb * 1024;
    const int img = (lane % S::LPE) * VW;
    float lost[VW];
#pragma unroll
    for (int k = 0; k < VW; ++k) acc[k] = lost[k] = 0.f;
    uint2 w = make_uint2(0u, 0u);
    if (part < T.nblk) w = __ldg(walk + (int64_t)part * T.nbp);
    for (int blk = part; blk < T.nblk; blk += PARTS) {
        const uint2 now = w;
        if (blk + PARTS < T.nblk) {
            w = __ldg(walk + (int64_t)(blk + PARTS) * T.nbp);
            // q streams from DRAM: the next tile is brought into L2 meanwhile
            if (threadIdx.x % (32 * S::LPE) == 0) l2_prefetch(T.q + T.at(v, (blk + PARTS) * 32, gb * 32), 4096u);
        }
        if (__all_sync(0xffffffffu, (now.x & kWalkOut) != 0u)) continue;
        const float *x = ((now.x & kWalkCls1) ? srcT : src) + img;
        const float *qt = q + blk * tile;
        float sum[VW];
#pragma unroll
        for (int k = 0; k < VW; ++k) sum[k] = 0.f;
        if (!__any_sync(0xffffffffu, (now.x & kWalkEdge) != 0u))
            line_block<NB>(x, qt, n, blk * 32, now, sum);
        else
            line_block_edge<NB>(x, qt, n, blk * 32, now, sum);
#pragma unroll
        for (int k = 0; k < VW; ++k) comp_add(acc[k], lost[k], sum[k]);
    }
    bool fine = true;
#pragma unroll
    for (int k = 0; k < VW; ++k) {
        acc[k] = comp_value(acc[k], lost[k]);
        fine = fine && isfinite(acc[k]);
    }
    if (fine) return;
    float sum[VW];
#pragma unroll
    for (int k = 0; k < VW; ++k) sum[k] = 0.f;
    for (int blk = part; blk < T.nblk; blk += PARTS) {
        const uint2 now = __ldg(walk + (int64_t)blk * T.nbp);
        line_block_careful<NB>(((now.x & kWalkCls1) ? srcT : src) + img, q + blk * tile, n, blk * 32, now, sum);
    }
#pragma unroll
    for (int k = 0; k < VW; ++k)  // images that are finite keep their sums
        if (!isfinite(acc[k])) acc[k] = sum[k];
}

// The block's sums of all 32 rays, [part][ray][NB].
template <int NB>
using LineSums = float[kLineParts][32 * NB];

template <int NB>
__device__ __forceinline__ void line_ray_store(LineSums<NB> &sm, const float (&acc)[LineShape<NB>::VW])
{
    using S = LineShape<NB>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ray = (warp % S::LPE) * S::PER + lane / S::LPE;
#pragma unroll
    for (int t = 0; t < S::VW; ++t) sm[warp / S::LPE][ray * NB + (lane % S::LPE) * S::VW + t] = acc[t];
}
// (A x) of the ray of length L and the image of element e = ray * NB + image
template <int NB>
__device__ __forceinline__ float line_ray_value(const LineSums<NB> &sm, int e, const float2 &L)
{
    static_assert(kLineParts == 4, "pairwise");
    // two words to the end: one rounding at the size of the ray's sum instead of
    // four (A x of two images at 512^2 / 60 views against 64 bits: 5.0e-8 -> 3.4e-8)
    float a = sm[0][e], b = sm[2][e], lost = 0.f;
    comp_pair(a, lost, sm[1][e]);
    comp_pair(b, lost, sm[3][e]);
    comp_pair(a, lost, b);
    if (!isfinite(lost)) lost = 0.f;
    const float y = L.x * a;
    return isfinite(y) ? y + (fmaf(L.x, a, -y) + fmaf(L.x, lost, L.y * a)) : y;
}

// blocks that take `items` items evenly, at most `most`
inline int even_grid(int items, int most)
{
    const int per = (items + most - 1) / most;
    return per > 0 ? (items + per - 1) / per : 1;
}

// Interleaved [n][n][NB] -> transposed [n][n][NB] (32 x 32 pixel tiles).
template <int NB>
__global__ void __launch_bounds__(256) k_line_transpose(const float *__restrict__ src, float *__restrict__ dst, int n)
{
    constexpr int VW = Batch<NB>::VW;
    __shared__ float tile[32][33][VW];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, j0 = blockIdx.x * 32, i0 = blockIdx.y * 32;
    for (int k = 0; k < NB; k += VW) {
        for (int r = ty; r < 32; r += 8)
            if (i0 + r < n && j0 + tx < n) {
                const Vec<VW> v = ld_v<VW>(src + ((int64_t)(i0 + r) * n + j0 + tx) * NB + k);
#pragma unroll
                for (int c = 0; c < VW; ++c) tile[r][tx][c] = v.v[c];
            }
        __syncthreads();
        for (int r = ty; r < 32; r += 8)
            if (j0 + r < n && i0 + tx < n) {
                Vec<VW> v;
#pragma unroll
                for (int c = 0; c < VW; ++c) v.v[c] = tile[tx][r][c];
                st_v<VW>(dst + ((int64_t)(j0 + r) * n + i0 + tx) * NB + k, v);
            }
        __syncthreads();
    }
}

inline dim3 transpose_grid(int n) { return dim3((unsigned)((n + 31) / 32), (unsigned)((n + 31) / 32)); }

}  // namespace dect
