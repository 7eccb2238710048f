// Fan-beam filtered backprojection: the analytic reconstruction the paper
// uses in Sec. 2.4 and Sec. 3, here as an initial image for the ADM
// (dect_adm_tv with warm_start = 1).  Textbook algorithm for an equally
// spaced flat detector over a full 360-degree scan:
//   1. bins moved to a virtual detector through the isocentre,
//      s_b = u_b SOD / SDD, spacing ds = pitch SOD / SDD;
//   2. cosine pre-weight q = p SOD / sqrt(SOD^2 + s_b^2);
//   3. Ram-Lak ramp filter sampled at ds: h(0) = 1 / (4 ds^2), h(k) = 0 for
//      even k != 0, h(k) = -1 / (pi^2 k^2 ds^2) for odd k, qf = ds (q * h);
//   4. back-projection: for pixel P and view v (source S, central-ray
//      direction c, lateral direction e of increasing bin index),
//      L = (P - S).c = SOD + P.c, s = (P.e) SOD / L, and
//      f(P) = sum_v (dtheta / 2) (SOD / L)^2 qf(v, s), linear between bins,
//      0 outside them.
// The filtered projections are FP32, laid out [view][bin][image] so that one
// interpolation serves all images of a pass (up to 64) with contiguous loads.
//
// Filter.  The taps cancel the projections' large mean, so the sums need more
// than FP32.  FP64 runs at 1/64 of the FP32 rate (direct FP64 sums: 4.9 ms for
// 64 images of 60 x 736), so the convolution runs on the tensor cores with
// integer arithmetic: the odd taps couple bins of one parity to bins of
// the other, a product with a Toeplitz matrix T(|d|) = 1 / d^2, d odd.  A
// row of q (below 2^e) is rounded to 2^(e-46), T to 2^-46;
// both are cut into six signed 8-bit digits, which BF16 holds exactly, and
// the 21 digit products of weight 2^(e-52) and above are summed by mma.sync in
// FP32, one accumulator per weight: the sums are integers below 2^24, so these
// sums are not rounded.  What is dropped leaves an error of the row's
// magnitude, about sqrt(n_bins) 2^(e-47) rms (736 bins: 1.6e-13 of 2^e, at most
// 7e-13 in 17664 sums), whatever the size of the output.  The
// accumulators, the cosine weight and the h(0) term are then joined in two FP32
// words and rounded once; an output so small that the error could show beside
// that rounding (below 2^27 of the rms, 3e-5 of 2^e at 736 bins: about one in
// 150 of a CT row, more than half of a row with one bin 100 times the others) is
// summed again in FP64.  (Five digits and no second sum were 8.7e-9 off
// before the rounding on CT rows, and 2.5e-7 beside such a bin.)
//
// Back-projection.  The bin coordinate t reaches n_bins - 1 and its rounding
// moves the interpolation weights, so the per-pixel geometry (t and the weight
// (SOD / L)^2 dtheta / 2) is formed in two FP32 words (about 2^-44 of t) and rounded
// once, once per pixel and view for all images (it was FP64, once per four
// images: 10.4 ms of the above case).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "dect_internal.cuh"
#include "kernels.cuh"

namespace dect {
namespace {

// A value in two FP32 words, hi + lo with |lo| <= ulp(hi) / 2 where it matters.
struct FF {
    float h, l;
};
__host__ __device__ __forceinline__ FF ff_of(double v)
{
    FF r;
    r.h = (float)v;
    r.l = (float)(v - (double)r.h);
    return r;
}
__device__ __forceinline__ FF two_sum(float a, float b)
{
    FF r;
    r.h = __fadd_rn(a, b);
    const float bv = __fsub_rn(r.h, a);
    r.l = __fadd_rn(__fsub_rn(a, __fsub_rn(r.h, bv)), __fsub_rn(b, bv));
    return r;
}
__device__ __forceinline__ FF ff_mul(const FF &a, const FF &b)
{
    FF r;
    r.h = __fmul_rn(a.h, b.h);
    r.l = __fadd_rn(fmaf(a.h, b.h, -r.h), fmaf(a.h, b.l, __fmul_rn(a.l, b.h)));
    return r;
}
__device__ __forceinline__ FF ff_add(const FF &a, const FF &b)
{
    FF r = two_sum(a.h, b.h);
    r.l = __fadd_rn(r.l, __fadd_rn(a.l, b.l));
    return r;
}

// Per view, in two words: the lateral direction e times SOD / (isocentre bin
// spacing), and the central-ray direction c (source -> isocentre).
struct ViewGeo {
    FF ex, ey, cx, cy;
};

// cosine weight of bin b
__device__ __forceinline__ double cos_weight(const dect_geometry &g, int b)
{
    const double u = ((double)b - 0.5 * (double)(g.n_bins - 1)) * g.pitch_mm + g.det_offset_mm;
    const double sb = u * (g.sod_mm / g.sdd_mm);
    return g.sod_mm / sqrt(g.sod_mm * g.sod_mm + sb * sb);
}
// tap h(k), k odd
__device__ __forceinline__ double odd_tap(double k, double ds)
{
    const double pi = 3.14159265358979323846;
    return -1.0 / (pi * pi * k * k * ds * ds);
}

// ---------------------------------------------------------------------------
// FP64 filter: one block per (view, image); shared memory q[nb] and the odd
// taps.  For detectors of more than kTcMaxBins bins.
// ---------------------------------------------------------------------------
constexpr int kFbpBlock = 256;

__global__ void __launch_bounds__(kFbpBlock) k_fbp_filter(const float *__restrict__ m, float *__restrict__ qf,
                                                       dect_geometry g, int width)
{
    const int nb = g.n_bins, v = blockIdx.x, img = blockIdx.y;
    extern __shared__ double sm[];
    double *q = sm, *hodd = sm + nb;
    const double ds = g.pitch_mm * (g.sod_mm / g.sdd_mm);
    const int64_t row = ((int64_t)img * g.n_views + v) * nb;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) q[b] = (double)m[row + b] * cos_weight(g, b);
    const int nodd = nb / 2 + 1;
    for (int j = threadIdx.x; j < nodd; j += blockDim.x) hodd[j] = odd_tap(2.0 * j + 1.0, ds);
    __syncthreads();
    const double h0 = 1.0 / (4.0 * ds * ds);
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        // taps at odd distances 2 j + 1 on both sides, farthest first
        const int jmax = max(b, nb - 1 - b) / 2;  // 2 jmax + 1 reaches past the farther end
        double acc = 0.0;
        for (int j = jmax; j >= 0; --j) {
            const int d = 2 * j + 1;
            double pair = 0.0;
            if (b - d >= 0) pair += q[b - d];
            if (b + d < nb) pair += q[b + d];
            acc = fma(hodd[j], pair, acc);
        }
        acc = fma(h0, q[b], acc);
        qf[((int64_t)v * nb + b) * width + img] = (float)(ds * acc);
    }
}

// ---------------------------------------------------------------------------
// Tensor-core filter (see the file header).  A block takes 16 rows (row R =
// view R / nimg, image R % nimg) and all bins: the digits of one parity at a time
// stay in shared memory (96 bytes per bin), 16 warps share the 8-bin output
// tiles.  B fragments come from a table of T's digits by n - k (Toeplitz), two
// neighbouring taps per 32-bit word.  T's first digit is zero from d = 13 on
// and its second from d = 183 on (1 / d^2 below half a unit of it), so tiles
// farther from the diagonal leave out the products with it.  27 k MMAs per
// block at 736 bins; two blocks' worth per SM at 64 images of 60 views.
//   The sum of one weight's products is at most the sum of |T digit| over both
// sides' taps times 128: 0.92 2^24 at 1152 bins, below 2^24 up to 1270.
// ---------------------------------------------------------------------------
constexpr int kTcRows = 16, kTcWarps = 16, kTcThreads = 32 * kTcWarps, kDig = 6, kTcTiles = 3;
constexpr int kTcMaxBins = 1270;

struct FilterShape {
    int half[2];  // bins of each parity
    int kpad;     // padded to a multiple of 16, for both
    int ld;       // row stride of a digit plane (BF16), 16 bytes off a multiple of 32
    int tn;       // words of one digit of the tap table
    int nw;       // words of a row's bits
    size_t dig;   // bytes of the digits and taps
    size_t smem;
};
__host__ __device__ inline FilterShape filter_shape(int nb)
{
    FilterShape f;
    f.half[0] = (nb + 1) / 2;
    f.half[1] = nb / 2;
    f.kpad = (f.half[0] + 15) & ~15;
    f.ld = f.kpad + 8;
    f.tn = 2 * f.kpad + 32;
    f.nw = (nb + 31) / 32;
    const size_t digits = ((size_t)kDig * kTcRows * f.ld * 2 + (size_t)kDig * f.tn * 4 + 15) & ~(size_t)15;
    const size_t rows = (size_t)kTcRows * nb * sizeof(double);  // of the second sums, over the digits and taps
    f.dig = digits > rows ? digits : rows;
    f.smem = f.dig + (size_t)nb * sizeof(FF) + (size_t)kTcRows * f.nw * 4;
    return f;
}
constexpr size_t kTcSmemMax = 176 * 1024;  // kTcMaxBins: 171 KB

__device__ __forceinline__ void ldsm_a(unsigned (&r)[4], const void *p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_u32(p)));
}
__device__ __forceinline__ void mma_exact(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// the six signed 8-bit digits of |Q| <= 2^46, most significant first, as BF16
__device__ __forceinline__ void digits(long long Q, __nv_bfloat16 (&d)[kDig])
{
#pragma unroll
    for (int k = kDig - 1; k >= 0; --k) {
        const int lo = (int)(signed char)(Q & 255);
        d[k] = __int2bfloat16_rn(lo);
        Q = (Q - lo) >> 8;
    }
}

// The views' directions, and for k_fbp_filter_tc the cosine weights [n_bins], the taps
// at odd distances 2 j + 1 [n_bins / 2 + 1] and the words of T's digits [kDig][tn]: word w
// holds (T(w - kpad - 16), T(w - kpad - 17)) of the even outputs, T(x) = 1 / (2 j +
// 1)^2, j = x - 1 for x > 0 and -x otherwise.  (Formed by every block, the digits' FP64
// divisions were a tenth of the filter.)
// And the pixel coordinates along an axis [n].  A table per blockIdx.y: one after the
// other in a thread their FP64 divisions and sines took 12 us.
constexpr int kTables = 4, kTableBlock = 64;
__global__ void __launch_bounds__(kTableBlock) k_fbp_tables(dect_geometry g, ViewGeo *vg, double *cwd, double *tap,
                                                            unsigned *tw, FF *pos)
{
    const int t = blockIdx.x * kTableBlock + threadIdx.x;
    const FilterShape F = filter_shape(g.n_bins);
    if (blockIdx.y == 0) {
        if (t < g.n_bins) cwd[t] = cos_weight(g, t);
        if (t < g.n) pos[t] = ff_of(((double)t + 0.5 - 0.5 * (double)g.n) * g.pixel_mm);
    } else if (blockIdx.y == 1) {
        if (t <= g.n_bins / 2) tap[t] = odd_tap(2.0 * t + 1.0, g.pitch_mm * (g.sod_mm / g.sdd_mm));
    } else if (blockIdx.y == 2) {
        if (t >= F.tn) return;
        __nv_bfloat16 d0[kDig], d1[kDig];
        const int x = t - F.kpad - 16, j0 = x > 0 ? x - 1 : -x, j1 = x - 1 > 0 ? x - 2 : 1 - x;
        const double k0 = 2.0 * j0 + 1.0, k1 = 2.0 * j1 + 1.0;
        digits(__double2ll_rn(0x1p46 / (k0 * k0)), d0);
        digits(__double2ll_rn(0x1p46 / (k1 * k1)), d1);
#pragma unroll
        for (int k = 0; k < kDig; ++k)
            tw[k * F.tn + t] = (unsigned)__bfloat16_as_ushort(d0[k]) | ((unsigned)__bfloat16_as_ushort(d1[k]) << 16);
    } else {
        if (t >= g.n_views) return;
        const double th = g.start_rad + (double)t * (g.arc_rad / (double)g.n_views);
        const double c = cos(th), s = sin(th), k = g.sdd_mm / g.pitch_mm;  // SOD / ds
        vg[t] = ViewGeo{ff_of(-s * k), ff_of(c * k), ff_of(-c), ff_of(-s)};
    }
}

// Numbers of a call that every thread would divide for.
struct FilterConst {
    double ds, h0;  // bin spacing at the isocentre, h(0)
    FF ipi2, ids;   // 1 / pi^2, 1 / ds
};

__global__ void __launch_bounds__(kTcThreads) k_fbp_filter_tc(const float *__restrict__ m, float *__restrict__ qf,
                                                              const double *__restrict__ cwd,
                                                              const double *__restrict__ tap,
                                                              const uint4 *__restrict__ tw, dect_geometry g,
                                                              FilterConst K, int nimg, int width)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ float sscale[kTcRows];  // 2^(e - 12) of the row
    __shared__ float slim[kTcRows];    // smaller outputs (times ds) are left to FP64; NaN: all of them
    const int nb = g.n_bins, nv = g.n_views;
    const FilterShape F = filter_shape(nb);
    __nv_bfloat16 *A = reinterpret_cast<__nv_bfloat16 *>(dyn);  // [digit][row][ld], the inputs of one parity
    unsigned *T = reinterpret_cast<unsigned *>(A + (size_t)kDig * kTcRows * F.ld);  // [digit][tn]
    FF *cw = reinterpret_cast<FF *>(dyn + F.dig);
    unsigned *todo = reinterpret_cast<unsigned *>(cw + nb);  // [row][nw] a bit per bin left to FP64
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t R0 = (int64_t)blockIdx.x * kTcRows, rows = (int64_t)nv * nimg;
    for (int b = threadIdx.x; b < nb; b += kTcThreads) cw[b] = ff_of(cwd[b]);
    for (int b = threadIdx.x; b < kTcRows * F.nw; b += kTcThreads) todo[b] = 0u;
    for (int w = threadIdx.x; w < kDig * F.tn / 4; w += kTcThreads) reinterpret_cast<uint4 *>(T)[w] = tw[w];
    __syncthreads();
    // a warp per row: its scale, later its digits
    const bool on = R0 + warp < rows;
    const int vw = on ? (int)((R0 + warp) / nimg) : 0, iw = on ? (int)((R0 + warp) % nimg) : 0;
    const float *mine = m + ((int64_t)iw * nv + vw) * nb;
    float sc;
    {
        float mx = 0.f;
        bool finite = true;
        for (int b = lane; b < nb && on; b += 32) {
            const float q = fabsf(mine[b] * cw[b].h);
            finite &= isfinite(q);
            mx = fmaxf(mx, q);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
        finite = __all_sync(0xffffffffu, finite);
        // q < 2^e; rows whose scaled words would leave FP32's range go to FP64
        int e = 0;
        frexpf(mx, &e);
        e += 1;  // the rounded product above may lie a rounding below q
        const bool bad = !finite || (mx > 0.f && (mx < 0x1p-60f || mx > 0x1p60f));
        sc = mx > 0.f && !bad ? ldexpf(1.f, 46 - e) : 0.f;
        if (lane == 0) {
            sscale[warp] = ldexpf(1.f, sc > 0.f ? e - 12 : 0);
            slim[warp] = bad ? NAN : mx > 0.f ? ldexpf(sqrtf((float)nb), e - 23) : 0.f;
        }
    }
    const int gid = lane >> 2, t4 = lane & 3;
    // outputs of parity par from inputs of the other: both, or (two blocks per 16 rows) one
    const int par0 = gridDim.y == 2 ? (int)blockIdx.y : 0, par1 = gridDim.y == 2 ? par0 + 1 : 2;
    for (int par = par0; par < par1; ++par) {
        __syncthreads();  // the scales are written; the other parity's digits have been read
        for (int i = lane; i < F.kpad; i += 32) {
            __nv_bfloat16 d[kDig];
            const int b = 2 * i + 1 - par;
            long long Q = 0;
            if (on && b < nb && sc > 0.f) {
                const FF q = ff_mul(FF{mine[b], 0.f}, cw[b]);
                Q = __float2ll_rn(q.h * sc) + __float2ll_rn(q.l * sc);
            }
            digits(Q, d);
#pragma unroll
            for (int k = 0; k < kDig; ++k) A[((size_t)k * kTcRows + warp) * F.ld + i] = d[k];
        }
        __syncthreads();
        const int nt = (F.half[par] + 7) / 8, per = (nt + kTcWarps - 1) / kTcWarps;
        const int ksteps = (F.half[1 - par] + 15) / 16;
        for (int base = 0; base < per; base += kTcTiles) {
            float acc[kTcTiles][kDig][4];
#pragma unroll
            for (int t = 0; t < kTcTiles; ++t)
#pragma unroll
                for (int k = 0; k < kDig; ++k)
#pragma unroll
                    for (int c = 0; c < 4; ++c) acc[t][k][c] = 0.f;
            const int tile0 = warp * per + base, ntl = min(min(kTcTiles, per - base), nt - tile0);
            for (int ks = 0; ks < ksteps && ntl > 0; ++ks) {
                unsigned af[kDig][4];
#pragma unroll
                for (int k = 0; k < kDig; ++k)
                    ldsm_a(af[k], A + ((size_t)k * kTcRows + (lane & 15)) * F.ld + ks * 16 + (lane >> 4) * 8);
#pragma unroll
                for (int t = 0; t < kTcTiles; ++t) {
                    if (t >= ntl) break;
                    // x = n - k (odd outputs: + 1) of this lane's first element
                    const int xb = (tile0 + t) * 8 - ks * 16 + par;
                    const int w0 = xb + gid - 2 * t4 + F.kpad + 16;
                    const int far = max(xb - 16, -xb - 8);  // |d| of the whole tile is at least 2 far + 1
                    const int l0 = far > 90 ? 2 : far > 5 ? 1 : 0;
#pragma unroll
                    for (int l = 0; l < kDig; ++l) {
                        if (l < l0) continue;
                        const unsigned b0 = T[l * F.tn + w0], b1 = T[l * F.tn + w0 - 8];
#pragma unroll
                        for (int k = 0; k + l < kDig; ++k) mma_exact(acc[t][k + l], af[k], b0, b1);
                    }
                }
            }
#pragma unroll
            for (int t = 0; t < kTcTiles; ++t)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int row = gid + (c >> 1) * 8, n = (tile0 + t) * 8 + 2 * t4 + (c & 1);
                    const int64_t R = R0 + row;
                    if (t >= ntl || n >= F.half[par] || R >= rows) continue;
                    const int b = 2 * n + par, v = (int)(R / nimg), img = (int)(R % nimg);
                    const FF s1 = two_sum(acc[t][0][c], acc[t][1][c] * 0x1p-8f);
                    const FF s2 = two_sum(s1.h, acc[t][2][c] * 0x1p-16f);
                    const FF s3 = two_sum(s2.h, acc[t][3][c] * 0x1p-24f);
                    const float scale = sscale[row];
                    const FF sum = two_sum(s3.h, __fadd_rn(__fadd_rn(s1.l, __fadd_rn(s2.l, s3.l)),
                                                           fmaf(acc[t][5][c], 0x1p-40f, acc[t][4][c] * 0x1p-32f)));
                    const FF far = ff_mul(FF{sum.h * scale, sum.l * scale}, K.ipi2);
                    const FF q = ff_mul(FF{m[((int64_t)img * nv + v) * nb + b], 0.f}, cw[b]);
                    const FF d = ff_add(FF{0.25f * q.h, 0.25f * q.l}, FF{-far.h, -far.l});
                    if (fabsf(d.h) >= slim[row]) {
                        const FF o = ff_mul(d, K.ids);
                        qf[((int64_t)v * nb + b) * width + img] = __fadd_rn(o.h, o.l);
                    } else {
                        atomicOr(&todo[row * F.nw + (b >> 5)], 1u << (b & 31));
                    }
                }
        }
    }
    // What is left to FP64: the rows' q in place of the digits, a warp per row; then a warp
    // per output, its lanes over the taps, 32 bins after 32 to one warp after the other.
    __syncthreads();  // every warp has set its bits and read the digits
    double *q = reinterpret_cast<double *>(dyn);  // [row][nb]
    {
        bool any = false;
        for (int w = lane; w < F.nw; w += 32) any |= todo[warp * F.nw + w] != 0u;
        if (__any_sync(0xffffffffu, any))
            for (int b = lane; b < nb; b += 32) q[warp * nb + b] = (double)mine[b] * cwd[b];
    }
    __syncthreads();
    for (int w = warp; w < kTcRows * F.nw; w += kTcWarps) {
        const int row = w / F.nw;
        const double *qr = q + row * nb;
        const int v = (int)((R0 + row) / nimg), img = (int)((R0 + row) % nimg);
        for (unsigned left = todo[w]; left != 0u; left &= left - 1u) {
            const int b = (w - row * F.nw) * 32 + __ffs(left) - 1;
            double acc = 0.0;
#pragma unroll 4
            for (int i = 1 - (b & 1) + 2 * lane; i < nb; i += 64) acc = fma(tap[abs(i - b) >> 1], qr[i], acc);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            if (lane == 0)
                qf[((int64_t)v * nb + b) * width + img] = (float)(K.ds * fma(K.h0, qr[b], acc));
        }
    }
}

// ---------------------------------------------------------------------------
// Back-projection of W interleaved images (nimg of them real).  A lane holds
// 8 images of a pixel (all of them below 8), W / 8 lanes a pixel, and a warp
// a run of pixels of one row; a block's pixels form a tile, whose bins of a
// view share an L1.  The lanes of a pixel form the geometry of different views
// and hand it round by shuffles.  Per pixel and view two bins x W x 4 bytes
// come back from L1, which bounds the pass: 64 images of 512^2 from 60 views
// are 8 GB, 200 us at the L1 rate (128 bytes per cycle and SM); measured 332
// us (10.4 ms with FP64 geometry repeated for every four images).
// ---------------------------------------------------------------------------
constexpr int kBpBlock = 512;
template <int W>
struct BpShape {
    static constexpr int IPL = W < 8 ? W : 8, LPP = W / IPL;  // images per lane, lanes per pixel
    static constexpr int PX = kBpBlock / LPP;                   // pixels per block
    static constexpr int TW = PX >= 256 ? 32 : 8, TH = PX / TW;
    static constexpr int VW = IPL >= 4 ? 4 : IPL;
    static constexpr int GV = LPP < 4 ? 4 : LPP, GPL = GV / LPP;  // views of a group, of a lane's geometry
};

// Numbers of a call, in two words (these and the pixel coordinates, formed in FP64 by
// every thread, took 47 us of the above case).
struct BpConst {
    int n, nv, nb;
    FF sod, half_dth, t0;  // t0: the isocentre's bin coordinate, negated
};

template <int W>
__global__ void __launch_bounds__(kBpBlock, 2) k_fbp_bp(const float *__restrict__ qf, float *__restrict__ x,
                                                        const ViewGeo *__restrict__ vg, const FF *__restrict__ pos,
                                                        BpConst K, int nimg)
{
    using S = BpShape<W>;
    constexpr int NV = S::IPL / S::VW;
    const int n = K.n, nv = K.nv, nb = K.nb;
    const FF sod = K.sod, half_dth = K.half_dth, t0 = K.t0;
    const int p = threadIdx.x / S::LPP, sub = threadIdx.x % S::LPP;
    const int i = blockIdx.y * S::TH + p / S::TW, j = blockIdx.x * S::TW + p % S::TW;
    const bool in = i < n && j < n;
    const FF px = pos[min(j, n - 1)], py = pos[min(i, n - 1)];
    const float tmax = (float)(nb - 1);
    float acc[S::IPL];
#pragma unroll
    for (int k = 0; k < S::IPL; ++k) acc[k] = 0.f;
    for (int v0 = 0; v0 < nv; v0 += S::GV) {
        int ray[S::GPL];  // first of the two rays, -1: the pixel lies outside the view's detector
        float wa[S::GPL], wb[S::GPL];
#pragma unroll
        for (int e = 0; e < S::GPL; ++e) {
            ray[e] = -1;
            wa[e] = wb[e] = 0.f;
            const int v = v0 + e * S::LPP + sub;
            if (v >= nv || !in) continue;
            const float4 E = __ldg(reinterpret_cast<const float4 *>(vg + v));
            const float4 C = __ldg(reinterpret_cast<const float4 *>(vg + v) + 1);
            const FF num = ff_add(ff_mul(px, FF{E.x, E.y}), ff_mul(py, FF{E.z, E.w}));
            const FF L = ff_add(sod, ff_add(ff_mul(px, FF{C.x, C.y}), ff_mul(py, FF{C.z, C.w})));
            // t = num / L - t0
            const float rc = __frcp_rn(L.h), q0 = __fmul_rn(num.h, rc);
            const float rem = __fadd_rn(fmaf(-q0, L.h, num.h), fmaf(-q0, L.l, num.l));
            FF t = two_sum(q0, -t0.h);
            t.l = __fadd_rn(t.l, __fsub_rn(__fmul_rn(rem, rc), t0.l));
            t = two_sum(t.h, t.l);
            float b0 = floorf(t.h), w = __fadd_rn(__fsub_rn(t.h, b0), t.l);
            if (w < 0.f) {  // t.h is an integer and t.l < 0
                b0 -= 1.f;
                w += 1.f;
            }
            if (b0 >= 0.f && (b0 < tmax || (b0 == tmax && w == 0.f))) {
                if (b0 == tmax) {
                    b0 -= 1.f;
                    w = 1.f;
                }
                // weight half_dth (sod / L)^2, rounded once
                FF r;
                r.h = __fmul_rn(sod.h, rc);
                r.l = __fmul_rn(rc, __fadd_rn(fmaf(-r.h, L.h, sod.h), fmaf(-r.h, L.l, sod.l)));
                const FF wt2 = ff_mul(half_dth, ff_mul(r, r));
                const float wt = __fadd_rn(wt2.h, wt2.l);
                int bi = (int)b0;
                if (!DECT_IDX_OK(bi, nb - 1, CHK_FBP_BIN)) bi = 0;
                ray[e] = v * nb + bi;
                wb[e] = wt * w;
                wa[e] = wt - wb[e];
            }
        }
        // the group's views are summed on their own first: fewer roundings at
        // the size of the running sum than one per view
        float part[S::IPL];
#pragma unroll
        for (int k = 0; k < S::IPL; ++k) part[k] = 0.f;
#pragma unroll
        for (int u = 0; u < S::GV; ++u) {
            const int e = u / S::LPP, src = (threadIdx.x & 31 & ~(S::LPP - 1)) + u % S::LPP;
            const int ru = S::LPP > 1 ? __shfl_sync(0xffffffffu, ray[e], src) : ray[e];
            const float a = S::LPP > 1 ? __shfl_sync(0xffffffffu, wa[e], src) : wa[e];
            const float b = S::LPP > 1 ? __shfl_sync(0xffffffffu, wb[e], src) : wb[e];
            if (ru < 0) continue;
            // load k covers images 4 (k LPP + sub) .. + 3: the pixel's lanes read contiguous bytes
            const float *q = qf + (int64_t)ru * W + sub * S::VW;
            Vec<S::VW> lo[NV], hi[NV];
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                lo[k] = ld_il<S::VW>(q + k * S::LPP * S::VW);
                hi[k] = ld_il<S::VW>(q + W + k * S::LPP * S::VW);
            }
#pragma unroll
            for (int k = 0; k < NV; ++k)
#pragma unroll
                for (int c = 0; c < S::VW; ++c)
                    part[k * S::VW + c] = fmaf(a, lo[k].v[c], fmaf(b, hi[k].v[c], part[k * S::VW + c]));
        }
#pragma unroll
        for (int k = 0; k < S::IPL; ++k) acc[k] += part[k];
    }
    if (!in) return;
    const int64_t N = (int64_t)n * n, pix = (int64_t)i * n + j;
#pragma unroll
    for (int k = 0; k < NV; ++k)
#pragma unroll
        for (int c = 0; c < S::VW; ++c) {
            const int img = (k * S::LPP + sub) * S::VW + c;
            if (img < nimg) x[(int64_t)img * N + pix] = acc[k * S::VW + c];
        }
}

template <int W>
void launch_bp(const float *qf, float *x, const ViewGeo *vg, const FF *pos, const BpConst &K, int nimg, cudaStream_t s)
{
    using S = BpShape<W>;
    const dim3 grid((unsigned)((K.n + S::TW - 1) / S::TW), (unsigned)((K.n + S::TH - 1) / S::TH));
    k_fbp_bp<W><<<grid, kBpBlock, 0, s>>>(qf, x, vg, pos, K, nimg);
}

}  // namespace
}  // namespace dect

using namespace dect;

extern "C" dect_status dect_fbp(const dect_plan *plan, const float *m, float *x, int batch, dect_stream stream)
{
    if (!plan || batch < 0 || plan->nz > 0) return DECT_ERR_INVALID_ARG;  // fan-beam plans only
    if (batch == 0) return DECT_OK;
    if (!m || !x) return DECT_ERR_INVALID_ARG;
    const dect_geometry &g = plan->g;
    if (std::fabs(g.arc_rad - 6.283185307179586) > 1e-9) {
        set_error_text("dect_fbp: the fan-beam FBP needs a full 360-degree scan (arc_rad = 2 pi)");
        return DECT_ERR_INVALID_ARG;
    }
    if (g.n_bins < 2) {
        set_error_text("dect_fbp: at least 2 detector bins");
        return DECT_ERR_INVALID_ARG;
    }
    const size_t smem = sizeof(double) * ((size_t)g.n_bins + (size_t)(g.n_bins / 2 + 1));
    if (smem > 200 * 1024) {
        set_error_text("dect_fbp: too many detector bins for the shared-memory filter");
        return DECT_ERR_INVALID_ARG;
    }
    DECT_CUDA(cudaSetDevice(plan->device));
    cudaStream_t s = (cudaStream_t)stream;
    int width = 1;  // images per pass: the next power of two >= min(batch, 64)
    while (width < std::min(batch, kMaxBatchImages)) width *= 2;
    const size_t nr = (size_t)g.n_views * g.n_bins, qbytes = (sizeof(float) * nr * width + 255) & ~(size_t)255;
    const int nodd = g.n_bins / 2 + 1;
    char *base = nullptr;
    const FilterShape F = filter_shape(g.n_bins);
    const size_t vbytes = sizeof(ViewGeo) * (size_t)g.n_views, wbytes = sizeof(unsigned) * (size_t)kDig * F.tn;
    DECT_CUDA(cudaMallocAsync((void **)&base,
                              qbytes + vbytes + wbytes + sizeof(double) * (size_t)(g.n_bins + nodd) + sizeof(FF) * g.n, s));
    float *qf = (float *)base;
    ViewGeo *vg = (ViewGeo *)(base + qbytes);
    unsigned *tw = (unsigned *)(base + qbytes + vbytes);  // (16-byte aligned: both sizes are multiples of 32)
    double *cwd = (double *)(base + qbytes + vbytes + wbytes), *tap = cwd + g.n_bins;
    FF *pos = (FF *)(tap + nodd);
    FilterConst K;
    K.ds = g.pitch_mm * (g.sod_mm / g.sdd_mm);
    K.h0 = 1.0 / (4.0 * K.ds * K.ds);
    K.ipi2 = ff_of(1.0 / (3.14159265358979323846 * 3.14159265358979323846));
    K.ids = ff_of(1.0 / K.ds);
    const bool tc = g.n_bins <= kTcMaxBins;
    cudaError_t e = cudaFuncSetAttribute(k_fbp_filter, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_fbp_filter_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmemMax);
    const BpConst B{g.n, g.n_views, g.n_bins, ff_of(g.sod_mm), ff_of(0.5 * g.arc_rad / (double)g.n_views),
                    ff_of(-0.5 * (double)(g.n_bins - 1) + g.det_offset_mm / g.pitch_mm)};
    if (e == cudaSuccess) {
        const int most = std::max({g.n, g.n_views, g.n_bins, F.tn});
        k_fbp_tables<<<dim3((unsigned)((most + kTableBlock - 1) / kTableBlock), kTables), kTableBlock, 0, s>>>(
            g, vg, cwd, tap, tw, pos);
        count_launches(1);
    }
    for (int done = 0; done < batch && e == cudaSuccess; done += kMaxBatchImages) {
        const int k = std::min(kMaxBatchImages, batch - done);
        const float *mk = m + (size_t)done * nr;
        float *xk = x + (int64_t)done * plan->N;
        int w = 1;
        while (w < k) w *= 2;
        if (tc) {
            // few rows leave most of the chip idle: a block per parity then (call on one image of
            // 512^2 / 60 views, 8 blocks instead of 4: 186 -> 147 us)
            const unsigned blocks = (unsigned)(((int64_t)g.n_views * k + kTcRows - 1) / kTcRows);
            k_fbp_filter_tc<<<dim3(blocks, blocks <= (unsigned)kSMs / 2 ? 2 : 1), kTcThreads, F.smem, s>>>(
                mk, qf, cwd, tap, (const uint4 *)tw, g, K, k, w);
        } else
            k_fbp_filter<<<dim3(g.n_views, k), kFbpBlock, smem, s>>>(mk, qf, g, w);
        switch (w) {
        case 1: launch_bp<1>(qf, xk, vg, pos, B, k, s); break;
        case 2: launch_bp<2>(qf, xk, vg, pos, B, k, s); break;
        case 4: launch_bp<4>(qf, xk, vg, pos, B, k, s); break;
        case 8: launch_bp<8>(qf, xk, vg, pos, B, k, s); break;
        case 16: launch_bp<16>(qf, xk, vg, pos, B, k, s); break;
        case 32: launch_bp<32>(qf, xk, vg, pos, B, k, s); break;
        default: launch_bp<64>(qf, xk, vg, pos, B, k, s); break;
        }
        count_launches(2);
        e = cudaGetLastError();
    }
    cudaFreeAsync(base, s);
    if (e != cudaSuccess) {
        set_error("dect_fbp", e);
        return e == cudaErrorMemoryAllocation ? DECT_ERR_OOM : DECT_ERR_CUDA;
    }
    return DECT_OK;
}
