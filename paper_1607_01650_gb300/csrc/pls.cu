// PLS image-domain decomposition, Eq. (11)-(15) (Sec. 2.3).
//
//   d   = D^{-1} x per pixel, D = [[eta_1H, eta_2H], [eta_1L, eta_2L]]     Eq. (11)-(12)
//         (closed-form 2x2 inverse in FP64)
//   e_ik= edge_eps if pixel i or k is an edge, else 1                     Eq. (14)
//         (edge: 3x3 Prewitt magnitude of x_h or x_l over its maximum > tau)
//   (I + gamma L_e) u_m = d_m,  (L_e u)_i = sum_{k in N_i} e_ik (u_i - u_k)
//         -- Eq. (15) with Hessian R = 2 L_e -- by Jacobi-preconditioned CG
//         from u = d, FP32 vectors, FP64 scalars.
//
// Vectors: v = 2 s + m (slice s, material m) at u + v N (the [slice][2][n][n]
// layout of the input and output); the CG runs all vectors of the batch in
// lockstep with per-vector step sizes and stop flags.  The edge decision is
// taken in FP32 (the precision of the reconstructed images; the paper fixes
// none for it): it can differ from the FP64 decision only at pixels whose
// normalised magnitude lies within FP32 rounding of the threshold.
//
// The CG keeps u, z = r / diag and p per vector (r = z diag is not stored),
// and one 16-bit link code per pixel of a slice.  A p is formed twice per
// iteration from p (once for <p, A p>, once for the z step) rather than
// stored, so an iteration moves 8 values per pixel and material: memory
// bandwidth bounds it (32 slices of 512^2: 58 + 72 us per iteration, 4.1 TB/s;
// storing r, z and A p and forming the diagonal from the mask took 189 + 176).
// On one slice an iteration is two launches of 7 to 9 us.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "dect_internal.cuh"

namespace dect {
namespace {

constexpr int kBlock = 256;

struct PlsDev {
    // scalars per vector
    double *part;     // [nvec][3][gx] block partials
    unsigned *ctr;    // [nvec] last-block tickets
    double *alpha, *beta, *rz, *bnorm;  // [nvec]
    int *done;        // [nvec]
    int *maxbits;     // [nvec] float bits of max Prewitt magnitude (slice, energy)
    // read back by the host in one copy: relres, iters, ndone
    double *relres;   // [nvec]
    int *iters;       // [nvec]
    int *ndone;       // [1] vectors that have stopped
};

struct PlsConst {
    int n, nz;   // nz = 1: 2-D images (4 neighbours); nz > 1: volumes (6 neighbours)
    int64_t N;
    float gamma, eps;
    double tol;
};

// Sums of K values over the blocks of vector v = blockIdx.y: FP32 inside a
// warp, FP64 across warps and blocks, always in the same order.  The vector's
// last block (a ticket per vector) returns true, with the totals in out[] of
// thread 0.  A vector's partials (at most 1216, cg_blocks) are summed by one warp
// per value, lanes in fixed strides, then a fixed butterfly: summing them one
// after the other in a single thread cost 40 of the 45 us of each launch on
// one 512^2 slice.
template <int K>
__device__ bool reduce_vec(const float (&v)[K], double *part, unsigned *counter, double (&out)[K])
{
    constexpr int NW = kBlock / 32;
    __shared__ double smem[NW * K];
    __shared__ double tot[K];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned gx = gridDim.x, y = blockIdx.y;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        float w = v[k];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) w += __shfl_xor_sync(0xffffffffu, w, off);
        if (lane == 0) smem[warp * K + k] = (double)w;
    }
    __syncthreads();
    double *mine = part + (size_t)y * gx * K;
    if (threadIdx.x < 32) {  // the partials' stores, the fence and the ticket in one warp
        if (lane < K) {
            double t = 0.0;
            for (int q = 0; q < NW; ++q) t += smem[q * K + lane];
            mine[(size_t)lane * gx + blockIdx.x] = t;
            __threadfence();
        }
        __syncwarp();
        if (lane == 0) last = atomicAdd(&counter[y], 1u) == gx - 1;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    if (warp < K) {
        double t = 0.0;
        for (unsigned b = lane; b < gx; b += 32) t += __ldcg(&mine[(size_t)warp * gx + b]);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
        if (lane == 0) tot[warp] = t;
    }
    if (threadIdx.x == 0) counter[y] = 0u;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) out[k] = tot[k];
    return true;
}

__device__ __forceinline__ int clampi(int a, int lo, int hi) { return a < lo ? lo : (a > hi ? hi : a); }

// 3-D Prewitt magnitude (volumes of nz > 1 slices), FP32, each component
// summed in the order of the two outer offsets s, t = -1, 0, 1.
__device__ __forceinline__ float prewitt3_at(const float *__restrict__ x, int n, int nz, int k, int i, int j)
{
    auto X = [&](int kk, int ii, int jj) {
        return x[((int64_t)clampi(kk, 0, nz - 1) * n + clampi(ii, 0, n - 1)) * n + clampi(jj, 0, n - 1)];
    };
    float gx = 0.f, gy = 0.f, gz = 0.f;
    for (int a = -1; a <= 1; ++a)
        for (int b = -1; b <= 1; ++b) {
            gx = __fadd_rn(gx, __fsub_rn(X(k + a, i + b, j + 1), X(k + a, i + b, j - 1)));
            gy = __fadd_rn(gy, __fsub_rn(X(k + a, i + 1, j + b), X(k + a, i - 1, j + b)));
            gz = __fadd_rn(gz, __fsub_rn(X(k + 1, i + a, j + b), X(k - 1, i + a, j + b)));
        }
    return __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(gx, gx), __fmul_rn(gy, gy)), __fmul_rn(gz, gz)));
}

// Volumes (nz > 1): d = D^{-1} x (FP64), written as the initial u (skipped
// when u is null); 3-D Prewitt magnitudes, stored, and their maxima.
__global__ void k_prep3(const float *__restrict__ x, int n, int nz, int64_t N, double a, double b, double c,
                       double e, float *__restrict__ u, float *__restrict__ mh,
                       float *__restrict__ ml, int *__restrict__ maxbits)
{
    const int s = blockIdx.y;
    const float *xs = x + (int64_t)(2 * s) * N, *ls = xs + N;
    float lmax_h = 0.f, lmax_l = 0.f;
    const double det = __dsub_rn(__dmul_rn(a, e), __dmul_rn(b, c));
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < N;
         p += (int64_t)gridDim.x * blockDim.x) {
        const double h = xs[p], l = ls[p];
        const double d1 = __ddiv_rn(__dsub_rn(__dmul_rn(e, h), __dmul_rn(b, l)), det);
        const double d2 = __ddiv_rn(__dadd_rn(__dmul_rn(-c, h), __dmul_rn(a, l)), det);
        if (u) {
            u[(int64_t)(2 * s) * N + p] = (float)d1;
            u[(int64_t)(2 * s + 1) * N + p] = (float)d2;
        }
        const int64_t plane = (int64_t)n * n;
        const int k = (int)(p / plane), i = (int)((p % plane) / n), j = (int)(p % n);
        const float g1 = prewitt3_at(xs, n, nz, k, i, j);
        const float g2 = prewitt3_at(ls, n, nz, k, i, j);
        mh[(int64_t)s * N + p] = g1;
        ml[(int64_t)s * N + p] = g2;
        lmax_h = fmaxf(lmax_h, g1);
        lmax_l = fmaxf(lmax_l, g2);
    }
    // maxima of non-negative floats: integer max of their bit patterns
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        lmax_h = fmaxf(lmax_h, __shfl_xor_sync(0xffffffffu, lmax_h, off));
        lmax_l = fmaxf(lmax_l, __shfl_xor_sync(0xffffffffu, lmax_l, off));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&maxbits[2 * s], __float_as_int(lmax_h));
        atomicMax(&maxbits[2 * s + 1], __float_as_int(lmax_l));
    }
}

__global__ void k_mask3(const float *__restrict__ mh, const float *__restrict__ ml, int64_t N,
                       const int *__restrict__ maxbits, float tau, unsigned char *__restrict__ mask)
{
    const int s = blockIdx.y;
    const float Mh = __int_as_float(maxbits[2 * s]), Ml = __int_as_float(maxbits[2 * s + 1]);
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < N;
         p += (int64_t)gridDim.x * blockDim.x) {
        const int64_t q = (int64_t)s * N + p;
        const bool eh = Mh > 0.f && __fdiv_rn(mh[q], Mh) > tau;
        const bool el = Ml > 0.f && __fdiv_rn(ml[q], Ml) > tau;
        mask[q] = (unsigned char)(eh || el);
    }
}

// ---------------------------------------------------------------------------
// 2-D images.  A thread walks kRows rows down one column, the Prewitt terms of
// the rows above and below in registers (3 loads per pixel and energy).  The
// magnitudes are not stored: the maxima pass (k_prep) and the mask pass
// (k_mask) each form them from x, which costs less than writing and reading
// two more arrays.
// ---------------------------------------------------------------------------
constexpr int kRows = 16, kPrepBlock = 128;

// the 3 pixels of a row around column j (replicate padding)
struct Row3 {
    float l, c, r;
};
__device__ __forceinline__ Row3 ld_row3(const float *__restrict__ x, int n, int i, int jl, int j, int jr)
{
    const float *row = x + (int64_t)clampi(i, 0, n - 1) * n;
    return Row3{row[jl], row[j], row[jr]};
}
// Prewitt magnitude, FP32, explicit rounding: gx sums the rows' right - left
// differences from the upper row down, gy the columns' lower - upper
// differences from the left column on.
__device__ __forceinline__ float prewitt_rows(const Row3 &u, const Row3 &c, const Row3 &d)
{
    const float gx = __fadd_rn(__fadd_rn(__fsub_rn(u.r, u.l), __fsub_rn(c.r, c.l)), __fsub_rn(d.r, d.l));
    const float gy = __fadd_rn(__fadd_rn(__fsub_rn(d.l, u.l), __fsub_rn(d.c, u.c)), __fsub_rn(d.r, u.r));
    return __fsqrt_rn(__fadd_rn(__fmul_rn(gx, gx), __fmul_rn(gy, gy)));
}

// (e0 p - e1 q) / det rounded once from its FP64 value, where the caller's
// FP64 form is exact64().  The quotient is first formed in two FP32 words
// (coefficients split in two, error below 2^-42 of the terms), which decides
// the FP32 rounding unless the value lies that near a rounding boundary; then
// (about once in 10^5 pixels), and for zeros, denormals and non-finite values,
// the FP64 form decides.  FP64 runs at 1/64 of the FP32 rate: with it alone
// this pass was bound by its two divisions (500 us on 32 slices of 512^2).
struct Coef {
    float hi, lo;
};
template <typename F>
__device__ __forceinline__ float solve2(const Coef &A, float p, const Coef &B, float q, F exact64)
{
    const float p1 = A.hi * p, e1 = fmaf(A.lo, p, fmaf(A.hi, p, -p1));
    const float p2 = B.hi * q, e2 = fmaf(B.lo, q, fmaf(B.hi, q, -p2));
    const float s = __fsub_rn(p1, p2), bv = __fsub_rn(s, p1);
    const float err = __fadd_rn(__fsub_rn(p1, __fsub_rn(s, bv)), -__fadd_rn(p2, bv));  // p1 - p2 = s + err
    const float lo = __fadd_rn(err, __fsub_rn(e1, e2));
    const float r = __fadd_rn(s, lo), rv = __fsub_rn(r, s);
    const float t = __fadd_rn(__fsub_rn(s, __fsub_rn(r, rv)), __fsub_rn(lo, rv));      // s + lo = r + t
    const unsigned bits = __float_as_uint(r), ex = (bits >> 23) & 255u;
    const float half = __uint_as_float((ex > 24u ? ex - 24u : 0u) << 23);              // half an ulp of r
    const float bound = 0x1p-42f * (fabsf(p1) + fabsf(p2));
    const bool ok = ex > 60u && ex < 255u && (bits & 0x7fffffu) != 0u && fabsf(t) + bound < half;
    return ok ? r : exact64();
}

struct Solve2 {  // D^{-1} in FP64 (a, b, c, e, det) and divided by det in two FP32 words
    double a, b, c, e, det;
    Coef ed, bd, ad, cd;
};

// d = D^{-1} x, written as the initial u (skipped when u is null), and the
// maxima of the Prewitt magnitudes.
__global__ void __launch_bounds__(kPrepBlock) k_prep(const float *__restrict__ x, int n, Solve2 S,
                                                     float *__restrict__ u, int *__restrict__ maxbits)
{
    const int s = blockIdx.z, j = blockIdx.x * kPrepBlock + threadIdx.x, i0 = blockIdx.y * kRows;
    const int64_t N = (int64_t)n * n;
    const float *xs = x + (int64_t)(2 * s) * N, *ls = xs + N;
    float mx[2] = {0.f, 0.f};
    if (j < n) {
        const int jl = max(j - 1, 0), jr = min(j + 1, n - 1), i1 = min(i0 + kRows, n);
        Row3 hu = ld_row3(xs, n, i0 - 1, jl, j, jr), hc = ld_row3(xs, n, i0, jl, j, jr);
        Row3 lu = ld_row3(ls, n, i0 - 1, jl, j, jr), lc = ld_row3(ls, n, i0, jl, j, jr);
#pragma unroll 4
        for (int i = i0; i < i1; ++i) {
            const Row3 hd = ld_row3(xs, n, i + 1, jl, j, jr), ld = ld_row3(ls, n, i + 1, jl, j, jr);
            mx[0] = fmaxf(mx[0], prewitt_rows(hu, hc, hd));
            mx[1] = fmaxf(mx[1], prewitt_rows(lu, lc, ld));
            if (u) {
                const float h = hc.c, l = lc.c;
                float *o = u + (int64_t)(2 * s) * N + (int64_t)i * n + j;
                o[0] = solve2(S.ed, h, S.bd, l, [&]() {
                    return (float)__ddiv_rn(__dsub_rn(__dmul_rn(S.e, h), __dmul_rn(S.b, l)), S.det);
                });
                o[N] = solve2(S.ad, l, S.cd, h, [&]() {
                    return (float)__ddiv_rn(__dadd_rn(__dmul_rn(-S.c, h), __dmul_rn(S.a, l)), S.det);
                });
            }
            hu = hc;
            hc = hd;
            lu = lc;
            lc = ld;
        }
    }
    // maxima of non-negative floats: integer max of their bit patterns, one atomic per block
    __shared__ int bm[2];
    if (threadIdx.x < 2) bm[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int m = __reduce_max_sync(0xffffffffu, __float_as_int(mx[e]));
        if ((threadIdx.x & 31) == 0) atomicMax(&bm[e], m);
    }
    __syncthreads();
    if (threadIdx.x < 2) atomicMax(&maxbits[2 * s + threadIdx.x], bm[threadIdx.x]);
}

__global__ void __launch_bounds__(kPrepBlock) k_mask(const float *__restrict__ x, int n,
                                                     const int *__restrict__ maxbits, float tau,
                                                     unsigned char *__restrict__ mask)
{
    const int s = blockIdx.z, j = blockIdx.x * kPrepBlock + threadIdx.x, i0 = blockIdx.y * kRows;
    if (j >= n) return;
    const int64_t N = (int64_t)n * n;
    const float *xs = x + (int64_t)(2 * s) * N, *ls = xs + N;
    const float Mh = __int_as_float(maxbits[2 * s]), Ml = __int_as_float(maxbits[2 * s + 1]);
    const int jl = max(j - 1, 0), jr = min(j + 1, n - 1), i1 = min(i0 + kRows, n);
    Row3 hu = ld_row3(xs, n, i0 - 1, jl, j, jr), hc = ld_row3(xs, n, i0, jl, j, jr);
    Row3 lu = ld_row3(ls, n, i0 - 1, jl, j, jr), lc = ld_row3(ls, n, i0, jl, j, jr);
#pragma unroll 4
    for (int i = i0; i < i1; ++i) {
        const Row3 hd = ld_row3(xs, n, i + 1, jl, j, jr), ld = ld_row3(ls, n, i + 1, jl, j, jr);
        const bool eh = Mh > 0.f && __fdiv_rn(prewitt_rows(hu, hc, hd), Mh) > tau;
        const bool el = Ml > 0.f && __fdiv_rn(prewitt_rows(lu, lc, ld), Ml) > tau;
        mask[(int64_t)s * N + (int64_t)i * n + j] = (unsigned char)(eh || el);
        hu = hc;
        hc = hd;
        lu = lc;
        lc = ld;
    }
}

// ---------------------------------------------------------------------------
// Link codes.  Bit m of a pixel's code: its m-th neighbour lies in the image
// and the link has weight 1; bit 6 + m: the link has weight edge_eps (Eq.
// (14); out-of-image links are omitted and have neither bit).  Neighbours in
// the order (slice - 1, slice + 1, row - 1, row + 1, column - 1, column + 1).
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool has_link(unsigned code, int m) { return (code & (0x41u << m)) != 0u; }
__device__ __forceinline__ float link_w(unsigned code, int m, float eps)
{
    return (code >> m) & 1u ? 1.f : ((code >> (6 + m)) & 1u ? eps : 0.f);
}
__device__ __forceinline__ float jacobi_diag(unsigned code, float gamma, float eps)
{
    float wsum = 0.f;
#pragma unroll
    for (int m = 0; m < 6; ++m) wsum += link_w(code, m, eps);
    return 1.f + gamma * wsum;
}

template <int VEC>
struct Px {
    float v[VEC];
};
template <int VEC>
__device__ __forceinline__ Px<VEC> ld_px(const float *p)
{
    Px<VEC> r;
    if constexpr (VEC == 4) {
        const float4 t = *reinterpret_cast<const float4 *>(p);
        r.v[0] = t.x, r.v[1] = t.y, r.v[2] = t.z, r.v[3] = t.w;
    } else {
        r.v[0] = *p;
    }
    return r;
}
template <int VEC>
__device__ __forceinline__ void st_px(float *p, const Px<VEC> &a)
{
    if constexpr (VEC == 4)
        *reinterpret_cast<float4 *>(p) = make_float4(a.v[0], a.v[1], a.v[2], a.v[3]);
    else
        *p = a.v[0];
}
template <int VEC>
__device__ __forceinline__ void ld_code(const unsigned short *p, unsigned (&c)[VEC])
{
    if constexpr (VEC == 4) {
        const ushort4 t = *reinterpret_cast<const ushort4 *>(p);
        c[0] = t.x, c[1] = t.y, c[2] = t.z, c[3] = t.w;
    } else {
        c[0] = *p;
    }
}

// (I + gamma L_e) applied to the VEC pixels q .. q + VEC - 1 of one row;
// val(q) gives the vector's VEC values at q, val1(q) one value, c those at q.
template <int VEC, typename F, typename F1>
__device__ __forceinline__ Px<VEC> apply_op(const PlsConst &C, int64_t q, const unsigned (&code)[VEC], const Px<VEC> &c,
                                            F val, F1 val1)
{
    Px<VEC> acc;
#pragma unroll
    for (int t = 0; t < VEC; ++t) acc.v[t] = 0.f;
    const int64_t off[4] = {-(int64_t)C.n * C.n, (int64_t)C.n * C.n, -(int64_t)C.n, (int64_t)C.n};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        if (!has_link(code[0], m)) continue;  // the same for all pixels of the row
        int64_t k = q + off[m];
        if (!DECT_IDX_OK(k, C.N - VEC + 1, CHK_PLS_STENCIL)) k = q;
        const Px<VEC> o = val(k);
#pragma unroll
        for (int t = 0; t < VEC; ++t) acc.v[t] += link_w(code[t], m, C.eps) * (c.v[t] - o.v[t]);
    }
    float left = c.v[0], right = c.v[VEC - 1];
    if (has_link(code[0], 4)) left = val1(DECT_IDX_OK(q - 1, C.N, CHK_PLS_STENCIL) ? q - 1 : q);
    if (has_link(code[VEC - 1], 5)) right = val1(DECT_IDX_OK(q + VEC, C.N, CHK_PLS_STENCIL) ? q + VEC : q);
#pragma unroll
    for (int t = 0; t < VEC; ++t) {
        const float l = t > 0 ? c.v[t > 0 ? t - 1 : 0] : left, r = t + 1 < VEC ? c.v[t + 1 < VEC ? t + 1 : 0] : right;
        if (has_link(code[t], 4)) acc.v[t] += link_w(code[t], 4, C.eps) * (c.v[t] - l);
        if (has_link(code[t], 5)) acc.v[t] += link_w(code[t], 5, C.eps) * (c.v[t] - r);
        acc.v[t] = c.v[t] + C.gamma * acc.v[t];
    }
    return acc;
}

// z = (d - A d) / diag of vector v and (from the first material's blocks) the
// slice's link codes; reductions <r, z>, <r, r> (r = z diag) and <d, d>.
template <int VEC>
__global__ void __launch_bounds__(kBlock) k_init(const float *__restrict__ uall, const unsigned char *__restrict__ mask,
                                                 unsigned short *__restrict__ codes, float *__restrict__ zall,
                                                 PlsConst C, PlsDev D)
{
    const int v = blockIdx.y, s = v >> 1;
    const unsigned char *mk = mask + (int64_t)s * C.N;
    const float *u = uall + (int64_t)v * C.N;
    const int64_t plane = (int64_t)C.n * C.n;
    float acc[3] = {0.f, 0.f, 0.f};
    for (int64_t q = ((int64_t)blockIdx.x * kBlock + threadIdx.x) * VEC; q < C.N; q += (int64_t)gridDim.x * kBlock * VEC) {
        int k, i, j;
        if (C.N <= 0xffffffffll) {  // 64-bit division costs more than the rest of the pass
            const unsigned q32 = (unsigned)q, row = q32 / (unsigned)C.n;
            j = (int)(q32 - row * (unsigned)C.n);
            k = (int)(row / (unsigned)C.n);
            i = (int)(row - (unsigned)k * (unsigned)C.n);
        } else {
            k = (int)(q / plane);
            i = (int)((q % plane) / C.n);
            j = (int)(q % C.n);
        }
        const bool in[4] = {k > 0, k + 1 < C.nz, i > 0, i + 1 < C.n};
        const int64_t off[4] = {-plane, plane, -(int64_t)C.n, (int64_t)C.n};
        unsigned code[VEC];
        unsigned char me[VEC + 2];  // the row's masks, one pixel more on either side
#pragma unroll
        for (int t = 0; t < VEC + 2; ++t) {
            const bool ok = (t > 0 || j > 0) && (t <= VEC || j + VEC < C.n);
            me[t] = mk[ok && DECT_IDX_OK(q + t - 1, C.N, CHK_PLS_STENCIL) ? q + t - 1 : q];
        }
#pragma unroll
        for (int t = 0; t < VEC; ++t) {
            code[t] = 0u;
            if (t > 0 || j > 0) code[t] |= ((me[t + 1] | me[t]) ? 0x40u : 1u) << 4;
            if (t + 1 < VEC || j + VEC < C.n) code[t] |= ((me[t + 1] | me[t + 2]) ? 0x40u : 1u) << 5;
        }
#pragma unroll
        for (int m = 0; m < 4; ++m)
            if (in[m])
#pragma unroll
                for (int t = 0; t < VEC; ++t) {
                    const int64_t nb = q + t + off[m];
                    code[t] |= ((me[t + 1] | mk[DECT_IDX_OK(nb, C.N, CHK_PLS_STENCIL) ? nb : q]) ? 0x40u : 1u) << m;
                }
        if (!(v & 1)) {
            if constexpr (VEC == 4)
                *reinterpret_cast<ushort4 *>(codes + (int64_t)s * C.N + q) =
                    make_ushort4((unsigned short)code[0], (unsigned short)code[1], (unsigned short)code[2], (unsigned short)code[3]);
            else
                codes[(int64_t)s * C.N + q] = (unsigned short)code[0];
        }
        const Px<VEC> c = ld_px<VEC>(u + q);
        const Px<VEC> Ad = apply_op<VEC>(C, q, code, c, [&](int64_t t) { return ld_px<VEC>(u + t); },
                                         [&](int64_t t) { return u[t]; });
        Px<VEC> z;
#pragma unroll
        for (int t = 0; t < VEC; ++t) {
            const float rr = c.v[t] - Ad.v[t];
            z.v[t] = rr / jacobi_diag(code[t], C.gamma, C.eps);
            acc[0] = fmaf(rr, z.v[t], acc[0]);
            acc[1] = fmaf(rr, rr, acc[1]);
            acc[2] = fmaf(c.v[t], c.v[t], acc[2]);
        }
        st_px<VEC>(zall + (int64_t)v * C.N + q, z);
    }
    double out[3];
    if (!reduce_vec<3>(acc, D.part, D.ctr, out) || threadIdx.x > 0) return;
    D.rz[v] = out[0];
    D.bnorm[v] = sqrt(out[2]);
    D.relres[v] = D.bnorm[v] > 0.0 ? sqrt(out[1]) / D.bnorm[v] : 0.0;
    D.beta[v] = 0.0;
    D.alpha[v] = 0.0;
    D.iters[v] = 0;
    D.done[v] = (C.tol > 0.0 && D.relres[v] < C.tol) || D.bnorm[v] == 0.0;
    if (D.done[v]) atomicAdd(D.ndone, 1);
}

// A vector that has stopped (its flag is set by its last block, after all its
// blocks of that launch have read it) leaves the launches at once.

// p_new = z + beta p_old (FIRST: p_new = z, p_old is not read), reduction
// <p, A p>, alpha.
template <int VEC, bool FIRST>
__global__ void __launch_bounds__(kBlock) k_cg_a(const float *__restrict__ zall, const float *__restrict__ pold,
                                                 float *__restrict__ pnew, const unsigned short *__restrict__ codes,
                                                 PlsConst C, PlsDev D)
{
    const int v = blockIdx.y;
    if (D.done[v]) return;
    const unsigned short *cs = codes + (int64_t)(v >> 1) * C.N;
    const float beta = (float)D.beta[v];
    const float *zv = zall + (int64_t)v * C.N, *pv = pold + (int64_t)v * C.N;
    float *pn = pnew + (int64_t)v * C.N;
    float acc[1] = {0.f};
    for (int64_t q = ((int64_t)blockIdx.x * kBlock + threadIdx.x) * VEC; q < C.N; q += (int64_t)gridDim.x * kBlock * VEC) {
        unsigned code[VEC];
        ld_code<VEC>(cs + q, code);
        auto val = [&](int64_t k) {
            Px<VEC> z = ld_px<VEC>(zv + k);
            if (!FIRST) {
                const Px<VEC> p = ld_px<VEC>(pv + k);
#pragma unroll
                for (int t = 0; t < VEC; ++t) z.v[t] = fmaf(beta, p.v[t], z.v[t]);
            }
            return z;
        };
        const Px<VEC> pc = val(q);
        const Px<VEC> Ap = apply_op<VEC>(C, q, code, pc, val,
                                         [&](int64_t k) { return FIRST ? zv[k] : fmaf(beta, pv[k], zv[k]); });
        st_px<VEC>(pn + q, pc);
#pragma unroll
        for (int t = 0; t < VEC; ++t) acc[0] = fmaf(pc.v[t], Ap.v[t], acc[0]);
    }
    double out[1];
    if (!reduce_vec<1>(acc, D.part, D.ctr, out) || threadIdx.x > 0) return;
    D.alpha[v] = out[0] > 0.0 ? D.rz[v] / out[0] : 0.0;
}

// u += alpha p, z -= alpha A p / diag; reductions <r, z>, <r, r> (r = z diag);
// beta and the stop test.
template <int VEC>
__global__ void __launch_bounds__(kBlock) k_cg_b(float *__restrict__ uall, const float *__restrict__ pall,
                                                 float *__restrict__ zall, const unsigned short *__restrict__ codes,
                                                 PlsConst C, PlsDev D)
{
    const int v = blockIdx.y;
    if (D.done[v]) return;
    const unsigned short *cs = codes + (int64_t)(v >> 1) * C.N;
    const float alpha = (float)D.alpha[v];
    const float *pv = pall + (int64_t)v * C.N;
    float *uv = uall + (int64_t)v * C.N, *zv = zall + (int64_t)v * C.N;
    float acc[2] = {0.f, 0.f};
    for (int64_t q = ((int64_t)blockIdx.x * kBlock + threadIdx.x) * VEC; q < C.N; q += (int64_t)gridDim.x * kBlock * VEC) {
        unsigned code[VEC];
        ld_code<VEC>(cs + q, code);
        const Px<VEC> pc = ld_px<VEC>(pv + q);
        Px<VEC> z = ld_px<VEC>(zv + q), u = ld_px<VEC>(uv + q);
        const Px<VEC> Ap = apply_op<VEC>(C, q, code, pc, [&](int64_t k) { return ld_px<VEC>(pv + k); },
                                         [&](int64_t k) { return pv[k]; });
#pragma unroll
        for (int t = 0; t < VEC; ++t) {
            const float diag = jacobi_diag(code[t], C.gamma, C.eps);
            u.v[t] = fmaf(alpha, pc.v[t], u.v[t]);
            const float rr = fmaf(-alpha, Ap.v[t], z.v[t] * diag), zz = rr / diag;
            z.v[t] = zz;
            acc[0] = fmaf(rr, zz, acc[0]);
            acc[1] = fmaf(rr, rr, acc[1]);
        }
        st_px<VEC>(uv + q, u);
        st_px<VEC>(zv + q, z);
    }
    double out[2];
    if (!reduce_vec<2>(acc, D.part, D.ctr, out) || threadIdx.x > 0) return;
    D.beta[v] = D.rz[v] != 0.0 ? out[0] / D.rz[v] : 0.0;
    D.rz[v] = out[0];
    D.relres[v] = D.bnorm[v] > 0.0 ? sqrt(out[1]) / D.bnorm[v] : 0.0;
    D.iters[v] += 1;
    if (C.tol > 0.0 && D.relres[v] < C.tol) {
        D.done[v] = 1;
        atomicAdd(D.ndone, 1);
    }
}

}  // namespace
}  // namespace dect

using namespace dect;

namespace dect {
namespace {

// Initial u (unless null) and the edge mask: k_prep and k_mask for images, the
// stored-magnitude kernels for volumes.  maxbits must be zero.
void prep_and_mask(const float *x, int n, int nz, int batch, const dect_pls_params *prm, float tau, float *u,
                   float *mh, float *ml, int *maxbits, unsigned char *mask, cudaStream_t s)
{
    Solve2 S{};
    if (prm) {
        S.a = prm->eta[0][0], S.b = prm->eta[1][0], S.c = prm->eta[0][1], S.e = prm->eta[1][1];
        S.det = S.a * S.e - S.b * S.c;
        auto split = [&](double v) {
            // outside 2^-60 .. 2^60 the two words would not hold 48 bits: NaN, so that FP64 decides
            const double q = v / S.det;
            const bool in = q == 0.0 || (std::fabs(q) > 0x1p-60 && std::fabs(q) < 0x1p60);
            Coef k;
            k.hi = in ? (float)q : NAN;
            k.lo = (float)(q - (double)k.hi);
            return k;
        };
        S.ed = split(S.e), S.bd = split(S.b), S.ad = split(S.a), S.cd = split(S.c);
    }
    const int64_t N = (int64_t)n * n * nz;
    if (nz > 1) {
        const int64_t want = (N + kBlock - 1) / kBlock;
        const int gx = (int)std::max<int64_t>(1, std::min<int64_t>(want, std::max(1, (kSMs * 8) / batch)));
        const dim3 gs((unsigned)gx, (unsigned)batch);
        k_prep3<<<gs, kBlock, 0, s>>>(x, n, nz, N, S.a, S.b, S.c, S.e, u, mh, ml, maxbits);
        k_mask3<<<gs, kBlock, 0, s>>>(mh, ml, N, maxbits, tau, mask);
    } else {
        const dim3 g((unsigned)((n + kPrepBlock - 1) / kPrepBlock), (unsigned)((n + kRows - 1) / kRows), (unsigned)batch);
        k_prep<<<g, kPrepBlock, 0, s>>>(x, n, S, u, maxbits);
        k_mask<<<g, kPrepBlock, 0, s>>>(x, n, maxbits, tau, mask);
    }
}

constexpr int kMaxBlocks = kSMs * 16;  // blocks of a CG launch, over all vectors

int cg_blocks(int64_t N, int batch)
{
    return (int)std::max<int64_t>(1, std::min<int64_t>((N + 4 * kBlock - 1) / (4 * kBlock), kMaxBlocks / (2 * batch)));
}

// Device scratch of a decomposition.
struct PlsWork {
    float *z, *pa, *pb;      // [2 batch][N]
    float *mh, *ml;          // [batch][N] magnitudes, volumes only
    unsigned short *codes;   // [batch][N]
    unsigned char *mask;     // [batch][N]
    PlsDev D;
    size_t zero_off, zero_bytes;  // what must start at zero: tickets, maxima, done count
    size_t report_bytes;          // relres, iters, ndone, from D.relres on
};

// Lays the scratch out from `base` (null: only the size).
size_t pls_layout(PlsWork &W, char *base, int64_t N, int nz, int batch)
{
    size_t o = 0;
    auto take = [&](size_t nb) { char *p = base ? base + o : nullptr; o = (o + nb + 255) & ~(size_t)255; return p; };
    const size_t nvec = 2 * (size_t)batch, nf = nvec * (size_t)N;
    W.z = (float *)take(nf * 4);
    W.pa = (float *)take(nf * 4);
    W.pb = (float *)take(nf * 4);
    W.mh = W.ml = nullptr;
    if (nz > 1) {
        W.mh = (float *)take((size_t)batch * N * 4);
        W.ml = (float *)take((size_t)batch * N * 4);
    }
    W.codes = (unsigned short *)take((size_t)batch * N * 2);
    W.mask = (unsigned char *)take((size_t)batch * N);
    W.D.part = (double *)take(nvec * cg_blocks(N, batch) * 3 * 8);
    W.D.alpha = (double *)take(nvec * 8);
    W.D.beta = (double *)take(nvec * 8);
    W.D.rz = (double *)take(nvec * 8);
    W.D.bnorm = (double *)take(nvec * 8);
    W.D.done = (int *)take(nvec * 4);
    W.zero_off = o;
    W.D.ctr = (unsigned *)take(nvec * 4);
    W.D.maxbits = (int *)take(nvec * 4);
    W.report_bytes = nvec * 12 + 4;
    W.D.relres = (double *)take(W.report_bytes);
    W.D.iters = (int *)(W.D.relres + nvec);
    W.D.ndone = W.D.iters + nvec;
    W.zero_bytes = o - W.zero_off;
    return o;
}

// The decomposition of `batch` images (nz = 1) or volumes (nz slices), all on
// stream s, with its scratch laid out at `base`; `host` holds report_bytes.
// With a tolerance the CG is enqueued in bursts; vectors that have stopped
// leave the launches at once (their blocks return), and one copy per burst
// brings the count of stopped vectors together with the reports.  Six
// iterations in the first burst: the workload's gamma needs five or six, and
// an iteration that finds every vector stopped costs two empty launches.
cudaError_t pls_core(const float *x, int n, int nz, int batch, const dect_pls_params *prm, float *u, char *base,
                     char *host, cudaStream_t s)
{
    const int64_t N = (int64_t)n * n * nz;
    PlsWork W;
    pls_layout(W, base, N, nz, batch);
    const PlsDev &D = W.D;
    cudaError_t e = cudaMemsetAsync(base + W.zero_off, 0, W.zero_bytes, s);
    if (e != cudaSuccess) return e;
    PlsConst C;
    C.n = n;
    C.nz = nz;
    C.N = N;
    C.gamma = (float)prm->gamma;
    C.eps = (float)prm->edge_eps;
    C.tol = prm->tol;
    prep_and_mask(x, n, nz, batch, prm, (float)prm->edge_tau, u, W.mh, W.ml, D.maxbits, W.mask, s);
    const dim3 g((unsigned)cg_blocks(N, batch), (unsigned)(2 * batch));
    // four pixels of a row per thread where rows split into fours (16-byte
    // aligned vectors); the caller's u is 4-byte aligned at least
    const bool vec4 = n % 4 == 0 && ((uintptr_t)u & 15u) == 0;
    if (vec4) k_init<4><<<g, kBlock, 0, s>>>(u, W.mask, W.codes, W.z, C, D);
    else k_init<1><<<g, kBlock, 0, s>>>(u, W.mask, W.codes, W.z, C, D);
    count_launches(3);
    const int K = prm->max_iter;
    const bool use_tol = prm->tol > 0.0;
    auto iteration = [&](int it) {
        const float *po = it & 1 ? W.pa : W.pb;
        float *pn = it & 1 ? W.pb : W.pa;
        if (vec4) {
            if (it == 0) k_cg_a<4, true><<<g, kBlock, 0, s>>>(W.z, po, pn, W.codes, C, D);
            else k_cg_a<4, false><<<g, kBlock, 0, s>>>(W.z, po, pn, W.codes, C, D);
            k_cg_b<4><<<g, kBlock, 0, s>>>(u, pn, W.z, W.codes, C, D);
        } else {
            if (it == 0) k_cg_a<1, true><<<g, kBlock, 0, s>>>(W.z, po, pn, W.codes, C, D);
            else k_cg_a<1, false><<<g, kBlock, 0, s>>>(W.z, po, pn, W.codes, C, D);
            k_cg_b<1><<<g, kBlock, 0, s>>>(u, pn, W.z, W.codes, C, D);
        }
        count_launches(2);
    };
    for (int it = 0; e == cudaSuccess;) {
        const int burst = use_tol ? (it == 0 ? 6 : 10) : K;
        for (int q = 0; q < burst && it < K; ++q, ++it) iteration(it);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(host, D.relres, W.report_bytes, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        int ndone = 0;
        std::memcpy(&ndone, host + (size_t)2 * batch * 12, sizeof(int));
        if (it >= K || (use_tol && ndone == 2 * batch)) break;
    }
    return e;
}

void pls_reports(const char *host, int batch, dect_pls_report *reports)
{
    if (!reports) return;
    for (int sl = 0; sl < batch; ++sl)
        for (int m = 0; m < 2; ++m) {
            std::memcpy(&reports[sl].relres[m], host + (size_t)(2 * sl + m) * 8, 8);
            std::memcpy(&reports[sl].iters[m], host + (size_t)2 * batch * 8 + (size_t)(2 * sl + m) * 4, 4);
        }
}

// Arguments common to the decomposition entry points.
bool pls_args_ok(const float *x, int n, int nz, int batch, const dect_pls_params *prm, const float *u)
{
    const size_t span = (size_t)batch * 2 * n * n * nz * sizeof(float);
    const char *xa = (const char *)x, *ua = (const char *)u;
    if (xa < ua + span && ua < xa + span) return false;
    if (!(prm->gamma >= 0) || !(prm->edge_eps >= 0) || prm->max_iter < 0 || !std::isfinite(prm->gamma)) return false;
    const double det = prm->eta[0][0] * prm->eta[1][1] - prm->eta[1][0] * prm->eta[0][1];
    return std::fabs(det) > 0 && std::isfinite(det);
}

dect_status pls_run(const float *x, int n, int nz, int batch, const dect_pls_params *prm, float *u,
                    dect_pls_report *reports, dect_stream stream)
{
    if (!prm || n < 1 || batch < 0 || n > 16384 || nz < 1 || nz > 4096) return DECT_ERR_INVALID_ARG;
    if (batch == 0) return DECT_OK;
    if (!x || !u) return DECT_ERR_INVALID_ARG;
    if (!pls_args_ok(x, n, nz, batch, prm, u)) return DECT_ERR_INVALID_ARG;
    if (batch > 65535 / 2) return DECT_ERR_INVALID_ARG;  // grid.y holds a vector index
    cudaStream_t s = (cudaStream_t)stream;
    PlsWork W;
    const size_t bytes = pls_layout(W, nullptr, (int64_t)n * n * nz, nz, batch);
    char *base = nullptr;
    DECT_CUDA(cudaMallocAsync((void **)&base, bytes, s));
    std::vector<char> host(W.report_bytes);
    const cudaError_t err = pls_core(x, n, nz, batch, prm, u, base, host.data(), s);
    cudaFreeAsync(base, s);
    if (err != cudaSuccess) {
        set_error("dect_pls_decompose", err);
        return err == cudaErrorMemoryAllocation ? DECT_ERR_OOM : DECT_ERR_CUDA;
    }
    pls_reports(host.data(), batch, reports);
    return DECT_OK;
}

}  // namespace
}  // namespace dect

extern "C" dect_status dect_pls_decompose(const float *x, int n, int batch, const dect_pls_params *prm,
                                          float *u, dect_pls_report *reports, dect_stream stream)
{
    return dect::pls_run(x, n, 1, batch, prm, u, reports, stream);
}

extern "C" dect_status dect_pls_decompose_cone(const float *x, int n, int nz, int batch, const dect_pls_params *prm,
                                               float *u, dect_pls_report *reports, dect_stream stream)
{
    return dect::pls_run(x, n, nz, batch, prm, u, reports, stream);
}

namespace dect {
namespace {

dect_status edge_mask_run(const float *x, int n, int nz, int batch, double edge_tau, uint8_t *mask,
                          dect_stream stream)
{
    if (n < 1 || batch < 0 || n > 16384 || nz < 1 || nz > 4096 || !std::isfinite(edge_tau))
        return DECT_ERR_INVALID_ARG;
    if (batch == 0) return DECT_OK;
    if (!x || !mask || batch > 65535) return DECT_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t mag_bytes = nz > 1 ? ((size_t)batch * n * n * nz * 4 + 255) & ~(size_t)255 : 0;  // volumes only
    char *base = nullptr;
    DECT_CUDA(cudaMallocAsync((void **)&base, 2 * mag_bytes + (size_t)2 * batch * 4, s));
    float *mh = (float *)base, *ml = (float *)(base + mag_bytes);
    int *maxbits = (int *)(base + 2 * mag_bytes);
    cudaError_t err = cudaMemsetAsync(maxbits, 0, (size_t)2 * batch * 4, s);
    if (err == cudaSuccess) {
        prep_and_mask(x, n, nz, batch, nullptr, (float)edge_tau, nullptr, mh, ml, maxbits, mask, s);
        count_launches(2);
        err = cudaGetLastError();
    }
    cudaFreeAsync(base, s);
    if (err != cudaSuccess) {
        set_error("dect_pls_edge_mask", err);
        return DECT_ERR_CUDA;
    }
    return DECT_OK;
}

}  // namespace
}  // namespace dect

extern "C" dect_status dect_pls_edge_mask(const float *x, int n, int batch, double edge_tau, uint8_t *mask,
                                          dect_stream stream)
{
    return dect::edge_mask_run(x, n, 1, batch, edge_tau, mask, stream);
}

extern "C" dect_status dect_pls_edge_mask_cone(const float *x, int n, int nz, int batch, double edge_tau,
                                               uint8_t *mask, dect_stream stream)
{
    return dect::edge_mask_run(x, n, nz, batch, edge_tau, mask, stream);
}

// ---------------------------------------------------------------------------
// Allocation-free variant of dect_pls_decompose.
//
// Some callers cannot allocate device memory while they run: for example an
// inline reconstruction service that reserves the whole device pool at
// start-up and must keep its footprint fixed, or a plug-in hosted by a
// process whose own allocator owns the GPU.  This entry point takes its
// scratch from one fixed array in the library image instead of the
// stream-ordered allocator, creates no stream, event or graph, and pins no
// host memory.
// ---------------------------------------------------------------------------
namespace dect {
namespace {

// Upper bounds of the allocation-free path (see dect.h).
constexpr int64_t kNoAllocMaxPixels = DECT_PLS_NOALLOC_MAX_PIXELS;
constexpr int kNoAllocMaxBatch = DECT_PLS_NOALLOC_MAX_BATCH;
constexpr size_t kNoAllocBytes = (size_t)14 << 20;

// The scratch itself: every device that loads the library holds it until
// the process exits.  In host code this name is only a stand-in; the device
// address comes from cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_pls_scratch[kNoAllocBytes];

std::mutex g_scratch_mu;
void *g_scratch_addr[256];  // per device ordinal, filled on the first call

cudaError_t scratch_address(int dev, void **out)
{
    std::lock_guard<std::mutex> lk(g_scratch_mu);
    if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
    if (!g_scratch_addr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_pls_scratch);
        if (e != cudaSuccess) return e;
        g_scratch_addr[dev] = p;
    }
    *out = g_scratch_addr[dev];
    return cudaSuccess;
}

}  // namespace
}  // namespace dect

extern "C" dect_status dect_pls_decompose_noalloc(const float *x, int n, int batch,
                                                  const dect_pls_params *prm, float *u,
                                                  dect_pls_report *reports, dect_stream stream)
{
    if (!prm || n < 1 || batch < 0 || n > 16384) return DECT_ERR_INVALID_ARG;
    if (batch == 0) return DECT_OK;
    if (!x || !u) return DECT_ERR_INVALID_ARG;
    if ((int64_t)batch * n * n > kNoAllocMaxPixels || batch > kNoAllocMaxBatch) {
        set_error_text("dect_pls_decompose_noalloc: batch * n * n must be <= " +
                       std::to_string(kNoAllocMaxPixels) + " and batch <= " +
                       std::to_string(kNoAllocMaxBatch) + " (use dect_pls_decompose for larger work)");
        return DECT_ERR_INVALID_ARG;
    }
    if (!pls_args_ok(x, n, 1, batch, prm, u)) return DECT_ERR_INVALID_ARG;
    int dev = 0;
    DECT_CUDA(cudaGetDevice(&dev));
    void *scratch = nullptr;
    DECT_CUDA(scratch_address(dev, &scratch));
    PlsWork W;
    if (pls_layout(W, nullptr, (int64_t)n * n, 1, batch) > kNoAllocBytes) {  // cannot happen within the limits above
        set_error_text("dect_pls_decompose_noalloc: scratch layout exceeds the fixed array");
        return DECT_ERR_INVALID_ARG;
    }
    // the array keeps the previous call's contents: pls_core zeroes what must start at zero
    char host[2 * kNoAllocMaxBatch * 12 + 4];
    DECT_CUDA(pls_core(x, n, 1, batch, prm, u, (char *)scratch, host, (cudaStream_t)stream));
    pls_reports(host, batch, reports);
    return DECT_OK;
}
