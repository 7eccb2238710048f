// A x and A^T y on caller-owned planar batches (Eq. (1); the A^T of G_f in
// Eq. (9)).  A batch is split into passes of up to 64 images; each pass packs its
// images pixel-major ([index][NB], zero-padded to the width NB), streams the
// table once with every entry gathering one contiguous vector of all NB images,
// and unpacks the result to the planar output.  A of narrow passes streams the
// line table instead (lines.cuh), whose kernel writes the planar result itself.
#include <cuda_runtime.h>

#include <algorithm>

#include "dect_internal.cuh"
#include "kernels.cuh"
#include "lines.cuh"

namespace dect {
namespace {

constexpr int kOpBlock = 1024;  // one block per SM
// Lanes per row (ray or pixel).  Narrow passes are bound by the cache lines that
// a warp's gathers touch: with 8 lanes a warp takes four adjacent rows, whose
// entries meet the same lines (A^T of two images at 512^2 / 60 views: 117 -> 65
// us against a warp per row; 4 lanes 64 us, but 20 % slower on small images;
// cone-beam 256^2 x 64, 60 views of 64 x 368, one volume: A 1275 -> 971 us, A^T
// 1821 -> 974; 16 volumes 3485 -> 3382 and 3864 -> 2759).  A fan-beam ray's pixels lie
// apart from its neighbours', and a warp per ray stays ahead (16 images, 512^2 / 60:
// 214 us against 262).
template <int NB>
constexpr int kLanes = NB <= 16 ? 8 : 32;

// Whether a row takes a whole warp.  Eight lanes take its entries four times as
// long one after the other, so on few rows a warp each is ahead: A^T up to two turns
// of the grid, three where a row has 256 entries or more (8 images of 96^2, 60 views:
// 20 us against 23; 112^2, 60 views: 22 and 23; 112^2, 180 views: 33 and 35; 128^2, 60
// views: 25 and 23); cone-beam A up to five (8 images of 128^2 x 4, 22080 rays: 34
// and 38; 64^2 x 16, 44160 rays: 37 and 34).
bool warp_rows(bool tiled, int nz, int64_t rows, int64_t nnz)
{
    if (!tiled && nz == 0) return true;  // fan-beam A
    const int turns = !tiled ? 5 : nnz < 256 * rows ? 2 : 3;
    return rows <= (int64_t)turns * kSMs * (kOpBlock / 32);
}
constexpr int kTileW = 8;  // A^T: tiles of 8 columns, so a tile's sinogram lines stay in one L1

// Packing and unpacking, bound by memory.  Up to 4 images a thread takes a row of
// all images (coalesced on both sides); above, a block turns a tile of kTileRows
// rows in shared memory.  (An element a thread read, or wrote, 4 bytes of each image's
// line: of operators over 64 images of 512^2 / 60 views 206 us went there, now
// 75; of a 256^2 x 64 volume and its 60 projections 67 us, now 41.)
constexpr int kPackBlock = 256;
template <int NB>
constexpr int kTileRows = NB <= 4 ? kPackBlock : NB >= 32 ? 64 : 2048 / NB;

// planar src [nimg][rows] -> interleaved dst [rows][NB] (images >= nimg are 0)
template <int NB>
__global__ void __launch_bounds__(kPackBlock) k_to_il(const float *__restrict__ src, float *__restrict__ dst,
                                                      int64_t rows, int nimg)
{
    constexpr int VW = Batch<NB>::VW, TR = kTileRows<NB>;
    const int64_t r0 = (int64_t)blockIdx.x * TR;
    if constexpr (NB <= 4) {
        const int64_t row = r0 + threadIdx.x;
        if (row >= rows) return;
        Vec<VW> v;
#pragma unroll
        for (int c = 0; c < NB; ++c) v.v[c] = c < nimg ? src[(int64_t)c * rows + row] : 0.f;
        st_v<VW>(dst + row * NB, v);
    } else {
        __shared__ float tile[TR][NB + 1];
        const int nr = (int)(rows - r0 < TR ? rows - r0 : TR);
#pragma unroll 8
        for (int e = threadIdx.x; e < TR * NB; e += kPackBlock) {
            const int r = e % TR, c = e / TR;
            tile[r][c] = c < nimg && r < nr ? src[(int64_t)c * rows + r0 + r] : 0.f;
        }
        __syncthreads();
        for (int e = threadIdx.x; e < nr * (NB / 4); e += kPackBlock) {
            const int r = e / (NB / 4), c = e % (NB / 4) * 4;
            st_v<4>(dst + (r0 + r) * NB + c, {tile[r][c], tile[r][c + 1], tile[r][c + 2], tile[r][c + 3]});
        }
    }
}

// The table and the interleaved images that k_rows_il has summed.
struct RowTable {
    const int64_t *ptr;
    const Entry *ent;
    const float *src;
    int64_t src_rows;
    unsigned site;
};

// v, image c of a row of sums; where it is not finite, the row's sum without the
// padded entries of row_dot, whose product 0 times a value at index 0 that is not
// finite is not 0.  (Tested in k_rows_il itself the comparison cost ptxas the order of
// its gathers: A of 16 volumes of 256^2 x 64 3.16 -> 4.00 ms, A^T of 64 images at
// 1024^2 / 360 views 10.3 -> 11.9.)
template <int NB>
__device__ __forceinline__ float unpadded(float v, const RowTable &T, int64_t row, int c)
{
    if (isfinite(v)) return v;
    float s = 0.f;
#pragma unroll 1
    for (int64_t k = T.ptr[row], e = T.ptr[row + 1]; k < e; ++k) {
        const Entry en = ld_entry(T.ent + k);
        int at = en.x;
        if (!DECT_IDX_OK(at, T.src_rows, T.site)) at = 0;
        s = fmaf(__int_as_float(en.y), T.src[(int64_t)at * NB + c], s);
    }
    return s;
}

// interleaved src [rows][NB] -> planar dst [nimg][rows]
template <int NB>
__global__ void __launch_bounds__(kPackBlock, 8) k_from_il(const float *__restrict__ src, float *__restrict__ dst,
                                                           int64_t rows, int nimg, RowTable T)
{
    constexpr int VW = Batch<NB>::VW, TR = kTileRows<NB>;
    const int64_t r0 = (int64_t)blockIdx.x * TR;
    if constexpr (NB <= 4) {
        const int64_t row = r0 + threadIdx.x;
        if (row >= rows) return;
        const Vec<VW> v = ld_il<VW>(src + row * NB);
#pragma unroll
        for (int c = 0; c < NB; ++c)
            if (c < nimg) dst[(int64_t)c * rows + row] = unpadded<NB>(v.v[c], T, row, c);
    } else {
        __shared__ float tile[TR][NB + 1];
        const int nr = (int)(rows - r0 < TR ? rows - r0 : TR);
        float zero = 0.f;  // stays 0 while every sum is finite
#pragma unroll 4
        for (int e = threadIdx.x; e < nr * (NB / 4); e += kPackBlock) {
            const int r = e / (NB / 4), c = e % (NB / 4) * 4;
            const Vec<4> v = ld_il<4>(src + (r0 + r) * NB + c);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                tile[r][c + k] = v.v[k];
                zero = fmaf(v.v[k], 0.f, zero);
            }
        }
        const bool fine = __syncthreads_and(zero == 0.f);
        for (int e = threadIdx.x; e < TR * nimg; e += kPackBlock) {
            const int r = e % TR, c = e / TR;
            if (r < nr) dst[(int64_t)c * rows + r0 + r] = fine ? tile[r][c] : unpadded<NB>(tile[r][c], T, r0 + r, c);
        }
    }
}

// dst[row][NB] = sum over the row's entries of len * src[index][NB], G
// lanes per row.  TILED (pixel-major table of an n x n image): the block's
// consecutive rows walk pixel tiles of 8 columns, so that pixels sharing rays
// share an L1; otherwise rows are taken in order (adjacent rays of a view share
// pixels).  Lanes gather 8 images of an entry above 16 images (row_dot_w), 4
// below (row_dot_g, its partial sums with their rounding errors).  Rows are padded with entries of weight 0 at
// index 0: where the value there is not finite, k_from_il forms the sum again.
template <int NB, int G, bool TILED>
__global__ void __launch_bounds__(kOpBlock) k_rows_il(const int64_t *__restrict__ ptr, const Entry *__restrict__ ent,
                                                      int64_t rows, int n, int nz, const float *__restrict__ src,
                                                      int64_t src_rows, float *__restrict__ dst)
{
    constexpr int VW = Batch<NB>::VW, LPE = Batch<NB>::CPB;
    constexpr int TW = kTileW, TH = kOpBlock / G > 64 ? kOpBlock / G / TW : 8;
    const int lr = threadIdx.x % G, grp = lr / LPE, vl = lr % LPE;
    const int64_t rpb = kOpBlock / G;
    const int tiles_x = (n + TW - 1) / TW, tiles_y = (n + TH - 1) / TH;
    const int64_t per_slice = (int64_t)tiles_x * tiles_y * TW * TH;
    const int64_t vrows = TILED ? per_slice * nz : rows;
    const unsigned long long pol = l2_evict_last_policy();
    for (int64_t v0 = (int64_t)blockIdx.x * rpb; v0 < vrows; v0 += (int64_t)gridDim.x * rpb) {
        const int64_t v = v0 + threadIdx.x / G;
        int64_t row = v;
        bool ok = v < vrows;
        if (TILED && ok) {  // slice k, tile of the slice, pixel of the tile
            const int64_t k = v / per_slice, vs = v % per_slice;
            const int64_t tile = vs / (TW * TH);
            const int w = (int)(vs % (TW * TH));
            const int i = (int)(tile / tiles_x) * TH + w / TW, j = (int)(tile % tiles_x) * TW + w % TW;
            ok = i < n && j < n;
            row = (k * n + i) * n + j;
        }
        int64_t b = 0, e = 0;
        if (ok) {
            b = ptr[row];
            e = ptr[row + 1];
        }
        Vec<VW> acc;
        if constexpr (NB > 16)
            acc = row_dot_w<NB, G, 8, 2>(ent, b, e, lr, src, pol, src_rows, TILED ? CHK_GATHER_AT : CHK_GATHER_A);
        else
            acc = row_dot<NB, G, true, false, true>(ent, b, e, src, src_rows, lr, TILED ? CHK_GATHER_AT : CHK_GATHER_A);
        if (ok && grp == 0) st_v<VW>(dst + row * NB + vl * VW, acc);
    }
}

template <int NB>
cudaError_t pass(const int64_t *ptr, const Entry *ent, int64_t rows_in, int64_t rows_out, int n, int nz, bool tiled,
                 int64_t nnz, const float *src, float *dst, int nimg, float *buf, cudaStream_t s)
{
    float *in_il = buf, *out_il = buf + rows_in * NB;
    constexpr int TR = kTileRows<NB>;
    const unsigned bi = (unsigned)((rows_in + TR - 1) / TR), bo = (unsigned)((rows_out + TR - 1) / TR);
    k_to_il<NB><<<bi, kPackBlock, 0, s>>>(src, in_il, rows_in, nimg);
    auto rows = [&](auto kernel) {
        kernel<<<kSMs, kOpBlock, 0, s>>>(ptr, ent, rows_out, n, std::max(nz, 1), in_il, rows_in, out_il);
    };
    if (warp_rows(tiled, nz, rows_out, nnz))
        tiled ? rows(k_rows_il<NB, 32, true>) : rows(k_rows_il<NB, 32, false>);
    else
        tiled ? rows(k_rows_il<NB, kLanes<NB>, true>) : rows(k_rows_il<NB, kLanes<NB>, false>);
    const RowTable T{ptr, ent, in_il, rows_in, tiled ? CHK_GATHER_AT : CHK_GATHER_A};
    k_from_il<NB><<<bo, kPackBlock, 0, s>>>(out_il, dst, rows_out, nimg, T);
    count_launches(3);
    return cudaGetLastError();
}

// Passes of up to 64 images over the table (ptr, ent) mapping src rows
// (rows_in per image) to dst rows (rows_out per image).
cudaError_t run_batched(const int64_t *ptr, const Entry *ent, int64_t rows_in, int64_t rows_out, int n, int nz,
                        bool tiled, int64_t nnz, const float *src, float *dst, int batch, cudaStream_t s)
{
    int width0 = 2;  // widest pass: the next power of two >= min(batch, 64), at least 2
    while (width0 < std::min(batch, kMaxBatchImages)) width0 *= 2;
    float *buf = nullptr;
    cudaError_t e = cudaMallocAsync((void **)&buf, sizeof(float) * (size_t)(rows_in + rows_out) * width0, s);
    if (e != cudaSuccess) return e;
    for (int done = 0; done < batch && e == cudaSuccess;) {
        const int k = std::min(kMaxBatchImages, batch - done);
        const float *sp = src + (int64_t)done * rows_in;
        float *dp = dst + (int64_t)done * rows_out;
        if (k <= 2) e = pass<2>(ptr, ent, rows_in, rows_out, n, nz, tiled, nnz, sp, dp, k, buf, s);
        else if (k <= 4) e = pass<4>(ptr, ent, rows_in, rows_out, n, nz, tiled, nnz, sp, dp, k, buf, s);
        else if (k <= 8) e = pass<8>(ptr, ent, rows_in, rows_out, n, nz, tiled, nnz, sp, dp, k, buf, s);
        else if (k <= 16) e = pass<16>(ptr, ent, rows_in, rows_out, n, nz, tiled, nnz, sp, dp, k, buf, s);
        else if (k <= 32) e = pass<32>(ptr, ent, rows_in, rows_out, n, nz, tiled, nnz, sp, dp, k, buf, s);
        else e = pass<64>(ptr, ent, rows_in, rows_out, n, nz, tiled, nnz, sp, dp, k, buf, s);
        done += k;
    }
    cudaError_t f = cudaFreeAsync(buf, s);
    return e != cudaSuccess ? e : f;
}

// ---------------------------------------------------------------------------
// A on the line table
// ---------------------------------------------------------------------------
// planar src [nimg][n][n] -> interleaved dst and its transpose dstT (images >= nimg are 0)
template <int NB>
__global__ void __launch_bounds__(256) k_line_pack(const float *__restrict__ src, float *__restrict__ dst,
                                                   float *__restrict__ dstT, int n, int nimg)
{
    constexpr int VW = Batch<NB>::VW;
    __shared__ float tile[VW][32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, j0 = blockIdx.x * 32, i0 = blockIdx.y * 32;
    const int64_t N = (int64_t)n * n;
    for (int k = 0; k < NB; k += VW) {
        for (int r = ty; r < 32; r += 8)
            if (i0 + r < n && j0 + tx < n) {
                const int64_t p = (int64_t)(i0 + r) * n + j0 + tx;
                Vec<VW> v;
#pragma unroll
                for (int c = 0; c < VW; ++c) {
                    v.v[c] = k + c < nimg ? src[(int64_t)(k + c) * N + p] : 0.f;
                    tile[c][r][tx] = v.v[c];
                }
                st_v<VW>(dst + p * NB + k, v);
            }
        __syncthreads();
        for (int r = ty; r < 32; r += 8)
            if (j0 + r < n && i0 + tx < n) {
                Vec<VW> v;
#pragma unroll
                for (int c = 0; c < VW; ++c) v.v[c] = tile[c][tx][r];
                st_v<VW>(dstT + ((int64_t)(j0 + r) * n + i0 + tx) * NB + k, v);
            }
        __syncthreads();
    }
}

// y[img][ray] = (A x)(ray): a block per group of 32 rays
template <int NB>
__global__ void __launch_bounds__(LineShape<NB>::BLOCK, LineShape<NB>::BLOCKS)
    k_line_project(LineTable T, const float *__restrict__ x, const float *__restrict__ xT, float *__restrict__ y, int nimg)
{
    __shared__ LineSums<NB> sm;
    const int64_t M = (int64_t)T.nv * T.nb;
    const int v = blockIdx.x / T.ngb, gb = blockIdx.x % T.ngb;
    float acc[LineShape<NB>::VW];
    line_ray_sums<NB>(T, v, gb, x, xT, acc);
    line_ray_store<NB>(sm, acc);
    __syncthreads();
    for (int e = threadIdx.x; e < 32 * NB; e += LineShape<NB>::BLOCK) {
        const int r = e & 31, k = e >> 5;
        if (gb * 32 + r >= T.nb || k >= nimg) continue;
        const int64_t ray = (int64_t)v * T.nb + gb * 32 + r;
        y[(int64_t)k * M + ray] = line_ray_value<NB>(sm, r * NB + k, __ldg(T.len + ray));
    }
}

template <int NB>
void line_pass(const LineTable &T, const float *x, float *y, int nimg, float *buf, cudaStream_t s)
{
    const int64_t N = (int64_t)T.n * T.n;
    k_line_pack<NB><<<transpose_grid(T.n), 256, 0, s>>>(x, buf, buf + N * NB, T.n, nimg);
    k_line_project<NB><<<line_groups(T), LineShape<NB>::BLOCK, 0, s>>>(T, buf, buf + N * NB, y, nimg);
    count_launches(2);
}

// A of up to kLineMaxImages images
cudaError_t run_lines(const LineTable &T, const float *x, float *y, int batch, cudaStream_t s)
{
    int width = 2;
    while (width < batch) width *= 2;
    float *buf = nullptr;
    cudaError_t e = cudaMallocAsync((void **)&buf, sizeof(float) * 2 * (size_t)T.n * T.n * width, s);
    if (e != cudaSuccess) return e;
    switch (width) {
    case 2: line_pass<2>(T, x, y, batch, buf, s); break;
    case 4: line_pass<4>(T, x, y, batch, buf, s); break;
    case 8: line_pass<8>(T, x, y, batch, buf, s); break;
    default: line_pass<16>(T, x, y, batch, buf, s); break;
    }
    e = cudaGetLastError();
    const cudaError_t f = cudaFreeAsync(buf, s);
    return e != cudaSuccess ? e : f;
}

// Images of a batch that A takes through the line table: the last pass, where it is
// narrow enough.  Above four images a small matrix does not fill the chip with the
// table's blocks, and a warp per ray is ahead up to about 3.5 million elements: 16 images
// of 64^2 / 60 views 21 us against 25, 160^2 / 60 (2.8 million) 36 against 44, 256^2 / 30
// (3.6) 46 both, 192^2 / 60 (4.0) 48 against 46, 384^2 / 30 (8.0) 83 against 64; 8 images of
// 160^2 / 60 26 against 29, 256^2 / 30 30 both, 192^2 / 60 32 against 31.
constexpr int64_t kLineElements = 3500000;
int line_tail(const dect_plan *p, int batch)
{
    const int rest = batch % kMaxBatchImages;
    return p->lines.ok && rest <= kLineMaxImages && (rest <= 4 || p->nnz >= kLineElements) ? rest : 0;
}

}  // namespace

cudaError_t launch_project_planar(const dect_plan *p, const float *x, float *y, int batch, cudaStream_t s)
{
    const int tail = line_tail(p, batch), head = batch - tail;
    cudaError_t e = cudaSuccess;
    if (head > 0) e = run_batched(p->rowptr, p->ent, p->N, p->M, p->n, p->nz, false, p->nnz, x, y, head, s);
    if (e == cudaSuccess && tail > 0) e = run_lines(p->lines, x + head * p->N, y + head * p->M, tail, s);
    return e;
}

cudaError_t launch_backproject_planar(const dect_plan *p, const float *y, float *x, int batch, cudaStream_t s)
{
    return run_batched(p->colptr, p->tent, p->M, p->N, p->n, p->nz, true, p->nnz, y, x, batch, s);
}

}  // namespace dect

using namespace dect;

extern "C" dect_status dect_project(const dect_plan *plan, const float *x, float *y, int batch,
                                    dect_stream stream)
{
    if (!plan || batch < 0) return DECT_ERR_INVALID_ARG;
    if (batch == 0) return DECT_OK;
    if (!x || !y) return DECT_ERR_INVALID_ARG;
    DECT_CUDA(cudaSetDevice(plan->device));
    DECT_CUDA(launch_project_planar(plan, x, y, batch, (cudaStream_t)stream));
    return DECT_OK;
}

extern "C" dect_status dect_backproject(const dect_plan *plan, const float *y, float *x, int batch,
                                        dect_stream stream)
{
    if (!plan || batch < 0) return DECT_ERR_INVALID_ARG;
    if (batch == 0) return DECT_OK;
    if (!x || !y) return DECT_ERR_INVALID_ARG;
    DECT_CUDA(cudaSetDevice(plan->device));
    DECT_CUDA(launch_backproject_planar(plan, y, x, batch, (cudaStream_t)stream));
    return DECT_OK;
}
