// Build of the line table (lines.cuh) from the columns that the Siddon walk
// wrote: the walk words of A.  A ray whose columns do not advance by at most one
// per line, always in one direction, is reported, and the plan then keeps to
// the CSR kernels.
#include <cuda_runtime.h>

#include "dect_internal.cuh"
#include "lines.cuh"

namespace dect {
namespace {

constexpr short kColOut = -32768;  // as in plan.cu
constexpr int kMaxN = 4096;

// One thread per (view, block of 32 lines, bin).  A line outside the image
// counts as column -1 (q = 1: -0) or n - 1 (q = 0), neither of which adds anything.
__global__ void __launch_bounds__(256) k_line_walk(LineTable T, const short *__restrict__ col, int *__restrict__ bad)
{
    const int b = blockIdx.x * 256 + threadIdx.x, blk = blockIdx.y, v = blockIdx.z;
    if (b >= T.nb) return;
    const int64_t at = T.at(v, blk * 32, b);
    const int ns = min(32, T.n - blk * 32);
    auto column = [&](int k) {
        const short c = col[at + k * 32];
        return c != kColOut ? (int)c : __float_as_int(T.q[at + k * 32]) < 0 ? -1 : T.n - 1;
    };
    int prev = column(0), sign = 0;
    const unsigned first = (unsigned)(prev + 1);
    unsigned bits = 0u;
    bool edge = prev < 0 || prev + 1 >= T.n || ns < 32, wrong = false, out = col[at] == kColOut;
    for (int k = 1; k < ns; ++k) {
        const int c = column(k), d = c - prev;
        edge = edge || c < 0 || c + 1 >= T.n;
        out = out && col[at + k * 32] == kColOut;
        if (d != 0) {
            wrong = wrong || (sign != 0 && d != sign) || d < -1 || d > 1;
            sign = d;
            bits |= 1u << (k - 1);
        }
        prev = c;
    }
    const bool c1 = T.cls[(int64_t)v * T.nb + b] != 0;
    T.walk[((int64_t)v * T.nblk + blk) * T.nbp + b] =
        make_uint2(first | (sign < 0 ? kWalkFalls : 0u) | (edge ? kWalkEdge : 0u) | (c1 ? kWalkCls1 : 0u) |
                       (out ? kWalkOut : 0u), bits);
    if (wrong) atomicOr(bad, 2);
}

}  // namespace

void lines_free(LineTable &T)
{
    cudaFree(T.q);
    cudaFree(T.walk);
    cudaFree(T.len);
    cudaFree(T.cls);
    T = LineTable{};
}

cudaError_t lines_alloc(LineTable &T, int n, int nv, int nb)
{
    T = LineTable{};
    if (n < 4 || n > kMaxN || nv > 65535) return cudaSuccess;
    T.n = n;
    T.nv = nv;
    T.nb = nb;
    T.nbp = (nb + 31) & ~31;
    T.ngb = T.nbp / 32;
    T.nblk = (n + 31) / 32;
    const size_t nq = (size_t)nv * T.nblk * T.ngb * 1024;
    cudaError_t e = cudaMalloc((void **)&T.q, sizeof(float) * nq);
    if (e == cudaSuccess) e = cudaMalloc((void **)&T.walk, sizeof(uint2) * (size_t)nv * T.nblk * T.nbp);
    if (e == cudaSuccess) e = cudaMalloc((void **)&T.len, sizeof(float2) * (size_t)nv * nb);
    if (e == cudaSuccess) e = cudaMalloc((void **)&T.cls, (size_t)nv * nb);
    if (e == cudaErrorMemoryAllocation) {  // the plan works without the table
        cudaGetLastError();
        lines_free(T);
        return cudaSuccess;
    }
    if (e != cudaSuccess) return e;
    T.ok = 1;
    return cudaSuccess;
}

cudaError_t lines_finish(LineTable &T, const short *d_col, int *d_bad, cudaStream_t s)
{
    k_line_walk<<<dim3((unsigned)((T.nb + 255) / 256), (unsigned)T.nblk, (unsigned)T.nv), 256, 0, s>>>(T, d_col, d_bad);
    return cudaGetLastError();
}

}  // namespace dect
