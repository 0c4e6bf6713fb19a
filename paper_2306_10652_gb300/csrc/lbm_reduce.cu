// lbm_reduce.cu -- deterministic per-component reductions over the lattice.
//
// Mass: M_i = sum_r rho_i(r).  Convergence: max_{i,r} |rho_i(r) - snap_i(r)|.
// Two launches: a grid of (chunks, components) CTAs, each reducing a fixed
// contiguous chunk of nodes of one component (per-thread strided sums, then a
// warp-shuffle tree and a shared-memory tree in a fixed order) into
// partials[chunk][i]; then one warp per component sums its partials, strided
// over the lanes and by a shuffle tree.  The result is bitwise reproducible for
// a given lattice size.  A non-finite density sets *nonfinite.
// Both launches are bound by memory latency: the second summed all partials of a
// component in one thread before, 85-115 us at any lattice size (128 x 4, Nc = 2:
// 95 us for both, now 11), and the first had one CTA walk a chunk of every
// component in turn (2048^2, Nc = 10, 335 MB: 312 us for both, now 136).
#include "lbm_internal.h"

namespace lbmfug {
namespace {

template <bool MAXDIFF> __device__ __forceinline__ double join(double a, double b)
{
    return MAXDIFF ? (b > a ? b : a) : a + b;
}

template <bool MAXDIFF>
__global__ void __launch_bounds__(kReduceThreads)
    k_partials(int nc, long long N, const double *__restrict__ rho, const double *__restrict__ snap,
               double *__restrict__ partials, int *__restrict__ nonfinite)
{
    __shared__ double sh[kReduceThreads / 32];
    const int i = blockIdx.y;
    const long long chunk = (N + gridDim.x - 1) / gridDim.x;
    const long long lo = blockIdx.x * chunk;
    const long long hi = lo + chunk < N ? lo + chunk : N;
    rho += (long long)i * N;
    if (MAXDIFF) snap += (long long)i * N;
    double acc = 0.0;
    bool bad = false;
#pragma unroll 4
    for (long long r = lo + threadIdx.x; r < hi; r += kReduceThreads) {
        const double v = __ldg(rho + r);
        bad |= (__double2hiint(v) & 0x7ff00000) == 0x7ff00000;  // infinite or NaN
        acc = join<MAXDIFF>(acc, MAXDIFF ? fabs(v - __ldg(snap + r)) : v);
    }
    if (bad) atomicExch(nonfinite, 1);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc = join<MAXDIFF>(acc, __shfl_down_sync(0xffffffffu, acc, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = sh[0];
        for (int w = 1; w < kReduceThreads / 32; ++w) s = join<MAXDIFF>(s, sh[w]);
        partials[(long long)blockIdx.x * nc + i] = s;
    }
}

// one warp per component
template <bool MAXDIFF>
__global__ void k_final(int nc, int nblocks, const double *__restrict__ partials, double *__restrict__ out)
{
    const int i = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s = 0.0;
#pragma unroll 8
    for (int b = lane; b < nblocks; b += 32) s = join<MAXDIFF>(s, __ldg(partials + (long long)b * nc + i));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s = join<MAXDIFF>(s, __shfl_down_sync(0xffffffffu, s, o));
    if (lane == 0) out[i] = s;
}

// chunks of at least four values per thread, at most kReduceBlocks
int chunks_for(long long N)
{
    const long long b = (N + 4 * kReduceThreads - 1) / (4 * kReduceThreads);
    return (int)(b < kReduceBlocks ? b : kReduceBlocks);
}

template <bool MAXDIFF>
int launch(int nc, long long N, const double *rho, const double *snap, double *partials, double *out,
           int *nonfinite, cudaStream_t s)
{
    const int b = chunks_for(N);
    k_partials<MAXDIFF><<<dim3(b, nc), kReduceThreads, 0, s>>>(nc, N, rho, snap, partials, nonfinite);
    k_final<MAXDIFF><<<1, 32 * nc, 0, s>>>(nc, b, partials, out);
    return (int)cudaGetLastError();
}

}  // namespace

int launch_mass(int nc, long long N, const double *rho, double *partials, double *out,
                int *nonfinite, cudaStream_t s)
{
    return launch<false>(nc, N, rho, nullptr, partials, out, nonfinite, s);
}

int launch_maxdiff(int nc, long long N, const double *rho, const double *snap, double *partials,
                   double *out, int *nonfinite, cudaStream_t s)
{
    return launch<true>(nc, N, rho, snap, partials, out, nonfinite, s);
}

}  // namespace lbmfug
