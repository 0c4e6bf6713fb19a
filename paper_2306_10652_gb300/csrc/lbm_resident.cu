// lbm_resident.cu -- dispatch of the resident schedule (many steps of a small
// D2Q9 problem in one cluster launch).
#include "lbm_resident.cuh"

namespace lbmfug {
namespace rs {
namespace {

using Kernel = void (*)(Par, StateBufs, Work);

template <typename E, bool TAU1, int MAXT> Kernel pick(int g)
{
    switch (g) {
    case 1: return k_resident<1, E, TAU1, MAXT>;
    case 2: return k_resident<2, E, TAU1, MAXT>;
    case 4: return k_resident<4, E, TAU1, MAXT>;
    case 8: return k_resident<8, E, TAU1, MAXT>;
    default: return k_resident<16, E, TAU1, MAXT>;
    }
}

template <typename E> Kernel pick32(int g, bool tau1, int threads)
{
    if (threads <= 512) return tau1 ? pick<E, true, 512>(g) : pick<E, false, 512>(g);
    return tau1 ? pick<E, true, 1024>(g) : pick<E, false, 1024>(g);
}

Kernel kernel_of(int prec, int g, bool tau1, int threads)
{
    if (prec == 0) return tau1 ? pick<double, true, 512>(g) : pick<double, false, 512>(g);
    return prec == 1 ? pick32<df::F2>(g, tau1, threads) : pick32<float>(g, tau1, threads);
}

int group(int nc)
{
    int g = 1;
    while (g < nc) g *= 2;
    return g;
}

// CTAs and threads of a problem: all 16 CTAs of the largest cluster, so that its
// warps spread over as many SMs as a barrier can span.
void shape(int nc, long long N, int ctas, int *threads)
{
    const long long items = N * group(nc);
    *threads = (int)(((items + ctas - 1) / ctas + 31) / 32 * 32);
}

cudaLaunchConfig_t config(int ctas, int threads, cudaStream_t s, cudaLaunchAttribute *attr)
{
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(ctas);
    c.blockDim = dim3(threads);
    c.stream = s;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = ctas;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    c.attrs = attr;
    c.numAttrs = 1;
    return c;
}

}  // namespace
}  // namespace rs

size_t resident_scratch_bytes(int prec, int nc, long long N)
{
    const size_t items = (size_t)N * rs::group(nc);
    const size_t s = prec == 0 ? 8 : 4;
    // rho, populations; mu; psi (8 bytes each at most), 16-byte aligned parts
    return items * s * 9 + items * 8 + (size_t)N * 8 + 64;
}

// CTAs of the cluster, 0 if the problem is not one for this schedule.  A thread
// holds one component of one node, so a problem has to fit 16 CTAs of 1024 threads
// (binary64: 512, for its registers).  Whatever fits is faster here in binary32
// (Nc = 2-10, 32 x 4 to 64 x 64: 2.4-13.5 us per step against 6.3-18.7 us fused).
// Binary64 has the binary64 pipes of 16 SMs only, 15.6-17.6 us at 4096 threads,
// against the three passes' latency of about 5 + 5.5 Nc us: 4096 threads, and all
// from six components on.
int resident_ctas(int lat, int prec, int nc, long long N, bool tau1)
{
    if (lat != 0) return 0;
    const long long items = N * rs::group(nc);
    const int most = prec == 0 ? 512 : 1024;
    if (items > (long long)rs::kMaxCluster * most) return 0;
    if (prec == 0 && nc < 6 && items > 4096) return 0;
    int threads = 0;
    rs::shape(nc, N, rs::kMaxCluster, &threads);
    // only the kernel that will run: a query loads it
    auto k = rs::kernel_of(prec, rs::group(nc), tau1, threads);
    cudaLaunchAttribute a;
    cudaLaunchConfig_t c = rs::config(rs::kMaxCluster, threads, 0, &a);
    int n = 0;
    if (cudaFuncSetAttribute((const void *)k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, (const void *)k, &c) != cudaSuccess || n < 1) {
        cudaGetLastError();
        return 0;
    }
    return rs::kMaxCluster;
}

int launch_resident(int prec, int nc, const Params &P, const Par64 *p64, const df::ParMu *pm, const df::MuTab *mtab,
                    const Log64 *ltab, StateBufs st, void *scratch, int ctas, int steps, cudaStream_t s)
{
    rs::Par q{};
    q.nx = P.nx;
    q.ny = P.ny;
    q.nc = nc;
    q.steps = steps;
    q.N = (int)P.N;
    q.omega = P.omega;
    q.RT = P.RT;
    D2 iRT, c2;
    rt_constants(P.RT, &iRT, &c2);
    auto narrow = [](D2 v) {
        const float h = (float)v.hi;
        return make_float2(h, (float)((v.hi - (double)h) + v.lo));
    };
    q.iRT = make_double2(iRT.hi, iRT.lo);
    q.c2 = make_double2(c2.hi, c2.lo);
    q.fiRT = narrow(iRT);
    q.fc2 = narrow(c2);
    q.p64 = p64;
    q.pm = pm;
    q.mtab = mtab;
    q.ltab = ltab;
    const size_t items = (size_t)P.N * rs::group(nc);
    auto up = [](size_t b) { return (b + 15) & ~(size_t)15; };
    char *b = (char *)scratch;
    rs::Work w;
    w.mu = b;
    b += up(items * 8);
    w.psi = b;
    b += up((size_t)P.N * 8);
    w.rho = b;
    b += up(items * (prec == 0 ? 8 : 4));
    w.g = b;
    int threads = 0;
    rs::shape(nc, P.N, ctas, &threads);
    cudaLaunchAttribute a;
    cudaLaunchConfig_t c = rs::config(ctas, threads, s, &a);
    return (int)cudaLaunchKernelEx(&c, rs::kernel_of(prec, rs::group(nc), P.omega == 1.0, threads), q, st, w);
}

}  // namespace lbmfug
