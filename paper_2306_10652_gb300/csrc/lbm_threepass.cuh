// lbm_threepass.cuh -- the three-pass time step (any lattice, any Nc <= 16).
//
// Pass 1 (k_sums):    rho_i, the momentum sum_i sum_a e_a g_{a,i} and
//                     psi = sum_j sqrt(kappa_j) rho~_j.
// Pass 2 (k_eos):     ln f_i (Eqs. 9-12), lap psi with the isotropic lattice
//                     Laplacian and mu_i = RT ln f_i - sqrt(kappa_i) lap psi.
// Pass 3 (k_collide): F_i = -rho~_i grad mu_i (Eq. 5 with kappa_ij =
//                     sqrt(kappa_i kappa_j), Eq. 4, so sum_j kappa_ij lap rho~_j =
//                     sqrt(kappa_i) lap psi),
//                     u = (sum e g + F/2) / rho, the equilibrium (Eq. 1b) and
//                     forcing term (Eq. 1c), BGK (Eq. 1a) and push streaming
//                     g_{a,i}(r + e_a) <- g*_{a,i}(r).
//
// All thermodynamics, forces and the collision run in binary64, whose pipe
// (two multiply-adds per clock and SM) is what bounds passes 2 and 3: memory
// would allow some ten times their traffic.  So the passes are shaped by the number of
// binary64 operations and nothing else: one node per thread (no halo is
// computed twice), mu formed once so that one gradient per component serves
// the force, the collision evaluated as one quadratic form per component
// (below), reciprocals of 3 operations and a table-driven logarithm of 8.
//
// State formats (post-streaming populations, the convention of Eq. 1a):
//  * binary64 (S = double): all Q populations g[i][a][node].
//  * binary32 (S = float): the Q-1 moving populations g[i][a-1][node] (a >= 1)
//    and the density rho_i as an unevaluated binary32 sum hi + lo.  The rest
//    population is never needed: rho_i is the state, and the collision of
//    a >= 1 uses only rho_i, u, F_i and grad rho_i.  Pass 4 (k_rupdate) moves
//    the density by exactly the populations that left and arrived,
//    rho(t+1) = rho(t) - sum_{a>=1} g*_a(r) + sum_{a>=1} g_a(t+1)(r), with
//    compensated sums of the stored binary32 values, so the component mass
//    is conserved to the rounding of the pair.
#pragma once
#include "lbm_internal.h"

namespace lbmfug {

namespace tp {

constexpr int kThreads = 256;

// Periodic neighbours r + e_a of node r.  Boxes below 2^31 nodes take 32-bit
// divisions.
template <int LAT>
__device__ __forceinline__ void neighbours(const Par64 &P, long long r, long long (&nb)[Lattice<LAT>::Q])
{
    using L = Lattice<LAT>;
    int x, y, z;
    if (P.N < (1LL << 31)) {
        const unsigned q = (unsigned)r / (unsigned)P.nx;
        x = (int)((unsigned)r - q * (unsigned)P.nx);
        z = (int)(q / (unsigned)P.ny);
        y = (int)(q - (unsigned)z * (unsigned)P.ny);
    } else {
        x = (int)(r % P.nx);
        const long long t = r / P.nx;
        y = (int)(t % P.ny);
        z = (int)(t / P.ny);
    }
    const int xs[3] = {x == 0 ? P.nx - 1 : x - 1, x, x == P.nx - 1 ? 0 : x + 1};
    const int ys[3] = {y == 0 ? P.ny - 1 : y - 1, y, y == P.ny - 1 ? 0 : y + 1};
    const int zs[3] = {z == 0 ? P.nz - 1 : z - 1, z, z == P.nz - 1 ? 0 : z + 1};
#pragma unroll
    for (int a = 0; a < L::Q; ++a)
        nb[a] = xs[L::e(a, 0) + 1] +
                (long long)P.nx * (ys[L::e(a, 1) + 1] + (long long)P.ny * (L::D == 3 ? zs[L::e(a, 2) + 1] : z));
}

// 12 grad X(r) = 36 sum_a w_a e_a X(r + e_a), summed over opposite pairs:
// the weights become the small integers 4 (D2Q9) or 2 (D3Q19) for the faces
// and 1 for the diagonals or edges, so the sum takes one operation per
// difference and one or two per axis.
template <int LAT>
__device__ __forceinline__ void grad12(const double *__restrict__ X, const long long (&nb)[Lattice<LAT>::Q],
                                       double (&G)[Lattice<LAT>::D])
{
    auto d = [&](int a) { return __ldg(X + nb[a]) - __ldg(X + nb[a + 1]); };
    if constexpr (LAT == 0) {
        const double ne = d(5), se = d(7);
        G[0] = fma(4.0, d(1), ne + se);
        G[1] = fma(4.0, d(3), ne - se);
    } else {
        const double a = d(7), b = d(9), c = d(11), e = d(13), f = d(15), g = d(17);
        G[0] = fma(2.0, d(1), (a + b) + (c + e));
        G[1] = fma(2.0, d(3), (a - b) + (f + g));
        G[2] = fma(2.0, d(5), (c - e) + (f - g));
    }
}

// population slot of direction a in the storage format of S (-1: not stored)
template <int LAT, typename S> __host__ __device__ constexpr int slot(int a)
{
    return sizeof(S) == 8 ? a : a - 1;
}
template <int LAT, typename S> __host__ __device__ constexpr int nslots()
{
    return sizeof(S) == 8 ? Lattice<LAT>::Q : Lattice<LAT>::Q - 1;
}

// g = g^eq(rho, u) (Eq. 1b, rho^c = 0); at rest (u null) that is (rho_i, 0, ..., 0).
// Bound by its stores: one node per thread, no arithmetic on the binary64 pipe
// at rest (2048^2, Nc = 10, binary32 storage, 1.7 GB written: 0.32 ms, 0.76 ms
// when every population was formed in binary64).
template <int LAT, typename S>
__global__ void __launch_bounds__(kThreads)
    k_init(const int nc, const long long N, const double *__restrict__ rho, const double *__restrict__ u,
           StateBufs st)
{
    using L = Lattice<LAT>;
    constexpr int NS = nslots<LAT, S>();
    S *__restrict__ g = (S *)st.g;
    float *__restrict__ rh = (float *)st.rhi;
    float *__restrict__ rl = st.rlo;
    const long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (r >= N) return;
    double B[L::Q];
    if (u) {
        double uu[L::D], u2 = 0.0;
#pragma unroll
        for (int d = 0; d < L::D; ++d) uu[d] = __ldg(u + d * N + r);
#pragma unroll
        for (int d = 0; d < L::D; ++d) u2 += uu[d] * uu[d];
#pragma unroll
        for (int a = 0; a < L::Q; ++a) {
            double ue = 0.0;
#pragma unroll
            for (int d = 0; d < L::D; ++d) ue += L::e(a, d) * uu[d];
            B[a] = 3.0 * ue + 4.5 * ue * ue - 1.5 * u2;
        }
    }
    if (sizeof(S) == 4) {  // both components of a pair with one store
        float2 *g2 = (float2 *)st.g, *rh2 = (float2 *)st.rhi, *rl2 = (float2 *)st.rlo;
#pragma unroll 2
        for (int p = 0; p < st.paired / 2; ++p) {
            const double r0 = __ldg(rho + 2 * p * N + r), r1 = __ldg(rho + (2 * p + 1) * N + r);
#pragma unroll
            for (int a = 1; a < L::Q; ++a)
                g2[(p * NS + a - 1) * N + r] = u ? make_float2((float)(L::w(a) * r0 * B[a]), (float)(L::w(a) * r1 * B[a]))
                                                 : make_float2(0.0f, 0.0f);
            const float2 hi = make_float2((float)r0, (float)r1);
            rh2[p * N + r] = hi;
            rl2[p * N + r] = make_float2((float)(r0 - (double)hi.x), (float)(r1 - (double)hi.y));
        }
    }
#pragma unroll 2
    for (int i = st.paired; i < nc; ++i) {
        const double ri = __ldg(rho + i * N + r);
#pragma unroll
        for (int a = 0; a < L::Q; ++a) {
            if (slot<LAT, S>(a) < 0) continue;
            S *o = g + (i * NS + slot<LAT, S>(a)) * N + r;
            if (u)
                *o = (S)(L::w(a) * ri * B[a] + (a == 0 ? ri : 0.0));
            else
                *o = a == 0 ? (S)ri : (S)0;
        }
        if (sizeof(S) == 4) {
            const float hi = (float)ri;
            rh[i * N + r] = hi;
            rl[i * N + r] = (float)(ri - (double)hi);
        }
    }
}

// Densities, and for kFull psi and the momentum (jm may be null).  kFull = false (only the
// densities are asked for): binary32 storage reads its pairs and no population.
template <int LAT, typename S, bool kFull>
__global__ void __launch_bounds__(kThreads)
    k_sums(const Par64 P, StateBufs st, double *__restrict__ rho, double *__restrict__ psi,
           double *__restrict__ jm)
{
    using L = Lattice<LAT>;
    constexpr int NS = nslots<LAT, S>();
    const S *__restrict__ g = (const S *)st.g;
    const float *__restrict__ rh = sizeof(S) == 4 ? st.rhi_f() : nullptr;
    const float *__restrict__ rl = st.rlo;
    const long long N = P.N;
    const long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (r >= N) return;
    if constexpr (!kFull && sizeof(S) == 4) {
        // both components of a pair with one load
        const float2 *__restrict__ h2 = (const float2 *)st.rhi, *__restrict__ l2 = (const float2 *)st.rlo;
#pragma unroll 4
        for (int p = 0; p < st.paired / 2; ++p) {
            const float2 h = __ldg(h2 + p * N + r), l = __ldg(l2 + p * N + r);
            rho[2 * p * N + r] = widen(h.x) + widen(l.x);
            rho[(2 * p + 1) * N + r] = widen(h.y) + widen(l.y);
        }
#pragma unroll 2
        for (int i = st.paired; i < P.nc; ++i) rho[i * N + r] = widen(__ldg(rh + i * N + r)) + widen(__ldg(rl + i * N + r));
        return;
    }
    // momentum: binary64 storage sums the differences of opposite directions over
    // all components, binary32 storage each component in binary32 first
    constexpr int kJ = sizeof(S) == 8 ? L::Q / 2 : L::D;
    double jp[kJ];
#pragma unroll
    for (int k = 0; k < kJ; ++k) jp[k] = 0.0;
    double ps = 0.0;
#pragma unroll 2
    for (int i = 0; i < P.nc; ++i) {
        S v[L::Q];
        if constexpr (kFull || sizeof(S) == 8) {
#pragma unroll
            for (int a = 0; a < L::Q; ++a)
                if (slot<LAT, S>(a) >= 0) v[a] = __ldg(g + st.at(i, slot<LAT, S>(a), NS, N, r));
        }
        double ri;
        if constexpr (sizeof(S) == 8) {
            // the moving populations first: they are small beside the resting one, which
            // carries the density, so one addition rounds at its size instead of Q - 1
            double m = v[1];
#pragma unroll
            for (int a = 2; a < L::Q; ++a) m += v[a];
            ri = v[0] + m;
        } else {
            ri = widen(__ldg(rh + st.at(i, N, r))) + widen(__ldg(rl + st.at(i, N, r)));
        }
        rho[i * N + r] = ri;
        if constexpr (kFull) {
            ps = fma(P.pk[i], ri, ps);
            if constexpr (sizeof(S) == 8) {
#pragma unroll
                for (int k = 0; k < kJ; ++k) jp[k] += v[2 * k + 1] - v[2 * k + 2];
            } else {
                float ji[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
                for (int a = 1; a < L::Q; ++a)
#pragma unroll
                    for (int d = 0; d < L::D; ++d)
                        if (L::e(a, d) > 0) ji[d] += v[a];
                        else if (L::e(a, d) < 0) ji[d] -= v[a];
#pragma unroll
                for (int d = 0; d < L::D; ++d) jp[d] += widen(ji[d]);
            }
        }
    }
    if constexpr (kFull) {
        psi[r] = ps;
        if (!jm) return;
        if constexpr (sizeof(S) == 8) {
            double j[3] = {0.0, 0.0, 0.0};
#pragma unroll
            for (int k = 0; k < kJ; ++k)
#pragma unroll
                for (int d = 0; d < L::D; ++d)
                    if (L::e(2 * k + 1, d) > 0) j[d] += jp[k];
                    else if (L::e(2 * k + 1, d) < 0) j[d] -= jp[k];
#pragma unroll
            for (int d = 0; d < L::D; ++d) jm[d * N + r] = j[d];
        } else {
#pragma unroll
            for (int d = 0; d < L::D; ++d) jm[d * N + r] = jp[d];
        }
    }
}

// Equation of state of every node (Eqs. 9-12).  STEP: out[i] = mu_i / (M_i RT).  Else
// the fields: out[i] = ln f_i (may be null), p (may be null) and lap psi (may
// be null).
template <int LAT, int NC, bool STEP>
__global__ void __launch_bounds__(kThreads)
    k_eos(const Par64 P, const double *__restrict__ rho, const double *__restrict__ psi,
          double *__restrict__ out, double *__restrict__ pout, double *__restrict__ lapout)
{
    using L = Lattice<LAT>;
    const long long N = P.N;
    const long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (r >= N) return;
    double ri[NC];
#pragma unroll
    for (int i = 0; i < NC; ++i) ri[i] = __ldg(rho + i * N + r);
    double lap = 0.0;
    if (STEP || lapout) {
        long long nb[L::Q];
        neighbours<LAT>(P, r, nb);
        // lap X = (2/cs2) sum_a w_a (X(r + e_a) - X(r)): D2Q9 (4 faces + diagonals - 20 X)/6,
        // D3Q19 (2 faces + edges - 24 X)/6
        const double c = __ldg(psi + nb[0]);
        constexpr int kFaces = 2 * L::D;
        double f = 0.0, e = 0.0;
#pragma unroll
        for (int a = 1; a <= kFaces; ++a) f += __ldg(psi + nb[a]);
#pragma unroll
        for (int a = kFaces + 1; a < L::Q; ++a) e += __ldg(psi + nb[a]);
        lap = fma(LAT == 0 ? 4.0 : 2.0, f, fma(LAT == 0 ? -20.0 : -24.0, c, e)) * (1.0 / 6.0);
        if (!STEP) lapout[r] = lap;
    }
    if (!STEP && !out && !pout) return;
    PrNode<NC> e;
    e.eval(P, ri);
    if constexpr (STEP) {
#pragma unroll
        for (int i = 0; i < NC; ++i) out[i * N + r] = e.mu(P, ri, lap, i);
    } else {
        if (out)
#pragma unroll
            for (int i = 0; i < NC; ++i) out[i * N + r] = e.lnf(P, ri, i);
        if (pout) pout[r] = e.pressure(P);
    }
}

// Pass 3.  STEP = false: only the velocity of Eq. (5)'s forced step, from X =
// ln f and lap (the fields); STEP: X = mu / (M RT).
//
// Per component, with r3 = 3 w rho_i / 36, f = 3 (1 - w/2) F_i / 36 and
// G = (1 - w/2) grad rho_i / 36 (w = 1/tau, and 36 w_a an integer), the
// change of population a, w g^eq_a + (1 - w/2) F_a (Eqs. 1b, 1c), is
//   36 w_a [ (u.e)(H.e) + base + e^2 K + e.V ],   V = r3 u + f,
//   H = 3/2 (V + f) + 3 G,  K = 3/2 G.u,  base = -r3 u^2/2 - f.u - (D/2 + 1) G.u:
// the products of Eqs. (1b) and (1c) with e collected into one quadratic
// form, so a pair of opposite directions takes 2 operations for its even and
// odd part and the two populations 2 each.  Written direction by direction the
// same terms take about 20 operations per population, and the kernel is bound
// by the binary64 pipe.  Whole step, with passes 1 and 2 as they stand now and
// as they were: D2Q9 512^2, Nc = 4, 0.260 ms (the fused kernel that ran there:
// 0.794 ms); D3Q19 51x47x45, Nc = 6, 0.290 ms (0.575 ms).  The pipe is 84 %
// active in passes 2 and 3, 70 % in pass 1, which waits for its loads too.
//
// TAU1 (tau = 1, the paper's value): (1 - w) g_a vanishes, so the moving
// populations are w g^eq + F/2 and the old ones are not read.
template <int LAT, typename S, bool STEP, bool TAU1>
__global__ void __launch_bounds__(kThreads)
    k_collide(const Par64 P, StateBufs in, StateBufs out, const double *__restrict__ rho,
              const double *__restrict__ X, const double *__restrict__ lap,
              const double *jm, double *uout /* may be jm */, float *__restrict__ osum,
              float *__restrict__ ocmp)
{
    using L = Lattice<LAT>;
    constexpr int D = L::D, Q = L::Q;
    constexpr int NS = nslots<LAT, S>();
    extern __shared__ double FS[];  // STEP: [nc][D][threads] the thread's f
    const S *__restrict__ gin = (const S *)in.g;
    S *__restrict__ gout = (S *)out.g;
    const long long N = P.N;
    const int t = threadIdx.x, T = blockDim.x;
    const long long r = blockIdx.x * (long long)T + t;
    if (r >= N) return;
    long long nb[Q];
    neighbours<LAT>(P, r, nb);
    const double om = TAU1 ? 1.0 : P.omega, om1 = 1.0 - om, sf = (1.0 - 0.5 * om) / 36.0;
    // Eq. (5): f_i = -3 sf rho~_i grad mu_i.  The fields need the sum of f_i alone, so
    // the part of lap psi, common to all components, is taken once.
    double Fs[D];
#pragma unroll
    for (int d = 0; d < D; ++d) Fs[d] = 0.0;
    double rt = 0.0, kl = 0.0;
    const double cf = -0.25 * sf * P.RT;
#pragma unroll 2
    for (int i = 0; i < P.nc; ++i) {
        double G[D];
        grad12<LAT>(X + i * N, nb, G);
        const double ri = __ldg(rho + i * N + r);
        rt += ri;
        if constexpr (STEP) {
            const double c = cf * ri;
#pragma unroll
            for (int d = 0; d < D; ++d) {
                const double f = c * G[d];
                Fs[d] += f;
                FS[(i * D + d) * T + t] = f;
            }
        } else {
            const double c = P.invM[i] * ri;
            kl = fma(P.sqk[i], c, kl);
#pragma unroll
            for (int d = 0; d < D; ++d) Fs[d] = fma(c, G[d], Fs[d]);
        }
    }
    if constexpr (!STEP) {
        double GL[D];
        grad12<LAT>(lap, nb, GL);
        kl *= P.iRT;
#pragma unroll
        for (int d = 0; d < D; ++d) Fs[d] = cf * fma(-kl, GL[d], Fs[d]);
    }
    const double irt = rcp64(rt), cs = 0.5 / (3.0 * sf);
    double u[D];
#pragma unroll
    for (int d = 0; d < D; ++d) u[d] = fma(cs, Fs[d], jm[d * N + r]) * irt;
    if constexpr (!STEP) {
#pragma unroll
        for (int d = 0; d < D; ++d) uout[d * N + r] = u[d];
        return;
    }
    double hu2 = 0.0;
#pragma unroll
    for (int d = 0; d < D; ++d) hu2 = fma(u[d], u[d], hu2);
    hu2 *= -0.5;
    const double sg = sf / 12.0, so3 = om / 12.0;
#pragma unroll 1
    for (int i = 0; i < P.nc; ++i) {
        S v[Q];
#pragma unroll
        for (int a = 0; a < Q; ++a)
            if (slot<LAT, S>(a) >= 0 && !TAU1) v[a] = __ldg(gin + (i * NS + slot<LAT, S>(a)) * N + r);
        double G[D];
        grad12<LAT>(rho + i * N, nb, G);
        const double ri = __ldg(rho + i * N + r);
        const double r3 = so3 * ri;
        double V[D], H[D];
        double fu = 0.0, gu = 0.0;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const double f = FS[(i * D + d) * T + t];
            V[d] = fma(r3, u[d], f);
            H[d] = fma(3.0 * sg, G[d], 1.5 * (V[d] + f));
            fu = fma(f, u[d], fu);
            gu = fma(G[d], u[d], gu);
        }
        gu *= sg;
        const double base = fma(-(0.5 * D + 1.0), gu, fma(r3, hu2, -fu));
        const double K = 1.5 * gu;
        S *__restrict__ go = gout + (long long)i * NS * N;
        float os = 0.0f, oc = 0.0f;  // binary32: compensated sum of what leaves the node
        // Eq. (1a) for the two populations of a pair, c = 36 w_a
        auto pair = [&](int a, double c, double even, double odd) {
            const double p = even + odd, m = even - odd;
            if constexpr (sizeof(S) == 8) {
                auto relax = [&](double x, S g) { return c == 1.0 ? fma(om1, g, x) : fma(c, x, om1 * g); };
                go[a * N + nb[a]] = TAU1 ? c * p : relax(p, v[a]);
                go[(a + 1) * N + nb[a + 1]] = TAU1 ? c * m : relax(m, v[a + 1]);
            } else {  // binary32 populations: the change rounded once, the relaxation in binary32
                const float gp = TAU1 ? (float)(c * p) : fmaf((float)om1, v[a], (float)(c * p));
                const float gm = TAU1 ? (float)(c * m) : fmaf((float)om1, v[a + 1], (float)(c * m));
                go[(a - 1) * N + nb[a]] = gp;
                go[a * N + nb[a + 1]] = gm;
                acc_add(os, oc, gp);
                acc_add(os, oc, gm);
            }
        };
        const double b1 = base + K;
        double q[D];  // u_d H_d
#pragma unroll
        for (int d = 0; d < D; ++d) {
            q[d] = u[d] * H[d];
            pair(2 * d + 1, LAT == 0 ? 4.0 : 2.0, b1 + q[d], V[d]);
        }
        const double b2 = b1 + K;
#pragma unroll
        for (int a = 2 * D + 1; a < Q; a += 4) {  // (a, a+1) = +-(e_k + e_l), (a+2, a+3) = +-(e_k - e_l)
            const int k = L::e(a, 0) ? 0 : 1, l = L::e(a, 2) ? 2 : 1;
            const double s = b2 + (q[k] + q[l]);
            const double x = fma(u[k], H[l], u[l] * H[k]);
            pair(a, 1.0, s + x, V[k] + V[l]);
            pair(a + 2, 1.0, s - x, V[k] - V[l]);
        }
        if constexpr (sizeof(S) == 8) {  // at rest: w g^eq_0 carries the density
            go[nb[0]] = fma(36.0 * L::w(0), base, TAU1 ? ri : fma(om, ri - v[0], (double)v[0]));
        } else {
            osum[i * N + r] = os;
            ocmp[i * N + r] = oc;
        }
    }
}

// binary32 pass 4: rho(t+1) = rho(t) - (left) + (arrived), all compensated.
template <int LAT, int NC>
__global__ void __launch_bounds__(kThreads)
    k_rupdate(const Params P, StateBufs in, StateBufs out, const float *__restrict__ osum,
              const float *__restrict__ ocmp)
{
    using L = Lattice<LAT>;
    constexpr int NS = L::Q - 1;
    const float *g = (const float *)out.g;
    const long long N = P.N;
    for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < N;
         r += (long long)gridDim.x * blockDim.x) {
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            float s = -osum[i * N + r], c = -ocmp[i * N + r];
#pragma unroll
            for (int k = 0; k < NS; ++k) acc_add(s, c, __ldg(g + (i * NS + k) * N + r));
            float hi = in.rhi_f()[i * N + r], lo = in.rlo[i * N + r];
            pair_add(hi, lo, s, c);
            out.rhi_f()[i * N + r] = hi;
            out.rlo[i * N + r] = lo;
        }
    }
}

template <int LAT, int NC, typename S>
__global__ void k_to_f64(const Params P, StateBufs st, double *__restrict__ out)
{
    using L = Lattice<LAT>;
    constexpr int NS = nslots<LAT, S>();
    const S *g = (const S *)st.g;
    const long long N = P.N;
    for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < N;
         r += (long long)gridDim.x * blockDim.x) {
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            double moving = 0.0;
#pragma unroll
            for (int a = 0; a < L::Q; ++a) {
                if (slot<LAT, S>(a) < 0) continue;
                const double v = (double)g[st.at(i, slot<LAT, S>(a), NS, N, r)];
                out[(i * L::Q + a) * N + r] = v;
                moving += a > 0 ? v : 0.0;
            }
            if (sizeof(S) == 4)
                out[(i * L::Q) * N + r] =
                    (double)st.rhi_f()[st.at(i, N, r)] + (double)st.rlo[st.at(i, N, r)] - moving;
        }
    }
}

template <int LAT, int NC, typename S>
__global__ void k_from_f64(const Params P, const double *__restrict__ in, StateBufs st)
{
    using L = Lattice<LAT>;
    constexpr int NS = nslots<LAT, S>();
    S *g = (S *)st.g;
    const long long N = P.N;
    for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < N;
         r += (long long)gridDim.x * blockDim.x) {
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            double rho = 0.0;
#pragma unroll
            for (int a = 0; a < L::Q; ++a) {
                const double v = in[(i * L::Q + a) * N + r];
                rho += v;
                if (slot<LAT, S>(a) >= 0) g[st.at(i, slot<LAT, S>(a), NS, N, r)] = (S)v;
            }
            if (sizeof(S) == 4) {
                const float hi = (float)rho;
                st.rhi_f()[st.at(i, N, r)] = hi;
                st.rlo[st.at(i, N, r)] = (float)(rho - (double)hi);
            }
        }
    }
}

inline unsigned grid_for(long long n)
{
    long long b = (n + kThreads - 1) / kThreads;
    if (b > 152LL * 64) b = 152LL * 64;
    if (b < 1) b = 1;
    return (unsigned)b;
}

// One node per thread.  Small boxes take small CTAs, down to one warp, so that
// their warps spread over the SMs and share no binary64 pipe.
inline int threads_for(long long n)
{
    constexpr long long kSms = 152;
    return n <= kSms * 32 ? 32 : n <= kSms * 64 ? 64 : 128;
}
inline unsigned blocks_for(long long n, int threads) { return (unsigned)((n + threads - 1) / threads); }

template <int LAT, int NC, typename S> struct Impl {
    static int init(const Params &P, const double *rho, const double *u, StateBufs st, cudaStream_t s)
    {
        k_init<LAT, S><<<blocks_for(P.N, kThreads), kThreads, 0, s>>>(NC, P.N, rho, u, st);
        return (int)cudaGetLastError();
    }
    static int step(const Params &P, StateBufs in, StateBufs out, const ThreePassWork &w,
                    cudaStream_t s)
    {
        const int T = threads_for(P.N);
        const unsigned G = blocks_for(P.N, T);
        const size_t sm = (size_t)NC * Lattice<LAT>::D * T * sizeof(double);
        auto collide = P.omega == 1.0 ? k_collide<LAT, S, true, true> : k_collide<LAT, S, true, false>;
        static_assert(kMaxNc * 3 * 128 * sizeof(double) <= 48 * 1024, "the forces fit the default limit");
        k_sums<LAT, S, true><<<G, T, 0, s>>>(w.par, in, w.rho, w.psi, w.jm);
        k_eos<LAT, NC, true><<<G, T, 0, s>>>(w.par, w.rho, w.psi, w.lnf, nullptr, nullptr);
        collide<<<G, T, sm, s>>>(w.par, in, out, w.rho, w.lnf, nullptr, w.jm, nullptr, w.osum, w.ocmp);
        if (sizeof(S) == 4)
            k_rupdate<LAT, NC><<<grid_for(P.N), kThreads, 0, s>>>(P, in, out, w.osum, w.ocmp);
        return (int)cudaGetLastError();
    }
    static int fields(const Params &P, StateBufs st, const ThreePassWork &w, double *rho,
                      double *u, double *p, double *lnf, cudaStream_t s)
    {
        const int T = threads_for(P.N);
        const unsigned G = blocks_for(P.N, T);
        // the caller's buffers are written by the kernels themselves; the scratch
        // fields stand in for those that are needed on the way but not asked for
        double *r = rho ? rho : w.rho;
        if (!u && !p && !lnf) {
            k_sums<LAT, S, false><<<G, T, 0, s>>>(w.par, st, r, nullptr, nullptr);
            return (int)cudaGetLastError();
        }
        double *lf = lnf ? lnf : (u ? w.lnf : nullptr);
        // (the momentum of a node waits in the place of its velocity)
        k_sums<LAT, S, true><<<G, T, 0, s>>>(w.par, st, r, w.psi, u);
        k_eos<LAT, NC, false><<<G, T, 0, s>>>(w.par, r, w.psi, lf, p, u ? w.lap : nullptr);
        if (u)
            k_collide<LAT, S, false, false>
                <<<G, T, 0, s>>>(w.par, st, StateBufs{}, r, lf, w.lap, u, u, nullptr, nullptr);
        return (int)cudaGetLastError();
    }
    static int to_f64(const Params &P, StateBufs st, double *out, cudaStream_t s)
    {
        if constexpr (sizeof(S) == 8) return (int)cudaErrorInvalidValue;  // the layouts are the same: a copy
        else k_to_f64<LAT, NC, S><<<grid_for(P.N), kThreads, 0, s>>>(P, st, out);
        return (int)cudaGetLastError();
    }
    static int from_f64(const Params &P, const double *in, StateBufs st, cudaStream_t s)
    {
        if constexpr (sizeof(S) == 8) return (int)cudaErrorInvalidValue;
        else k_from_f64<LAT, NC, S><<<grid_for(P.N), kThreads, 0, s>>>(P, in, st);
        return (int)cudaGetLastError();
    }
    static int launches_per_step() { return sizeof(S) == 4 ? 4 : 3; }
};

// Function table of one (lattice, storage, Nc) instantiation.
struct Ops {
    int (*init)(const Params &, const double *, const double *, StateBufs, cudaStream_t);
    int (*step)(const Params &, StateBufs, StateBufs, const ThreePassWork &, cudaStream_t);
    int (*fields)(const Params &, StateBufs, const ThreePassWork &, double *, double *, double *,
                  double *, cudaStream_t);
    int (*to_f64)(const Params &, StateBufs, double *, cudaStream_t);
    int (*from_f64)(const Params &, const double *, StateBufs, cudaStream_t);
    int (*launches_per_step)();
};

template <int LAT, int NC, typename S> const Ops *ops_of()
{
    static const Ops o = {&Impl<LAT, NC, S>::init,   &Impl<LAT, NC, S>::step,
                          &Impl<LAT, NC, S>::fields, &Impl<LAT, NC, S>::to_f64,
                          &Impl<LAT, NC, S>::from_f64, &Impl<LAT, NC, S>::launches_per_step};
    return &o;
}

// Table of one translation unit: lattice LAT, storage S, Nc in [LO, HI].
template <int LAT, typename S, int LO, int HI> const Ops *ops_range(int nc)
{
    if constexpr (LO > HI) {
        return nullptr;
    } else {
        if (nc == LO) return ops_of<LAT, LO, S>();
        return ops_range<LAT, S, LO + 1, HI>(nc);
    }
}

}  // namespace tp

#define LBM_TP_TU(NAME, LAT, S, LO, HI) \
    namespace lbmfug { namespace tp { \
    const Ops *NAME(int nc) { return ops_range<LAT, S, LO, HI>(nc); } \
    } }

}  // namespace lbmfug
