// lbm_fused2d.cuh -- single-pass D2Q9 time step.
//
// One launch per step.  The state is the post-streaming population set g(t)
// (Eq. 1a) plus the density state R(t) = sum_a g_{a,i}(t) per node and
// component, which the previous step produced on chip.  Each CTA owns a strip
// of W interior columns (one thread per column, plus one halo column on each
// side) and a segment of H rows, which it walks row by row:
//
//   row k   : load R(k) on columns [-3, W+3) -> psi(k) = sum_j sqrt(kappa_j) rho~_j
//   row k-1 : ln f_i (Eqs. 9-12) and mu_i = RT ln f_i - sqrt(kappa_i) lap psi
//             on columns [-2, W+2)   (Eq. 5 with Eq. 4: sum_j kappa_ij lap rho~_j
//             = sqrt(kappa_i) lap psi)
//   row k-2 : F_i = -rho~_i grad mu_i, grad rho_i, u = (sum e g + F/2)/rho,
//             equilibrium (Eq. 1b), forcing (Eq. 1c), BGK (Eq. 1a) on columns
//             [-1, W+1); push streaming of the interior columns to g(t+1);
//             the new densities R(t+1) of the interior are gathered from the
//             collided values of rows k-3..k-1 and columns -1..W in a fixed
//             order (no atomics), so R(t+1) needs no second pass over g.
//
// DRAM traffic per node-step: g read + g written (the algorithmic bytes) plus
// R read + R written (Nc values each); halo rows and columns come from L2.
// Storage S (double, or float deviation h = g - delta_a0 rhobar_i), EOS and
// force arithmetic E (double or float), collision arithmetic S.
#pragma once

#include <type_traits>

#include "lbm_internal.h"
#include "lbm_thermo_df.cuh"

namespace lbmfug {
namespace fz {

constexpr int kT = 128;     // threads per CTA: one column each
constexpr int kWmax = kT - 2;

__host__ __device__ constexpr size_t align16(size_t b) { return (b + 15) & ~(size_t)15; }

template <int NC, typename S, typename E> struct Smem {
    static __host__ __device__ constexpr size_t rs(int W) { return align16((size_t)4 * NC * (W + 6) * sizeof(S)); }
    static __host__ __device__ constexpr size_t ps(int W) { return align16((size_t)3 * (W + 6) * sizeof(E)); }
    static __host__ __device__ constexpr size_t mu(int W) { return align16((size_t)3 * NC * (W + 4) * sizeof(E)); }
    static __host__ __device__ constexpr size_t xc() { return align16((size_t)6 * NC * kT * sizeof(S)); }
    static __host__ __device__ constexpr size_t red() { return align16((size_t)(kT / 32) * NC * sizeof(double)); }
    static __host__ __device__ constexpr size_t total(int W) { return rs(W) + ps(W) + mu(W) + xc() + red(); }
};

__device__ __forceinline__ int wrapc(int v, int n)
{
    if (v >= 0 && v < n) return v;
    v %= n;
    return v < 0 ? v + n : v;
}

template <int NC, typename S, typename E>
__global__ void __launch_bounds__(kT)
    k_fused(const Params P, const int W, const int H, const S *__restrict__ gin,
            S *__restrict__ gout, const S *__restrict__ rin, S *__restrict__ rout,
            double *__restrict__ mass_partials)
{
    using L = Lattice<0>;
    using V = PV<E>;
    using VS = PV<S>;
    constexpr bool kDev = sizeof(S) == 4;                 // deviation storage
    constexpr bool kKeep = 9 * NC * sizeof(S) <= 360;     // populations held in registers
    extern __shared__ __align__(16) unsigned char smem[];
    using SM = Smem<NC, S, E>;
    S *RS = (S *)smem;                                   // [4][NC][W+6]  R rows
    E *PS = (E *)(smem + SM::rs(W));                     // [3][W+6]      psi rows
    E *MU = (E *)(smem + SM::rs(W) + SM::ps(W));         // [3][NC][W+4]  mu rows
    S *XC = (S *)(smem + SM::rs(W) + SM::ps(W) + SM::mu(W));  // [6][NC][kT] exchange
    double *RED = (double *)(smem + SM::rs(W) + SM::ps(W) + SM::mu(W) + SM::xc());

    const int nx = P.nx, ny = P.ny;
    const long long N = P.N;
    const int CW = W + 6, CM = W + 4;
    const int x0 = blockIdx.x * W;
    const int w = min(W, nx - x0);
    const int y0 = blockIdx.y * H;
    const int h = min(H, ny - y0);
    const int t = threadIdx.x;
    const int col = t - 1;                 // collision column of this thread
    const bool active = t < w + 2;         // columns -1 .. w
    const bool interior = col >= 0 && col < w;
    const int xg = wrapc(x0 + col, nx);
    const int xd[3] = {wrapc(xg - 1, nx), xg, wrapc(xg + 1, nx)};  // destination columns, ex = -1, 0, 1
    // phase (A) columns of this thread: c = t - 3 and c = t - 3 + kT
    const int cA0 = t - 3, cA1 = t - 3 + kT;
    const bool hasA0 = cA0 < w + 3, hasA1 = cA1 < w + 3;
    const int xA0 = wrapc(x0 + cA0, nx), xA1 = hasA1 ? wrapc(x0 + cA1, nx) : 0;
    const E RT = V::RT(P);
    const S om = (S)P.omega, cF = (S)(1.0 - 0.5 * P.omega);

    S msum[NC], mcmp[NC];      // per-thread mass of the written rows (compensated)
    S accA[NC], accB[NC];
    S rp0[NC], rp1[NC];        // prefetched density state of the next row
#pragma unroll
    for (int i = 0; i < NC; ++i) {
        msum[i] = 0;
        mcmp[i] = 0;
        accA[i] = 0;
        accB[i] = 0;
    }
    {
        const long long rowb = (long long)wrapc(y0 - 3, ny) * nx;
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            rp0[i] = hasA0 ? __ldg(rin + i * N + rowb + xA0) : (S)0;
            rp1[i] = hasA1 ? __ldg(rin + i * N + rowb + xA1) : (S)0;
        }
    }

    const int nrows = h + 6;  // rows y0-3 .. y0+h+2
    for (int kk = 0; kk < nrows; ++kk) {
        const int k = y0 - 3 + kk;
        // ---- (0) populations of the collision row k-2, in flight during (A), (B) ----
        const int crow = k - 2;
        const int yc = wrapc(crow, ny);
        const long long rc = (long long)yc * nx + xg;
        S hv[kKeep ? NC : 1][9];
        if (kKeep && kk >= 4 && active) {
#pragma unroll
            for (int i = 0; i < NC; ++i)
#pragma unroll
                for (int a = 0; a < 9; ++a) hv[kKeep ? i : 0][a] = __ldg(gin + (i * 9 + a) * N + rc);
        }
        // ---- (A) density state and psi of row k --------------------------------
        {
            const int s4 = kk & 3, s3 = kk % 3;
            if (hasA0) {
                E ps = 0;
#pragma unroll
                for (int i = 0; i < NC; ++i) {
                    RS[(s4 * NC + i) * CW + cA0 + 3] = rp0[i];
                    ps = fma(V::sqk(P, i), (V::rhobar(P, i) + (E)rp0[i]) * V::invM(P, i), ps);
                }
                PS[s3 * CW + cA0 + 3] = ps;
            }
            if (hasA1) {
                E ps = 0;
#pragma unroll
                for (int i = 0; i < NC; ++i) {
                    RS[(s4 * NC + i) * CW + cA1 + 3] = rp1[i];
                    ps = fma(V::sqk(P, i), (V::rhobar(P, i) + (E)rp1[i]) * V::invM(P, i), ps);
                }
                PS[s3 * CW + cA1 + 3] = ps;
            }
        }
        __syncthreads();
        // ---- (B) ln f and mu of row k-1 ------------------------------------------
        if (kk >= 2) {
            const int q = kk - 1;
            const int s4 = q & 3;
            const E *p0 = PS + ((q + 2) % 3) * CW;  // row q-1
            const E *p1 = PS + (q % 3) * CW;        // row q
            const E *p2 = PS + ((q + 1) % 3) * CW;  // row q+1
            for (int c = t - 2; c < w + 2; c += kT) {
                const int cc = c + 3;
                E rm[NC], lf[NC];
#pragma unroll
                for (int i = 0; i < NC; ++i)
                    rm[i] = (V::rhobar(P, i) + (E)RS[(s4 * NC + i) * CW + cc]) * V::invM(P, i);
                pr_lnf<NC, E>(P, rm, lf, nullptr);
                const E c0 = p1[cc];
                const E faces = (p1[cc + 1] - c0) + (p1[cc - 1] - c0) + (p2[cc] - c0) + (p0[cc] - c0);
                const E diags = (p2[cc + 1] - c0) + (p0[cc - 1] - c0) + (p0[cc + 1] - c0) + (p2[cc - 1] - c0);
                const E lap = (E)6 * fma((E)(1.0 / 9.0), faces, (E)(1.0 / 36.0) * diags);
#pragma unroll
                for (int i = 0; i < NC; ++i)
                    MU[((q % 3) * NC + i) * CM + c + 2] = fma(RT, lf[i], -V::sqk(P, i) * lap);
            }
        }
        __syncthreads();
        // ---- prefetch the density state of row k+1 (in flight during (C)) ---------
        if (kk + 1 < nrows) {
            const long long rowb = (long long)wrapc(k + 1, ny) * nx;
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                if (hasA0) rp0[i] = __ldg(rin + i * N + rowb + xA0);
                if (hasA1) rp1[i] = __ldg(rin + i * N + rowb + xA1);
            }
        }
        if (kk < 4) continue;
        // ---- (C) collision of row k-2 --------------------------------------------
        const int q = kk - 2;
        const bool own_row = crow >= y0 && crow < y0 + h;
        S ownv[3][NC];  // collided values with dx = 0, by dy = -1, 0, +1
        if (active) {
            const long long yd[3] = {(long long)wrapc(yc - 1, ny) * nx, (long long)yc * nx,
                                     (long long)wrapc(yc + 1, ny) * nx};
            const int cc = col + 3, cm = col + 2;
            const S *R0 = RS + ((q + 3) & 3) * NC * CW;  // row q-1
            const S *R1 = RS + (q & 3) * NC * CW;        // row q
            const S *R2 = RS + ((q + 1) & 3) * NC * CW;  // row q+1
            const E *M0 = MU + ((q + 2) % 3) * NC * CM;
            const E *M1 = MU + (q % 3) * NC * CM;
            const E *M2 = MU + ((q + 1) % 3) * NC * CM;
            // momentum sum_i sum_a e_a g_{a,i}
            S jx = 0, jy = 0;
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                S v[9];
#pragma unroll
                for (int a = 0; a < 9; ++a)
                    v[a] = kKeep ? hv[kKeep ? i : 0][a] : __ldg(gin + (i * 9 + a) * N + rc);
                jx += (v[1] - v[2]) + (v[5] - v[6]) + (v[7] - v[8]);
                jy += (v[3] - v[4]) + (v[5] - v[6]) + (v[8] - v[7]);
            }
            // Eq. (5): F_i = -rho~_i grad mu_i
            S Fx[NC], Fy[NC];
            E Fsx = 0, Fsy = 0, rt = 0;
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                const E *m0 = M0 + i * CM, *m1 = M1 + i * CM, *m2 = M2 + i * CM;
                // grad X = 3 sum_pairs w e (X(r+e) - X(r-e)): faces 1/9, diagonals 1/36
                const E dE = m1[cm + 1] - m1[cm - 1];
                const E dN = m2[cm] - m0[cm];
                const E dNE = m2[cm + 1] - m0[cm - 1];
                const E dSE = m0[cm + 1] - m2[cm - 1];
                const E gx = (E)3 * fma((E)(1.0 / 9.0), dE, (E)(1.0 / 36.0) * (dNE + dSE));
                const E gy = (E)3 * fma((E)(1.0 / 9.0), dN, (E)(1.0 / 36.0) * (dNE - dSE));
                const E ri = V::rhobar(P, i) + (E)R1[i * CW + cc];
                rt += ri;
                const E rmi = ri * V::invM(P, i);
                const E fx = -rmi * gx, fy = -rmi * gy;
                Fsx += fx;
                Fsy += fy;
                Fx[i] = (S)fx;
                Fy[i] = (S)fy;
            }
            const E irt = (E)1 / rt;
            const S ux = (S)(fma((E)0.5, Fsx, (E)jx) * irt);
            const S uy = (S)(fma((E)0.5, Fsy, (E)jy) * irt);
            const S u2 = ux * ux + uy * uy;
            // per-direction scalars (component independent)
            S ue[9], Bq[9], c9[9];
#pragma unroll
            for (int a = 0; a < 9; ++a) {
                ue[a] = (S)L::e(a, 0) * ux + (S)L::e(a, 1) * uy;
                Bq[a] = ue[a] * fma((S)4.5, ue[a], (S)3) - (S)1.5 * u2;
                c9[a] = fma((S)9, ue[a], (S)3);
            }
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                const S *r0 = R0 + i * CW, *r1 = R1 + i * CW, *r2 = R2 + i * CW;
                const S dE = r1[cc + 1] - r1[cc - 1];
                const S dN = r2[cc] - r0[cc];
                const S dNE = r2[cc + 1] - r0[cc - 1];
                const S dSE = r0[cc + 1] - r2[cc - 1];
                const S Gx = (S)3 * fma((S)(1.0 / 9.0), dE, (S)(1.0 / 36.0) * (dNE + dSE));
                const S Gy = (S)3 * fma((S)(1.0 / 9.0), dN, (S)(1.0 / 36.0) * (dNE - dSE));
                const S dri = r1[cc];                          // rho_i - rhobar_i
                const S ri = VS::rhobar(P, i) + dri;
                const S Fu3 = (S)3 * (Fx[i] * ux + Fy[i] * uy);
                const S Gu = Gx * ux + Gy * uy;
                S v[9];
#pragma unroll
                for (int a = 0; a < 9; ++a)
                    v[a] = kKeep ? hv[kKeep ? i : 0][a] : __ldg(gin + (i * 9 + a) * N + rc);
                S others = 0;  // sum of the moving populations of this node
                if (kDev)
#pragma unroll
                    for (int a = 1; a < 9; ++a) others += v[a];
#pragma unroll
                for (int a = 0; a < 9; ++a) {
                    const int ex = L::e(a, 0), ey = L::e(a, 1);
                    const S wa = (S)L::w(a);
                    const S Fe = (S)ex * Fx[i] + (S)ey * Fy[i];
                    const S Ge = (S)ex * Gx + (S)ey * Gy;
                    const S cW = (S)(0.5 * (3.0 * (ex * ex + ey * ey) - 2.0) - 1.0);
                    // Eq. (1c): F.[(e-u)/cs2 + (u.e)e/cs4] + grad rho.[-u + (u.e)e/cs2 + (e^2/cs2 - D)u/2]
                    const S Fa = wa * (fma(Fe, c9[a], -Fu3) + fma((S)3 * ue[a], Ge, cW * Gu));
                    S gs;
                    if (kDev && a == 0) {
                        // Eq. (1a) at rest with Eq. (1b): h0 + w (sum_a h_a - h0 + w0 rho B0) + cF F0,
                        // the node's own populations carrying its mass exactly
                        gs = v[0] + fma(om, others + wa * ri * Bq[0], cF * Fa);
                    } else {
                        const S geq = wa * ri * Bq[a] + (a == 0 ? dri : (S)0);
                        gs = fma(om, geq - v[a], v[a]) + cF * Fa;
                    }
                    if (interior && own_row) gout[(i * 9 + a) * N + yd[ey + 1] + xd[ex + 1]] = gs;
                    if (ex == 0)
                        ownv[ey + 1][i] = gs;
                    else
                        XC[(((ey + 1) * 2 + (ex > 0 ? 0 : 1)) * NC + i) * kT + t] = gs;
                }
            }
        }
        __syncthreads();
        // ---- gather R(t+1) of the interior columns ---------------------------------
        if (interior) {
            const bool write_row = (crow - 1) >= y0 && (crow - 1) < y0 + h;
            const long long rw = (long long)wrapc(crow - 1, ny) * nx + xg;
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                S Pd[3];
#pragma unroll
                for (int dy = 0; dy < 3; ++dy)
                    Pd[dy] = (XC[((dy * 2 + 0) * NC + i) * kT + t - 1] + ownv[dy][i]) +
                             XC[((dy * 2 + 1) * NC + i) * kT + t + 1];
                accA[i] += Pd[0];  // row crow-1 now complete
                if (write_row) {
                    rout[i * N + rw] = accA[i];
                    // compensated (Kahan) running sum of the written densities
                    const S yv = accA[i] - mcmp[i];
                    const S tv = msum[i] + yv;
                    mcmp[i] = (tv - msum[i]) - yv;
                    msum[i] = tv;
                }
                accA[i] = accB[i] + Pd[1];
                accB[i] = Pd[2];
            }
        }
    }
    if (mass_partials) {
        // deterministic block reduction of the mass of the rows written
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            double v = (double)msum[i] - (double)mcmp[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if ((t & 31) == 0) RED[(t >> 5) * NC + i] = v;
        }
        __syncthreads();
        if (t < NC) {
            double s = 0.0;
            for (int wv = 0; wv < kT / 32; ++wv) s += RED[wv * NC + t];
            s += P.rhobar[t] * (double)w * (double)h;
            mass_partials[((long long)blockIdx.y * gridDim.x + blockIdx.x) * NC + t] = s;
        }
    }
}

// Thermodynamics arithmetic of the binary32-state kernel: binary32 (LBM_FP32,
// evaluated inside the step kernel) or double-binary32 (LBM_FP32DEV: a
// separate pass, k_mu32, writes grad mu, which the step kernel reads).
struct DF64 {};

// Constants of the binary32 step (a small kernel argument).  With w = 1/tau:
// r3 = 3 w rho / 36, f = 3 (1 - w/2) F / 36, sg = (1 - w/2) / (12 * 36).
struct Par32 {
    int nx, ny;
    long long N;
    float om1;           // 1 - w
    float2 so3;          // 3 w / 36 in two words: one is off by up to 2^-25, the same in every
                         // node and step, and so would be the momentum that a step hands on
    float sg, cs;        // (1 - w/2)/432; F/2 from f: 0.5 * 36 / (3 (1 - w/2))
    float RT, lnRT;
    float2 cf[kMaxNc / 2], cfl[kMaxNc / 2];  // f_i / (rho_i X), X = grad mu_i (double-binary32) or 12 grad mu_i: two words
    float invM[kMaxNc], sqk[kMaxNc], b[kMaxNc], A[kMaxNc * kMaxNc];
};

inline Par32 make_par32(const Params &P, bool df)
{
    Par32 q{};
    const double cF = 1.0 - 0.5 * P.omega;
    q.nx = P.nx;
    q.ny = P.ny;
    q.N = P.N;
    q.om1 = (float)(1.0 - P.omega);
    q.so3.x = (float)(P.omega / 12.0);
    q.so3.y = (float)(P.omega / 12.0 - (double)q.so3.x);
    q.sg = (float)(cF / 432.0);
    q.cs = (float)(6.0 / cF);
    q.RT = P.fRT;
    q.lnRT = P.flnRT;
    for (int i = 0; i < P.nc; ++i) {
        const double c = -cF / (df ? 12.0 : 144.0) * P.invM[i];
        (i & 1 ? q.cf[i / 2].y : q.cf[i / 2].x) = (float)c;
        (i & 1 ? q.cfl[i / 2].y : q.cfl[i / 2].x) = (float)(c - (double)(float)c);
        q.invM[i] = P.finvM[i];
        q.sqk[i] = P.fsqk[i];
        q.b[i] = P.fb[i];
    }
    for (int k = 0; k < kMaxNc * kMaxNc; ++k) q.A[k] = P.fA[k];
    return q;
}

struct View32 {
    const Par32 &P;
    __device__ float A(int i, int j) const { return P.A[i * kMaxNc + j]; }
    __device__ float b(int i) const { return P.b[i]; }
    __device__ float RT() const { return P.RT; }
    __device__ float lnRT() const { return P.lnRT; }
};

// Shared memory of the binary32 kernel.  Components go in pairs (the two lanes
// of a packed operation), and every row has a fixed pitch of kT entries, so all
// offsets are compile-time constants.  XC holds the collided values that move to
// a neighbouring column (6 slots: row below, same row, row above; to the right
// or left), XJ the same values summed over the components, for the momentum; G
// and J the grad mu and momentum of the row collided next.
template <int NC, typename E> struct Smem32 {
    static constexpr bool kDF = std::is_same<E, DF64>::value;
    static constexpr int NP = (NC + 1) / 2;
    static constexpr int kHalo = kDF ? 2 : 3;  // density columns and rows beyond the strip
    static constexpr int kRing = 4;            // density rows kept
    static __host__ __device__ constexpr size_t rs() { return (size_t)kRing * NP * kT * sizeof(float2); }
    static __host__ __device__ constexpr size_t g() { return kDF ? (size_t)NP * kT * sizeof(float4) : 0; }
    static __host__ __device__ constexpr size_t mu() { return kDF ? 0 : (size_t)3 * NP * kT * sizeof(float2); }
    static __host__ __device__ constexpr size_t xc() { return (size_t)6 * NP * kT * sizeof(float2); }
    static __host__ __device__ constexpr size_t j() { return (size_t)kT * sizeof(float2); }
    static __host__ __device__ constexpr size_t xj() { return (size_t)6 * kT * sizeof(float); }
    static __host__ __device__ constexpr size_t ps() { return kDF ? 0 : (size_t)3 * kT * sizeof(float); }
    // CTAs per SM that the registers are cut for.  At general tau the largest odd number of
    // components of a class, whose last pair has addresses of its own, waits less with one
    // CTA fewer and no spilled registers (2048 x 1024, tau = 0.8, LBM_FP32: Nc = 5 212 us,
    // 223 with four; Nc = 9 408 us, 447 with three; Nc = 7 304 us, 340 with two).
    static __host__ __device__ constexpr int ctas(bool tau1)
    {
        const bool odd = !tau1 && (NC == 5 || NC == 9);
        return NC == 1 ? 6 : NC <= 6 ? (odd ? 3 : 4) : NC <= 10 ? (odd ? 2 : 3) : 2;
    }
    // General tau: the old populations of the next pair are copied ahead of it.  More
    // pairs than two hide their loads behind each other, and lose registers by it (same
    // box, with and without: LBM_FP32 Nc = 2 86 and 99 us, Nc = 3 130 and 138, Nc = 6
    // 254 and 213, Nc = 8 331 and 297).
    static __host__ __device__ constexpr bool ahead(bool tau1) { return !tau1 && NC <= 4; }
    static __host__ __device__ constexpr size_t v() { return (size_t)8 * kT * sizeof(float2); }
    static __host__ __device__ constexpr size_t base() { return rs() + g() + mu() + xc() + j() + xj() + ps(); }
    static __host__ __device__ constexpr size_t total(bool tau1) { return base() + (ahead(tau1) ? v() : 0); }
};
// *a = x where `on` (a predicated store, no branch)
__device__ __forceinline__ void store_if(bool on, float2 *a, float2 x)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %3, 0;\n\t@p st.global.v2.f32 [%0], {%1, %2};\n\t}" ::"l"(a),
                 "f"(x.x), "f"(x.y), "r"((int)on)
                 : "memory");
}
__device__ __forceinline__ void store_if(bool on, float *a, float x)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p st.global.f32 [%0], %1;\n\t}" ::"l"(a), "f"(x),
                 "r"((int)on)
                 : "memory");
}
// store_pair where `on`
__device__ __forceinline__ void store_pair_if(bool on, void *base, bool one, int p, int a, int ns, long long N, unsigned o,
                                              float2 v)
{
    if (one) store_if(on, (float *)base + (2LL * p * ns + a) * N + o, v.x);
    else store_if(on, (float2 *)base + ((long long)p * ns + a) * N + o, v);
}
template <typename E> constexpr int wmax32() { return kT - 2 * (std::is_same<E, DF64>::value ? 2 : 3); }

// asynchronous copies to shared memory (no register holds the data in flight)
template <int BYTES> __device__ __forceinline__ void copy_async(void *dst, const void *src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}
// node o of pair p into *dst (an odd last component: into its first word)
__device__ __forceinline__ void copy_pair(float2 *dst, const void *base, bool one, int p, long long N, unsigned o)
{
    if (one) copy_async<4>(dst, (const float *)base + 2LL * p * N + o);
    else copy_async<8>(dst, (const float2 *)base + (long long)p * N + o);
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Double-binary32 chemical potentials and their gradients (LBM_FP32DEV), one
// pass before the step kernel.  Each CTA walks a segment of rows of a strip
// of W <= kT - 4 columns; for row k it forms
//   psi(k) (Eq. 4) on columns [-2, W + 1] from the state's exact density pairs,
//     with B(k) = b_m rho~ (Eq. 11) in the same packed sum,
//   mu(k-1) (Eqs. 5, 9-12 through lbm_thermo_df.cuh) on columns [-1, W] from
//     psi rows k-2..k and the pairs and B of row k-1 kept from the previous row,
//   grad mu(k-2) on the interior columns from mu rows k-3..k-1, every
//     difference mu(r + e) - mu(r - e) taken on the (hi, lo) pairs and
//     rounded once (so it carries the df64 accuracy of mu), written in binary32
//     to G[p][node], (d/dx, d/dx, d/dy, d/dy) of components 2p and 2p + 1, or
//     (d/dx, d/dy) of an odd last one.
// The step kernel forms F_i = -rho~_i G_i.  psi and mu rows live in rings of
// three: a slot is rewritten only after the barrier that follows its last
// reader.
// Bound by the FMA pipe, which takes two cycles per packed operation (67 % active
// before the next row was copied ahead); the evaluation is straight-line code that
// packs two components per operation.  2048^2, Nc = 10: 0.379 ms; 0.423 ms with the
// row loaded where it is used, and 0.54 ms with scalar logarithms and closing sums
// and TwoProd plus ordered FastTwoSum in the Nc^2 mixing sums.
constexpr int kWmaxMu = kT - 4;

template <int NC> struct SmemMu {
    static constexpr int NP = (NC + 1) / 2;
    static __host__ __device__ constexpr size_t bytes()
    {
        // logarithm tables, psi ring, mu ring (pairs of components), the next row's density pairs
        return sizeof(df::MuTab) + 3 * kT * sizeof(float2) + (size_t)3 * NP * kT * sizeof(float4) +
               (size_t)2 * NP * kT * sizeof(float2);
    }
};

template <int NC>
__global__ void __launch_bounds__(kT, NC <= 10 && NC != 9 ? 4 : 3)
    k_mu32(const df::ParMu P, const int W, const int H, StateBufs in, float4 *__restrict__ G)
{
    constexpr int NP = SmemMu<NC>::NP, CW = NP * kT;
    auto one = [](int p) { return 2 * p + 1 == NC; };  // an odd last component
    extern __shared__ __align__(16) unsigned char smem[];
    float4 *TV = (float4 *)smem;      // [128] logarithm tables
    float2 *TK = (float2 *)(TV + 128);  // [512]
    float2 *PS = TK + 512;            // [3][kT]
    float4 *MU = (float4 *)(PS + 3 * kT);  // [3][NP][kT] (hi, hi, lo, lo)
    float2 *NX = (float2 *)(MU + 3 * CW);  // [2][NP][kT] density pairs of row k
    const int nx = P.nx, ny = P.ny;
    const long long N = P.N;
    const int x0 = blockIdx.x * W;
    const int w = min(W, nx - x0);
    const int y0 = blockIdx.y * H;
    const int h = min(H, ny - y0);
    const int t = threadIdx.x;
    const int c = t - 2;  // column of this thread, -2 .. w + 1
    const bool hasP = c <= w + 1;
    const bool hasM = c >= -1 && c <= w;
    const bool interior = c >= 0 && c < w;
    const unsigned xg = (unsigned)wrapc(x0 + c, nx);
    df::load_mu_tab(P.tab, TV, TK);
    auto copy_row = [&](int y) {  // asynchronous, the thread's own column
        const unsigned o = (unsigned)wrapc(y, ny) * (unsigned)nx + xg;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            copy_pair(NX + p * kT + t, in.rhi, one(p), p, N, o);
            copy_pair(NX + (NP + p) * kT + t, in.rlo, one(p), p, N, o);
        }
    };
    if (hasP) copy_row(y0 - 2);
    float ph[NC], pl[NC];      // density pairs of row k-1 at this column
    df::F2 Bp = {0.0f, 0.0f};  // and its B (Eq. 11)
#pragma unroll
    for (int i = 0; i < NC; ++i) ph[i] = pl[i] = 0.0f;
    for (int kk = 0; kk < h + 4; ++kk) {
        const int k = y0 - 2 + kk;
        float hh[NC], ll[NC];
        df::F2 Bk = {0.0f, 0.0f};
        if (hasP) {
            copy_async_wait();
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const float2 a = NX[p * kT + t], b = NX[(NP + p) * kT + t];
                hh[2 * p] = a.x, ll[2 * p] = b.x;
                if (!one(p)) hh[2 * p + 1] = a.y, ll[2 * p + 1] = b.y;
            }
            df::F2 ps;
            df::psi_and_B<NC>(P, hh, ll, ps, Bk);
            if (kk + 1 < h + 4) copy_row(k + 1);  // the values above are consumed
            PS[(kk % 3) * kT + t] = make_float2(ps.hi, ps.lo);
        }
        __syncthreads();
        if (kk >= 2 && hasM) {
            const float2 *p0 = PS + ((kk - 2) % 3) * kT + t, *p1 = PS + ((kk - 1) % 3) * kT + t, *p2 = PS + (kk % 3) * kT + t;
            const df::F2 lap = df::lap9x6(p1[0], p1[1], p1[-1], p2[0], p0[0], p2[1], p2[-1], p0[1], p0[-1]);
            float4 *out = MU + ((kk - 1) % 3) * CW + t;
            df::mu_pairs<NC, false>(P, TV, TK, ph, pl, Bp, lap, [&](int p, df::P2 m) {
                out[p * kT] = make_float4(m.hi.x, m.hi.y, m.lo.x, m.lo.y);
            });
        }
        if (hasP) {
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                ph[i] = hh[i];
                pl[i] = ll[i];
            }
            Bp = Bk;
        }
        __syncthreads();
        if (kk >= 4 && interior) {
            // gradient of mu at row k-2: rows k-3 (south), k-2, k-1 (north)
            const float4 *S = MU + ((kk - 3) % 3) * CW + t, *C = MU + ((kk - 2) % 3) * CW + t,
                         *Nr = MU + ((kk - 1) % 3) * CW + t;
            const unsigned ob = (unsigned)wrapc(k - 2, ny) * (unsigned)nx + xg;
            // grad X = 3 sum_pairs w e (X(r+e) - X(r-e)): faces 1/9, diagonals 1/36
            auto diff = [](float4 a, float4 b) {
                return df::vadd(df::vsub(make_float2(a.x, a.y), make_float2(b.x, b.y)),
                                df::vsub(make_float2(a.z, a.w), make_float2(b.z, b.w)));
            };
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const float4 *s0 = S + p * kT, *c0 = C + p * kT, *n0 = Nr + p * kT;
                const float2 dE = diff(c0[1], c0[-1]), dN = diff(n0[0], s0[0]);
                const float2 dNE = diff(n0[1], s0[-1]), dSE = diff(s0[1], n0[-1]);
                const float2 f = df::vbc(1.0f / 9.0f), d = df::vbc(1.0f / 36.0f), three = df::vbc(3.0f);
                const float2 gx = df::vmul(three, df::vfma(f, dE, df::vmul(d, df::vadd(dNE, dSE))));
                const float2 gy = df::vmul(three, df::vfma(f, dN, df::vmul(d, df::vsub(dNE, dSE))));
                if (one(p)) ((float2 *)(G + p * N))[ob] = make_float2(gx.x, gy.x);
                else G[p * N + ob] = make_float4(gx.x, gx.y, gy.x, gy.y);
            }
        }
    }
}

// Binary32 state: the 8 moving populations (a = 1..8), the density rho_i = hi + lo
// and the momentum j = sum_i sum_a e_a g_{a,i}; components in pairs, g[p][a-1][node][2]
// and rhi, rlo[p][node][2], so that a load or store serves two (an odd last one alone,
// StateBufs).  Collision arithmetic in binary32; thermodynamics and forces in E.  The new density of a
// node is its old density minus the populations that left it plus those that
// arrived: every stored binary32 population is added once where it arrives and
// subtracted once where it left, each by an error-free Fast2Sum into the (hi, lo)
// pair of the node, so the component mass is conserved to the rounding of the
// pairs.  Fast2Sum is exact when |hi| >= |term|, i.e. when no single moving
// population exceeds the density of the node it leaves or enters.  The pairs are
// normalised, so hi is the density rounded to binary32 and the collision, the
// gradients and the binary32 thermodynamics use hi alone.
//
// The momentum of the new state is gathered like the densities, from the sums
// over the components of what arrives.  The velocity is then known before any
// population is read, so the collision takes the components one pair after the
// other and reads each old population once, and none at tau = 1 (TAU1), where
// (1 - w) g vanishes.
//
// A thread owns one column.  For each row k the CTA has the densities of rows
// k - 2 .. k in shared memory and, with one row of lag (two for binary32
// thermodynamics, which form mu of row k - 1 first), collides row q on columns
// -1 .. W, pushes it, and updates rows q - 1 (complete: written), q and q + 1.
// The inputs of the next row are copied to shared memory asynchronously during
// the collision of this one.  Two components share every instruction of the
// collision and of the density update (packed FP32x2, lbm_df64.cuh).  The
// collision is the quadratic form in e of lbm_multipass.cuh; at tau = 1 the sums
// over the components that make the momentum follow from the sums of rho_i, F_i
// and grad rho_i, in which the form is linear.
// 2048^2, Nc = 10, tau = 1, double-binary32: 0.43 ms per launch.  0.52 ms with
// the components of a pair stored apart (twice the stores and addresses), 0.67 ms
// with that and the inputs loaded into registers (spills, and every row waits for
// its loads), 0.81 ms when it held the 80 populations of a node in registers,
// component by component.  LBM_FP32 1021 x 1531, Nc = 6: 0.117 ms with four CTAs
// per SM, 0.134 ms with three, 0.141 ms with three and the components apart, 0.260 ms
// at first; Nc = 10 needs more than the 128 registers that four leave it.
template <int NC, typename E, bool TAU1>
__global__ void __launch_bounds__(kT, (Smem32<NC, E>::ctas(TAU1)))
    k_fused32(const Par32 P, const int W, const int H, StateBufs in, StateBufs out,
              const float4 *__restrict__ mug /* DF64: grad mu of a pair of components (x, x, y, y); an odd last one (x, y) */)
{
    using L = Lattice<0>;
    using SM = Smem32<NC, E>;
    using df::vbc;
    // one component alone: the other lane stays zero and costs nothing
    auto vadd = [](float2 a, float2 b) { return NC == 1 ? make_float2(__fadd_rn(a.x, b.x), 0.0f) : df::vadd(a, b); };
    auto vmul = [](float2 a, float2 b) { return NC == 1 ? make_float2(__fmul_rn(a.x, b.x), 0.0f) : df::vmul(a, b); };
    auto vfma = [](float2 a, float2 b, float2 c) {
        return NC == 1 ? make_float2(__fmaf_rn(a.x, b.x, c.x), 0.0f) : df::vfma(a, b, c);
    };
    constexpr bool kDF = SM::kDF, AHEAD = SM::ahead(TAU1);
    constexpr int NP = SM::NP, kHalo = SM::kHalo, kRing = SM::kRing, kLag = kDF ? 1 : 2;
    constexpr int CW = NP * kT;  // a ring slot
    auto one = [](int p) { return 2 * p + 1 == NC; };  // an odd last component
    extern __shared__ __align__(16) unsigned char smem[];
    float2 *RS = (float2 *)smem;                              // [kRing][NP][kT] rho hi rows
    float4 *GS = (float4 *)(RS + kRing * CW);                 // [NP][kT] grad mu of row q
    float2 *MU = (float2 *)((unsigned char *)GS + SM::g());   // [3][NP][kT] mu rows (binary32)
    float2 *XC = (float2 *)((unsigned char *)MU + SM::mu());  // [6][NP][kT] exchange
    float2 *JS = XC + 6 * CW;                                 // [kT] momentum of row q
    float2 *VS = JS + kT;                                     // [8][kT] AHEAD: old populations of a pair
    float *XJ = (float *)(VS + (AHEAD ? 8 * kT : 0));         // [6][kT]
    float *PS = XJ + 6 * kT;                                  // [3][kT] psi rows (binary32)
    const void *__restrict__ gin = in.g;
    void *__restrict__ gout = out.g;
    const void *__restrict__ rhin = in.rhi;
    const void *__restrict__ rlin = in.rlo;
    void *__restrict__ rhout = out.rhi;
    void *__restrict__ rlout = out.rlo;
    const float2 *__restrict__ jin = in.j;
    float2 *__restrict__ jout = out.j;

    const int nx = P.nx, ny = P.ny;
    const long long N = P.N;
    const int x0 = blockIdx.x * W;
    const int w = min(W, nx - x0);
    const int y0 = blockIdx.y * H;
    const int h = min(H, ny - y0);
    const int t = threadIdx.x;
    const int c = t - kHalo;  // column of this thread
    const bool loads = c < w + kHalo;
    const bool active = c >= -1 && c <= w;
    const bool interior = c >= 0 && c < w;
    // node offsets are unsigned: a box has at most 4e9 nodes
    const unsigned xg = (unsigned)wrapc(x0 + c, nx);
    const unsigned xl = xg == 0 ? nx - 1 : xg - 1, xr = xg + 1 == (unsigned)nx ? 0 : xg + 1;
    const float2 m1 = vbc(-1.0f);

    // (hi, lo) += x and -= x by Fast2Sum, two components at once
    auto arrive = [&](float2 &hi, float2 &lo, float2 x) {
        const float2 s = vadd(hi, x);
        lo = vadd(lo, vfma(vfma(hi, m1, s), m1, x));
        hi = s;
    };
    auto leave = [&](float2 &hi, float2 &lo, float2 x) {
        const float2 s = vfma(x, m1, hi);
        lo = vfma(vadd(vfma(hi, m1, s), x), m1, lo);
        hi = s;
    };
    auto row = [&](int y) { return (unsigned)wrapc(y, ny) * (unsigned)nx; };
    // asynchronous copies of the thread's own column
    auto copy_density = [&](int y, int slot) {
        if (!loads) return;
        const unsigned o = row(y) + xg;
        float2 *dst = RS + slot * CW + t;
#pragma unroll
        for (int p = 0; p < NP; ++p) copy_pair(dst + p * kT, rhin, one(p), p, N, o);
    };
    auto copy_collision = [&](int y) {
        if (!active) return;
        const unsigned o = row(y) + xg;
        copy_async<8>(JS + t, jin + o);
        if constexpr (kDF) {
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                if (one(p)) copy_async<8>(GS + p * kT + t, (const float2 *)(mug + p * N) + o);
                else copy_async<16>(GS + p * kT + t, mug + p * N + o);
            }
        }
    };

    // the old populations of a pair, one pair ahead of its collision
    auto copy_populations = [&](int p, unsigned o) {
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            if (one(p)) copy_async<4>(VS + a * kT + t, (const float *)gin + (16LL * p + a) * N + o);
            else copy_async<8>(VS + a * kT + t, (const float2 *)gin + (8LL * p + a) * N + o);
        }
    };

    // an odd last component shares its operations with a zero: the copies leave its words
    // in the density rows alone
    if constexpr (NC & 1) {
#pragma unroll
        for (int k = 0; k < kRing; ++k) RS[k * CW + (NP - 1) * kT + t].y = 0.0f;
    }
    if (!loads)  // columns beyond the strip feed psi rows only
#pragma unroll
        for (int p = 0; p < kRing * NP; ++p) RS[p * kT + t] = vbc(0.0f);
    copy_density(y0 - kHalo, 0);
    float2 aH[NP], aL[NP], bH[NP], bL[NP];  // density pairs being updated: rows q-1, q
    float2 nL[NP];                          // lo of row q+1
    float2 ja = vbc(0.0f), jb = vbc(0.0f);  // momentum being gathered: rows q-1, q
#pragma unroll
    for (int p = 0; p < NP; ++p) aH[p] = aL[p] = bH[p] = bL[p] = nL[p] = vbc(0.0f);

    const int nrows = h + 2 * kHalo;
    for (int kk = 0; kk < nrows; ++kk) {
        const int k = y0 - kHalo + kk;
        const int crow = k - kLag;
        const bool collide = kk >= 2 * kLag;
        copy_async_wait();
        if constexpr (kDF) {
            // row k+1 into the slot of row k-3, which no thread reads any more
            if (kk + 1 < nrows) copy_density(k + 1, (kk + 1) % kRing);
        } else {
            const float2 *R = RS + (kk % kRing) * CW + t;
            float ps = 0.0f;
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const float2 v = R[p * kT];
                ps = fmaf(P.sqk[2 * p], v.x * P.invM[2 * p], ps);
                if (2 * p + 1 < NC) ps = fmaf(P.sqk[2 * p + 1], v.y * P.invM[2 * p + 1], ps);
            }
            PS[(kk % 3) * kT + t] = ps;
        }
        __syncthreads();
        // ---- binary32 thermodynamics: mu of row k-1 on columns -2 .. W+1 ---------------
        if constexpr (!kDF) {
            if (kk >= 2 && c >= -2 && c <= w + 1) {
                const float *p0 = PS + ((kk + 1) % 3) * kT + t;  // row k-2
                const float *p1 = PS + ((kk + 2) % 3) * kT + t;  // row k-1
                const float *p2 = PS + (kk % 3) * kT + t;        // row k
                float rm[NC], lf[NC];
                const float2 *R = RS + ((kk + 3) % kRing) * CW + t;
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    const float2 v = R[p * kT];
                    rm[2 * p] = v.x * P.invM[2 * p];
                    if (2 * p + 1 < NC) rm[2 * p + 1] = v.y * P.invM[2 * p + 1];
                }
                pr_lnf_v<NC, float>(View32{P}, rm, lf, nullptr);
                const float c0 = p1[0];
                const float faces = (p1[1] - c0) + (p1[-1] - c0) + (p2[0] - c0) + (p0[0] - c0);
                const float diags = (p2[1] - c0) + (p0[-1] - c0) + (p0[1] - c0) + (p2[-1] - c0);
                const float lap = 6.0f * fmaf(1.0f / 9.0f, faces, (1.0f / 36.0f) * diags);
                float2 *M = MU + ((kk + 2) % 3) * CW + t;
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    float2 v;
                    v.x = fmaf(P.RT, lf[2 * p], -P.sqk[2 * p] * lap);
                    v.y = 2 * p + 1 < NC ? fmaf(P.RT, lf[2 * p + 1], -P.sqk[2 * p + 1] * lap) : 0.0f;
                    M[p * kT] = v;
                }
            }
            __syncthreads();
        }
        const int s1 = (kk + kRing - kLag) % kRing;  // slot of row q
        float2 own2[NP], jn = vbc(0.0f);             // what arrives in row q+1 from below
        if (collide && active) {
            // 12 grad X from three rows: faces 4, diagonals 1
            auto grad12 = [&](const float2 *r0, const float2 *r1, const float2 *r2, float2 &Gx, float2 &Gy) {
                const float2 dE = vfma(r1[-1], m1, r1[1]), dN = vfma(r0[0], m1, r2[0]);
                const float2 ne = vfma(r0[-1], m1, r2[1]), se = vfma(r2[-1], m1, r0[1]);
                Gx = vfma(vbc(4.0f), dE, vadd(ne, se));
                Gy = vfma(vbc(4.0f), dN, vfma(se, m1, ne));
            };
            const float2 *R0 = RS + ((s1 + kRing - 1) % kRing) * CW + t;
            const float2 *R1 = RS + s1 * CW + t;
            const float2 *R2 = RS + ((s1 + 1) % kRing) * CW + t;
            const float2 jq = JS[t];
            // Eq. (5): f_i ~ -rho~_i grad mu_i
            float2 fx[NP], fy[NP], Fsx = vbc(0.0f), Fsy = vbc(0.0f), rs = vbc(0.0f);
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const float2 ri = R1[p * kT];
                rs = vadd(rs, ri);
                const float2 cr = vfma(P.cf[p], ri, vmul(P.cfl[p], ri));
                float2 gx, gy;
                if constexpr (kDF) {
                    if (one(p)) {
                        const float2 g = *(const float2 *)(GS + p * kT + t);
                        gx = make_float2(g.x, 0.0f);
                        gy = make_float2(g.y, 0.0f);
                    } else {
                        const float4 g = GS[p * kT + t];
                        gx = make_float2(g.x, g.y);
                        gy = make_float2(g.z, g.w);
                    }
                } else {
                    const int q1 = (kk + 1) % 3;  // mu row q = k-2
                    grad12(MU + ((q1 + 2) % 3) * CW + p * kT + t, MU + q1 * CW + p * kT + t,
                           MU + ((q1 + 1) % 3) * CW + p * kT + t, gx, gy);
                }
                fx[p] = vmul(cr, gx);
                fy[p] = vmul(cr, gy);
                Fsx = vadd(Fsx, fx[p]);
                Fsy = vadd(Fsy, fy[p]);
            }
            const float rt = rs.x + rs.y, Fx = Fsx.x + Fsx.y, Fy = Fsy.x + Fsy.y;
            const float irt = rcp32(rt);
            const float u0 = fmaf(P.cs, Fx, jq.x) * irt;
            const float u1 = fmaf(P.cs, Fy, jq.y) * irt;
            const float h2 = -0.5f * fmaf(u0, u0, u1 * u1);
            if (kk + 1 < nrows) copy_collision(crow + 1);  // G and J of this row are consumed
            const float2 ux = vbc(u0), uy = vbc(u1), hu2 = vbc(h2);
            const bool st = interior && crow >= y0 && crow < y0 + h;
            const unsigned rq = row(crow), rn = row(crow + 1), rsn = row(crow - 1);
            const unsigned rc = rq + xg;
            const unsigned dst[9] = {rc, rq + xr, rq + xl, rn + xg, rsn + xg, rn + xr, rsn + xl, rsn + xr, rn + xl};
            float2 S[TAU1 && NC > 1 ? 1 : 9];  // general tau, one component: collided values summed over the components
            float2 Gsx = vbc(0.0f), Gsy = vbc(0.0f);  // tau = 1: sum of 12 grad rho
            if constexpr (!TAU1)
#pragma unroll
                for (int a = 1; a < 9; ++a) S[a] = vbc(0.0f);
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                float2 v[9];
                if constexpr (!TAU1 && !AHEAD) {
#pragma unroll
                    for (int a = 1; a < 9; ++a) v[a] = load_pair(gin, one(p), p, a - 1, 8, N, rc);
                }
                if constexpr (AHEAD) {
                    if (p > 0) copy_async_wait();
#pragma unroll
                    for (int a = 1; a < 9; ++a) {
                        v[a] = VS[(a - 1) * kT + t];
                        if (one(p)) v[a].y = 0.0f;
                    }
                    if (p + 1 < NP) copy_populations(p + 1, rc);
                    else if (kk + 1 < nrows) copy_populations(0, rn + xg);  // of the next row
                }
                float2 Gx, Gy;
                grad12(R0 + p * kT, R1 + p * kT, R2 + p * kT, Gx, Gy);
                if constexpr (TAU1) {
                    Gsx = vadd(Gsx, Gx);
                    Gsy = vadd(Gsy, Gy);
                }
                const float2 r3 = vfma(vbc(P.so3.x), R1[p * kT], vmul(vbc(P.so3.y), R1[p * kT]));
                const float2 Vx = vfma(r3, ux, fx[p]), Vy = vfma(r3, uy, fy[p]);
                const float2 sg3 = vbc(3.0f * P.sg);
                const float2 Hx = vfma(sg3, Gx, vmul(vbc(1.5f), vadd(Vx, fx[p])));
                const float2 Hy = vfma(sg3, Gy, vmul(vbc(1.5f), vadd(Vy, fy[p])));
                const float2 fu = vfma(fx[p], ux, vmul(fy[p], uy));
                const float2 gu = vmul(vbc(P.sg), vfma(Gx, ux, vmul(Gy, uy)));
                const float2 base = vfma(gu, vbc(-2.0f), vfma(r3, hu2, vmul(fu, m1)));
                const float2 b1 = vfma(gu, vbc(1.5f), base);  // faces: base + K, K = 3/2 G.u
                const float2 qx = vmul(ux, Hx), qy = vmul(uy, Hy);
                float2 *X = XC + p * kT + t;
                auto out1 = [&](int a, float2 g) {  // population a of the pair: Eq. (1a)
                    if constexpr (!TAU1) g = vfma(vbc(P.om1), v[a], g);
                    if constexpr (NC == 1) S[a] = g;
                    else if constexpr (!TAU1) S[a] = vadd(S[a], g);
                    store_pair_if(st, gout, one(p), p, a - 1, 8, N, dst[a], g);
                    leave(bH[p], bL[p], g);
                    const int ex = L::e(a, 0), ey = L::e(a, 1);
                    if (ex != 0) X[((ey + 1) * 2 + (ex > 0 ? 0 : 1)) * CW] = g;
                    else if (ey < 0) arrive(aH[p], aL[p], g);
                    else own2[p] = g;
                };
                const float2 b4 = vmul(vbc(4.0f), b1);
                {
                    const float2 ev = vfma(vbc(4.0f), qx, b4), od = vmul(vbc(4.0f), Vx);
                    out1(1, vadd(ev, od));
                    out1(2, vfma(od, m1, ev));
                }
                {
                    const float2 ev = vfma(vbc(4.0f), qy, b4), od = vmul(vbc(4.0f), Vy);
                    out1(3, vadd(ev, od));
                    out1(4, vfma(od, m1, ev));
                }
                const float2 sd = vadd(vfma(gu, vbc(1.5f), b1), vadd(qx, qy));
                const float2 xy = vfma(ux, Hy, vmul(uy, Hx));
                {
                    const float2 ev = vadd(sd, xy), od = vadd(Vx, Vy);
                    out1(5, vadd(ev, od));
                    out1(6, vfma(od, m1, ev));
                }
                {
                    const float2 ev = vfma(xy, m1, sd), od = vfma(Vy, m1, Vx);
                    out1(7, vadd(ev, od));
                    out1(8, vfma(od, m1, ev));
                }
            }
            float s[9];  // collided values summed over the components
            if constexpr (NC == 1) {
#pragma unroll
                for (int a = 1; a < 9; ++a) s[a] = S[a].x;
            } else if constexpr (TAU1) {
                const float Gx = Gsx.x + Gsx.y, Gy = Gsy.x + Gsy.y, r3 = fmaf(P.so3.x, rt, P.so3.y * rt);
                const float Vx = fmaf(r3, u0, Fx), Vy = fmaf(r3, u1, Fy);
                const float Hx = fmaf(3.0f * P.sg, Gx, 1.5f * (Vx + Fx)), Hy = fmaf(3.0f * P.sg, Gy, 1.5f * (Vy + Fy));
                const float fu = fmaf(Fx, u0, Fy * u1), gu = P.sg * fmaf(Gx, u0, Gy * u1);
                const float b1 = fmaf(-0.5f, gu, fmaf(r3, h2, -fu)), qx = u0 * Hx, qy = u1 * Hy;
                const float ex = 4.0f * (b1 + qx), ey = 4.0f * (b1 + qy), xy = fmaf(u0, Hy, u1 * Hx);
                const float sd = fmaf(1.5f, gu, b1) + (qx + qy), sp = Vx + Vy, sm = Vx - Vy;
                s[1] = fmaf(4.0f, Vx, ex), s[2] = fmaf(-4.0f, Vx, ex);
                s[3] = fmaf(4.0f, Vy, ey), s[4] = fmaf(-4.0f, Vy, ey);
                s[5] = (sd + xy) + sp, s[6] = (sd + xy) - sp;
                s[7] = (sd - xy) + sm, s[8] = (sd - xy) - sm;
            } else {
#pragma unroll
                for (int a = 1; a < 9; ++a) s[a] = S[a].x + S[a].y;
            }
            XJ[0 * kT + t] = s[7];
            XJ[1 * kT + t] = s[6];
            XJ[2 * kT + t] = s[1];
            XJ[3 * kT + t] = s[2];
            XJ[4 * kT + t] = s[5];
            XJ[5 * kT + t] = s[8];
            ja.y -= s[4];
            jn.y = s[3];
        } else if (kk == 2 * kLag - 1) {
            copy_collision(crow + 1);  // of the first row that is collided
            if (AHEAD && active) copy_populations(0, row(crow + 1) + xg);
        }
        __syncthreads();
        if constexpr (!kDF)  // into the slot of row k-3, whose last reader was this collision
            if (kk + 1 < nrows) copy_density(k + 1, (kk + 1) % kRing);
        // ---- what arrives from the neighbouring columns ---------------------------------
        if (collide && interior) {
            const bool write_row = crow - 1 >= y0 && crow - 1 < y0 + h;
            const unsigned rw = row(crow - 1) + xg;
            {
                const float dr = XJ[0 * kT + t - 1], dl = XJ[1 * kT + t + 1];
                const float er = XJ[2 * kT + t - 1], el = XJ[3 * kT + t + 1];
                const float ur = XJ[4 * kT + t - 1], ul = XJ[5 * kT + t + 1];
                ja.x += dr - dl;
                ja.y -= dr + dl;
                if (write_row) jout[rw] = ja;
                ja = make_float2(jb.x + (er - el), jb.y);
                jb = make_float2(ur - ul, jn.y + (ur + ul));
            }
            const float2 *Rn = RS + ((s1 + 1) % kRing) * CW + t;  // row q+1
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const float2 *X = XC + p * kT + t;
                // row q-1 is complete
                arrive(aH[p], aL[p], X[0 * CW - 1]);
                arrive(aH[p], aL[p], X[1 * CW + 1]);
                const float2 hi = vadd(aH[p], aL[p]);
                const float2 lo = vfma(vfma(aH[p], m1, hi), m1, aL[p]);
                store_pair_if(write_row, rhout, one(p), p, 0, 1, N, rw, hi);
                store_pair_if(write_row, rlout, one(p), p, 0, 1, N, rw, lo);
                aH[p] = bH[p];
                aL[p] = bL[p];
                arrive(aH[p], aL[p], X[2 * CW - 1]);
                arrive(aH[p], aL[p], X[3 * CW + 1]);
                bH[p] = Rn[p * kT];
                bL[p] = nL[p];
                arrive(bH[p], bL[p], X[4 * CW - 1]);
                arrive(bH[p], bL[p], own2[p]);
                arrive(bH[p], bL[p], X[5 * CW + 1]);
            }
        }
        // lo of the row that the next iteration starts to update
        if (interior && kk + 1 < nrows && kk + 1 >= 2 * kLag) {
            const unsigned o = row(crow + 2) + xg;
#pragma unroll
            for (int p = 0; p < NP; ++p) nL[p] = load_pair(rlin, one(p), p, N, o);
        }
    }
}

// R(0) = sum_a g_{a,i} for every node (fixed order a = 0..8).
template <int NC, typename S>
__global__ void k_density(const Params P, const S *__restrict__ g, S *__restrict__ R)
{
    const long long N = P.N;
    for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < N;
         r += (long long)gridDim.x * blockDim.x) {
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            S s = 0;
#pragma unroll
            for (int a = 0; a < 9; ++a) s += g[(i * 9 + a) * N + r];
            R[i * N + r] = s;
        }
    }
}

struct Ops {
    int wmax;
    int (*density)(const Params &, StateBufs, cudaStream_t);
    // one step; mu: the gradient buffer of the double-binary32 chemical
    // potentials, [nc][N] (d/dx, d/dy) (LBM_FP32DEV), else unused.  Returns the launches made through *launches.
    int (*step)(const Params &, const df::ParMu &, const FusedGeom &, StateBufs, StateBufs, double *, float2 *mu, int *launches,
                KernelTimer *, cudaStream_t);
    size_t (*smem)(bool tau1, int W);
    int (*occupancy)(bool tau1, size_t smem);  // CTAs per SM of the step kernel that will run
    int (*occupancy_mu)();  // CTAs per SM of the mu pass (0: the form has none)
};

// S = double: binary64 kernel (all populations, binary64 densities).
// S = float:  binary32 kernel with thermodynamics in E (DF64: a mu pass first).
template <int NC, typename S, typename E> struct Impl {
    static constexpr bool k64 = sizeof(S) == 8;
    static constexpr bool kDF = std::is_same<E, DF64>::value;
    static auto kernel(bool tau1)
    {
        if constexpr (k64) return k_fused<NC, double, double>;
        else return tau1 ? k_fused32<NC, E, true> : k_fused32<NC, E, false>;
    }
    static constexpr int wmax()
    {
        if constexpr (k64) return kWmax;
        else return wmax32<E>();
    }
    static int density(const Params &P, StateBufs st, cudaStream_t s)
    {
        if constexpr (k64) {
            long long b = (P.N + 255) / 256;
            if (b > 152 * 32) b = 152 * 32;
            k_density<NC, double><<<(unsigned)b, 256, 0, s>>>(P, (const double *)st.g, st.rhi_d());
        }
        return (int)cudaGetLastError();
    }
    static size_t smem(bool tau1, int W)
    {
        if constexpr (k64) return Smem<NC, double, double>::total(W);
        else return Smem32<NC, E>::total(tau1);
    }
    static int occupancy(bool tau1, size_t bytes)
    {
        // the limit is the widest strip's need, so that problems of other
        // widths launched later keep fitting under it
        if (cudaFuncSetAttribute(kernel(tau1), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem(tau1, wmax())) != cudaSuccess)
            return 0;
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel(tau1), kT, bytes) != cudaSuccess)
            return 0;
        return n;
    }
    static int occupancy_mu()
    {
        if constexpr (kDF) {
            const size_t b = SmemMu<NC>::bytes();
            if (cudaFuncSetAttribute(k_mu32<NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b) != cudaSuccess)
                return 0;
            int n = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_mu32<NC>, kT, b) != cudaSuccess) return 0;
            return n;
        } else {
            return 0;
        }
    }
    static int step(const Params &P, const df::ParMu &pm, const FusedGeom &g, StateBufs in, StateBufs out, double *mp, float2 *mu,
                    int *launches, KernelTimer *kt, cudaStream_t s)
    {
        dim3 grid(g.nstrips, g.segs);
        *launches = 1;
        if constexpr (k64) {
            kt_begin(kt, kKtStep, s);
            k_fused<NC, double, double><<<grid, kT, g.smem, s>>>(
                P, g.strip, g.seg_h, (const double *)in.g, (double *)out.g, in.rhi_d(),
                out.rhi_d(), mp);
            kt_end(kt, s);
        } else {
            if constexpr (kDF) {
                if (!mu) return (int)cudaErrorInvalidValue;
                dim3 mgrid(g.mnstrips, g.msegs);
                const size_t b = SmemMu<NC>::bytes();
                kt_begin(kt, kKtMuPass, s);
                k_mu32<NC><<<mgrid, kT, b, s>>>(pm, g.mstrip, g.mseg_h, in, (float4 *)mu);
                kt_end(kt, s);
                *launches = 2;
            }
            const Par32 q = make_par32(P, kDF);
            auto step32 = kernel(P.omega == 1.0);
            kt_begin(kt, kKtStep, s);
            step32<<<grid, kT, g.smem, s>>>(q, g.strip, g.seg_h, in, out, (const float4 *)mu);
            kt_end(kt, s);
        }
        return (int)cudaGetLastError();
    }
};

template <int NC, typename S, typename E> const Ops *ops_of()
{
    static const Ops o = {Impl<NC, S, E>::wmax(),     &Impl<NC, S, E>::density,
                          &Impl<NC, S, E>::step,      &Impl<NC, S, E>::smem,
                          &Impl<NC, S, E>::occupancy, &Impl<NC, S, E>::occupancy_mu};
    return &o;
}

template <typename S, typename E, int LO, int HI> const Ops *ops_range(int nc)
{
    if constexpr (LO > HI) {
        return nullptr;
    } else {
        if (nc == LO) return ops_of<LO, S, E>();
        return ops_range<S, E, LO + 1, HI>(nc);
    }
}

}  // namespace fz
}  // namespace lbmfug

#define LBM_FZ_TU(NAME, S, E, LO, HI)                                                          \
    namespace lbmfug {                                                                         \
    namespace fz {                                                                             \
    const Ops *NAME(int nc) { return ops_range<S, E, LO, HI>(nc); }                            \
    }                                                                                          \
    }
