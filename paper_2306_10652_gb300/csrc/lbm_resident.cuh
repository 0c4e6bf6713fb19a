// lbm_resident.cuh -- many time steps of a small D2Q9 problem in one launch.
//
// A slab of a few hundred nodes (the paper's 400 x 2 and 128 x 4 interfaces) is
// bound by latency: every kernel of a step costs some 3 us however little it does,
// and a row walk is a serial chain on top.  Here one cluster of CTAs keeps the
// problem: thread (node, component) holds the component's density and populations
// in registers for the whole launch, and a step is three phases with a cluster
// barrier after each (Sec. 2.1, Eqs. 1a-1c, 5; Sec. 2.3, Eqs. 9-12):
//   P2  mu_i from rho_j of the node (lanes of the node's group) and lap psi
//   P3  F_i, grad rho_i, u = (j + F/2)/rho, collision, push
//   P4  the arrived populations: new density, j, psi
// A node's components are G consecutive lanes of a warp (G the power of two >= Nc),
// so sums over components are butterflies and the rows of T_i take rho_j by
// shuffles.  What neighbours need (rho, mu, psi and the pushed populations, [node][G])
// goes through a scratch area that stays in L2, stored and loaded past L1.  Every
// buffer has one write phase and one read phase per step with a barrier between
// them in either order.
//
// Arithmetic by form: float (LBM_FP32), double (LBM_FP64), df::F2 (LBM_FP32DEV:
// double-binary32 thermodynamics, binary32 collision, exact density pairs), with
// the equations in the forms of the other kernels.
// Per step: 400 x 2, Nc = 10, LBM_FP32 6.6 us (the fused kernel in a graph: 14.4 us),
// LBM_FP32DEV 8.7 us (18.8 us); 128 x 4, Nc = 2, LBM_FP64 8.6 us (three passes:
// 16.9 us).  The floor, at a few hundred threads, is 2.4-3 us: three barriers and
// the L2 round trips around them.
#pragma once

#include "lbm_internal.h"

namespace lbmfug {
namespace rs {

constexpr int kMaxCluster = 16;

// Constants (a kernel argument); tables indexed [j * kMaxNc + i] so that the lanes
// of a group read neighbouring words.
template <typename E> struct Real { using T = E; };   // type of mu and psi
template <> struct Real<df::F2> { using T = float2; };

struct Par {
    int nx, ny, nc, steps;
    int N;
    double omega, RT;
    double2 iRT, c2;      // 1 / RT and -1 / (sqrt2 RT) as unevaluated sums,
    float2 fiRT, fc2;     // in binary32
    const Par64 *p64;     // device copies: binary64 constants,
    const df::ParMu *pm;  // double-binary32 constants
    const df::MuTab *mtab;
    const Log64 *ltab;
};

// scratch of one problem
struct Work {
    void *rho, *mu, *psi, *g;
};

__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int G, typename T> __device__ __forceinline__ T bfly(T v)
{
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, 32);
    return v;
}
template <int G> __device__ __forceinline__ df::F2 bfly(df::F2 v)
{
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1)
        v = df::add(v, {__shfl_xor_sync(0xffffffffu, v.hi, o, 32), __shfl_xor_sync(0xffffffffu, v.lo, o, 32)});
    return v;
}
template <int G> __device__ __forceinline__ float bfly_max(float v)
{
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o, 32));
    return v;
}

// (binary32: the chain of a step hides most of logf, and __logf, whose absolute error is
// 2^-21.4, is the largest rounding of mu: 400 x 2, Nc = 10, 200 steps, error of the
// densities 5.3e-8 with logf, 1.1e-7 with __logf, at 6.6 and 6.3 us per step)
__device__ __forceinline__ float lane_log(float x, const Log64 *) { return logf(x); }
__device__ __forceinline__ double lane_log(double x, const Log64 *t) { return log64(x, t); }
__device__ __forceinline__ float lane_rcp(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ double lane_rcp(double x) { return rcp64(x); }

// ---- thermodynamics of a lane --------------------------------------------------
// mu_i / (M_i RT) up to a constant, and psi: binary32 and binary64 (PrNode of
// lbm_core.cuh with the components in lanes).
template <int G, typename E> struct Thermo {
    E bM, invM, kM, pk;
    const E *A;  // shared, [j][G]
    const Log64 *tab;
    __device__ __forceinline__ void init(const Par &P, int i, E *sh, float4 *, float2 *)
    {
        const Par64 &q = *P.p64;
        const bool on = i < P.nc;
        bM = on ? (E)q.bM[i] : (E)0;
        invM = on ? (E)q.invM[i] : (E)0;
        kM = on ? (E)q.kM[i] : (E)0;
        pk = on ? (E)q.pk[i] : (E)0;
        tab = P.ltab;
        for (int k = threadIdx.x; k < G * G; k += blockDim.x) {
            const int j = k / G, c = k % G;
            sh[k] = j < P.nc && c < P.nc ? (E)q.A[c * kMaxNc + j] : (E)0;
        }
        A = sh + i;
    }
    __device__ __forceinline__ E psi(E r, float, float) const { return bfly<G>(pk * r); }
    template <typename At> __device__ __forceinline__ E mu(const Par &P, bool on, E r, float, float, At psi_at) const
    {
        const E kS2 = (E)1.4142135623730951;
        const E c0 = psi_at(0);
        const E faces = (psi_at(1) - c0) + (psi_at(2) - c0) + (psi_at(3) - c0) + (psi_at(4) - c0);
        const E diags = (psi_at(5) - c0) + (psi_at(6) - c0) + (psi_at(7) - c0) + (psi_at(8) - c0);
        const E lap = (E)6 * fma((E)(1.0 / 9.0), faces, (E)(1.0 / 36.0) * diags);
        const E B = bfly<G>(bM * r), rho = bfly<G>(invM * r);
        E T = 0;
        for (int j = 0; j < P.nc; ++j) T = fma(A[j * G], __shfl_sync(0xffffffffu, r, j, G), T);
        const E Q = bfly<G>(r * T);
        const E omB = (E)1 - B, den = fma(B, (E)2 - B, (E)1);
        const E u = lane_rcp(B), vb = lane_rcp(omB), vd = lane_rcp(den);
        const E n1 = fma((E)1 + kS2, B, (E)1), n2 = fma((E)1 - kS2, B, (E)1), w = n1 * vd;
        E q = n1 * w;
        q = fma(fma(-q, n2, n1), w, q);
        const E Lu = lane_log(q, tab) * u;
        const E C0 = -lane_log(omB, tab);
        const E qu = Q * u;
        E iRT, iRTl, c2, c2l;
        if constexpr (sizeof(E) == 8)
            iRT = P.iRT.x, iRTl = P.iRT.y, c2 = P.c2.x, c2l = P.c2.y;
        else
            iRT = P.fiRT.x, iRTl = P.fiRT.y, c2 = P.fc2.x, c2l = P.fc2.y;
        const E C1 = fma(fma(qu, iRT, qu * iRTl), fma((E)0.5 / kS2, Lu, -vd), rho * vb);
        const E C2 = fma(Lu, c2, Lu * c2l);
        const E lr = lane_log(on ? r : (E)1, tab);
        return fma(invM, lr + C0, fma(bM, C1, fma(T, C2, -kM * lap)));
    }
    static __device__ __forceinline__ E diff(E a, E b) { return a - b; }
};

// mu_i up to a constant in double-binary32 (MuNode of lbm_thermo_df.cuh with the
// components in lanes).
template <int G> struct Thermo<G, df::F2> {
    df::F2 bM, iM, b, k6, pk, RT, c1, c2;
    float CT;
    const float2 *A;  // shared, [j][G]
    const float4 *tv;
    const float2 *tk;
    __device__ __forceinline__ void init(const Par &P, int i, float2 *sh, float4 *shv, float2 *shk)
    {
        const df::ParMu &q = *P.pm;
        auto get = [&](const float4 *a) -> df::F2 {
            const float4 v = a[i / 2];
            return i < P.nc ? (i & 1 ? df::F2{v.y, v.w} : df::F2{v.x, v.z}) : df::F2{0.0f, 0.0f};
        };
        const float4 pb = i < P.nc ? q.PB[i] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        pk = {pb.x, pb.z};
        bM = {pb.y, pb.w};
        iM = get(q.iM);
        b = get(q.b);
        k6 = get(q.k6);
        RT = df::f2(q.RT);
        c1 = df::f2(q.c1);
        c2 = df::f2(q.c2);
        CT = i < P.nc ? (i & 1 ? q.CT[i / 2].y : q.CT[i / 2].x) : 0.0f;
        for (int k = threadIdx.x; k < G * G; k += blockDim.x) {
            const int j = k / G, c = k % G;
            const float4 v = q.A[c / 2 * kMaxNc + j];
            sh[k] = j < P.nc && c < P.nc ? (c & 1 ? make_float2(v.y, v.w) : make_float2(v.x, v.z))
                                         : make_float2(0.0f, 0.0f);
        }
        A = sh + i;
        df::load_mu_tab(P.mtab, shv, shk);
        tv = shv;
        tk = shk;
    }
    __device__ __forceinline__ float2 psi(float, float h, float l) const
    {
        const df::F2 v = bfly<G>(df::mul(pk, {h, l}));
        return make_float2(v.hi, v.lo);
    }
    template <typename At>
    __device__ __forceinline__ float2 mu(const Par &P, bool on, float, float h, float l, At psi_at) const
    {
        using namespace df;
        constexpr double kS2 = 1.41421356237309504880168872421;
        const F2 lap = lap9x6(psi_at(0), psi_at(1), psi_at(2), psi_at(3), psi_at(4), psi_at(5), psi_at(8), psi_at(7),
                              psi_at(6));
        const F2 x = {h, l};
        const F2 B = bfly<G>(df::mul(bM, x)), y = df::mul(iM, x), rho = bfly<G>(y);
        // T_i from a bound on its terms (see lbm_thermo_df.cuh)
        float C = __fmul_rn(CT, bfly_max<G>(__fmul_rn(bM.hi, h)));
        const float C12 = __fmul_rn(C, 4097.0f);
        C = __fsub_rn(C12, __fsub_rn(C12, C));
        float s = C, c = 0.0f;
        for (int j = 0; j < P.nc; ++j) {
            const float2 a = A[j * G];
            const float xh = __shfl_sync(0xffffffffu, h, j, G), xl = __shfl_sync(0xffffffffu, l, j, G);
            const float t = fmaf(a.x, xh, s);
            c = __fadd_rn(c, fmaf(a.x, xl, fmaf(a.y, xh, fmaf(a.x, xh, __fsub_rn(s, t)))));
            s = t;
        }
        const F2 T = fast_two_sum(__fsub_rn(s, C), c);
        const F2 Q = bfly<G>(df::mul(y, T));
        const F2 omB = one_plus(neg(B));
        const F2 tmB = fast_two_sum(2.0f, -B.hi);
        const F2 den = one_plus(df::mul(B, {tmB.hi, __fsub_rn(tmB.lo, B.lo)}));
        const F2 n1 = df::add(df::mul(B, {hi_of(1.0 + kS2), lo_of(1.0 + kS2)}), {1.0f, 0.0f});
        const F2 u = rcp(B), w = rcp(den), vb = rcp(omB);
        // RT ln of rho_i / (1 - B) and of the ratio in Lr, in the two lanes of a packed evaluation
        const F2 ra = df::mul(df::mul(n1, n1), w), xv = df::mul(on ? x : F2{1.0f, 0.0f}, vb);
        Sum2 lg = rtlog(RT, tv, tk, {make_float2(xv.hi, ra.hi), make_float2(xv.lo, ra.lo)});
        const F2 Lu = df::mul(lane_y(lg.value()), u);
        const F2 RC1 = df::add(df::mul(df::mul(RT, rho), vb),
                               df::mul(df::mul(Q, u), df::add(df::mul(Lu, c1), neg(w))));
        const F2 RC2 = df::mul(Lu, c2);
        // b_i RC1 beside -sqrt(kappa_i) lap psi, then T_i RC2
        lg.s.y = lg.c.y = lg.l.y = 0.0f;
        lg.two_sum(mul_u({make_float2(b.hi, k6.hi), make_float2(b.lo, k6.lo)},
                         {make_float2(RC1.hi, lap.hi), make_float2(RC1.lo, lap.lo)}));
        lg.two_sum(mul_u({make_float2(T.hi, 0.0f), make_float2(T.lo, 0.0f)},
                         {make_float2(RC2.hi, 0.0f), make_float2(RC2.lo, 0.0f)}));
        const P2 v = lg.value();
        const F2 m = df::add(lane_x(v), lane_y(v));
        return make_float2(m.hi, m.lo);
    }
    static __device__ __forceinline__ float diff(float2 a, float2 b) { return (a.x - b.x) + (a.y - b.y); }
};

// S: type of the populations and of the collision; MAXT: threads per CTA at most
// (512 leaves a thread 128 registers)
template <int G, typename E, bool TAU1, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_resident(const Par P, StateBufs st, const Work W)
{
    using L = Lattice<0>;
    using S = typename std::conditional<std::is_same<E, double>::value, double, float>::type;
    using R = typename Real<E>::T;  // type of mu and psi
    constexpr bool kDF = std::is_same<E, df::F2>::value;
    constexpr bool k64 = sizeof(S) == 8;
    __shared__ R shA[G * G];
    __shared__ float4 shv[kDF ? 128 : 1];
    __shared__ float2 shk[kDF ? 512 : 1];
    const int item = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = item & (G - 1);
    const bool here = item / G < P.N, on = here && i < P.nc;
    const int n = here ? item / G : 0;
    const long long N = P.N;
    int nb[9];
    {
        const int x = n % P.nx, y = n / P.nx;
#pragma unroll
        for (int a = 0; a < 9; ++a) {
            const int xx = x + L::e(a, 0), yy = y + L::e(a, 1);
            nb[a] = (xx < 0 ? xx + P.nx : xx >= P.nx ? xx - P.nx : xx) +
                    P.nx * (yy < 0 ? yy + P.ny : yy >= P.ny ? yy - P.ny : yy);
        }
    }
    Thermo<G, E> th;
    th.init(P, i, shA, shv, shk);
    S *rho = (S *)W.rho + i;
    R *mu = (R *)W.mu + i;
    R *psi = (R *)W.psi;
    S *gx = (S *)W.g + i;  // [8][N][G]
    const S om = TAU1 ? (S)1 : (S)P.omega, om1 = (S)1 - om;
    const S sf = (S)((1.0 - 0.5 * (TAU1 ? 1.0 : P.omega)) / 36.0), sg = sf / (S)12;
    // w/12 in two words in binary32: one is off by up to 2^-25, the same in every step, and so
    // would be the momentum that a step hands on
    const double w12 = (TAU1 ? 1.0 : P.omega) / 12.0;
    const S so3 = (S)w12, so3l = k64 ? (S)0 : (S)(w12 - (double)so3);
    const S cs = (S)0.5 / ((S)3 * sf);
    // f_i from 12 grad(mu): mu / (M RT) for binary32 and binary64, mu for double-binary32
    const S cf = kDF ? (S)(-0.25) * sf * (S)(on ? P.p64->invM[i] : 0.0) : (S)(-0.25 * P.RT) * sf;

    // the thread's own state
    S v[9];               // arrived populations (binary32: v[0] unused)
    S r = 0;              // density (binary32: the pair's hi)
    float lo = 0.0f;
    S jx, jy, rt;         // momentum and total density of the node
    const S *__restrict__ gin = (const S *)st.g;
    constexpr int NS = k64 ? 9 : 8;
#pragma unroll
    for (int a = 0; a < 9; ++a) v[a] = on && (k64 || a > 0) ? gin[((long long)i * NS + a - (9 - NS)) * N + n] : (S)0;
    if (on && !k64) {
        r = (S)st.rhi_f()[i * N + n];
        lo = st.rlo[i * N + n];
    }
    // density (binary64), momentum, psi and total density of a state
    auto close = [&]() {
        if constexpr (k64) {
            r = v[1];  // (the resting one last, see k_sums)
#pragma unroll
            for (int a = 2; a < 9; ++a) r += v[a];
            r = v[0] + r;
        }
        jx = bfly<G>((v[1] - v[2]) + (v[5] - v[6]) + (v[7] - v[8]));
        jy = bfly<G>((v[3] - v[4]) + (v[5] - v[6]) + (v[8] - v[7]));
        rt = bfly<G>(r);
        const R ps = th.psi(r, (float)r, lo);
        if (on) __stcg(rho + n * G, r);
        if (here && i == 0) __stcg(psi + n, ps);
    };
    __syncthreads();
    close();
    cluster_barrier();
    for (int s = 0; s < P.steps; ++s) {
        // (the neighbours' addresses are formed anew each step: kept, they would
        // take more registers than a thread has)
#pragma unroll
        for (int a = 0; a < 9; ++a) asm volatile("" : "+r"(nb[a]));
        // P2
        const R m = th.mu(P, on, r, (float)r, lo, [&](int a) { return __ldcg(psi + nb[a]); });
        if (on) __stcg(mu + n * G, m);
        cluster_barrier();
        // P3: the quadratic form in e of lbm_threepass.cuh / lbm_multipass.cuh
        S fx = 0, fy = 0, Gx = 0, Gy = 0;
        if (on) {
            S d[9], q[9];
#pragma unroll
            for (int a = 1; a < 9; a += 2) {
                d[a] = Thermo<G, E>::diff(__ldcg(mu + nb[a] * G), __ldcg(mu + nb[a + 1] * G));
                q[a] = __ldcg(rho + nb[a] * G) - __ldcg(rho + nb[a + 1] * G);
            }
            const S c = cf * r;
            fx = c * fma((S)4, d[1], d[5] + d[7]);
            fy = c * fma((S)4, d[3], d[5] - d[7]);
            Gx = fma((S)4, q[1], q[5] + q[7]);
            Gy = fma((S)4, q[3], q[5] - q[7]);
        }
        const S Fx = bfly<G>(fx), Fy = bfly<G>(fy);
        S irt;
        if constexpr (k64) irt = rcp64(rt);
        else irt = rcp32(rt);
        const S ux = fma(cs, Fx, jx) * irt, uy = fma(cs, Fy, jy) * irt;
        if (on) {
            const S hu2 = (S)(-0.5) * fma(ux, ux, uy * uy);
            const S r3 = k64 ? so3 * r : fma(so3, r, so3l * r);
            const S Vx = fma(r3, ux, fx), Vy = fma(r3, uy, fy);
            const S Hx = fma((S)3 * sg, Gx, (S)1.5 * (Vx + fx)), Hy = fma((S)3 * sg, Gy, (S)1.5 * (Vy + fy));
            const S fu = fma(fx, ux, fy * uy), gu = sg * fma(Gx, ux, Gy * uy);
            const S base = fma((S)(-2), gu, fma(r3, hu2, -fu));
            const S b1 = fma((S)1.5, gu, base);
            const S qx = ux * Hx, qy = uy * Hy, xy = fma(ux, Hy, uy * Hx);
            const S sd = fma((S)1.5, gu, b1) + (qx + qy), sp = Vx + Vy, sm = Vx - Vy;
            const S ex = (S)4 * (b1 + qx), ey = (S)4 * (b1 + qy);
            S g[9];
            g[1] = fma((S)4, Vx, ex), g[2] = fma((S)(-4), Vx, ex);
            g[3] = fma((S)4, Vy, ey), g[4] = fma((S)(-4), Vy, ey);
            g[5] = (sd + xy) + sp, g[6] = (sd + xy) - sp;
            g[7] = (sd - xy) + sm, g[8] = (sd - xy) - sm;
            if constexpr (k64) v[0] = fma((S)16, base, TAU1 ? r : fma(om, r - v[0], v[0]));
#pragma unroll
            for (int a = 1; a < 9; ++a) {
                if (!TAU1) g[a] = fma(om1, v[a], g[a]);
                if constexpr (!k64) pair_acc(r, lo, -g[a]);
                __stcg(gx + ((a - 1) * P.N + nb[a]) * G, g[a]);
            }
        }
        cluster_barrier();
        // P4
        if (on) {
#pragma unroll
            for (int a = 1; a < 9; ++a) v[a] = __ldcg(gx + ((a - 1) * P.N + n) * G);
            if constexpr (!k64) {
#pragma unroll
                for (int a = 1; a < 9; ++a) pair_acc(r, lo, v[a]);
                const float h = r + lo;
                lo = lo - (h - r);
                r = h;
            }
        }
        close();
        cluster_barrier();
    }
    if (on) {
        S *go = (S *)st.g;
#pragma unroll
        for (int a = 9 - NS; a < 9; ++a) go[((long long)i * NS + a - (9 - NS)) * N + n] = v[a];
        if constexpr (!k64) {
            st.rhi_f()[i * N + n] = r;
            st.rlo[i * N + n] = lo;
        }
    }
}

}  // namespace rs
}  // namespace lbmfug
