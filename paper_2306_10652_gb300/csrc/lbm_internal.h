// lbm_internal.h -- host-side interface between the C ABI (lbm_api.cu) and
// the kernel translation units.  Not installed; not part of the ABI.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>
#include <vector>

#include "lbm_core.cuh"
#include "lbm_thermo_df.cuh"

namespace lbmfug {

// Optional CUDA-event timing of the kernels of a step (lbm_timing_enable /
// lbm_timing_read): a launch site records an event before and after its
// launch on the launching stream.  A null timer records nothing.
enum KtSlot : int {
    kKtMuPass = 0,   // k_mu32: double-binary32 chemical potentials and their gradients
    kKtStep,         // k_fused32 / k_fused: the fused step kernel
    kKtMass,         // k_mass32, k_mass_final: monitored mass of a fused step
    kKtMpPsi,        // k_mp_psi
    kKtMpMu,         // k_mp_mu
    kKtMpCollide,    // k_mp_collide
    kKtMpUpdate,     // k_mp_update
    kKtThreePass,    // the three-pass step (k_sums, k_eos, k_collide, k_rupdate)
    kKtResident,     // k_resident: many steps of a small problem in one launch
    kKtMonitor,      // densities and mass of a monitored multi- or three-pass step
    kKtSlots
};
struct KernelTimer {
    struct Rec {
        int slot;
        cudaEvent_t a, b;
        bool a_shared;  // a is the previous record's b (recycled with that record)
    };
    std::vector<cudaEvent_t> pool;  // recycled events
    std::vector<Rec> pending;       // recorded, not yet read
    long long launches[kKtSlots] = {};
    double ms[kKtSlots] = {};
    int open = -1;  // slot between begin and end
    cudaEvent_t open_ev = nullptr;
    bool open_shared = false;
    // The end event of the last timed launch, while nothing else has been
    // enqueued after it: the next begin() takes it as its start event, so
    // back-to-back launches cost one event each.  lbm_step clears it on entry.
    cudaEvent_t last_end = nullptr;
    int err = 0;    // a CUDA error met while recording
    void begin(int slot, cudaStream_t s);
    void end(cudaStream_t s);
    // read every pending pair (their stream has completed) and recycle the events
    int collect();
    void release();
};
inline void kt_begin(KernelTimer *t, int slot, cudaStream_t s)
{
    if (t) t->begin(slot, s);
}
inline void kt_end(KernelTimer *t, cudaStream_t s)
{
    if (t) t->end(s);
}

// Captures what record(stream) enqueues as a graph and instantiates it.  `own` is a
// stream that nobody but the caller's object uses, created here if null: a capture
// belongs to its stream, so on a stream of the user's the launches of other threads
// (and of other handles) made meanwhile would go into this graph instead of running.
// The nodes do not depend on the stream; the graph may be launched on any.  Relaxed
// mode, for the stream and the thread: no call here touches a capture that another
// thread has under way, and none of theirs ends this one.  Returns 0, or -1 with
// *exec null if the work could not be captured.
template <typename Record> int capture_graph(cudaStream_t *own, Record record, cudaGraphExec_t *exec)
{
    *exec = nullptr;
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    if (cudaThreadExchangeStreamCaptureMode(&mode) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    cudaGraph_t g = nullptr;
    bool ok = *own || cudaStreamCreateWithFlags(own, cudaStreamNonBlocking) == cudaSuccess;
    if (ok && cudaStreamBeginCapture(*own, cudaStreamCaptureModeRelaxed) == cudaSuccess) {
        ok = record(*own) == 0;
        ok = cudaStreamEndCapture(*own, &g) == cudaSuccess && ok && g &&
             cudaGraphInstantiate(exec, g, 0) == cudaSuccess;
    } else {
        ok = false;
    }
    if (g) cudaGraphDestroy(g);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (ok) return 0;
    cudaGetLastError();
    *exec = nullptr;
    return -1;
}

// True if work enqueued on `s` would go into a capture of the caller's (or if that
// cannot be told: the launches themselves then report what is wrong).
inline bool being_captured(cudaStream_t s)
{
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusNone) return false;
    cudaGetLastError();
    return true;
}

// Device state of one time level.
//  binary64 storage: g = all Q populations [nc][Q][N] (double); the fused
//    schedule also keeps the densities rhi = [nc][N] (double).
//  binary32 storage: g = the Q-1 moving populations [nc][Q-1][N] (float) and
//    the densities as the pair rhi + rlo ([nc][N] float each); the fused
//    schedule also keeps the momentum j = sum_i sum_a e_a g_{a,i} ([N]).
struct StateBufs {
    void *g = nullptr;
    void *rhi = nullptr;
    float *rlo = nullptr;
    float2 *j = nullptr;
    // binary32, multi-pass and fused schedules: this many components (an even number)
    // are stored in pairs, g[p][a][N][2] and rhi, rlo [p][N][2] (component 2p + k at
    // element k).  An odd last component follows alone, g[a][N] and rhi, rlo [N], which
    // is where it stands without pairs: it shares its packed operations with a zero that
    // no array holds.  (Paired with a stored zero, a state of Nc = 1 took twice its
    // bytes, and that zero turned into NaN with a diverged run.)
    int paired = 0;
    // element of component i, slot a of ns at node r
    __host__ __device__ long long at(int i, int a, int ns, long long N, long long r) const
    {
        return i < paired ? (((long long)(i >> 1) * ns + a) * N + r) * 2 + (i & 1) : ((long long)i * ns + a) * N + r;
    }
    __host__ __device__ long long at(int i, long long N, long long r) const { return at(i, 0, 1, N, r); }
    __host__ __device__ float *rhi_f() const { return (float *)rhi; }
    __host__ __device__ double *rhi_d() const { return (double *)rhi; }
};

// Node o of plane a (of ns) of pair p of components; `one`: an odd last component,
// stored alone, beside a zero.  (A constant where these are called.)
__device__ __forceinline__ float2 load_pair(const void *base, bool one, int p, int a, int ns, long long N, long long o)
{
    if (one) return make_float2(__ldg((const float *)base + (2LL * p * ns + a) * N + o), 0.0f);
    return __ldg((const float2 *)base + ((long long)p * ns + a) * N + o);
}
__device__ __forceinline__ float2 load_pair(const void *base, bool one, int p, long long N, long long o)
{
    return load_pair(base, one, p, 0, 1, N, o);
}
__device__ __forceinline__ void store_pair(void *base, bool one, int p, int a, int ns, long long N, long long o, float2 v)
{
    if (one)
        ((float *)base)[(2LL * p * ns + a) * N + o] = v.x;
    else
        ((float2 *)base)[((long long)p * ns + a) * N + o] = v;
}
__device__ __forceinline__ void store_pair(void *base, bool one, int p, long long N, long long o, float2 v)
{
    store_pair(base, one, p, 0, 1, N, o, v);
}

// Scratch fields of the three-pass schedule (device).
struct ThreePassWork {
    double *rho;  // [nc][N] mass densities rho_i
    double *lnf;  // [nc][N] ln f_i (the step: mu_i / (M_i RT)); followed by psi and lap
    double *psi;  // [N]     psi = sum_j sqrt(kappa_j) rho~_j
    double *lap;  // [N]     lap psi
    double *jm;   // [D][N]  sum_i sum_a e_a g_{a,i} (of a step: null in the other schedules)
    Par64 par;              // constants of the binary64 passes (its table is on the device)
    float *osum;  // [nc][N] binary32 storage: compensated sum of the populations
    float *ocmp;  //         that left each node in the last collision
};

// Fused single-pass D2Q9 schedule: density state and launch geometry.
struct FusedGeom {
    int strip;    // interior columns per CTA
    int nstrips;  // CTAs along x
    int segs;     // CTAs along y
    int seg_h;    // rows per CTA
    int threads;  // threads per CTA
    size_t smem;  // dynamic shared memory bytes
    // the chemical-potential pass of LBM_FP32DEV (0 for the other forms)
    int mstrip, mnstrips, msegs, mseg_h;
};

// All launchers return a cudaError_t cast to int (0 = success).
// Three-pass prec: 0 = binary64 storage, 1 = binary32 deviation storage
// (thermodynamics in binary64).  Fused prec: 0 = binary64, 1 = binary32
// deviation storage with binary64 thermodynamics, 2 = binary32 throughout.
int launch_init_equilibrium(int lat, int prec, int nc, const Params &P, const double *rho,
                            const double *u, StateBufs st, cudaStream_t s);
int launch_threepass_step(int lat, int prec, int nc, const Params &P, StateBufs in, StateBufs out,
                          const ThreePassWork &w, cudaStream_t s);
int threepass_launches_per_step(int lat, int prec, int nc);
// Macroscopic outputs of state st into device buffers (any may be null).
int launch_fields(int lat, int prec, int nc, const Params &P, StateBufs st,
                  const ThreePassWork &w, double *rho, double *u, double *p, double *lnf,
                  cudaStream_t s);
// Populations <-> binary64 post-streaming layout [nc][Q][N].
int launch_state_to_f64(int lat, int prec, int nc, const Params &P, StateBufs st, double *out,
                        cudaStream_t s);
int launch_state_from_f64(int lat, int prec, int nc, const Params &P, const double *in,
                          StateBufs st, cudaStream_t s);

// Fused D2Q9 schedule (lbm_fused2d.cu).  prec as the options: 0 binary64,
// 1 binary32 storage with binary64 thermodynamics, 2 binary32 throughout.
bool fused_supported(int lat, int prec, int nc);
FusedGeom fused_geometry(int prec, int nc, const Params &P, int num_sms, int extra_strips = 0,
                         int seg_mult = 1, int mseg_mult = 1);
FusedGeom fused_geometry_forced(int prec, int nc, const Params &P, int num_sms, int strip, int seg_h);
// binary64 only: densities of the fused state from the populations
int launch_fused_density(int prec, int nc, const Params &P, StateBufs st, cudaStream_t s);
// binary32 only: momentum of the state from its populations
int launch_fused_momentum(int nc, long long N, StateBufs st, cudaStream_t s);
// mu: grad mu_i of LBM_FP32DEV, nc x N (else unused); *launches receives the kernels
// launched.
int launch_fused_step(int prec, int nc, const Params &P, const df::ParMu &pm, const FusedGeom &geo, StateBufs in,
                      StateBufs out, double *mass_partials, float2 *mu, int *launches, KernelTimer *kt,
                      cudaStream_t s);
// Mass of the new state of a monitored fused step into out[nc] (partials: room
// for `parts` partial sums per component; binary64: the step kernel wrote them).
int launch_fused_mass(int prec, int nc, const Params &P, const FusedGeom &geo, StateBufs st, double *partials,
                      int parts, double *out, int *nonfinite, int *launches, cudaStream_t s);

// Binary32 multi-pass schedule of LBM_FP32DEV on any lattice
// (lbm_multipass.cu): psi [N] (hi, lo) of the current state, mu nc x N (hi, lo)
// scratch, jm [D][N] momentum of the current state.
bool multipass_supported(int lat, int prec, int nc, long long N);
int launch_multipass_psi(int lat, int nc, const Params &P, const df::ParMu &pm, StateBufs st, float2 *psi, float *jm,
                         cudaStream_t s);
int launch_multipass_step(int lat, int nc, const Params &P, const df::ParMu &pm, StateBufs in, StateBufs out, float2 *psi,
                          float2 *mu, float *jm, KernelTimer *kt, cudaStream_t s);

// Resident schedule (lbm_resident.cu): `steps` steps of a small D2Q9 problem in
// place, in one launch of a cluster of resident_ctas() CTAs (0: not for this
// problem).  p64, pm (with their tables) are device copies; prec as the options.
int resident_ctas(int lat, int prec, int nc, long long N, bool tau1);
size_t resident_scratch_bytes(int prec, int nc, long long N);
int launch_resident(int prec, int nc, const Params &P, const Par64 *p64, const df::ParMu *pm, const df::MuTab *mtab,
                    const Log64 *ltab, StateBufs st, void *scratch, int ctas, int steps, cudaStream_t s);

// Chemical potentials and forces of a D2Q9 state from its binary64 densities
// (lbm_fields_*.cu).  prec: 0 binary64, 1 double-binary32, 2 binary32
// thermodynamics.  scratch: (nc + 1) * N * 8 bytes; F [nc][2][N], mu [nc][N]
// (mu may be null).
int launch_forces_lo(int prec, int nc, const Params &P, const df::ParMu &pm, const double *rho, void *scratch, double *F,
                     double *mu, cudaStream_t s);
int launch_forces_hi(int prec, int nc, const Params &P, const df::ParMu &pm, const double *rho, void *scratch, double *F,
                     double *mu, cudaStream_t s);

// Deterministic reductions (lbm_reduce.cu).  Partials: [blocks][nc].
constexpr int kReduceBlocks = 1216;  // 8 x 152 SMs
constexpr int kReduceThreads = 256;
int launch_mass(int nc, long long N, const double *rho, double *partials, double *out,
                int *nonfinite, cudaStream_t s);
int launch_maxdiff(int nc, long long N, const double *rho, const double *snap, double *partials,
                   double *out, int *nonfinite, cudaStream_t s);

}  // namespace lbmfug
