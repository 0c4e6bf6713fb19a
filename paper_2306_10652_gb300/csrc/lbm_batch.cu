// lbm_batch.cu -- C ABI of the batched form (lbm_batch_*), its job table,
// the autotuner of the batched kernel and the captured CUDA graph of a round.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <tuple>
#include <vector>

#include "lbm_batch.cuh"
#include "lbmfug.h"

using namespace lbmfug;

namespace lbmfug {
namespace bt {
const Ops *f32_lo(int nc);
const Ops *f32_hi(int nc);
const Ops *f64_lo(int nc);
const Ops *f64_hi(int nc);
}  // namespace bt
}  // namespace lbmfug

struct lbm_batch {
    int nc = 0, njobs = 0, precision = LBM_FP32;
    bt::Shared S{};
    std::vector<bt::Job> jobs;
    std::vector<int> order;  // largest jobs first
    char *device = nullptr;  // one allocation for everything on the device
    char *pinned = nullptr;  // and one that the device writes on the host
    bt::Job *d_jobs = nullptr;
    bt::Status *d_status = nullptr;
    int *d_order = nullptr, *d_work = nullptr, *d_nconv = nullptr;
    int *h_nconv = nullptr;  // pinned
    // pinned, written by the device: a job's status and densities on their way out
    bt::Status *h_status = nullptr;
    double *h_rho = nullptr;
    float *pool = nullptr;
    size_t pool_floats = 0;
    long long maxN = 0;
    Log64 *d_log64 = nullptr;
    std::pair<int, size_t> tuned{0, 0};  // threads and shared memory per CTA that the tuner chose
    const bt::Ops *ops = nullptr;
    int threads = 0, ctas = 0;
    size_t smem = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    cudaStream_t cap = nullptr;  // where a round is captured: the batch's own stream, or one made for it
    cudaGraphExec_t exec = nullptr;
    int graph_steps = -1;
    double graph_tol = -1.0;
    long long launches = 0;
    long long rounds = 0;
};

namespace {

const bt::Ops *lookup(int prec, int nc)
{
    if (nc < 1 || nc > bt::kMaxNcBatch) return nullptr;
    const bool lo = nc <= 5;
    if (prec == LBM_FP32) return lo ? bt::f32_lo(nc) : bt::f32_hi(nc);
    if (prec == LBM_FP32DEV) return lo ? bt::f64_lo(nc) : bt::f64_hi(nc);
    return nullptr;
}

double alpha_of(double a, double b, double omega, double T, double R)
{
    const double Tc = (0.077796074 / 0.457235529) * a / (R * b);  // Sec. 2.3
    double m;
    if (omega <= 0.49)
        m = 0.374640 + 1.54226 * omega - 0.26992 * omega * omega;
    else
        m = 0.379642 + 1.48503 * omega - 0.164423 * omega * omega + 0.016666 * omega * omega * omega;
    const double s = 1.0 + m * (1.0 - std::sqrt(T / Tc));
    return s * s;
}

// autotuner cache: what the best (threads, shared memory) per CTA depends on: device,
// precision, Nc, the kernel (tau = 1 or not), the largest box, jobs per SM (how many CTAs
// should share one, up to four) and how far the boxes fill the largest on average (in
// quarters; smaller ones keep their exchange buffer on chip in less)
using TuneKey = std::tuple<int, int, int, bool, long long, int, int>;
std::mutex g_tune_mutex;
std::map<TuneKey, std::pair<int, size_t>> g_tune_cache;

TuneKey tune_key(const lbm_batch *b)
{
    int dev = 0, nsm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    long long nodes = 0;
    for (const bt::Job &J : b->jobs) nodes += J.N;
    return TuneKey(dev, b->precision, b->nc, b->S.omega == 1.0, b->maxN, std::min((b->njobs + nsm - 1) / nsm, 4),
                   (int)(4 * nodes / (b->njobs * b->maxN)));
}

void release(lbm_batch *b)
{
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->cap && !b->own_stream) cudaStreamDestroy(b->cap);
    cudaFree(b->device);
    if (b->pinned) cudaFreeHost(b->pinned);
    if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
}

int launch_round(lbm_batch *b, int steps, double tol)
{
    if (cudaMemsetAsync(b->d_work, 0, sizeof(int), b->stream) != cudaSuccess) return LBM_ECUDA;
    if (b->ops->launch(b->S, b->d_jobs, b->d_status, b->d_order, b->njobs, b->d_work, steps, tol, b->pool,
                       b->d_nconv, b->ctas, b->threads, b->smem, b->stream))
        return LBM_ECUDA;
    if (cudaMemcpyAsync(b->h_nconv, b->d_nconv, sizeof(int), cudaMemcpyDeviceToHost, b->stream) !=
        cudaSuccess)
        return LBM_ECUDA;
    return LBM_OK;
}

int configure(lbm_batch *b, int threads, size_t want)
{
    int dev = 0, nsm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const bool tau1 = b->S.omega == 1.0;
    size_t smem = std::max(want, b->ops->smem(b->maxN, false));
    int per_sm = b->ops->occupancy(tau1, threads, smem);
    if (per_sm < 1) {
        smem = b->ops->smem(b->maxN, false);
        per_sm = b->ops->occupancy(tau1, threads, smem);
    }
    if (per_sm < 1) return LBM_ENOTSUP;
    b->threads = threads;
    b->smem = smem;
    b->ctas = std::min((long long)nsm * per_sm, (long long)b->njobs);
    return LBM_OK;
}

// Shared memory per CTA worth trying: what the largest job needs without its
// exchange buffer, and a half or all of an SM's, with which the exchange buffers of
// more jobs stay on chip (never more than the largest job can use).
std::vector<size_t> smem_candidates(const lbm_batch *b)
{
    int dev = 0, sm = 0, opt = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&opt, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const size_t lo = b->ops->smem(b->maxN, false), hi = b->ops->smem(b->maxN, true);
    constexpr size_t kStatic = 4096;  // static shared memory and the reserved part of a CTA
    std::vector<size_t> c{lo};
    for (size_t v : {(size_t)sm / 2 - kStatic, (size_t)opt - kStatic}) {
        v = std::min(v, hi) & ~(size_t)15;
        if (v > c.back()) c.push_back(v);
    }
    return c;
}

// Time one short round per candidate on a copy of the state, keep the fastest.
int autotune(lbm_batch *b)
{
    const TuneKey key = tune_key(b);
    {
        std::lock_guard<std::mutex> lock(g_tune_mutex);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end()) {
            b->tuned = it->second;
            return configure(b, b->tuned.first, b->tuned.second);
        }
    }
    float *backup = nullptr;
    bt::Status *sbackup = nullptr;
    if (cudaMalloc(&backup, b->pool_floats * sizeof(float)) != cudaSuccess) return LBM_ENOMEM;
    if (cudaMalloc(&sbackup, b->njobs * sizeof(bt::Status)) != cudaSuccess) {
        cudaFree(backup);
        return LBM_ENOMEM;
    }
    cudaMemcpyAsync(backup, b->pool, b->pool_floats * sizeof(float), cudaMemcpyDeviceToDevice, b->stream);
    cudaMemcpyAsync(sbackup, b->d_status, b->njobs * sizeof(bt::Status), cudaMemcpyDeviceToDevice, b->stream);
    std::pair<int, size_t> best{0, 0};
    float best_ms = 1e30f;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    for (size_t want : smem_candidates(b))
        for (int th : {128, 256, 512, 1024}) {
            if (configure(b, th, want) != LBM_OK || b->smem < want) continue;
            float ms = 0.0f;
            for (int rep = 0; rep < 2; ++rep) {  // the first repetition warms up
                cudaEventRecord(e0, b->stream);
                if (launch_round(b, 20, -1.0) != LBM_OK) break;
                b->launches += 1;
                cudaEventRecord(e1, b->stream);
                cudaEventSynchronize(e1);
                cudaEventElapsedTime(&ms, e0, e1);
            }
            if (ms > 0.0f && ms < best_ms) {
                best_ms = ms;
                best = {th, want};
            }
        }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaMemcpyAsync(b->pool, backup, b->pool_floats * sizeof(float), cudaMemcpyDeviceToDevice, b->stream);
    cudaMemcpyAsync(b->d_status, sbackup, b->njobs * sizeof(bt::Status), cudaMemcpyDeviceToDevice, b->stream);
    cudaMemsetAsync(b->d_nconv, 0, sizeof(int), b->stream);
    cudaStreamSynchronize(b->stream);
    *b->h_nconv = 0;  // the trials' count
    cudaFree(backup);
    cudaFree(sbackup);
    if (!best.first) return LBM_ENOTSUP;
    {
        std::lock_guard<std::mutex> lock(g_tune_mutex);
        g_tune_cache[key] = best;
    }
    b->tuned = best;
    return configure(b, best.first, best.second);
}

int capture(lbm_batch *b, int steps, double tol)
{
    if (b->exec && b->graph_steps == steps && b->graph_tol == tol) return LBM_OK;
    if (b->exec) cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
    if (being_captured(b->stream)) return LBM_ECUDA;  // a run waits for its rounds
    cudaStream_t const user = b->stream;
    if (b->own_stream) b->cap = b->stream;  // nobody else has it
    const int st = capture_graph(
        &b->cap,
        [&](cudaStream_t s) {
            b->stream = s;
            return launch_round(b, steps, tol);
        },
        &b->exec);
    b->stream = user;
    if (st) return LBM_ECUDA;
    b->graph_steps = steps;
    b->graph_tol = tol;
    return LBM_OK;
}

}  // namespace

extern "C" {

int lbm_batch_create(lbm_batch **out, int Nc, const double *a, const double *b, const double *omega,
                     const double *kij, double tau, const lbm_options *opt, const lbm_job *jobs, int njobs)
{
    if (!out) return LBM_EINVAL;
    *out = nullptr;
    if (Nc < 1 || Nc > bt::kMaxNcBatch || !a || !b || !omega || !jobs || njobs < 1) return LBM_EINVAL;
    if (!(tau > 0.5) || !std::isfinite(tau)) return LBM_EINVAL;
    lbm_options o;
    lbm_options_default(&o);
    if (opt) o = *opt;
    if (o.precision == LBM_FP64) o.precision = LBM_FP32DEV;  // the batched form stores binary32
    if (o.precision != LBM_FP32 && o.precision != LBM_FP32DEV) return LBM_EINVAL;
    if (!(o.R > 0.0) || o.kappa_ref_index < 0 || o.kappa_ref_index >= Nc || !(o.kappa_ref >= 0.0))
        return LBM_EINVAL;
    for (int i = 0; i < Nc; ++i) {
        if (!(a[i] > 0.0) || !(b[i] > 0.0) || !std::isfinite(omega[i])) return LBM_EINVAL;
        if (o.M && !(o.M[i] > 0.0)) return LBM_EINVAL;
        if (kij)
            for (int j = 0; j < Nc; ++j)
                if (!(std::fabs(kij[i * Nc + j]) < 1.0) || kij[i * Nc + j] != kij[j * Nc + i] ||
                    (i == j && kij[i * Nc + j] != 0.0))
                    return LBM_EINVAL;
    }
    long long total = 0;
    for (int k = 0; k < njobs; ++k) {
        const lbm_job &J = jobs[k];
        if (J.nx < 1 || J.ny < 1 || !(J.T > 0.0) || !J.rho) return LBM_EINVAL;
        if ((long long)J.nx * J.ny > (1LL << 20)) return LBM_EINVAL;
        unsigned long long bad = 0;  // not positive and finite, on the bit patterns
        for (long long r = 0; r < (long long)Nc * J.nx * J.ny; ++r) {
            unsigned long long u;
            std::memcpy(&u, J.rho + r, 8);
            bad |= u - 1 >= 0x7ff0000000000000ull - 1;
        }
        if (bad) return LBM_EINVAL;
        total += (long long)J.nx * J.ny;
    }
    const bt::Ops *ops = lookup(o.precision, Nc);
    if (!ops) return LBM_ENOTSUP;

    lbm_batch *bt_ = new (std::nothrow) lbm_batch();
    if (!bt_) return LBM_ENOMEM;
    bt_->nc = Nc;
    bt_->njobs = njobs;
    bt_->precision = o.precision;
    bt_->ops = ops;
    bt_->S.nc = Nc;
    bt_->S.omega = 1.0 / tau;
    const double aref = a[o.kappa_ref_index];
    for (int i = 0; i < Nc; ++i) {
        bt_->S.b[i] = b[i];
        bt_->S.invM[i] = 1.0 / (o.M ? o.M[i] : 1.0);
        bt_->S.sqk[i] = std::sqrt(o.kappa_ref * a[i] / aref);  // Eqs. (4), (6)
    }
    // job table and pool: the density pairs [nc][N] hi, lo and the momentum of all
    // jobs (what a new batch fills, one copy), then per job the exchange buffer
    // [nc][8][N] and, at tau != 1, the populations
    const bool tau1 = bt_->S.omega == 1.0;
    bt_->jobs.resize(njobs);
    size_t init_floats = 0;
    for (int k = 0; k < njobs; ++k) {
        const size_t N = (size_t)jobs[k].nx * jobs[k].ny;
        bt::Job &J = bt_->jobs[k];
        std::memset(&J, 0, sizeof(J));
        J.rh = init_floats;
        J.rl = J.rh + Nc * N;
        J.j = (J.rl + Nc * N + 1) & ~1LL;
        init_floats = (J.j + 2 * N + 31) & ~(size_t)31;
    }
    size_t off = init_floats;
    for (int k = 0; k < njobs; ++k) {
        bt::Job &J = bt_->jobs[k];
        J.nx = jobs[k].nx;
        J.ny = jobs[k].ny;
        J.N = (long long)J.nx * J.ny;
        J.x = off;
        off += (size_t)Nc * 8 * J.N;
        J.g = off;
        if (!tau1) off += (size_t)Nc * 8 * J.N;
        off = (off + 31) & ~(size_t)31;
        J.RT = o.R * jobs[k].T;
        D2 iRT, c2;
        rt_constants(J.RT, &iRT, &c2);
        J.iRT = iRT.hi;
        J.iRTl = iRT.lo;
        J.c2 = c2.hi;
        J.c2l = c2.lo;
        double aa[bt::kMaxNcBatch];
        for (int i = 0; i < Nc; ++i) aa[i] = a[i] * alpha_of(a[i], b[i], omega[i], jobs[k].T, o.R);
        for (int i = 0; i < Nc; ++i)
            for (int j = 0; j < Nc; ++j)
                J.A[i * bt::kMaxNcBatch + j] = std::sqrt(aa[i] * aa[j]) * (1.0 - (kij ? kij[i * Nc + j] : 0.0));
        bt_->maxN = std::max(bt_->maxN, J.N);
    }
    bt_->pool_floats = off;
    bt_->order.resize(njobs);
    for (int k = 0; k < njobs; ++k) bt_->order[k] = k;
    std::stable_sort(bt_->order.begin(), bt_->order.end(),
                     [&](int x, int y) { return bt_->jobs[x].N > bt_->jobs[y].N; });
    int st = LBM_OK;
    if (o.stream) {
        bt_->stream = (cudaStream_t)o.stream;
    } else if (cudaStreamCreateWithFlags(&bt_->stream, cudaStreamNonBlocking) == cudaSuccess) {
        bt_->own_stream = true;
    } else {
        st = LBM_ECUDA;
    }
    // parts of the two allocations, 256-byte aligned
    size_t db = 0, hb = 0;
    auto part = [](size_t &at, size_t bytes) {
        const size_t o = at;
        at += (bytes + 255) & ~(size_t)255;
        return o;
    };
    const size_t o_pool = part(db, off * sizeof(float)), o_jobs = part(db, njobs * sizeof(bt::Job)),
                 o_status = part(db, njobs * sizeof(bt::Status)), o_order = part(db, njobs * sizeof(int)),
                 o_work = part(db, sizeof(int)), o_nconv = part(db, sizeof(int)), o_log = part(db, sizeof(Log64));
    const size_t h_nconv = part(hb, sizeof(int)), h_status = part(hb, sizeof(bt::Status)),
                 h_rho = part(hb, (size_t)Nc * bt_->maxN * sizeof(double));
    if (!st && (cudaMalloc(&bt_->device, db) != cudaSuccess ||
                cudaHostAlloc(&bt_->pinned, hb, cudaHostAllocMapped) != cudaSuccess))
        st = LBM_ENOMEM;
    if (!st) {
        bt_->pool = (float *)(bt_->device + o_pool);
        bt_->d_jobs = (bt::Job *)(bt_->device + o_jobs);
        bt_->d_status = (bt::Status *)(bt_->device + o_status);
        bt_->d_order = (int *)(bt_->device + o_order);
        bt_->d_work = (int *)(bt_->device + o_work);
        bt_->d_nconv = (int *)(bt_->device + o_nconv);
        bt_->d_log64 = (Log64 *)(bt_->device + o_log);
        bt_->h_nconv = (int *)(bt_->pinned + h_nconv);
        bt_->h_status = (bt::Status *)(bt_->pinned + h_status);
        bt_->h_rho = (double *)(bt_->pinned + h_rho);
        *bt_->h_nconv = 0;
    }
    if (!st) {
        cudaMemcpyAsync(bt_->d_log64, &log64_host(), sizeof(Log64), cudaMemcpyHostToDevice, bt_->stream);
        bt_->S.log64 = bt_->d_log64;
        cudaMemcpyAsync(bt_->d_jobs, bt_->jobs.data(), njobs * sizeof(bt::Job), cudaMemcpyHostToDevice, bt_->stream);
        cudaMemcpyAsync(bt_->d_order, bt_->order.data(), njobs * sizeof(int), cudaMemcpyHostToDevice, bt_->stream);
        cudaMemsetAsync(bt_->d_status, 0, njobs * sizeof(bt::Status), bt_->stream);
        cudaMemsetAsync(bt_->d_nconv, 0, sizeof(int), bt_->stream);
        // at rest: the exact density pairs, no momentum, no populations
        std::unique_ptr<float[]> init(new (std::nothrow) float[init_floats]());
        if (!init) st = LBM_ENOMEM;
        for (int k = 0; !st && k < njobs; ++k) {
            const bt::Job &J = bt_->jobs[k];
            float *hi = init.get() + J.rh, *lo = init.get() + J.rl;
            const double *rho = jobs[k].rho;
            for (long long r = 0; r < Nc * J.N; ++r) {
                hi[r] = (float)rho[r];
                lo[r] = (float)(rho[r] - (double)hi[r]);
            }
            if (!tau1) cudaMemsetAsync(bt_->pool + J.g, 0, (size_t)Nc * 8 * J.N * sizeof(float), bt_->stream);
        }
        if (!st)
            cudaMemcpyAsync(bt_->pool, init.get(), init_floats * sizeof(float), cudaMemcpyHostToDevice, bt_->stream);
        if (cudaStreamSynchronize(bt_->stream) != cudaSuccess || cudaGetLastError() != cudaSuccess) st = LBM_ECUDA;
    }
    if (!st) st = autotune(bt_);
    if (st) {
        release(bt_);
        delete bt_;
        return st;
    }
    *out = bt_;
    return LBM_OK;
}

int lbm_batch_run(lbm_batch *b, long long max_steps, int check_every, double tol, int *n_converged)
{
    if (!b || check_every < 1 || max_steps < 0 || !(tol >= 0.0)) return LBM_EINVAL;
    int st = capture(b, check_every, tol);
    if (st) return st;
    long long done = 0;
    for (;;) {
        if (cudaStreamSynchronize(b->stream) != cudaSuccess) return LBM_ECUDA;
        const int nconv = *b->h_nconv;
        if (n_converged) *n_converged = nconv;
        if (nconv >= b->njobs || done + check_every > max_steps) break;
        if (cudaGraphLaunch(b->exec, b->stream) != cudaSuccess) return LBM_ECUDA;
        b->launches += 1;
        b->rounds += 1;
        done += check_every;
    }
    return LBM_OK;
}

int lbm_batch_job_state(lbm_batch *b, int job, double *rho, long long *steps, double *last_drho,
                        int *converged)
{
    if (!b || job < 0 || job >= b->njobs) return LBM_EINVAL;
    const bt::Job &J = b->jobs[job];
    const long long n = rho ? b->nc * J.N : 0;
    bt::k_batch_job<<<(unsigned)std::min<long long>((n + 255) / 256 + 1, 256), 256, 0, b->stream>>>(
        b->d_status + job, b->pool + J.rh, b->pool + J.rl, n, b->h_status, b->h_rho);
    b->launches += 1;
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(b->stream) != cudaSuccess) return LBM_ECUDA;
    const bt::Status s = *b->h_status;
    if (steps) *steps = s.steps;
    if (last_drho) *last_drho = s.last_drho;
    if (converged) *converged = s.converged;
    if (rho) std::memcpy(rho, b->h_rho, (size_t)n * sizeof(double));
    return LBM_OK;
}

int lbm_batch_info(const lbm_batch *b, int *threads, int *ctas, long long *rounds, long long *launches)
{
    if (!b) return LBM_EINVAL;
    if (threads) *threads = b->threads;
    if (ctas) *ctas = b->ctas;
    if (rounds) *rounds = b->rounds;
    if (launches) *launches = b->launches;
    return LBM_OK;
}

int lbm_batch_set_threads(lbm_batch *b, int threads)
{
    if (!b || (threads != 128 && threads != 256 && threads != 512 && threads != b->tuned.first)) return LBM_EINVAL;
    if (b->exec) cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
    b->graph_steps = -1;
    // the shared memory the tuner chose goes with its CTA size; small CTAs need company on their SM
    return configure(b, threads, threads == b->tuned.first ? b->tuned.second : 0);
}

int lbm_batch_destroy(lbm_batch *b)
{
    if (!b) return LBM_OK;
    if (b->stream) cudaStreamSynchronize(b->stream);
    release(b);
    delete b;
    return LBM_OK;
}

}  // extern "C"
