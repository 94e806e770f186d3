// Stateless entry points of the C ABI: each phase kernel on caller-owned device
// memory, for tests, the autograd binding and custom drivers.  Temporaries are
// allocated stream-ordered on the caller's stream, one block per call, from the
// library's memory pool, and freed before returning.
#include "../../include/smc.h"
#include "kernels.cuh"
#include "mala.cuh"
#include "phase.cuh"

#include <cmath>
#include <cstring>
#include <mutex>

namespace smc {
void count_launch();
}
using namespace smc;

namespace {

void model_dev(const smc_model& m, ModelDev& d)
{
    std::memset(&d, 0, sizeof d);
    d.kind = m.model;
    d.K = m.K;
    d.I = m.I;
    d.gamma = m.gamma;
    d.eps0_zero = m.eps0_zero;
    d.p = m.p;
    d.sigma = m.sigma;
    d.d_full = m.d_full;
    d.d = m.n_free > 0 ? m.n_free : m.d_full;
    d.has_free = m.n_free > 0;
    for (int i = 0; i < SMC_MAX_D; ++i) {
        d.free_idx[i] = m.free_idx[i];
        d.theta_fixed[i] = m.theta_fixed[i];
        d.prior_mean[i] = m.prior_mean[i];
        const double sd = m.prior_sd[i] > 0.0 ? m.prior_sd[i] : 1.0;
        d.prior_isd[i] = 1.0 / sd;
        d.prior_c[i] = -0.5 * kLog2Pi - std::log(sd);
        d.prior_lo[i] = m.prior_lo[i];
        d.prior_mean_f[i] = (float)d.prior_mean[i];
        d.prior_isd_f[i] = (float)d.prior_isd[i];
        d.prior_c_f[i] = (float)d.prior_c[i];
        d.prior_lo_f[i] = (float)d.prior_lo[i];
    }
}

bool model_ok(const smc_model* m, int precision)
{
    if (!m) return false;
    if (m->model == SMC_EGARCH) {
        if (m->K < 1 || m->K > kMaxK || m->I < 1 || m->I > kMaxI) return false;
        if (precision != SMC_FP32 && precision != SMC_FP64) return false;
    } else if (m->model == SMC_LINREG) {
        if (m->p < 1 || m->p > 7 || precision != SMC_FP64) return false;
    } else {
        return false;
    }
    return m->d_full >= 1 && m->d_full <= SMC_MAX_D && m->n_free >= 0 && m->n_free <= m->d_full;
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

// The pool of the stateless calls' temporaries, one per device, made at the
// first call.  It keeps up to kPoolKeep bytes across synchronisations: the
// device's default pool gives everything back at each one, and every call here
// that returns a number synchronises, so a call after a device-wide wait paid
// 200 us for mapping its memory again (random walk, K=2, I=2, 65,536 x 5,000:
// first call after a wait 545 -> 341 us; power search, S phase and covariance
// at 1,024 particles: 475 -> 250 us; calls in a row cost the same).  What is kept
// serves every stream and thread (the pool orders reuse between streams
// itself); smc_release_workspace() gives it back, and the driver takes it for an
// allocation of this process that would fail otherwise.  The handle lives as long
// as the process: after cudaDeviceReset it is stale, so no stateless call may
// follow one.
constexpr uint64_t kPoolKeep = 512ull << 20;
constexpr int kMaxPools = 64;
std::mutex g_pool_mu;
cudaMemPool_t g_pool[kMaxPools] = {};

cudaError_t pool_of_device(cudaMemPool_t* out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxPools) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_pool_mu);
    if (!g_pool[dev]) {
        cudaMemPoolProps props;
        std::memset(&props, 0, sizeof props);
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t pool = nullptr;
        // (the first call may be one that a stream capture records)
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
        e = cudaThreadExchangeStreamCaptureMode(&mode);
        if (e != cudaSuccess) return e;
        uint64_t keep = kPoolKeep;
        e = cudaMemPoolCreate(&pool, &props);
        if (e == cudaSuccess) e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        cudaThreadExchangeStreamCaptureMode(&mode);
        if (e != cudaSuccess) {
            if (pool) cudaMemPoolDestroy(pool);
            return e;
        }
        g_pool[dev] = pool;
    }
    *out = g_pool[dev];
    return cudaSuccess;
}

// One call's temporaries: a single stream-ordered block cut into 256-byte
// aligned parts, freed (stream-ordered) when it goes out of scope.  add() every
// part, then get(), then take() them in the same order.
class Scratch {
public:
    explicit Scratch(cudaStream_t s) : s_(s) {}
    ~Scratch()
    {
        if (base_) cudaFreeAsync(base_, s_);
    }
    Scratch(const Scratch&) = delete;
    Scratch& operator=(const Scratch&) = delete;
    void add(size_t bytes) { size_ += round(bytes); }
    cudaError_t get()
    {
        cudaMemPool_t pool = nullptr;
        const cudaError_t e = pool_of_device(&pool);
        if (e != cudaSuccess) return e;
        return cudaMallocFromPoolAsync((void**)&base_, size_ ? size_ : 256, pool, s_);
    }
    template <typename T>
    T* take(size_t bytes)
    {
        char* p = base_ + used_;
        used_ += round(bytes);
        return reinterpret_cast<T*>(p);
    }

private:
    static size_t round(size_t b) { return (b + 255) & ~(size_t)255; }
    cudaStream_t s_;
    char* base_ = nullptr;
    size_t size_ = 0, used_ = 0;
};

smc_status from_cuda(cudaError_t e) { return e == cudaSuccess ? SMC_OK : SMC_ECUDA; }

}  // namespace

#define CK(x)                                   \
    do {                                        \
        cudaError_t e_ = (x);                   \
        if (e_ != cudaSuccess) return SMC_ECUDA; \
    } while (0)

extern "C" {

smc_status smc_release_workspace(void)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return SMC_ECUDA;
    if (dev < 0 || dev >= kMaxPools) return SMC_OK;
    std::lock_guard<std::mutex> lock(g_pool_mu);
    return g_pool[dev] ? from_cuda(cudaMemPoolTrimTo(g_pool[dev], 0)) : SMC_OK;
}

smc_status smc_loglik(const smc_model* m, int precision, const void* obs, int T, const double* theta,
                      int P, double* ll, double* lp, double* state, void* stream)
{
    if (!model_ok(m, precision) || !obs || !theta || !ll || T < 1 || P < 1 || !aligned16(obs))
        return SMC_EINVAL;
    LoglikArgs a;
    a.m = ModelDev{};
    model_dev(*m, a.m);
    a.obs = obs;
    a.T = T;
    a.W = m->model == SMC_LINREG ? smc_linreg_width(m->p) : 1;
    a.theta = theta;
    a.ll = ll;
    a.lp = lp;
    a.state = m->model == SMC_EGARCH ? state : nullptr;
    a.P = P;
    a.ns = m->model == SMC_EGARCH ? m->K + 1 : 0;
    a.err = nullptr;
    a.by_size = 1;
    return from_cuda(launch_loglik(a, precision, (cudaStream_t)stream));
}

static smc_status mutate_impl(const smc_model* m, int precision, const void* obs, int T, double* theta,
                              double* ll, double* lp, double* state, int P, const double* qmean,
                              const double* L, double phi, uint64_t seed, uint64_t cycle, uint64_t iter,
                              uint64_t* accepted, void* stream)
{
    if (!model_ok(m, precision) || !obs || !theta || !ll || !lp || !L || T < 1 || P < 1 ||
        !aligned16(obs) || !(phi >= 0.0))
        return SMC_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int d = m->n_free > 0 ? m->n_free : m->d_full;
    const size_t n_thp = (size_t)P * d * sizeof(double), n_lq = qmean ? (size_t)P * sizeof(double) : 0;
    Scratch w(s);
    w.add(n_thp);
    w.add(sizeof(unsigned long long));
    w.add(n_lq);
    CK(w.get());
    double* thp = w.take<double>(n_thp);
    unsigned long long* cnt = w.take<unsigned long long>(sizeof(unsigned long long));
    double* lq = qmean ? w.take<double>(n_lq) : nullptr;
    CK(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), s));
    if (qmean) CK(launch_indep_logq(theta, d, P, L, qmean, lq, s));
    MutateArgs a;
    a.m = ModelDev{};
    model_dev(*m, a.m);
    a.obs = obs;
    a.T = T;
    a.W = m->model == SMC_LINREG ? smc_linreg_width(m->p) : 1;
    a.theta = theta;
    a.ll = ll;
    a.lp = lp;
    a.state = m->model == SMC_EGARCH ? state : nullptr;
    a.thp = thp;
    a.P = P;
    a.ns = m->model == SMC_EGARCH ? m->K + 1 : 0;
    a.L = L;
    a.qmean = qmean;
    a.lq = lq;
    a.covtile = nullptr;
    a.covshift = nullptr;
    a.ntiles = 0;
    a.phi = phi;
    a.seed = seed;
    a.cycle = cycle;
    a.iter = iter;
    a.acc_count = cnt;
    a.pending = nullptr;
    a.err = nullptr;
    int ppt, threads;
    mutate_default_shape(a.m, precision, qmean == nullptr, P, &ppt, &threads);
    cudaError_t e = ppt == 2 ? launch_mutate_x2(a, threads, s) : launch_mutate(a, precision, threads, s);
    unsigned long long h = 0;
    if (e == cudaSuccess && accepted) {
        e = cudaMemcpyAsync(&h, cnt, sizeof h, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        *accepted = h;
    }
    return from_cuda(e);
}

smc_status smc_mutate_rw(const smc_model* m, int precision, const void* obs, int T, double* theta,
                         double* ll, double* lp, double* state, int P, const double* L, double phi,
                         uint64_t seed, uint64_t cycle, uint64_t iter, uint64_t* accepted,
                         void* stream)
{
    return mutate_impl(m, precision, obs, T, theta, ll, lp, state, P, nullptr, L, phi, seed, cycle,
                       iter, accepted, stream);
}

smc_status smc_mutate_indep(const smc_model* m, int precision, const void* obs, int T, double* theta,
                            double* ll, double* lp, double* state, int P, const double* mean,
                            const double* L, double phi, uint64_t seed, uint64_t cycle, uint64_t iter,
                            uint64_t* accepted, void* stream)
{
    if (!mean) return SMC_EINVAL;
    return mutate_impl(m, precision, obs, T, theta, ll, lp, state, P, mean, L, phi, seed, cycle,
                       iter, accepted, stream);
}

smc_status smc_loglik_grad(const smc_model* m, int precision, const void* obs, int T,
                           const double* theta, int P, double* ll, double* grad, double* state,
                           void* stream)
{
    if (!model_ok(m, precision) || !obs || !theta || !ll || !grad || T < 1 || P < 1 || !aligned16(obs))
        return SMC_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    GradArgs a;
    a.m = ModelDev{};
    model_dev(*m, a.m);
    a.obs = obs;
    a.T = T;
    a.W = m->model == SMC_LINREG ? smc_linreg_width(m->p) : 1;
    a.theta = theta;
    a.P = P;
    a.ll = ll;
    a.grad = grad;
    a.state = m->model == SMC_EGARCH ? state : nullptr;
    const size_t n_ckpt = mala_ckpt_bytes(a.m, precision, T, P);
    Scratch w(s);
    w.add(n_ckpt);
    CK(w.get());
    a.ckpt = w.take<void>(n_ckpt);
    a.by_size = 1;
    return from_cuda(launch_loglik_grad(a, precision, s));
}

smc_status smc_mutate_mala(const smc_model* m, int precision, const void* obs, int T, double* theta,
                           double* ll, double* lp, double* grad, double* state, int P, const double* L,
                           double phi, uint64_t seed, uint64_t cycle, uint64_t iter, uint64_t* accepted,
                           void* stream)
{
    if (!model_ok(m, precision) || !obs || !theta || !ll || !lp || !grad || !L || T < 1 || P < 1 ||
        !aligned16(obs) || !(phi >= 0.0))
        return SMC_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    MalaArgs a;
    a.m = ModelDev{};
    model_dev(*m, a.m);
    a.obs = obs;
    a.T = T;
    a.W = m->model == SMC_LINREG ? smc_linreg_width(m->p) : 1;
    a.theta = theta;
    a.ll = ll;
    a.lp = lp;
    a.state = m->model == SMC_EGARCH ? state : nullptr;
    a.grad = grad;
    a.P = P;
    a.ns = m->model == SMC_EGARCH ? m->K + 1 : 0;
    a.L = L;
    a.phi = phi;
    a.seed = seed;
    a.cycle = cycle;
    a.iter = iter;
    a.pending = nullptr;
    a.err = nullptr;
    const size_t n_ckpt = mala_ckpt_bytes(a.m, precision, T, P);
    Scratch w(s);
    w.add(n_ckpt);
    w.add(sizeof(unsigned long long));
    CK(w.get());
    a.ckpt = w.take<void>(n_ckpt);
    unsigned long long* cnt = w.take<unsigned long long>(sizeof(unsigned long long));
    CK(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), s));
    a.acc_count = cnt;
    cudaError_t e = launch_mala(a, precision, s);
    unsigned long long h = 0;
    if (e == cudaSuccess && accepted) {
        e = cudaMemcpyAsync(&h, cnt, sizeof h, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        *accepted = h;
    }
    return from_cuda(e);
}

smc_status smc_cov_chol(const double* theta, int d, int P, int h_tenths, double* mean, double* cov,
                        double* L, void* stream)
{
    if (!theta || d < 1 || d > SMC_MAX_D || P < 2 || h_tenths < 0) return SMC_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int G = cov_grid(P);
    const size_t n = (size_t)(G + 1) * (d + d * (d + 1) / 2);
    Scratch w(s);
    w.add((n + 1) * sizeof(double));
    CK(w.get());
    double* part = w.take<double>((n + 1) * sizeof(double));
    unsigned int* counter = reinterpret_cast<unsigned int*>(part + n);
    CK(cudaMemsetAsync(counter, 0, sizeof(unsigned int), s));
    return from_cuda(launch_cov(theta, d, P, part, G, counter, nullptr, h_tenths, 0.0, 1, 10, mean, cov, L, s));
}

smc_status smc_power_search(const double* ll, int P, double phi, double d1, int passes, double* dphi,
                            double* rss, void* stream)
{
    if (!ll || P < 1 || !(phi >= 0.0 && phi < 1.0) || !(d1 > 0.0 && d1 < 1.0) || passes < 1)
        return SMC_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t n_part = search_part_len(P) * sizeof(double);
    struct Out {
        Ctl ctl;
        double gstat[3], lw, a;
    };
    Scratch w(s);
    w.add(n_part);
    w.add(sizeof(Out));
    CK(w.get());
    double* part = w.take<double>(n_part);
    Out* out = w.take<Out>(sizeof(Out));
    CK(cudaMemsetAsync(part, 0, search_bar_bytes(), s));
    Out h;
    std::memset(&h, 0, sizeof h);
    h.ctl.phi = phi;
    cudaError_t e = cudaMemcpyAsync(out, &h, sizeof h, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = launch_power_search(ll, P, d1, passes, part, &out->ctl, s);
    // FP64 RSS at the chosen power: the weights pass of the S phase over one
    // group holding all particles gives (max, sum w, sum w^2).
    if (e == cudaSuccess && P <= SMC_MAX_N) {
        SelectArgs sa;
        std::memset(&sa, 0, sizeof sa);
        sa.mode = 0;
        sa.ll = ll;
        sa.J = 1;
        sa.N = P;
        sa.a = &out->a;
        sa.lw = &out->lw;
        sa.gstat = out->gstat;
        sa.ctl = &out->ctl;
        sa.stats_only = 1;
        e = launch_select(sa, s);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, out, sizeof h, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess) {
        if (dphi) *dphi = h.ctl.dphi;
        if (rss) *rss = P <= SMC_MAX_N ? h.gstat[1] * h.gstat[1] / ((double)P * h.gstat[2]) : NAN;
    }
    return from_cuda(e);
}

smc_status smc_resample(const double* w, int J, int N, int resampler, uint64_t seed, uint64_t cycle,
                        int32_t* idx, void* stream)
{
    if (!w || !idx || J < 1 || N < 1 || N > SMC_MAX_N) return SMC_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    Scratch w_(s);
    w_.add(sizeof(int));
    CK(w_.get());
    int* err = w_.take<int>(sizeof(int));
    CK(cudaMemsetAsync(err, 0, sizeof(int), s));
    SelectArgs sa;
    std::memset(&sa, 0, sizeof sa);
    sa.mode = 2;
    sa.w = w;
    sa.J = J;
    sa.N = N;
    sa.scheme = resampler;
    sa.seed = seed;
    sa.cycle = cycle;
    sa.idx = idx;
    sa.err = err;
    cudaError_t e = launch_select(sa, s);
    int h = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, err, sizeof h, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return SMC_ECUDA;
    if (h & kErrDegenerate) return SMC_EDEGENERATE;
    return h ? SMC_ECUDA : SMC_OK;
}

smc_status smc_resample_logw(const double* logw, int J, int N, int resampler, uint64_t seed, uint64_t cycle,
                             int32_t* idx, double* lwbar, void* stream)
{
    if (!logw || !idx || J < 1 || N < 1 || N > SMC_MAX_N || resampler < 0 || resampler > 3) return SMC_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    // a [J] and the error word (cleared together), lw [J], gstat [3 J]
    const size_t Js = (size_t)J, n_buf = (5 * Js + 1) * sizeof(double);
    Scratch w(s);
    w.add(n_buf);
    CK(w.get());
    double* buf = w.take<double>(n_buf);
    int* err = reinterpret_cast<int*>(buf + Js);
    CK(cudaMemsetAsync(buf, 0, (Js + 1) * sizeof(double), s));
    SelectArgs sa;
    std::memset(&sa, 0, sizeof sa);
    sa.mode = 1;
    sa.logw = logw;
    sa.J = J;
    sa.N = N;
    sa.scheme = resampler;
    sa.seed = seed;
    sa.cycle = cycle;
    sa.a = buf;
    sa.lw = buf + Js + 1;
    sa.gstat = buf + 2 * Js + 1;
    sa.idx = idx;
    sa.err = err;
    cudaError_t e = launch_select(sa, s);
    int h = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, err, sizeof h, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && lwbar)
        e = cudaMemcpyAsync(lwbar, buf + Js + 1, Js * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return SMC_ECUDA;
    if (h & kErrDegenerate) return SMC_EDEGENERATE;
    return h ? SMC_ECUDA : SMC_OK;
}

smc_status smc_group_moments(const double* g, int nf, int J, int N, double* out, void* stream)
{
    if (!g || !out || nf < 1 || J < 2 || N < 1) return SMC_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t n_part = (size_t)nf * J * 2 * sizeof(double), n_out = (size_t)nf * 4 * sizeof(double);
    Scratch w(s);
    w.add(n_part);
    w.add(n_out);
    CK(w.get());
    double* part = w.take<double>(n_part);
    double* dout = w.take<double>(n_out);
    cudaError_t e = launch_moments(g, nf, J, N, part, dout, nullptr, 0, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(out, dout, (size_t)nf * 4 * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return from_cuda(e);
}

smc_status smc_ml_from_groups(const double* a, int J, double* log_ml, double* nse, void* stream)
{
    if (!a || J < 2) return SMC_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    Scratch w(s);
    w.add(3 * sizeof(double));
    CK(w.get());
    double* dout = w.take<double>(3 * sizeof(double));
    cudaError_t e = launch_ml(a, J, nullptr, dout, s);
    double h[3] = {0, 0, 0};
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, dout, sizeof h, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (log_ml) *log_ml = h[0];
    if (nse) *nse = h[1];
    return from_cuda(e);
}

}  // extern "C"
