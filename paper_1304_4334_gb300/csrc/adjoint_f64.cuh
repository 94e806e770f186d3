// FP64 log likelihood with its gradient by the adjoint recurrence of
// adjoint.cuh, on the integer pipes wherever FP64 is not needed.
//
// FP64 instructions bound it (about 64 cycles each per warp, whatever the
// occupancy), so they are what is saved here:
//   - the forward pass and each segment's recomputation run in the
//     fixed-point recursion (EgarchFx; the FP64 recursion takes particles out
//     of its ranges);
//   - the component weights r_i come from integer exponentials and an integer
//     reciprocal of their sum, assembled as FP64 numbers by integer instructions;
//   - the sums over t keep r_i, r_i z and r_i z^2 per component, z = eps - mu_i
//     (about mu_i, and combined every segment, so that no two large sums are
//     left to cancel at the end: the gradient's rms error at K = 1, I = 2, T = 150 is
//     0.96e-15 of its largest entry, 1.39e-15 with sums over the series,
//     0.98e-15 with FP64 throughout), from which d log p_i, d mu_i and d a_i
//     follow at the end (5 FP64 instructions per component and observation
//     instead of 11).
// About 40 FP64 instructions per particle and observation at K = 2, I = 2
// against 230 with FP64 exponentials and division.
// Measured (value and gradient, K = 2, I = 2, 2,049 particles x 1,037
// observations, a warp per scheduler at most): 7.9 ms in FP64 throughout, 2.42
// ms in AdjointF64, 1.33 ms in GradSplit.
#pragma once

#include "adjoint.cuh"

namespace smc {

struct GradArgs {
    ModelDev m;
    const void* obs;
    int T, W;
    const double* theta;   // [d][P]
    int P;
    double* ll;            // [P]
    double* grad;          // [d][P] d log p(y|theta) / d theta (free parameters)
    double* state;         // [K+1][P] (nullable)
    void* ckpt;            // segment checkpoints (gradient policy's layout)
    int by_size;           // the kernel may be chosen by P: the last bits of l and of the gradient
                           // differ between them, so a run, whose particles do not depend on how
                           // they are divided over launches, leaves it 0
};

// Gradient with respect to the full theta vector (Table 1 layout) from the
// natural parameters' (mu, log sigma, alpha, beta, gamma, log p_i, mu_i, a_i):
// the transforms and the mixture's normalisation taken backwards,
//   p_i = P_i / S,  m = sum p_i M_i,  V = sum p_i ((M_i - m)^2 + s_i^2),  c = V^-1/2,
//   mu_i = c (M_i - m),  1 / a_i = c s_i
// (about 15 FP64 instructions per component; forward-mode duals along each of
// the 3 I directions made the K=2, I=2 gradient of 4,096 particles 36 us
// longer, as long as some 60 observations).
template <int K, int I>
__device__ __forceinline__ void natural_to_theta_f64(const EgarchParams<double, K, I>& q, const double* gn,
                                                     const double* th, int has_gamma, double* gth)
{
    int j = 0;
    gth[j++] = gn[0] / 1000.0;
    gth[j++] = gn[1];
#pragma unroll
    for (int k = 0; k < K; ++k) gth[j++] = gn[2 + k] * (1.0 - q.alpha[k] * q.alpha[k]);
#pragma unroll
    for (int k = 0; k < K; ++k) gth[j++] = gn[2 + K + k] * q.beta[k];
    if (has_gamma) {
#pragma unroll
        for (int k = 0; k < K; ++k) gth[j++] = gn[2 + 2 * K + k];
    }
    if constexpr (I >= 2) {
        const double* glp = gn + 2 + 3 * K;
        const double* gmu = glp + I;
        const double* ga = gmu + I;
        double P[I], s[I], pb[I], m2b[I], S = 0.0;
#pragma unroll
        for (int i = 0; i < I; ++i) {
            P[i] = 2.0 / (1.0 + exp(-2.0 * th[j + i]));
            s[i] = exp(th[j + 2 * I + i]);
            S += P[i];
        }
        const double c = q.sig[0] / s[0], ic = 1.0 / c, c2 = c * c;
        double cb = 0.0;
#pragma unroll
        for (int i = 0; i < I; ++i) cb += gmu[i] * q.mu[i] - ga[i] / q.sig[i];   // c dL/dc
        const double Vb = -0.5 * c2 * cb;                                            // dL/dV
        double mb = 0.0, pp = 0.0;
#pragma unroll
        for (int i = 0; i < I; ++i) {
            const double m2 = q.mu[i] * ic;
            m2b[i] = c * gmu[i] + 2.0 * Vb * q.p[i] * m2;
            mb -= m2b[i];
            pb[i] = glp[i] / q.p[i] + Vb * (m2 * m2 + s[i] * s[i]);
            gth[j + 2 * I + i] = -ga[i] / q.sig[i] + 2.0 * Vb * q.p[i] * s[i] * s[i];
        }
#pragma unroll
        for (int i = 0; i < I; ++i) {
            gth[j + I + i] = m2b[i] + mb * q.p[i];
            pb[i] += mb * th[j + I + i];
            pp += pb[i] * q.p[i];
        }
#pragma unroll
        for (int i = 0; i < I; ++i) gth[j + i] = (pb[i] - pp) / S * (P[i] * (2.0 - P[i]));
    }
}

// r_i with the terms x_i formed in FP64 (any parameters and shock); returns
// log sum_i exp(x_i).  A term that is NaN makes all of them NaN.
template <int K, int I>
__device__ __noinline__ double weights_f64(const EgarchParams<double, K, I>& q, double eps, const uint64_t* tab,
                                           double* r)
{
    double x[I], mx = -INFINITY, s = 0.0;
#pragma unroll
    for (int i = 0; i < I; ++i) {
        const double z = (eps - q.mu[i]) / q.sig[i];
        x[i] = log(q.p[i]) - log(q.sig[i]) - 0.5 * z * z;
        mx = fmax(mx, x[i]);
    }
#pragma unroll
    for (int i = 0; i < I; ++i) {
        r[i] = fx_exp_neg(mx - x[i], tab);
        s += r[i];
    }
    const double is = 1.0 / s;
#pragma unroll
    for (int i = 0; i < I; ++i) r[i] *= is;
    return mx + log(s);
}

template <int K, int I, int kSeg>
struct AdjointF64 {
    EgarchFxSafe<K, I> mdl;
    double a2[I];                // a_i^2

    __device__ __forceinline__ void setup(const double* th, int has_gamma, int eps0_zero, const uint64_t* tab)
    {
        mdl.setup(th, has_gamma, eps0_zero, tab);
#pragma unroll
        for (int i = 0; i < I; ++i) {
            const double a = 1.0 / mdl.q.sig[i];
            a2[i] = a * a;
        }
    }

    // Forward pass with the state entering every segment but the first saved
    // in ckpt[seg - 1][v_1..v_K, eps][P]; returns l(theta), the end state in st.
    __device__ __forceinline__ double forward(const double* __restrict__ y, int T, double* ckpt, size_t P, int p,
                                              double* st)
    {
        EgarchFx<K, I> fx = mdl.fx;   // (in registers, as in the reverse sweep)
        for (int t0 = 0; t0 < T; t0 += kSeg) {
            const int n = min(kSeg, T - t0);
            if (t0 > 0) {
                double* c = ckpt + (size_t)(t0 / kSeg - 1) * (K + 1) * P + p;
                if (mdl.out) mdl.m.state_out(st);
                else fx.state_out(st, kLn2);
#pragma unroll
                for (int k = 0; k <= K; ++k) c[k * P] = st[k];
            }
            fx.block(y + t0, n, t0 == 0, mdl.tab);
            mdl.close(fx, y + t0, t0, n, T);
        }
        if (!mdl.out) mdl.fx.restore(mdl.saved);
        mdl.state_out(st, y + T - 1);
        return mdl.finish(T);
    }

    // Recomputes a segment's states in FP64 (out of the fixed-point ranges).
    __device__ __noinline__ void segment_f64(const double* __restrict__ y, int t0, int n, const double* vprev,
                                             double eprev, double* buf, int stride)
    {
        EgarchF64<K, I> w;
        w.setup(mdl.q, mdl.eps0_zero, mdl.tab);
#pragma unroll
        for (int k = 0; k < K; ++k) w.v[k] = vprev[k];
        w.eps = eprev;
        for (int r = 0; r < n; ++r) {
            uint64_t s;
            if (t0 + r == 0) w.template terms<true>(y[0], s);
            else w.template terms<false>(y[t0 + r], s);
            double vs = w.v[0];
#pragma unroll
            for (int k = 1; k < K; ++k) vs += w.v[k];
            put(buf + (size_t)r * (K + 2) * stride, stride, w.v, w.eps,
                fx_exp_neg(mdl.q.log_sigma_y + 0.5 * vs, mdl.tab));
        }
    }

    __device__ __forceinline__ static void put(double* b, int stride, const double* v, double eps, double inv)
    {
#pragma unroll
        for (int k = 0; k < K; ++k) b[k * stride] = v[k];
        b[K * stride] = eps;
        b[(K + 1) * stride] = inv;
    }

    // Reverse sweep; gn (EgarchNat<double, K, I>::kNp) receives d l / d natural
    // parameters.  buf: this thread's slab, [kSeg][v_1..v_K, eps, 1/h][stride].
    __device__ __forceinline__ void reverse(const double* __restrict__ y, int T, const double* ckpt, size_t P, int p,
                                            double* buf, int stride, double* gn)
    {
        constexpr int NS = 2 + 3 * K;      // mu, log sigma, alpha, beta, gamma
        constexpr int W = K + 2;
        double gs[NS], s0[I], s1[I], s2[I], vb[K];
        for (int i = 0; i < NS + 3 * I; ++i) gn[i] = 0.0;
#pragma unroll
        for (int i = 0; i < NS; ++i) gs[i] = 0.0;
#pragma unroll
        for (int i = 0; i < I; ++i) {
            s0[i] = s1[i] = s2[i] = 0.0;
        }
#pragma unroll
        for (int k = 0; k < K; ++k) vb[k] = 0.0;
        const EgarchParams<double, K, I>& q = mdl.q;
        double al[K], bp[K], bm[K], ga[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            al[k] = q.alpha[k];
            ga[k] = q.gamma[k];
            bp[k] = q.beta[k] + q.gamma[k];
            bm[k] = q.gamma[k] - q.beta[k];
        }
        const bool fixed = mdl.fixed;
        EgarchFx<K, I> fx = mdl.fx;
        fx.natural_shocks();
        auto back = [&](double eps, double inv, const double* vp, double ep, bool has_prev) {
            double eb = -eps;
            if constexpr (I >= 2) {
                double r[I];
                if (!(fixed && fx.weights(eps, r, mdl.tab))) weights_f64(mdl.q, eps, mdl.tab, r);
                eb = 0.0;
#pragma unroll
                for (int i = 0; i < I; ++i) {
                    const double z = eps - q.mu[i];
                    const double rz = r[i] * z;
                    eb = fma(-rz, a2[i], eb);
                    s0[i] += r[i];
                    s1[i] += rz;
                    s2[i] = fma(rz, z, s2[i]);
                }
            }
#pragma unroll
            for (int k = 0; k < K; ++k)
                eb = fma(vb[k], eps > 0.0 ? bp[k] : (eps < 0.0 ? bm[k] : ga[k]), eb);
            const double sb = fma(-eb, eps, -1.0);
            gs[0] = fma(-eb, inv, gs[0]);
            gs[1] += sb;
            const double h = 0.5 * sb;
            const double ae = fabs(ep) - kSqrt2OverPi;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                vb[k] = fma(al[k], vb[k], h);
                if (has_prev) {
                    gs[2 + k] = fma(vb[k], vp[k], gs[2 + k]);
                    gs[2 + K + k] = fma(vb[k], ae, gs[2 + K + k]);
                    gs[2 + 2 * K + k] = fma(vb[k], ep, gs[2 + 2 * K + k]);
                } else if (mdl.eps0_zero) {
                    gs[2 + K + k] = fma(vb[k], -kSqrt2OverPi, gs[2 + K + k]);
                }
            }
        };
        const int nseg = (T + kSeg - 1) / kSeg;
        for (int sg = nseg - 1; sg >= 0; --sg) {
            const int t0 = sg * kSeg, n = min(kSeg, T - t0);
            double vprev[K], eprev = 0.0;      // the state entering the segment
#pragma unroll
            for (int k = 0; k < K; ++k) vprev[k] = 0.0;
            if (sg > 0) {
                const double* c = ckpt + (size_t)(sg - 1) * (K + 1) * P + p;
#pragma unroll
                for (int k = 0; k < K; ++k) vprev[k] = c[k * P];
                eprev = c[K * P];
            }
            bool ok = fixed && (sg == 0 || fx.enter(vprev, eprev));
            fx.bad = 0;
            auto keep = [&](int r) {
                double s[K + 1];
                fx.state_out(s, kLn2);   // (its shock is not used)
                put(buf + (size_t)r * W * stride, stride, s, fx.eps(), fx.inv_h());
            };
            if (t0 == 0) fx.template chain<true>(y[0], mdl.tab);
            else fx.template chain<false>(y[t0], mdl.tab);
            keep(0);
#pragma unroll 2
            for (int r = 1; r < n; ++r) {
                fx.template chain<false>(y[t0 + r], mdl.tab);
                keep(r);
            }
            ok = ok && fx.bad == 0u;
            if (!ok) segment_f64(y, t0, n, vprev, eprev, buf, stride);
            const double* b = buf + (size_t)(n - 1) * W * stride;
#pragma unroll 2
            for (int r = n - 1; r >= 1; --r, b -= W * stride) {
                const double* bq = b - W * stride;
                double vp[K];
#pragma unroll
                for (int k = 0; k < K; ++k) vp[k] = bq[k * stride];
                back(b[K * stride], b[(K + 1) * stride], vp, bq[K * stride], true);
            }
            back(buf[K * stride], buf[(K + 1) * stride], vprev, eprev, t0 > 0);
            if ((sg & 7) == 0) {
#pragma unroll
                for (int i = 0; i < NS; ++i) {
                    gn[i] += gs[i];
                    gs[i] = 0.0;
                }
            }
            if constexpr (I >= 2) {
#pragma unroll
                for (int i = 0; i < I; ++i) {
                    gn[NS + i] += s0[i];
                    gn[NS + I + i] += s1[i];
                    gn[NS + 2 * I + i] += fma(-a2[i], s2[i], s0[i]);
                    s0[i] = s1[i] = s2[i] = 0.0;
                }
            }
        }
        // sum r_i, sum r_i z, sum r_i (1 - a^2 z^2) -> d log p_i, d mu_i, d a_i
        if constexpr (I >= 2) {
#pragma unroll
            for (int i = 0; i < I; ++i) {
                gn[NS + I + i] *= a2[i];
                gn[NS + 2 * I + i] *= q.sig[i];
            }
        }
    }
};

// ------------------------------------------- two warps per 32 particles
// The same computation split over two warps for particles too few to fill the
// SMs' schedulers (I >= 2): the first carries the volatility chain and the
// adjoint carry, the second everything about the mixture, a segment behind.
// A warp's own latency (about 4,000 cycles per observation in AdjointF64 at
// K=2, I=2) is what bounds such a launch; the two halves run side by side.
// Forward: warp 0 leaves each segment's shocks, warp 1 takes their mixture
// densities.  Backward, at step j: warp 0 recomputes segment n-1-j and runs the
// carry over segment n+1-j, warp 1 forms dl/deps and the component sums of
// segment n-j.  V_k is kept in units of 2^-55 and its sums scaled once at the
// end; sums of z^2 are in eps's own units, so they overflow where FP64's do.
// Measured at T=600, up to one block (of 32 particles) per SM, one warp ->
// two: K=1,I=2 1,298 -> 703 us, K=2,I=2 1,441 -> 823 us, K=3,I=4 2,604 ->
// 1,347 us, K=4,I=4 2,884 -> 1,364 us; with all the blocks an SM's shared
// memory holds 1,358 -> 822, 1,495 -> 976, 2,723 -> 1,645 us.  (With weights and
// shocks of all bits the two warps take 688, 773, 1,360 and 1,370 us.)  Beyond that
// a second wave would take what the split gains (k_loglik_grad then).
template <int K, int I>
struct GradSplit {
    static constexpr int kSeg = mala_seg<double>(), W = K + 2;   // (the caller's checkpoint block is sized from it)
    static constexpr double kVu = 0x1p55 * 0.5 / kLn2;   // V_k units of v_k
    struct Smem {
        double slab[3][kSeg][W][32];       // V_1..V_K, eps, 1/h
        double x[2][kSeg][32];             // forward: shocks (2^-53); backward: dl/deps
        double comb[3 * I + 2][32];        // warp 1's results
        uint64_t tab[256];
    };

    // Both warps, each from its own place in the code.
    __device__ __forceinline__ static void meet() { asm volatile("barrier.sync 1, 64;" ::: "memory"); }

    // A segment of warp 0 in FP64: shocks out, times `unit` (and V, 1/h for the
    // recomputation), log h summed; w carries the state.
    __device__ __noinline__ static double segment_f64(EgarchF64<K, I>& w, double lsy, const double* __restrict__ y,
                                                      int t0, int n, double unit, double* es, int es_stride, double* v, double* inv)
    {
        double sum = 0.0;
        for (int r = 0; r < n; ++r) {
            uint64_t s;
            if (t0 + r == 0) w.template terms<true>(y[0], s);
            else w.template terms<false>(y[t0 + r], s);
            double vs = w.v[0];
#pragma unroll
            for (int k = 1; k < K; ++k) vs += w.v[k];
            sum += lsy + 0.5 * vs;
            es[(size_t)r * es_stride] = w.eps * unit;
            if (v) {
#pragma unroll
                for (int k = 0; k < K; ++k) v[(size_t)r * es_stride + 32 * k] = w.v[k] * kVu;
                inv[(size_t)r * es_stride] = fx_exp_neg(lsy + 0.5 * vs, w.tab);
            }
        }
        return sum;
    }

    __device__ static void run(const GradArgs& a, Smem& sm)
    {
        const int lane = threadIdx.x & 31, role = threadIdx.x >> 5;
        for (int i = threadIdx.x; i < 256; i += blockDim.x) sm.tab[i] = g_exp2_neg256[i];
        const int p = blockIdx.x * 32 + lane;
        const bool active = p < a.P;
        const int pp = active ? p : a.P - 1;
        const size_t P = (size_t)a.P;
        const int T = a.T, nseg = (T + kSeg - 1) / kSeg;
        const double* __restrict__ y = (const double*)a.obs;
        double* ckpt = (double*)a.ckpt;
        double th[kMaxD], full[kMaxD];
        for (int i = 0; i < a.m.d; ++i) th[i] = a.theta[i * P + pp];
        full_theta<double>(a.m, th, full);
        EgarchParams<double, K, I> q;
        egarch_transform<double, K, I>(full, a.m.gamma, q);
        EgarchFx<K, I> fx;
        fx.setup(q.mu_y, q.log_sigma_y, q.alpha, q.beta, q.gamma, q.p, q.mu, q.sig, a.m.eps0_zero, kLog2e);
        const bool fixed = fx.bad == 0u;
        __syncthreads();
        if (role == 0) chain_warp(a, sm, fx, q, fixed, lane, p, pp, active, full, y, ckpt, P, T, nseg);
        else mixture_warp(sm, fx, q, fixed, lane, T, nseg);
    }

    __device__ __forceinline__ static void chain_warp(const GradArgs& a, Smem& sm, EgarchFx<K, I> fx,
                                                      const EgarchParams<double, K, I>& q, bool fixed, int lane,
                                                      int p, int pp, bool active, const double* full,
                                                      const double* __restrict__ y, double* ckpt, size_t P, int T,
                                                      int nseg)
    {
        EgarchF64<K, I> w;
        w.setup(q, a.m.eps0_zero, sm.tab);
        bool out = !fixed;
        double st[K + 1], lh64 = 0.0;      // state at the segment's start; log h summed in FP64
        int n64 = 0;
        unsigned __int128 sx = 0;
#pragma unroll
        for (int k = 0; k <= K; ++k) st[k] = 0.0;
        for (int sg = 0; sg <= nseg; ++sg) {
            if (sg < nseg) {
                const int t0 = sg * kSeg, n = min(kSeg, T - t0);
                if (sg > 0) {
                    double* c = ckpt + (size_t)(sg - 1) * (K + 1) * P + pp;
                    if (active)
#pragma unroll
                        for (int k = 0; k <= K; ++k) c[k * P] = st[k];
                }
                double* es = &sm.x[sg & 1][0][lane];
                fx.bad = 0;
                fx.sx = 0;
                if (t0 == 0) fx.template chain<true>(y[0], sm.tab);
                else fx.template chain<false>(y[t0], sm.tab);
                es[0] = (double)fx.shock();
#pragma unroll 2
                for (int r = 1; r < n; ++r) {
                    fx.template chain<false>(y[t0 + r], sm.tab);
                    es[r * 32] = (double)fx.shock();
                }
                if (fx.bad == 0u && !out) {
                    sx += fx.sx;
                    fx.state_out(st, kLn2);
                    st[K] = fx.eps();
                } else {
                    if (!out) w.load_state(st);
                    lh64 += segment_f64(w, q.log_sigma_y, y, t0, n, 0x1p53, es, 32, nullptr, nullptr);
                    n64 += n;
                    out = !(fixed && fx.enter(w.v, w.eps));
                    w.state_out(st);
                }
            }
            meet();
        }
        const double logh = lh64 + kLn2 * fx_to_double((__int128)sx - ((__int128)(T - n64) << 63), -55);
        if (active && a.state)
#pragma unroll
            for (int k = 0; k <= K; ++k) a.state[k * P + p] = st[k];

        constexpr int NS = 2 + 3 * K;
        double gn[NS + 3 * I], gs[NS], vb[K], al[K], bp[K], bm[K], ga[K];
#pragma unroll
        for (int i = 0; i < NS; ++i) gn[i] = gs[i] = 0.0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            vb[k] = 0.0;                   // 2 dL/dv_k,t+1
            al[k] = q.alpha[k];
            ga[k] = 0.5 * q.gamma[k];
            bp[k] = 0.5 * (q.beta[k] + q.gamma[k]);
            bm[k] = 0.5 * (q.gamma[k] - q.beta[k]);
        }
        auto carry = [&](double dle, double es, double inv, const double* vp, double ep, bool has_prev) {
            double eb = dle;               // dL/deps
#pragma unroll
            for (int k = 0; k < K; ++k) eb = fma(vb[k], es > 0.0 ? bp[k] : (es < 0.0 ? bm[k] : ga[k]), eb);
            const double sb = fma(-eb, es, -1.0);
            gs[0] = fma(-eb, inv, gs[0]);
            gs[1] += sb;
            const double ae = fabs(ep) - kSqrt2OverPi;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                vb[k] = fma(al[k], vb[k], sb);
                if (has_prev) {
                    gs[2 + k] = fma(vb[k], vp[k], gs[2 + k]);
                    gs[2 + K + k] = fma(vb[k], ae, gs[2 + K + k]);
                    gs[2 + 2 * K + k] = fma(vb[k], ep, gs[2 + 2 * K + k]);
                } else if (a.m.eps0_zero) {
                    gs[2 + K + k] = fma(vb[k], -kSqrt2OverPi, gs[2 + K + k]);
                }
            }
        };
        auto entering = [&](int sg, double* v, double& e) {   // the state entering segment sg
            if (sg > 0) {
                const double* c = ckpt + (size_t)(sg - 1) * (K + 1) * P + pp;
#pragma unroll
                for (int k = 0; k < K; ++k) v[k] = c[k * P];
                e = c[K * P];
            } else {
#pragma unroll
                for (int k = 0; k < K; ++k) v[k] = 0.0;
                e = 0.0;
            }
        };
        for (int j = 0; j < nseg + 2; ++j) {
            if (j < nseg) {                // recompute segment nseg - 1 - j
                const int sg = nseg - 1 - j, t0 = sg * kSeg, n = min(kSeg, T - t0);
                double v0[K], e0;
                entering(sg, v0, e0);
                bool ok = fixed && (sg == 0 || fx.enter(v0, e0));
                fx.bad = 0;
                double(*b)[W][32] = sm.slab[j % 3];
                auto put = [&](int r) {
#pragma unroll
                    for (int k = 0; k < K; ++k) b[r][k][lane] = (double)fx.V[k];
                    b[r][K][lane] = fx.eps();
                    b[r][K + 1][lane] = fx.inv_h();
                };
                if (t0 == 0) fx.template chain<true>(y[0], sm.tab);
                else fx.template chain<false>(y[t0], sm.tab);
                put(0);
#pragma unroll 2
                for (int r = 1; r < n; ++r) {
                    fx.template chain<false>(y[t0 + r], sm.tab);
                    put(r);
                }
                ok = ok && fx.bad == 0u;
                if (!ok) {
#pragma unroll
                    for (int k = 0; k < K; ++k) w.v[k] = v0[k];
                    w.eps = e0;
                    segment_f64(w, q.log_sigma_y, y, t0, n, 1.0, &b[0][K][lane], W * 32, &b[0][0][lane], &b[0][K + 1][lane]);
                }
            }
            if (j >= 2) {                  // carry over segment nseg + 1 - j
                const int sg = nseg + 1 - j, t0 = sg * kSeg, n = min(kSeg, T - t0);
                const double(*b)[W][32] = sm.slab[(j - 2) % 3];
                const double* dl = &sm.x[j & 1][0][lane];
#pragma unroll 2
                for (int r = n - 1; r >= 1; --r) {
                    double vp[K];
#pragma unroll
                    for (int k = 0; k < K; ++k) vp[k] = b[r - 1][k][lane];
                    carry(dl[r * 32], b[r][K][lane], b[r][K + 1][lane], vp, b[r - 1][K][lane], true);
                }
                double v0[K], e0;
                entering(sg, v0, e0);
#pragma unroll
                for (int k = 0; k < K; ++k) v0[k] *= kVu;
                carry(dl[0], b[0][K][lane], b[0][K + 1][lane], v0, e0, t0 > 0);
                if ((sg & 7) == 0) {
#pragma unroll
                    for (int i = 0; i < NS; ++i) {
                        gn[i] += gs[i];
                        gs[i] = 0.0;
                    }
                }
            }
            meet();
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            gn[2 + k] *= 0.5 / kVu;
            gn[2 + K + k] *= 0.5;
            gn[2 + 2 * K + k] *= 0.5;
        }
        meet();                            // warp 1's results
#pragma unroll
        for (int i = 0; i < 3 * I; ++i) gn[NS + i] = sm.comb[i][lane];
        double ll = sm.comb[3 * I][lane] - logh - 0.5 * kLog2Pi * (double)T;
        if (!(ll > -INFINITY)) ll = -INFINITY;
        double gfull[kMaxD];
        natural_to_theta_f64<K, I>(q, gn, full, a.m.gamma, gfull);
        if (!active) return;
        a.ll[p] = ll;
        for (int k = 0; k < a.m.d; ++k) a.grad[k * P + p] = gfull[a.m.has_free ? a.m.free_idx[k] : k];
    }

    __device__ __forceinline__ static void mixture_warp(Smem& sm, EgarchFx<K, I> fx,
                                                        const EgarchParams<double, K, I>& q, bool fixed, int lane,
                                                        int T, int nseg)
    {
        // forward: sum_t log mixture density
        double e1 = 0.0, e2 = 0.0, lm64 = 0.0;   // sums of eps, eps^2 (2^-53, 2^-106); densities in FP64
        int n64 = 0;
        unsigned __int128 scw = 0;
        meet();                            // (segment 0 is warp 0's alone)
        for (int sg = 0; sg < nseg; ++sg) {
            const int n = min(kSeg, T - sg * kSeg);
            const double* es = &sm.x[sg & 1][0][lane];
            double u1 = 0.0, u2 = 0.0;
            for (int h = 0; h < n; h += 8) {
                fx.sc = 0;
#pragma unroll 2
                for (int r = h; r < min(n, h + 8); ++r) {
                    const double e = es[r * 32];
                    const uint64_t pm = fx.pm, sc = fx.sc;
                    const int pe = fx.pe;
                    uint32_t over;
                    fx.mix_terms(e, sm.tab, over);
                    // (a shock past fixed point's range has its square taken in its own units)
                    const bool far = (fx_bits(e) << 1) >= (uint64_t)(1023 + 60) << 53;
                    if (over != 0u || !fixed || far) {
                        double r8[I];
                        fx.pm = pm;
                        fx.pe = pe;
                        fx.sc = sc;
                        lm64 += weights_f64(q, e * 0x1p-53, sm.tab, r8);
                        ++n64;
                    } else {
                        u1 += e;
                        u2 = fma(e, e, u2);
                    }
                }
                scw += fx.sc;
            }
            e1 += u1;
            e2 += u2;
            meet();
        }
        double lm = lm64;
        if (fixed) {
            const double nf = (double)(T - n64);
            lm += kLn2 * (fx_to_double((__int128)scw, -55) + (double)fx.pe + log2((double)fx.pm * 0x1p-62)) -
                  0.5 * (fx.a0 * fx.a0) * (e2 * 0x1p-106 - 2.0 * fx.m0 * (e1 * 0x1p-53) + nf * (fx.m0 * fx.m0)) +
                  nf * (kLn2 * fx.c0);
        }
        // backward: dl/deps and the component sums
        fx.natural_shocks();
        double a2[I], s0[I], s1[I], s2[I], g[3 * I];
#pragma unroll
        for (int i = 0; i < I; ++i) {
            const double ai = 1.0 / q.sig[i];
            a2[i] = ai * ai;
            s0[i] = s1[i] = s2[i] = 0.0;
            g[i] = g[I + i] = g[2 * I + i] = 0.0;
        }
        meet();                            // (step 0 is warp 0's alone)
        for (int j = 1; j < nseg + 2; ++j) {
            if (j <= nseg) {
                const int sg = nseg - j, n = min(kSeg, T - sg * kSeg);
                const double(*b)[W][32] = sm.slab[(j - 1) % 3];
                double* dl = &sm.x[(j - 1) & 1][0][lane];
#pragma unroll 2
                for (int r = n - 1; r >= 0; --r) {
                    const double es = b[r][K][lane];
                    double ri[I];
                    if (!(fixed && fx.weights(es, ri, sm.tab))) weights_f64(q, es, sm.tab, ri);
                    double d = 0.0;
#pragma unroll
                    for (int i = 0; i < I; ++i) {
                        const double z = es - q.mu[i];
                        const double rz = ri[i] * z;
                        d = fma(-rz, a2[i], d);
                        s0[i] += ri[i];
                        s1[i] += rz;
                        s2[i] = fma(rz, z, s2[i]);
                    }
                    dl[r * 32] = d;
                }
#pragma unroll
                for (int i = 0; i < I; ++i) {
                    g[i] += s0[i];
                    g[I + i] += s1[i];
                    g[2 * I + i] += fma(-a2[i], s2[i], s0[i]);
                    s0[i] = s1[i] = s2[i] = 0.0;
                }
            }
            meet();
        }
#pragma unroll
        for (int i = 0; i < I; ++i) {
            sm.comb[i][lane] = g[i];
            sm.comb[I + i][lane] = a2[i] * g[I + i];
            sm.comb[2 * I + i][lane] = q.sig[i] * g[2 * I + i];
        }
        sm.comb[3 * I][lane] = lm;
        meet();                            // warp 0 takes them
    }
};

}  // namespace smc
