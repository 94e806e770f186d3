// FP64 log likelihood with its gradient by the adjoint recurrence of
// adjoint.cuh, on the integer pipes wherever FP64 is not needed.
//
// FP64 instructions bound it (about 64 cycles each per warp, whatever the
// occupancy), so they are what is saved here:
//   - the forward pass and each segment's recomputation run in the
//     fixed-point recursion (EgarchFx; the FP64 recursion takes particles out
//     of its ranges);
//   - the component weights r_i come from integer exponentials and an integer
//     reciprocal of their sum;
//   - the sums over t keep r_i (exact integers), r_i eps and r_i eps^2 per
//     component, from which d log p_i, d mu_i and d a_i follow once at the end
//     (4 FP64 instructions per component and observation instead of 11).
// About 40 FP64 instructions per particle and observation at K = 2, I = 2
// against 230 with FP64 exponentials and division.
// Measured (value and gradient, K = 2, I = 2, 2,049 particles x 1,037
// observations, a warp per scheduler at most): 7.9 ms in FP64 throughout, 2.7 ms.
#pragma once

#include "adjoint.cuh"

namespace smc {

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

template <int K, int I, int kSeg>
struct AdjointF64 {
    EgarchFxSafe<K, I> mdl;
    double a2[I], m2[I];         // a_i^2, mu_i a_i^2, times 2^-59 (the units of r_i)

    __device__ __forceinline__ void setup(const double* th, int has_gamma, int eps0_zero, const uint64_t* tab)
    {
        mdl.setup(th, has_gamma, eps0_zero, tab);
#pragma unroll
        for (int i = 0; i < I; ++i) {
            const double a = 1.0 / mdl.q.sig[i];
            a2[i] = a * a * 0x1p-59;
            m2[i] = mdl.q.mu[i] * a2[i];
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
        mdl.state_out(st);
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

    // r_i (2^-59) with the terms x_i formed in FP64 (any parameters and shock).
    __device__ __noinline__ void weights_f64(double eps, uint64_t* r) const
    {
        double x[I], mx = -INFINITY;
#pragma unroll
        for (int i = 0; i < I; ++i) {
            const double z = (eps - mdl.q.mu[i]) / mdl.q.sig[i];
            x[i] = log(mdl.q.p[i]) - log(mdl.q.sig[i]) - 0.5 * z * z;
            mx = fmax(mx, x[i]);
        }
        uint64_t s = 0;
#pragma unroll
        for (int i = 0; i < I; ++i) {
            r[i] = fx_exp_q61(mx - x[i], mdl.tab);
            s += r[i];
        }
        const uint64_t Y = fx_rcp(s);
#pragma unroll
        for (int i = 0; i < I; ++i) r[i] = fx_mulhi(r[i], Y);
    }

    // Reverse sweep; gn (EgarchNat<double, K, I>::kNp) receives d l / d natural
    // parameters.  buf: this thread's slab, [kSeg][v_1..v_K, eps, 1/h][stride].
    __device__ __forceinline__ void reverse(const double* __restrict__ y, int T, const double* ckpt, size_t P, int p,
                                            double* buf, int stride, double* gn)
    {
        constexpr int NS = 2 + 3 * K;      // mu, log sigma, alpha, beta, gamma
        constexpr int W = K + 2;
        double gs[NS], s1[I], s2[I], vb[K];
        uint64_t s0[I];
        for (int i = 0; i < NS + 3 * I; ++i) gn[i] = 0.0;
#pragma unroll
        for (int i = 0; i < NS; ++i) gs[i] = 0.0;
#pragma unroll
        for (int i = 0; i < I; ++i) {
            s1[i] = s2[i] = 0.0;
            s0[i] = 0;
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
        auto back = [&](double eps, double inv, const double* vp, double ep, bool has_prev) {
            double eb = -eps;
            if constexpr (I >= 2) {
                uint64_t r[I];
                if (!(fixed && fx.weights(eps, r, mdl.tab))) weights_f64(eps, r);
                eb = 0.0;
#pragma unroll
                for (int i = 0; i < I; ++i) {
                    const double ri = (double)(int64_t)r[i];
                    const double re = ri * eps;
                    eb = fma(-re, a2[i], fma(ri, m2[i], eb));
                    s0[i] += r[i];
                    s1[i] += re;
                    s2[i] = fma(re, eps, s2[i]);
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
                fx.state_out(s, kLn2);
                put(buf + (size_t)r * W * stride, stride, s, s[K], fx.inv_h());
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
            if constexpr (I >= 2) {            // (r_i <= 2^59: the sum of 16 is at most 2^63)
                static_assert(kSeg <= 16);
#pragma unroll
                for (int i = 0; i < I; ++i) {
                    gn[NS + i] += (double)s0[i] * 0x1p-59;
                    s0[i] = 0;
                }
            }
            if ((sg & 7) == 0) {
#pragma unroll
                for (int i = 0; i < NS; ++i) {
                    gn[i] += gs[i];
                    gs[i] = 0.0;
                }
#pragma unroll
                for (int i = 0; i < I; ++i) {
                    gn[NS + I + i] += s1[i];
                    gn[NS + 2 * I + i] += s2[i];
                    s1[i] = s2[i] = 0.0;
                }
            }
        }
        // sum r_i, sum r_i eps, sum r_i eps^2 -> d log p_i, d mu_i, d a_i
        if constexpr (I >= 2) {
#pragma unroll
            for (int i = 0; i < I; ++i) {
                const double r0 = gn[NS + i], r1 = gn[NS + I + i] * 0x1p-59, r2 = gn[NS + 2 * I + i] * 0x1p-59;
                const double a = 1.0 / q.sig[i], mu = q.mu[i];
                gn[NS + I + i] = a * a * (r1 - mu * r0);
                gn[NS + 2 * I + i] = q.sig[i] * r0 - a * (r2 - mu * (2.0 * r1 - mu * r0));
            }
        }
    }
};

}  // namespace smc
