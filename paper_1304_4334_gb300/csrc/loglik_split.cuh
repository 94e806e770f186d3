// FP64 log likelihood of few particles with the work of 32 of them given to
// several warps (I >= 2).
//
// A launch with fewer warps than the SMs have schedulers (four each) is bound
// by one warp's time per observation, 1,190 cycles at K=3, I=4 in
// EgarchFxSafe, while most schedulers have nothing to issue.  Here the first
// warp carries the volatility chain and leaves each segment's shocks in shared
// memory, and one (I = 2) or two others take their mixture densities a segment
// behind, alternate observations each.  Sums stay exact integers, as in
// EgarchFx; only the product of the mixture sums is taken in another order.
// A segment in which a particle's state leaves the fixed-point ranges is taken
// in FP64 by the first warp, a shock whose mixture terms leave them by FP64
// terms relative to component 0.
// Measured at T=1000, one warp -> split: up to one block per SM K=1,I=2 389 ->
// 240 us, K=3,I=2 464 -> 356, K=2,I=3 563 -> 316, K=3,I=4 770 -> 381; 9,728
// particles at K=3,I=4 779 -> 452 us, 10,007 x 3,089 2.28 -> 1.47 ms.
#pragma once

#include "adjoint_f64.cuh"
#include "kernels.cuh"
#include "phase.cuh"

namespace smc {

template <int K, int I>
struct LoglikSplit {
    static constexpr int kSeg = 32, kMix = I > 2 ? 2 : 1, kThreads = 32 * (1 + kMix);
    static constexpr int kBlocks = I > 2 ? 4 : 6;   // 168 registers: at 218-250, without a cap, two fit an SM
    struct Smem {
        double x[2][kSeg][32];             // shocks (2^-53)
        double ys[2][kSeg];
        uint64_t lo[kMix][32], hi[kMix][32];   // sum of m_t (2^-55)
        double lm[kMix][32];               // log of the product; FP64 densities
        uint64_t tab[256];
    };

    // All warps, each from its own place in the code.
    __device__ __forceinline__ static void meet() { asm volatile("barrier.sync 1, %0;" ::"n"(kThreads) : "memory"); }

    // log of the mixture density relative to component 0's, in FP64.
    __device__ __noinline__ static double relative(const EgarchFx<K, I>& fx, double e)
    {
        double d[EgarchFx<K, I>::kM], mx = 0.0;
#pragma unroll
        for (int i = 0; i < I - 1; ++i) {
            d[i] = fma(fma(fx.A[i], e, fx.B[i]), e, fx.C[i]) * 0x1p-55;
            mx = fmax(mx, d[i]);
        }
        double s = exp2(-mx);
#pragma unroll
        for (int i = 0; i < I - 1; ++i) s += exp2(d[i] - mx);
        return kLn2 * mx + log(s);
    }

    // Observations r0, r0 + kMix, ... < r1 one by one, those out of range in FP64.
    __device__ __noinline__ static double singly(EgarchFx<K, I>& fx, const EgarchParams<double, K, I>& q, bool fixed,
                                                 const double* es, int r0, int r1, const uint64_t* tab)
    {
        double sum = 0.0;
        for (int r = r0; r < r1; r += kMix) {
            const double e = es[r * 32];
            const uint64_t pm = fx.pm, sc = fx.sc;
            const int pe = fx.pe;
            uint32_t over;
            fx.mix_terms(e, tab, over);
            if (over != 0u || !fixed) {
                fx.pm = pm;
                fx.pe = pe;
                fx.sc = sc;
                double ri[I];
                sum += fixed ? relative(fx, e) : weights_f64(q, e * 0x1p-53, tab, ri);
            }
        }
        return sum;
    }

    __device__ __forceinline__ static void mixture_warp(Smem& sm, EgarchFx<K, I> fx,
                                                        const EgarchParams<double, K, I>& q, bool fixed, int m,
                                                        int lane, int T, int nseg)
    {
        double lm64 = 0.0;
        unsigned __int128 scw = 0;
        meet();                            // (segment 0 is the first warp's alone)
        for (int sg = 0; sg < nseg; ++sg) {
            const int n = min(kSeg, T - sg * kSeg);
            const double* es = &sm.x[sg & 1][0][lane];
            for (int h = m; h < n; h += 8 * kMix) {
                const int end = min(n, h + 8 * kMix);
                const uint64_t pm = fx.pm;
                const int pe = fx.pe;
                uint32_t any = fixed ? 0u : 1u;
                fx.sc = 0;
#pragma unroll 2
                for (int r = h; r < end; r += kMix) {
                    uint32_t over;
                    fx.mix_terms(es[r * 32], sm.tab, over);
                    any |= over;
                }
                if (any != 0u) {
                    EgarchFx<K, I> f = fx;
                    f.pm = pm;
                    f.pe = pe;
                    f.sc = 0;
                    lm64 += singly(f, q, fixed, es, h, end, sm.tab);
                    fx.pm = f.pm;
                    fx.pe = f.pe;
                    fx.sc = f.sc;
                }
                scw += fx.sc;
            }
            meet();
        }
        sm.lo[m][lane] = (uint64_t)scw;
        sm.hi[m][lane] = (uint64_t)(scw >> 64);
        sm.lm[m][lane] = lm64 + (fixed ? kLn2 * ((double)fx.pe + log2((double)fx.pm * 0x1p-62)) : 0.0);
        meet();                            // the first warp takes them
    }

    // Returns log p(y_1:T | theta), the end state in st.
    __device__ __forceinline__ static double chain_warp(Smem& sm, EgarchFx<K, I> fx,
                                                        const EgarchParams<double, K, I>& q, int eps0_zero,
                                                        bool fixed, int lane, const double* __restrict__ y, int T,
                                                        int nseg, double* st)
    {
        EgarchF64<K, I> w;
        bool out = !fixed, ready = false;
        double lh64 = 0.0, q64 = 0.0;      // FP64 segments: log h; (eps - mu_0)^2
        int n64 = 0;
        unsigned __int128 sx = 0, s2 = 0;
        __int128 s1 = 0;
        double yn = lane < T ? y[lane] : 0.0;
        for (int sg = 0; sg < nseg; ++sg) {
            const int t0 = sg * kSeg, n = min(kSeg, T - t0);
            double* ys = sm.ys[sg & 1];
            ys[lane] = yn;
            __syncwarp();
            yn = t0 + kSeg + lane < T ? y[t0 + kSeg + lane] : 0.0;
            double* es = &sm.x[sg & 1][0][lane];
            int64_t V0[K];
            const uint64_t E0 = fx.E;
            const int32_t neg0 = fx.neg;
#pragma unroll
            for (int k = 0; k < K; ++k) V0[k] = fx.V[k];
            fx.bad = 0;
            fx.sx = fx.s2 = 0;
            fx.s1w = 0;
            auto put = [&](int r) {
                const int64_t e = fx.shock();
                fx.s1 += e;
                es[r * 32] = (double)e;
            };
            if (t0 == 0) fx.template chain<true>(ys[0], sm.tab);
            else fx.template chain<false>(ys[0], sm.tab);
            put(0);
            fx.flush();
            for (int h = 1; h < n; h += 8) {
                const int end = min(n, h + 8);
#pragma unroll 2
                for (int r = h; r < end; ++r) {
                    fx.template chain<false>(ys[r], sm.tab);
                    put(r);
                }
                fx.flush();
            }
            if (fx.bad == 0u && !out) {
                sx += fx.sx;
                s2 += fx.s2;
                s1 += fx.s1w;
            } else {
                if (!ready) w.setup(q, eps0_zero, sm.tab);
                ready = true;
                if (!out) {
#pragma unroll
                    for (int k = 0; k < K; ++k) fx.V[k] = V0[k];
                    fx.E = E0;
                    fx.neg = neg0;
                    fx.state_out(st, kLn2);
                    w.load_state(st);
                }
                lh64 += GradSplit<K, I>::segment_f64(w, q.log_sigma_y, y, t0, n, 0x1p53, es, 32, nullptr, nullptr);
                for (int r = 0; r < n; ++r) {
                    const double z = es[r * 32] * 0x1p-53 - fx.m0;
                    q64 = fma(z, z, q64);
                }
                n64 += n;
                out = !(fixed && fx.enter(w.v, w.eps));
            }
            meet();
        }
        meet();                            // nseg segments of the other warps
        if (out) {
            w.state_out(st);
        } else {
            fx.state_out(st, kLn2);
            st[K] = fx.shock_of(y[T - 1], sm.tab);
        }
        meet();                            // their results
        unsigned __int128 scw = 0;
        double lm = 0.0;
#pragma unroll
        for (int m = 0; m < kMix; ++m) {
            scw += ((unsigned __int128)sm.hi[m][lane] << 64) + sm.lo[m][lane];
            lm += sm.lm[m][lane];
        }
        const double sle = fx_to_double((__int128)(scw - sx) + ((__int128)(T - n64) << 63), -55);
        double ll = kLn2 * sle + lm - lh64 - 0.5 * kLog2Pi * (double)T;
        if (fixed) {
            const double nf = (double)(T - n64);
            const double qd = fx_to_double((__int128)s2, -86) - 2.0 * fx.m0 * fx_to_double(s1, -53) +
                              nf * (fx.m0 * fx.m0) + q64;
            ll += (double)T * (kLn2 * fx.c0) - 0.5 * (fx.a0 * fx.a0) * qd;
        }
        return ll;
    }
};

template <int K, int I>
__global__ void __launch_bounds__(LoglikSplit<K, I>::kThreads, LoglikSplit<K, I>::kBlocks) k_loglik_split(LoglikArgs a)
{
    __shared__ typename LoglikSplit<K, I>::Smem sm;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < 256; i += blockDim.x) sm.tab[i] = g_exp2_neg256[i];
    const int p = blockIdx.x * 32 + lane;
    const bool active = p < a.P;
    const int pp = active ? p : a.P - 1;
    const size_t P = (size_t)a.P;
    const int T = a.T, nseg = (T + LoglikSplit<K, I>::kSeg - 1) / LoglikSplit<K, I>::kSeg;
    double th[kMaxD], full[kMaxD];
    for (int i = 0; i < a.m.d; ++i) th[i] = a.theta[i * P + pp];
    full_theta<double>(a.m, th, full);
    EgarchParams<double, K, I> q;
    egarch_transform<double, K, I>(full, a.m.gamma, q);
    EgarchFx<K, I> fx;
    fx.setup(q.mu_y, q.log_sigma_y, q.alpha, q.beta, q.gamma, q.p, q.mu, q.sig, a.m.eps0_zero, kLog2e);
    const bool fixed = fx.bad == 0u;
    __syncthreads();
    if (warp > 0) {
        LoglikSplit<K, I>::mixture_warp(sm, fx, q, fixed, warp - 1, lane, T, nseg);
        return;
    }
    double st[K + 1];
    double ll = LoglikSplit<K, I>::chain_warp(sm, fx, q, a.m.eps0_zero, fixed, lane, (const double*)a.obs, T, nseg, st);
    if (isnan(ll)) ll = -INFINITY;
    if (active) {
        a.ll[p] = ll;
        if (a.lp) a.lp[p] = log_prior(a.m, th);
        if (a.state)
            for (int k = 0; k < K + 1; ++k) a.state[k * P + p] = st[k];
    }
}

// Up to four blocks per SM, what the register cap keeps resident (I > 2; I = 2
// would fit six): there the split is ahead at every I > 2 (19,456 particles,
// T=1000, one warp -> split: K=1,I=3 548 -> 406 us, K=4,I=4 803 -> 671) and at
// I = 2 for K <= 2 (K=2 425 -> 414); with a second wave it is not (K=2,I=3 780
// -> 807).  At I = 2 and K >= 3 the chain is the longer part and two of them
// already fill a scheduler's time: ahead to two blocks per SM (K=3, 9,728
// particles 465 -> 360 us; 12,000: 466 -> 483).
template <int K, int I>
cudaError_t launch_loglik_split(const LoglikArgs& a, cudaStream_t s, bool* taken)
{
    const int blocks = (a.P + 31) / 32;
    *taken = a.by_size && blocks <= (I == 2 && K >= 3 ? 2 : 4) * device_sm_count();
    if (!*taken) return cudaSuccess;
    k_loglik_split<K, I><<<blocks, LoglikSplit<K, I>::kThreads, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace smc
