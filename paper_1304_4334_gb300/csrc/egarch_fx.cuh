// The double-precision EGARCH(K, I) likelihood recursion in 64-bit fixed point.
//
// On this part an FP64 instruction holds its scheduler's FP64 pipe for about
// 64 cycles per warp (two lanes per clock and SM) while a 32 x 32 -> 64-bit
// integer multiply-add costs a few.  The recursion written in FP64 takes 141
// FP64 instructions per particle and observation at K = 2, I = 2 (most of
// them inside exp and log), so the FP64 pipe is its only bound.  Here the
// state and every exponential are 64-bit integers:
//   - volatility factors V_k = v_k log2(e) / 2 in units of 2^-55, the shock
//     |eps_t| in units of 2^-53 with its sign apart;
//   - log2 h_t = log2 sigma_Y + sum_k V_k is then an exact integer sum whose
//     integer and fraction parts index 2^-X = 2^-n 2^(-j/256) 2^-r directly,
//     r < 2^-8 by a degree-5 polynomial (2^-60 relative);
//   - mixture terms relative to component 0, the one with the largest sigma:
//     d_i = x_i - x_0 is a quadratic in eps (two FP64 FMAs; y_t - mu_Y and the
//     conversion of eps are the other FP64 work of an observation), brought to fixed
//     point; m = max(0, d_i), s_t = sum_i 2^(d_i - m) in [1, I], and one
//     logarithm of the running product of the s_t for the whole series;
//   - sums of log2 h_t, m, eps_t and eps_t^2 are exact integer sums; x_0's
//     own sum follows from the last two at the end.
// Ranges: |V_k| < 64 (log2 units; 32 at K = 4), |eps| < 128 (less where beta
// passes 1.3, so that no product leaves 64 bits), d_i < 16, parameters as
// setup() checks (one that is not finite fails).  A particle that leaves them
// sets `bad`: its owner repeats the observations since the last save() in the
// FP64 recursion (EgarchF64), which takes any value.  V_k and eps have absolute
// units, so the state's v_k carries 2^-55 of log2 h whatever its size; shocks
// and component weights that leave the recursion (end state, adjoint) are formed
// with all of FP64's bits.
//
// Measured, random-walk iteration at K = 2, I = 2, 65,536 particles x 5,000
// observations: 76.1 ms with the recursion in FP64, 5.06 ms (about 300
// instructions per particle and observation; x 500: the FP64 pipe 54% busy, the
// integer multiplier 44%, issue 41%, and a warp waits longest for its own
// dependent instructions, at 3.4 warps per scheduler); likelihood at K = 3,
// I = 4, 10,007 x 3,089: 17.8 ms, 2.28 ms with one warp per 32 particles (one
// warp per scheduler: the chain's latency), 1.47 ms with three (LoglikSplit);
// mutation of 1,024 x 500 at K = I = 1: 0.55 ms, 0.14 ms.  Errors against
// 113-bit arithmetic: log likelihood 2e-16 relative at T = 5,000 (2.5e-15 in
// FP64, whose running sum rounds), end state 0.4 to 1 of FP64's.
//
// Plain C++ apart from the intrinsics' names: the CPU test compiles this file
// with the host compiler and compares it with long double.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#if defined(__CUDACC__)
#define SMC_FX __device__ __forceinline__
#else
#define SMC_FX inline
#endif

namespace smc {

// round(ln2^k / k! * 2^s) for k = 1..5, s = 64, 56, 36, 32, 24
constexpr uint64_t kFxC1 = 12786308645202655660ull;
constexpr uint64_t kFxC2 = 17310144115608349ull;
constexpr uint32_t kFxC3 = 3814213304u;
constexpr uint32_t kFxC4 = 41309550u;
constexpr uint32_t kFxC5 = 22370u;
constexpr double kFxLn2 = 0.69314718055994530942;
constexpr double kFxLog2eLo = 0x1.777d0ffda0d24p-56;   // log2(e) less its FP64 rounding
constexpr uint64_t kFxAbsMean = 14718372293494604904ull;   // round((2 / pi)^1/2 * 2^64)

SMC_FX uint64_t fx_bits(double x)
{
#if defined(__CUDA_ARCH__)
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t b;
    std::memcpy(&b, &x, 8);
    return b;
#endif
}

SMC_FX bool fx_isnan(double x) { return (fx_bits(x) << 1) > 0xffe0000000000000ull; }

SMC_FX uint32_t fx_mulhi32(uint32_t a, uint32_t b)
{
#if defined(__CUDA_ARCH__)
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}

SMC_FX int fx_clz64(uint64_t x)
{
#if defined(__CUDA_ARCH__)
    return __clzll((long long)x);
#else
    return __builtin_clzll(x);
#endif
}

// x >> n for n >= 0, zero from 64 on.
SMC_FX uint64_t fx_shr(uint64_t x, int n)
{
#if defined(__CUDA_ARCH__)
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));   // clamps n at 64
    return r;
#else
    return n > 63 ? 0ull : x >> n;
#endif
}

// floor(a b / 2^64) less at most 2 units (the low halves' product is left out).
SMC_FX uint64_t fx_mulhi(uint64_t a, uint64_t b)
{
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    return (uint64_t)ah * bh + fx_mulhi32(al, bh) + fx_mulhi32(ah, bl);
}

// 2^-x for x = n + X 2^-55 (the low 55 bits of X used): M 2^-63, M in (2^62, 2^63];
// tab[j] = round(2^(63 - j/256)), M = tab[j] 2^-r.  With r = rho 2^-8 the fraction below the
// table's, 2^-r = 1 - rho (k1 - rho (k2 - rho (k3 - rho (k4 - rho k5)))),
// k_i = ln2^i / i! 2^-8i; k5, k4 in units of 2^-64, k3 of 2^-60, k2 and k1 of
// 2^-72: each level carries the bits that reach the result, and one shift
// at the end puts the sum into the table's units.
SMC_FX uint64_t fx_exp2neg_q(uint64_t X)   // 1 - 2^-r in units of 2^-72
{
    const uint64_t R = X << 17;
    const uint32_t rho = (uint32_t)(R >> 32);
    const uint32_t t4 = kFxC4 - fx_mulhi32(rho, kFxC5);
    const uint32_t t3 = kFxC3 - (fx_mulhi32(rho, t4) >> 4);
    const uint64_t t2 = kFxC2 - (((uint64_t)rho * t3) >> 20);
    const uint64_t t1 = kFxC1 - fx_mulhi(R, t2);
    return fx_mulhi(R, t1);
}
SMC_FX uint64_t fx_exp2neg(uint64_t X, const uint64_t* tab)
{
    const uint64_t T = tab[(uint32_t)(X >> 47) & 255u];
    return T - (fx_mulhi(T, fx_exp2neg_q(X)) >> 8);
}

// |x| in units of 2^-56 for |x| < 128 (truncated); false beyond, and for inf, NaN.
SMC_FX bool fx_fixed56(double x, uint64_t& X)
{
    const uint64_t b = fx_bits(x);
    const int s = 1030 - ((int)(b >> 52) & 0x7ff);
    const uint64_t m = (b << 11) | 0x8000000000000000ull;
    X = fx_shr(m, s > 0 ? s : 0);
    return s > 0;
}

constexpr uint64_t kFxLog2e = 13306513097844322492ull;   // round(log2(e) * 2^63)

// e^-w for w >= 0 in units of 2^-61 (0 for w >= 128, inf and NaN).
SMC_FX uint64_t fx_exp_q61(double w, const uint64_t* tab)
{
    uint64_t X;
    if (!fx_fixed56(w, X)) return 0ull;
    X = fx_mulhi(X, kFxLog2e);                       // w log2(e), units of 2^-55
    const int n = (int)(X >> 55) + 2;
    return fx_shr(fx_exp2neg(X, tab), n);
}

#if defined(__CUDACC__)
__device__ __noinline__ inline double fx_exp_library(double x) { return exp(x); }
#else
inline double fx_exp_library(double x) { return std::exp(x); }
#endif

// M 2^(-63 - n) for M in (2^62, 2^63] as FP64 (normal range).
SMC_FX double fx_pack(uint64_t M, int n)
{
    const uint64_t r = ((M + 512ull) >> 10) + ((uint64_t)(uint32_t)(1021 - n) << 52);
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((long long)r);
#else
    double d;
    std::memcpy(&d, &r, 8);
    return d;
#endif
}

// 2^123 / s for s in [2^61, 2^63], within a few units of 2^-59 relative.
SMC_FX uint64_t fx_rcp(uint64_t s)
{
    const uint32_t sh = (uint32_t)(s >> 32);
#if defined(__CUDA_ARCH__)
    const float y = __frcp_rn(__uint2float_rn(sh));
    const uint32_t yb = __float_as_uint(y);
#else
    const float y = 1.0f / (float)sh;
    uint32_t yb;
    std::memcpy(&yb, &y, 4);
#endif
    // y 2^91 = mantissa 2^(exponent - 127 - 23 + 91)
    uint64_t Y = (uint64_t)((yb & 0x7fffffu) | 0x800000u) << (((yb >> 23) - 59u) & 63u);
    int64_t e = (int64_t)((1ull << 59) - fx_mulhi(s, Y));                       // relative error 2^-59
    Y += (uint64_t)(((int64_t)(int32_t)(uint32_t)(Y >> 32) * (int32_t)(e >> 8)) >> 19);
    e = (int64_t)((1ull << 59) - fx_mulhi(s, Y));
    Y += (uint64_t)(((int64_t)(int32_t)(uint32_t)(Y >> 32) * (int32_t)e) >> 27);
    return Y;
}

// e^-x in FP64 without FP64 instructions for |x| < 700, within a unit in the
// last place (from 128 on x log2(e) has more than 64 bits: its full product is
// taken, log2(e)'s own rounding is 2^-54 of the exponent at most); the library's
// exponential where the result leaves the normal range, and its limits past that.
SMC_FX double fx_exp_neg(double x, const uint64_t* tab)
{
    const uint64_t sg = (uint64_t)((int64_t)fx_bits(x) >> 63);
    uint64_t X;
    int n;
    if (fx_fixed56(x, X)) {
        X = fx_mulhi(X, kFxLog2e);
        X = (X ^ sg) - sg;
        n = (int)((int64_t)X >> 55);
    } else if (std::fabs(x) < 700.0) {
        const uint64_t b = fx_bits(x);                // |x| = m 2^(e - 1023 - 63), e from 1030 to 1032
        const uint64_t m = (b << 11) | 0x8000000000000000ull;
        const unsigned __int128 w = ((unsigned __int128)m * kFxLog2e) >> (1094 - ((int)(b >> 52) & 0x7ff));
        const __int128 v = sg ? -(__int128)w : (__int128)w;   // units of 2^-55
        n = (int)(v >> 55);
        X = (uint64_t)v;
    } else if (std::fabs(x) < 1024.0) {
        return fx_exp_library(-x);
    } else {
        return x > 0.0 ? 0.0 : (x < 0.0 ? INFINITY : x);   // (a NaN stays one)
    }
    return fx_pack(fx_exp2neg(X, tab), n);            // e^-x = M 2^(-63 - n)
}

// |x| < c (c > 0); false for a NaN.  On the integer pipe: a comparison holds the
// FP64 pipe like any other FP64 instruction.
SMC_FX bool fx_below(double x, double c) { return (fx_bits(x) << 1) < (fx_bits(c) << 1); }

// Nearest integer to x 2^s (ties away from zero) for |x| 2^s < 2^62, from the
// bits of x: a product and a conversion on the FP64 pipe take 128 cycles per
// warp, and a setup has 2 + 3 K of them.
SMC_FX int64_t fx_scaled(double x, int s)
{
    const uint64_t b = fx_bits(x);
    const int sh = 1085 - s - ((int)(b >> 52) & 0x7ff);   // |x| 2^s = m 2^-(sh + 1)
    const uint64_t r = (fx_shr((b << 11) | 0x8000000000000000ull, sh > 0 ? sh : 0) + 1ull) >> 1;
    const uint64_t sg = (uint64_t)((int64_t)b >> 63);
    return (int64_t)((r ^ sg) - sg);
}

// v 2^e in FP64 (rounded once, normal range; zero for zero), likewise.
SMC_FX double fx_to_double(__int128 v, int e)
{
    const uint64_t sg = (uint64_t)(v >> 127);
    const unsigned __int128 m = sg ? -(unsigned __int128)v : (unsigned __int128)v;
    const uint64_t hi = (uint64_t)(m >> 64), lo = (uint64_t)m;
    if ((hi | lo) == 0ull) return 0.0;
    const int z = hi ? fx_clz64(hi) : 64 + fx_clz64(lo);
    const uint64_t t = hi ? (hi << z) | fx_shr(lo, 64 - z) : lo << (z - 64);   // m = t 2^(64 - z), bit 63 set
    const double d = fx_pack(t >> 1, z - 128 - e);
    return sg ? -d : d;
}

// Product of the mixture sums s (units 2^-61, in [1, 4]): pm 2^(pe - 62) with
// pm kept in [2^62, 2^63).
SMC_FX void fx_product(uint64_t& pm, int& pe, uint64_t s)
{
    const uint64_t v = fx_mulhi(pm, s);
    const int z = fx_clz64(v) - 1;
    pm = v << z;
    pe += 3 - z;
}

template <int K, int I>
struct EgarchFx {
    static constexpr int kM = I > 1 ? I - 1 : 1;
    // |V_k| < kVmax: with |log2 sigma_Y| < 256 - K kVmax, log2 h_t + 256 stays in [0, 512)
    static constexpr int kVmax = K < 4 ? 64 : 32;
    double mu;
    uint64_t ly;                         // log2 sigma_Y + 256
    int32_t ah[K], al[K];                // (1 + alpha_k) / 2 in 30-bit limbs (units 2^-61)
    int32_t cph[K], cpl[K];              // (beta_k +- gamma_k) log2(e)/2 2^-cs in 29-bit limbs (units
    int32_t cmh[K], cml[K];              //   2^-60), for a positive and a negative shock
    int cs;
    int64_t nb[K];                       // -beta_k (2/pi)^1/2 log2(e)/2
    int32_t nf[K];                       // the constant's fraction (2^-84) with the rounding half
    int32_t na[K];                       // rounding half of the other product (2^-85)
    int64_t v0[K];                       // state after the first update
    double A[kM], B[kM], C[kM];          // d_i 2^55 = (A E + B) E + C, E = eps 2^53
    // state
    int64_t V[K];
    uint64_t E;                          // |eps|
    int32_t eh, el;                      // |eps| 2^cs in 29-bit limbs
    int32_t neg;                         // 0, or -1 for a negative shock
    // sums over up to 8 observations
    uint64_t hh, hl, ll;                 // of the limb products of E^2
    uint64_t sc;                         // m_t (2^-55)
    int64_t s1;                          // eps_t (2^-53)
    uint64_t pm;                         // product of the s_t
    // sums over the series
    unsigned __int128 sx;                // log2 h_t + 256 (2^-55)
    unsigned __int128 s2;                // eps_t^2 (2^-86)
    unsigned __int128 scw;
    __int128 s1w;
    int pe;                              // product: pm 2^(pe - 62)
    double c0, m0, a0;                   // component 0: log2(p / sigma), mu, 1 / sigma
    int ref;                             // its place in the caller's order
    uint64_t M, X;                       // 1 / h_t = M 2^(-63 - n), n = (X >> 55) - 256
    double dy;                           // y_t - mu_Y
    uint32_t bad;

    // Natural parameters (EgarchParams) in; eps0_zero as in EgarchF64.
    SMC_FX void setup(double mu_y, double log_sigma_y, const double* alpha, const double* beta,
                      const double* gamma, const double* p, const double* mum, const double* sig, int eps0_zero,
                      double log2e)
    {
        bool ok = true;
        const double g = 0.5 * log2e;
        mu = mu_y;
        // (the product's rounding error and log2(e)'s own go in separately: a
        // constant error of log2 h_t scales every shock)
        const double lyd = log_sigma_y * log2e;
        ok = ok && fx_below(lyd, 40.0 < 255.0 - K * kVmax ? 40.0 : 255.0 - K * kVmax) && fx_below(mu_y, 1e30);
        const double lye = fma(log_sigma_y, log2e, -lyd) + log_sigma_y * kFxLog2eLo;
        ly = (uint64_t)(ok ? fx_scaled(lyd, 55) + fx_scaled(lye, 55) : 0) ^ (1ull << 63);
        bool c0ok = true, c2ok = true;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const double c = g * (beta[k] + std::fabs(gamma[k]));
            ok = ok && fx_below(c, 15.8);   // (each by itself: a NaN fails it)
            c0ok = c0ok && fx_below(c, 0.99);
            c2ok = c2ok && fx_below(c, 3.96);
        }
        cs = c0ok ? 0 : (c2ok ? 2 : 4);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            ok = ok && fx_below(alpha[k], 1.0 + 0x1p-52) && !(fx_bits(beta[k]) >> 63);
            int64_t as = fx_scaled(ok ? alpha[k] : 0.0, 60) + (1ll << 60);
            as = as < (1ll << 61) ? as : (1ll << 61) - 1;   // alpha = 1 to FP64 precision
            ah[k] = (int32_t)(as >> 30);
            al[k] = (int32_t)as & 0x3fffffff;
            const int64_t bi = fx_scaled(ok ? beta[k] * g : 0.0, 60 - cs);
            const int64_t gi = fx_scaled(ok ? gamma[k] * g : 0.0, 60 - cs);
            const int64_t cpi = bi + gi, cmi = bi - gi;
            cph[k] = (int32_t)(cpi >> 29);
            cpl[k] = (int32_t)cpi & 0x1fffffff;
            cmh[k] = (int32_t)(cmi >> 29);
            cml[k] = (int32_t)cmi & 0x1fffffff;
            // -beta c, from the rounded beta (the terms beta |eps| and beta c
            // nearly cancel on average, so both carry the same factor) and with
            // bits below the unit (a rounding of it would be amplified by
            // 1 / (1 - alpha)).  The means of what the products leave out are
            // made good here too: the shock's truncation (half a unit of
            // 2^-53) and the low limbs' products (cl el and al vl; el and vl
            // average half a limb).
            const uint64_t w = fx_mulhi((uint64_t)bi, kFxAbsMean) - (uint64_t)((bi >> 54) >> cs);
            const int sh = 5 - cs;                          // 2^-(60 - cs) to 2^-55
            nb[k] = -(int64_t)(w >> sh) - 1;
            const uint32_t fr = (uint32_t)w & ((1u << sh) - 1u);
            nf[k] = (int32_t)(((1u << sh) - fr) << (29 - sh)) + (1 << 28) + (cpl[k] >> 2) + (cml[k] >> 2);
            na[k] = (1 << 29) + (al[k] >> 1);
            v0[k] = eps0_zero ? -(int64_t)((w + ((1u << sh) >> 1)) >> sh) : 0;
        }
        c0 = m0 = 0.0;
        a0 = 1.0;
        ref = 0;
        if (I > 1) {
            // component 0: the one with the largest sigma (changes place with ref)
            double ps[I], ms[I], sg[I], top = sig[0];
#pragma unroll
            for (int i = 1; i < I; ++i) {
                ref = sig[i] > top ? i : ref;
                top = sig[i] > top ? sig[i] : top;
            }
#pragma unroll
            for (int i = 0; i < I; ++i) {
                const bool sw = i > 0 && i == ref;
                ps[i] = sw ? p[0] : p[i];
                ms[i] = sw ? mum[0] : mum[i];
                sg[i] = sw ? sig[0] : sig[i];
                if (sw) {
                    ps[0] = p[i];
                    ms[0] = mum[i];
                    sg[0] = sig[i];
                }
            }
            a0 = 1.0 / sg[0];
            m0 = ms[0];
            c0 = log2(ps[0] * a0);
            ok = ok && std::fabs(c0) < 1000.0 && std::fabs(m0) * a0 < 8.0;
#pragma unroll
            for (int i = 1; i < I; ++i) {
                const double ai = 1.0 / sg[i], u = ms[i] * ai, w = m0 * a0;
                const double q2 = -g * ((ai - a0) * (ai + a0)), q1 = 2.0 * g * (u * ai - w * a0);
                const double q0 = log2(ps[i] * ai) - c0 - g * ((u - w) * (u + w));
                ok = ok && std::fabs(u) < 8.0 && ai < 1e3 && std::fabs(q0) < 1000.0;
                A[i - 1] = q2 * 0x1p-51;
                B[i - 1] = q1 * 0x1p2;
                C[i - 1] = q0 * 0x1p55;
            }
        }
        bad = ok ? 0u : 0x80000000u;
        E = 0;
        eh = el = 0;
        neg = 0;
        hh = hl = ll = sc = 0;
        s1 = 0;
        sx = s2 = scw = 0;
        s1w = 0;
        pm = 1ull << 62;
        pe = 0;
    }

    // beta |eps| + gamma eps - beta c + (2 alpha_s - 1) V, each product to the
    // nearest unit of 2^-55 (nf and na carry the halves that round the shifts;
    // the low limbs' products enter by their means).
    SMC_FX void update_volatility()
    {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int32_t ch = neg ? cmh[k] : cph[k];
            const int32_t cl = neg ? cml[k] : cpl[k];
            const int64_t S = (int64_t)cl * eh + ((int64_t)ch * el + (int64_t)nf[k]);
            const int32_t vh = (int32_t)(V[k] >> 30), vl = (int32_t)((uint32_t)V[k] & 0x3fffffffu);
            const int64_t Q = (int64_t)al[k] * vh + ((int64_t)ah[k] * vl + (int64_t)na[k]);
            const int64_t off = ((int64_t)ah[k] * vh + (Q >> 30)) + (nb[k] - V[k]);   // (before the shock is known)
            V[k] = ((int64_t)ch * eh + off) + (S >> 29);
        }
    }

    // The volatility and the shock of one observation, with their sums.
    template <bool kFirst>
    SMC_FX void chain(double y, const uint64_t* tab)
    {
        if (kFirst) {
#pragma unroll
            for (int k = 0; k < K; ++k) V[k] = v0[k];
        } else {
            update_volatility();
        }
        X = ly;                          // log2 h_t + 256
#pragma unroll
        for (int k = 0; k < K; ++k) {
            X += (uint64_t)V[k];
            // |V_k| < kVmax
            bad |= ((uint32_t)((uint64_t)V[k] >> 32) + (kVmax << 23)) & ~(uint32_t)((kVmax << 24) - 1);
        }
        sx += X;
        const uint64_t T = tab[(uint32_t)(X >> 47) & 255u], q = fx_exp2neg_q(X);
        M = T - (fx_mulhi(T, q) >> 8);   // (kept only where inv_h() is used)
        // |eps| = |y - mu| 2^-X: the 53-bit significand times M, shifted; the
        // shift passes 63 for a zero return
        dy = y - mu;                     // (kept only where eps() is used)
        const uint64_t b = fx_bits(dy);
        const int ed = (int)(uint32_t)(b >> 52) & 0x7ff;
        const uint64_t p0 = fx_mulhi((b << 11) | 0x8000000000000000ull, T);   // beside the polynomial
        const uint64_t prod = p0 - (fx_mulhi(p0, q) >> 8);
        const int sh = (1032 - 256) + (int)(uint32_t)(X >> 55) - ed;
        bad |= (uint32_t)(sh - 3 - cs) & 0x80000000u;   // |eps| 2^cs < 128
        E = fx_shr(prod, sh);
        set_limbs(fx_shr(prod, sh - cs));
        neg = (int32_t)(uint32_t)(b >> 32) >> 31;
        const uint32_t h = (uint32_t)(E >> 31), l = (uint32_t)E & 0x7fffffffu;
        hh += (uint64_t)h * h;
        hl += (uint64_t)h * l;
        ll += (uint64_t)(l >> 4) * (l >> 4);
    }

    // d_i = x_i - x_0 (log2 units, 2^-55) for the shock ed (units 2^-53), -128
    // where it is below that (nothing to the sum).  over: bit 31 set for
    // d_i >= 2^(9 - lim).
    SMC_FX int64_t term(int i, double ed, int lim, uint32_t& over) const
    {
        const double d = fma(fma(A[i], ed, B[i]), ed, C[i]);
        const uint64_t db = fx_bits(d);   // |d| = significand 2^(e - 1023 - 63), shifted
        const int ds = 1086 - ((int)(uint32_t)(db >> 52) & 0x7ff);
        const int32_t nm = (int32_t)(uint32_t)(db >> 32) >> 31;
        uint64_t mag = fx_shr((db << 11) | 0x8000000000000000ull, ds);
        if (ds < 2) mag = 1ull << 62;
        over = (uint32_t)((ds - lim) & ~nm) & 0x80000000u;
        const uint64_t nm64 = (uint64_t)(int64_t)nm;
        return (int64_t)((mag ^ nm64) - nm64);
    }

    // Posterior weights r_i of the components (order of setup's arguments) for
    // the shock ed (units 2^-53); false where a d_i is out of range.  Each is
    // 2^-(m - d_i) / s with its own exponent, so a rare component's weight has
    // as many bits as the others' (0 below 2^-128 of the largest): 1 / s by two
    // Newton steps on integers from the FP32 reciprocal, no FP64 instruction.
    SMC_FX bool weights(double ed, double* r, const uint64_t* tab) const
    {
        int64_t D[I], cur = 0;
        uint32_t over = 0;
        D[0] = 0;
#pragma unroll
        for (int i = 1; i < I; ++i) {
            uint32_t o;
            D[i] = term(i - 1, ed, 2, o);
            over |= o;
            cur = D[i] > cur ? D[i] : cur;
        }
        uint64_t w[I], s = 0;                // 2^-(m - d_i) = w 2^(-63 - n)
        int n[I];
        if (I == 2) {   // one of the two is 1
            const uint64_t Y = (uint64_t)(2 * cur - D[1]);
            const uint64_t e = fx_exp2neg(Y, tab);
            const int ne = (int)(uint32_t)(Y >> 55);
            w[0] = cur > 0 ? e : 1ull << 63;
            w[1] = cur > 0 ? 1ull << 63 : e;
            n[0] = cur > 0 ? ne : 0;
            n[1] = cur > 0 ? 0 : ne;
            s = (1ull << 61) + fx_shr(e, ne + 2);
        } else {
#pragma unroll
            for (int i = 0; i < I; ++i) {
                const uint64_t Y = (uint64_t)(cur - D[i]);
                w[i] = fx_exp2neg(Y, tab);
                n[i] = (int)(uint32_t)(Y >> 55);
                s += fx_shr(w[i], n[i] + 2);
            }
        }
        const uint64_t Y = fx_rcp(s);
#pragma unroll
        for (int i = 0; i < I; ++i) {
            const uint64_t R = fx_mulhi(w[i], Y);   // in [2^58, 2^61]: r_i = R 2^(-61 - n)
            const int z = fx_clz64(R) - 1;
            r[i] = fx_pack(R << z, n[i] + z - 2);
            if (n[i] > 127) r[i] = 0.0;             // (term() gives -128 below it)
        }
#pragma unroll
        for (int i = 1; i < I; ++i) {
            const double r0 = r[0], ri = r[i];
            r[0] = i == ref ? ri : r0;
            r[i] = i == ref ? r0 : ri;
        }
        return over == 0u;
    }

    // From here on weights() takes eps itself in the place of eps 2^53 (and
    // mix_terms() must not be called).
    SMC_FX void natural_shocks()
    {
#pragma unroll
        for (int i = 0; i < kM; ++i) {
            A[i] *= 0x1p106;
            B[i] *= 0x1p53;
        }
    }

    // 1 / h_t and eps_t of the last chain(), the shock with all its bits (shock()
    // holds it in units of 2^-53).
    SMC_FX double inv_h() const { return fx_pack(M, (int)(uint32_t)(X >> 55) - 256); }
    SMC_FX double eps() const { return dy * inv_h(); }

    // The shock of an observation y whose volatility V is, as FP64 has it.
    SMC_FX double shock_of(double y, const uint64_t* tab) const
    {
        uint64_t x = ly;
#pragma unroll
        for (int k = 0; k < K; ++k) x += (uint64_t)V[k];
        return (y - mu) * fx_pack(fx_exp2neg(x, tab), (int)(uint32_t)(x >> 55) - 256);
    }

    // eps_t of the last chain() (units 2^-53).
    SMC_FX int64_t shock() const
    {
        const uint64_t sg = (uint64_t)(int64_t)neg;
        return (int64_t)((E ^ sg) - sg);
    }

    // The mixture part for the shock (E_, neg_): independent of the next
    // observation's chain.
    SMC_FX void mix(uint64_t E_, int32_t neg_, const uint64_t* tab)
    {
        if (I == 1) return;
        const uint64_t sg = (uint64_t)(int64_t)neg_;
        const int64_t es = (int64_t)((E_ ^ sg) - sg);
        s1 += es;
        uint32_t over;
        mix_terms((double)es, tab, over);
        bad |= over;
    }

    // m_t and s_t of the shock ed_ (units 2^-53) into their sums; over: bit 31
    // set (and the sums spoiled) where a d_i is out of range.
    SMC_FX void mix_terms(double ed_, const uint64_t* tab, uint32_t& over)
    {
        over = 0;
        int64_t D[kM];
        int64_t cur = 0;
#pragma unroll
        for (int i = 0; i < kM; ++i) {
            uint32_t o;
            const int64_t x = term(i, ed_, 5, o);   // 16 or more is out of range
            over |= o;
            // (cur, D_i) <- (max, min): the terms stay the same set, and cur
            // ends as the largest
            D[i] = x < cur ? x : cur;
            cur = x < cur ? cur : x;
        }
        sc += (uint64_t)cur;
        uint64_t s = 1ull << 61;
#pragma unroll
        for (int i = 0; i < kM; ++i) {
            const uint64_t Y = (uint64_t)(cur - D[i]);
            s += fx_shr(fx_exp2neg(Y, tab), (int)(uint32_t)(Y >> 55) + 2);
        }
        fx_product(pm, pe, s);
    }

    // One step of block(): the chain of an observation and the mixture part of
    // the one before, which do not depend on each other.
    SMC_FX void step(double y, const uint64_t* tab)
    {
        const uint64_t E0 = E;
        const int32_t neg0 = neg;
        chain<false>(y, tab);
        mix(E0, neg0, tab);
    }

    // n observations (first: they open the series), sums flushed.  Eight steps
    // between flushes without a test in between, unrolled by two: the pieces
    // of two steps interleave (K=3, I=4, one warp per scheduler:
    // 1,830 cycles an observation taken singly, 1,190 so; by three or four it is
    // slower again).
    SMC_FX void block(const double* y, int n, bool first, const uint64_t* tab)
    {
        if (first) chain<true>(y[0], tab);
        else chain<false>(y[0], tab);
        int r = 1;
        for (; r + 8 <= n; r += 8) {
#pragma unroll 2
            for (int u = 0; u < 8; ++u) step(y[r + u], tab);
            flush();
        }
#pragma unroll 2
        for (; r < n; ++r) step(y[r], tab);
        mix(E, neg, tab);
        flush();
    }

    // At least every 8 observations (9 of chain(): E < 2^60, so hl stays below
    // 2^64 and |s1| below 2^63).
    SMC_FX void flush()
    {
        s2 += ((unsigned __int128)hh << 42) + ((unsigned __int128)hl << 12) + (ll >> 12);
        hh = hl = ll = 0;
        if (I > 1) {
            scw += sc;
            s1w += s1;
            sc = 0;
            s1 = 0;
        }
    }

    // What a particle carries between observations (after a flush).
    struct Saved {
        int64_t V[K];
        uint64_t E, pm;
        int32_t eh, el, neg, pe;
        unsigned __int128 sx, s2, scw;
        __int128 s1w;
    };
    template <class To, class From>
    SMC_FX static void copy_state(To& o, const From& f)
    {
#pragma unroll
        for (int k = 0; k < K; ++k) o.V[k] = f.V[k];
        o.E = f.E;
        o.eh = f.eh;
        o.el = f.el;
        o.neg = f.neg;
        o.sx = f.sx;
        o.s2 = f.s2;
        if (I > 1) {
            o.pm = f.pm;
            o.pe = f.pe;
            o.scw = f.scw;
            o.s1w = f.s1w;
        }
    }
    SMC_FX void save(Saved& o) const { copy_state(o, *this); }
    template <class From>
    SMC_FX void restore(const From& o)   // Saved or EgarchFx
    {
        copy_state(*this, o);
        bad = 0;
    }

    // Takes up a state in FP64; false when it is out of range.
    SMC_FX bool enter(const double* v, double eps)
    {
        const double g = 0.5 / kFxLn2;
        bool ok = std::fabs(eps) * (double)(1 << cs) < 127.0;
#pragma unroll
        for (int k = 0; k < K; ++k) ok = ok && std::fabs(v[k] * g) < kVmax - 1.0;
        if (!ok) return false;
#pragma unroll
        for (int k = 0; k < K; ++k) V[k] = fx_scaled(v[k] * g, 55);
        E = (uint64_t)fx_scaled(std::fabs(eps), 53);
        set_limbs(E << cs);
        neg = eps < 0.0 ? -1 : 0;
        return true;
    }

    SMC_FX void set_limbs(uint64_t Es)
    {
        eh = (int32_t)(Es >> 29);
        el = (int32_t)((uint32_t)Es & 0x1fffffffu);
    }

    // log p(y_1:T | theta) after the last flush.
    SMC_FX double finish(int T, double ln2, double log2pi) const
    {
        const double sle = fx_to_double((__int128)(scw - sx) + ((__int128)T << 63), -55);
        const double s2d = fx_to_double((__int128)s2, -86);
        if (I == 1) return ln2 * sle - 0.5 * s2d - 0.5 * log2pi * (double)T;
        const double s1e = fx_to_double(s1w, -53);
        const double q = s2d - 2.0 * m0 * s1e + (double)T * (m0 * m0);
        return ln2 * (sle + (double)pe + log2((double)pm * 0x1p-62)) - 0.5 * (a0 * a0) * q +
               (double)T * (ln2 * c0 - 0.5 * log2pi);
    }

    // The shock is the recursion's own, in units of 2^-53: what the next
    // observation takes up.  A caller's end state takes shock_of().
    SMC_FX void state_out(double* st, double ln2) const
    {
#pragma unroll
        for (int k = 0; k < K; ++k) st[k] = (double)V[k] * (2.0 * ln2 * 0x1p-55);
        st[K] = (double)shock() * 0x1p-53;
    }
};

}  // namespace smc
