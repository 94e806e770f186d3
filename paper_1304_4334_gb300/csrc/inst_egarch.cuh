// Instantiation helpers: one translation unit per (precision, K) keeps each
// compile short and lets the build run them in parallel.
#pragma once

#include "kernels.cuh"
#include "loglik_split.cuh"
#include "phase.cuh"

namespace smc {

inline int mutate_grid(int P, int threads = kMutThreads) { return (P + threads - 1) / threads; }

// The kernel for P particles (one per thread): the policy's form for few
// particles (Few) up to the warps per SM that the policy gives.
template <class Pol>
struct KernelPick {
    static bool few(int P, int warps) { return P <= warps * 32 * device_sm_count(); }
    template <bool kIndep>
    static void (*mutate(int P))(MutateArgs)
    {
        constexpr int w = kIndep ? Pol::kFewIndep : Pol::kFewMutate;
        if constexpr (w > 0)
            if (few(P, w)) return k_mutate<typename Pol::Few, kIndep>;
        return k_mutate<Pol, kIndep>;
    }
    static void (*loglik(int P))(LoglikArgs)
    {
        if constexpr (Pol::kFewLoglik > 0)
            if (few(P, Pol::kFewLoglik)) return k_loglik<typename Pol::Few>;
        return k_loglik<Pol>;
    }
};

template <template <int, int> class Pol, int K, bool kIndep>
void (*mutate_kernel(int I, int P))(MutateArgs)
{
    switch (I) {
    case 1: return KernelPick<Pol<K, 1>>::template mutate<kIndep>(P);
    case 2: return KernelPick<Pol<K, 2>>::template mutate<kIndep>(P);
    case 3: return KernelPick<Pol<K, 3>>::template mutate<kIndep>(P);
    case 4: return KernelPick<Pol<K, 4>>::template mutate<kIndep>(P);
    }
    return nullptr;
}

// One particle per thread; threads = a multiple of 32 up to kMutMaxThreads (the caller checks).
template <template <int, int> class Pol, int K>
cudaError_t launch_mutate_k(const MutateArgs& a, int threads, cudaStream_t s)
{
    const int g = mutate_grid(a.P, threads);
    const auto k = a.qmean ? mutate_kernel<Pol, K, true>(a.m.I, a.P) : mutate_kernel<Pol, K, false>(a.m.I, a.P);
    if (!k) return cudaErrorInvalidValue;
    if (a.dependent && !a.qmean) return pdl_launch(k, g, threads, 0, s, a);
    k<<<g, threads, 0, s>>>(a);
    return cudaGetLastError();
}

// ppt = particles per thread (1 or 2; 2 only for the FP32 policy)
template <int K>
cudaError_t launch_mutate_x2_k(const MutateArgs& a, int threads, cudaStream_t s)
{
    const int g = (a.P + 2 * threads - 1) / (2 * threads);
    void (*k)(MutateArgs) = nullptr;
    switch (a.m.I) {
    case 1: k = k_mutate_x2<K, 1>; break;
    case 2: k = k_mutate_x2<K, 2>; break;
    case 3: k = k_mutate_x2<K, 3>; break;
    case 4: k = k_mutate_x2<K, 4>; break;
    default: return cudaErrorInvalidValue;
    }
    if (a.dependent) return pdl_launch(k, g, threads, 0, s, a);
    k<<<g, threads, 0, s>>>(a);
    return cudaGetLastError();
}

template <template <int, int> class Pol, int K>
cudaError_t launch_loglik_k(const LoglikArgs& a, cudaStream_t s)
{
    if constexpr (Pol<K, 2>::kExpTab) {   // FP64: the fixed-point recursion
        bool taken = false;
        cudaError_t e = cudaSuccess;
        switch (a.m.I) {
        case 2: e = launch_loglik_split<K, 2>(a, s, &taken); break;
        case 3: e = launch_loglik_split<K, 3>(a, s, &taken); break;
        case 4: e = launch_loglik_split<K, 4>(a, s, &taken); break;
        }
        if (taken) return e;
    }
    void (*k)(LoglikArgs) = nullptr;
    switch (a.m.I) {
    case 1: k = KernelPick<Pol<K, 1>>::loglik(a.P); break;
    case 2: k = KernelPick<Pol<K, 2>>::loglik(a.P); break;
    case 3: k = KernelPick<Pol<K, 3>>::loglik(a.P); break;
    case 4: k = KernelPick<Pol<K, 4>>::loglik(a.P); break;
    default: return cudaErrorInvalidValue;
    }
    k<<<mutate_grid(a.P), kMutThreads, 0, s>>>(a);
    return cudaGetLastError();
}

template <template <int, int> class Pol, int K>
cudaError_t launch_cdata_k(const CdataArgs& a, cudaStream_t s)
{
    const int g = mutate_grid(a.P);
    switch (a.m.I) {
    case 1: k_cdata<Pol<K, 1>><<<g, kMutThreads, 0, s>>>(a); break;
    case 2: k_cdata<Pol<K, 2>><<<g, kMutThreads, 0, s>>>(a); break;
    case 3: k_cdata<Pol<K, 3>><<<g, kMutThreads, 0, s>>>(a); break;
    case 4: k_cdata<Pol<K, 4>><<<g, kMutThreads, 0, s>>>(a); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace smc

// POL: the mutation kernels' policy; POL_EVAL: the stand-alone likelihood's;
// POL_CDATA: the data-tempering C phase's.
#define SMC_INSTANTIATE_EGARCH(TAG, POL, POL_EVAL, POL_CDATA, K)                                \
    namespace smc {                                                                             \
    cudaError_t launch_mutate_##TAG##_k##K(const MutateArgs& a, int threads, cudaStream_t s)    \
    {                                                                                           \
        return launch_mutate_k<POL, K>(a, threads, s);                                          \
    }                                                                                           \
    cudaError_t launch_loglik_##TAG##_k##K(const LoglikArgs& a, cudaStream_t s)                 \
    {                                                                                           \
        return launch_loglik_k<POL_EVAL, K>(a, s);                                              \
    }                                                                                           \
    cudaError_t launch_cdata_##TAG##_k##K(const CdataArgs& a, cudaStream_t s)                   \
    {                                                                                           \
        return launch_cdata_k<POL_CDATA, K>(a, s);                                               \
    }                                                                                           \
    }
