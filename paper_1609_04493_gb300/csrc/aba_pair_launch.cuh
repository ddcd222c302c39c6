// aba_pair_launch.cuh -- host launcher of the forward-dynamics kernels with two
// (aba_pair.cuh) or three (aba_tri.cuh) warps per 32 instances, or with three
// lanes per instance and four warps per 30 (aba_trio.cuh).
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <type_traits>

#include "aba_tri.cuh"
#include "aba_trio.cuh"
#include "rdyn_internal.h"

namespace rdyn {

// One block per 32 instances, WARPS warps per block (WARPS = 4: three lanes
// per instance, aba_trio.cuh). Workspace: the sweep-1
// state in the bias precision TB, then (256-byte aligned) the solve state in D.
// withhold: the two-warp kernel's test hook (aba_pair_kernel).
template <typename T, typename D, typename TB, int WARPS>
int launch_aba_multi(const rd_model *m, int B, const void *q, const void *qd, const void *tau,
                     void *qdd, int *status, void *ws, const double *base18, cudaStream_t stream,
                     bool withhold = false)
{
    static_assert(WARPS >= 2 && WARPS <= 4, "two, three or four warps per block");
    const int n = m->n;
    double bb[18];
    rd_convert_base_dh(m, base18, bb);
    BaseParams<T> bp;
    for (int k = 0; k < 6; ++k) {
        bp.V0[k] = (T)bb[k];
        bp.dV0[k] = (T)bb[6 + k];
        bp.Fn[k] = (T)bb[12 + k];
    }
    const T *sc = nullptr;
    if constexpr (sizeof(T) == 4) sc = reinterpret_cast<const T *>(m->d_dh32);
    else sc = reinterpret_cast<const T *>(m->d_dh64);
    const D *sd = nullptr;
    if constexpr (std::is_same<D, double>::value) sd = m->d_aba64;
    else sd = reinterpret_cast<const D *>(m->d_abadf);
    const DF *sdf = reinterpret_cast<const DF *>(m->d_abadf);
    const size_t a = (size_t)n * aba_bias_ws_scalars<T, TB>() * (size_t)B * sizeof(T);
    D *wsz = reinterpret_cast<D *>(static_cast<char *>(ws) + ((a + 255) & ~(size_t)255));
    constexpr int kPerBlock = WARPS < 4 ? 32
                              : std::is_same<TB, T>::value ? kTrioInstances : kTrioExtInstances;
    const unsigned grid = (unsigned)((B + kPerBlock - 1) / kPerBlock);
    // three lanes per instance: the records, and with bias in T the constants
    size_t smem = 0;
    if constexpr (WARPS == 4) {
        constexpr bool kExt = !std::is_same<TB, T>::value;
        smem = (size_t)n * (kAbaDh64 * sizeof(D) + (kExt ? 0 : kDhConsts * sizeof(T)));
        static std::atomic<uint64_t> configured{0};
        const uint64_t bit = 1ull << (m->device & 63);
        if (!(configured.load() & bit)) {
            const void *f = nullptr;
            if constexpr (kExt) f = reinterpret_cast<const void *>(aba_trio_ext_kernel<kTrigPoly>);
            else f = reinterpret_cast<const void *>(aba_trio_kernel<T, D, kTrigPoly>);
            constexpr int most = RD_MAX_LINKS * (int)(kAbaDh64 * sizeof(D) + kDhConsts * sizeof(T));
            cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
            if (e != cudaSuccess) return rd_cuda_fail(e, "cudaFuncSetAttribute");
            configured.fetch_or(bit);
        }
    }
    if constexpr (WARPS == 2)
        aba_pair_kernel<T, D, TB, kTrigPoly><<<grid, 64, 0, stream>>>(
            sc, sd, sdf, n, B, static_cast<const T *>(q), static_cast<const T *>(qd),
            static_cast<const T *>(tau), static_cast<T *>(qdd), status, static_cast<T *>(ws), wsz,
            bp, withhold ? 1 : 0);
    else if constexpr (WARPS == 4 && std::is_same<TB, T>::value)
        aba_trio_kernel<T, D, kTrigPoly><<<grid, 128, smem, stream>>>(
            sc, sd, n, B, static_cast<const T *>(q), static_cast<const T *>(qd),
            static_cast<const T *>(tau), static_cast<T *>(qdd), status, static_cast<T *>(ws), wsz,
            bp);
    else if constexpr (WARPS == 4)
        aba_trio_ext_kernel<kTrigPoly><<<grid, 128, smem, stream>>>(
            sc, sdf, n, B, static_cast<const float *>(q), static_cast<const float *>(qd),
            static_cast<const float *>(tau), static_cast<float *>(qdd), status,
            static_cast<float *>(ws), wsz, bp);
    else
        aba_tri_kernel<T, D, TB, kTrigPoly><<<grid, 96, 0, stream>>>(
            sc, sd, sdf, n, B, static_cast<const T *>(q), static_cast<const T *>(qd),
            static_cast<const T *>(tau), static_cast<T *>(qdd), status, static_cast<T *>(ws), wsz,
            bp);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return rd_cuda_fail(e, WARPS == 2   ? "aba two-warp kernel launch"
                               : WARPS == 3 ? "aba three-warp kernel launch"
                                            : "aba three-lane kernel launch");
    return RD_OK;
}

}  // namespace rdyn
