// se_fx64_launch.cuh -- host launchers of the kernels in se_fx64.cuh.
#pragma once
#include <algorithm>

#include "se_fx64.cuh"
#include "se_launch.cuh"

namespace se {

template <int P>
cudaError_t fx_scatter_P(const double* xyz, const double* q, const FxParams& fp, const FxBufs& b,
                         int c0, int c1, bool again, cudaStream_t s) {
    const long long n = again ? c1 - c0 : fp.kp.N;
    const int blocks = (int)std::max(1LL, std::min((n + 63) / 64, 1LL << 18));
    k_scatter_fx<P><<<dim3(blocks, 3), 64, 0, s>>>(xyz, q, fp, b.slot, b.tile_of, b.tile_start,
                                           (double*)b.sorted, b.perm, b.cells, (int4*)b.fac,
                                           (int2*)b.xq, b.acc, c0, c1, again);
    return cudaGetLastError();
}

template <int P>
cudaError_t fx_spread_P(const FxParams& fp, const FxBufs& b, int c0, int c1, cudaStream_t s) {
    const int per = (kFxThreads / 32) * kFxGPW<P>;
    const int blocks = std::max(1, std::min((c1 - c0 + per - 1) / per, 1 << 20));
    k_spread_fx<P><<<blocks, kFxThreads, 0, s>>>((const int4*)b.fac, (const int2*)b.xq, b.cells,
                                                 (const double*)b.sorted, (unsigned long long*)b.g64,
                                                 fp, b.acc, c0, c1);
    return cudaGetLastError();
}

template <int P>
cudaError_t fx_gather_P(const FxParams& fp, const FxBufs& b, double* phi, double* F, double e_scale,
                        double* E_out, const double* adj, int c0, int c1, cudaStream_t s) {
    const int warps_all = (c1 - c0 + kFxGPW<P> - 1) / kFxGPW<P>;
    const int warps = std::max(1, std::min(P <= 16 ? 8 : 16, warps_all / 152));
    const int blocks = std::max(1, std::min((warps_all + warps - 1) / warps, b.nparts));
    k_gather_fx<P><<<blocks, 32 * warps, 0, s>>>(
        (const int4*)b.fac, b.cells, (const double*)b.sorted, b.perm, (const int2*)b.split,
        b.top, phi, F, fp, b.parts, b.ticket, b.acc, e_scale, E_out, adj, c0, c1);
    return cudaGetLastError();
}

#define SE_FX_INSTANTIATE(P)                                                                      \
    template cudaError_t fx_scatter_P<P>(const double*, const double*, const FxParams&,           \
                                         const FxBufs&, int, int, bool, cudaStream_t);            \
    template cudaError_t fx_spread_P<P>(const FxParams&, const FxBufs&, int, int, cudaStream_t);  \
    template cudaError_t fx_gather_P<P>(const FxParams&, const FxBufs&, double*, double*, double, \
                                        double*, const double*, int, int, cudaStream_t);

}  // namespace se
