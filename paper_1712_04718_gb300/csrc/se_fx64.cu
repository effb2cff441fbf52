// se_fx64.cu -- the double-precision integer spread and gather (se_fx64.cuh):
// dispatch over the support and over ranges of particles.
#include <math_constants.h>

#include "se_fx64_launch.cuh"

namespace se {

#define SE_FX_EXTERN(P)                                                                           \
    extern template cudaError_t fx_scatter_P<P>(const double*, const double*, const FxParams&,    \
                                                const FxBufs&, int, int, bool, cudaStream_t);     \
    extern template cudaError_t fx_spread_P<P>(const FxParams&, const FxBufs&, int, int,          \
                                               cudaStream_t);                                     \
    extern template cudaError_t fx_gather_P<P>(const FxParams&, const FxBufs&, double*, double*,  \
                                               double, double*, const double*, int, int,          \
                                               cudaStream_t);
SE_P_LIST(SE_FX_EXTERN)

namespace {

// The padded integer grid (units of 2^-grid_bits of the largest charge, times
// c_g) -> FP64: every grid point is the sum of its images.  For FP64 sums the grid
// holds FP64 numbers in units of the largest charge's power of two.  A warp takes
// a row (x, y).  The scaling step clears the grid: clearing what was read here
// made the loads wait for the stores (113 us instead of 16 for 119^3 points).
__global__ void __launch_bounds__(256)
k_fx_fold(const long long* __restrict__ g, int Mp, int p0, const FxParams fp,
          const Acc* __restrict__ acc, double* __restrict__ grid) {
    const int bits = grid_bits(acc, fp);
    const bool tiny = acc->qunit < 0x1p-850;   // 2^kTinyExp
    const int up = tiny ? kTinyShift : 0;
    const double base = bits > 0 ? acc->qunit * pow2i(up - bits)
                                 : pow2i(((__double2hiint(acc->qunit) >> 20) & 0x7ff) - 1021 + up);
    // NaN or infinite input: NaN results
    const double unit = acc->nonfinite ? CUDART_NAN : fp.kp.qcg * base;
    const int M = fp.kp.M, warps = gridDim.x * (blockDim.x >> 5), lane = threadIdx.x & 31;
    // the images of index i: i + p0, and one more M above or below (P <= M)
    auto other = [&](int i) { return i <= p0 ? i + p0 + M : (i >= M - p0 ? i + p0 - M : -1); };
    auto rows = [&](auto zero, auto value, auto finish) {
        for (int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < M * M; r += warps) {
            const int x = r / M, y = r - x * M;
            const int xo = other(x), yo = other(y);
            for (int z = lane; z < M; z += 32) {
                const int zo = other(z);
                auto v = zero;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int px = j & 1 ? xo : x + p0, py = j & 2 ? yo : y + p0;
                    if (px < 0 || py < 0) continue;   // uniform over the warp
                    const long long* s = g + ((size_t)px * Mp + py) * Mp;
                    v += value(__ldg(s + z + p0));
                    if (zo >= 0) v += value(__ldg(s + zo));
                }
                grid[(size_t)r * M + z] = finish((double)v * unit);
            }
        }
    };
    // the branch outside the loops: within them it cost 6 us of 50 for 135^3 points
    auto word = [](long long v) { return v; };
    auto real = [](long long v) { return __longlong_as_double(v); };
    auto down = [up](double w) { return w * pow2i(-up); };
    if (bits == 0) rows(0.0, real, down);
    else if (tiny) rows(0LL, word, down);
    else rows(0LL, word, [](double w) { return w; });
}

// The grid split in units of 2^(E - hb), every |value| < 2^E, by integer
// operations on the bits, and padded by its periodic images to Mp^3 points,
// Mp = M + P - 1, point (x, y, z) being grid point (x - p0, y - p0, z - p0) mod M.
// E from the bound
//   |Ht(x)| <= sum_k G/M^3 |Hhat| <= (sum_k G)^1/2 (sum_k G |Hhat|^2)^1/2 / M^3
// (Cauchy and Schwarz; the second sum is the grid energy's, known from the
// scaling step).  It exceeds the largest value by about sqrt(N) / 3, 6 bits of
// the 60 at 21 642 atoms, and saves a pass over the grid.  Charges so large or
// small that the energy leaves the normal range (beyond about 1e+-145) take
//   |Ht(x)| <= sum_k G/M^3 sum_x |H(x)|,  sum_x |H| <= sum_n |q_n| c_g W^3
// instead, W a bound of the sum of a window's factors (gbound1).  Block 0 leaves
// the biased exponent E + 1022 in *top.  Inf and NaN values (finite charges whose
// grid or transform overflowed) have no place in the split grid: they set
// acc->overflow, and the gather gives NaN.
__global__ void __launch_bounds__(256)
k_grid_split(const double* __restrict__ grid, int M, int Mp, int p0, double gbound,
             double gbound1, Acc* acc, int* __restrict__ top, int hb, int2* __restrict__ out) {
    __shared__ int s_top;
    if (threadIdx.x == 0) {
        const double e = acc->e_grid;
        const double bound = e > 1e-290 && e < 1e300 ? gbound * sqrt(e) : gbound1 * acc->sum_absq;
        s_top = min(0x7fe, max(1, (__double2hiint(bound) >> 20) & 0x7ff));
        if (blockIdx.x == 0) *top = s_top;
    }
    __syncthreads();
    const int etop = s_top;
    const int warps = gridDim.x * (blockDim.x >> 5), lane = threadIdx.x & 31;
    for (int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < Mp * Mp; r += warps) {
        const int x = r / Mp, y = r - x * Mp;
        const double* src = grid + ((size_t)wrap_index(x - p0, M) * M + wrap_index(y - p0, M)) * M;
        for (int z = lane; z < Mp; z += 32) {
            const long long b = __double_as_longlong(__ldg(src + wrap_index(z - p0, M)));
            const int e = (int)(b >> 52) & 0x7ff;
            if (e == 0x7ff) acc->overflow = 1u;
            const long long mant = (b & 0xfffffffffffffLL) | (e ? 1LL << 52 : 0LL);   // < 2^53
            // |value| = mant 2^(max(e,1) - 1075); hb + 32 bits below 2^E, E = etop - 1022
            const int sh = max(0, etop - max(e, 1));
            long long f = hb + 32 >= 53 ? mant << (hb + 32 - 53) : mant >> (53 - hb - 32);
            f = sh < 63 ? f >> sh : 0;
            if (b < 0) f = -f;
            out[(size_t)r * Mp + z] = make_int2((int)((f + (1LL << 31)) >> 32), (int)f >> 2);
        }
    }
}

cudaError_t scatter(const double* xyz, const double* q, const FxParams& fp, const FxBufs& b, int c0,
                    int c1, bool again, cudaStream_t s) {
    switch (fp.kp.P) {
#define SE_CASE(PP) case PP: return fx_scatter_P<PP>(xyz, q, fp, b, c0, c1, again, s);
        SE_FOR_EACH_P(SE_CASE)
#undef SE_CASE
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t fx_spread(const double* xyz, const double* q, const FxParams& fp, const FxBufs& b,
                      bool only, cudaStream_t s, void (*mark)(void*, int), void* ctx) {
    const int N = fp.kp.N;
    cudaError_t e = cudaSuccess;
    for (int c0 = 0; c0 < N && e == cudaSuccess; c0 += b.cap) {
        const int c1 = (int)std::min<long long>(N, (long long)c0 + b.cap);
        e = scatter(xyz, q, fp, b, c0, c1, c0 > 0, s);
        if (e != cudaSuccess) break;
        if (c0 == 0) mark(ctx, 1);
        if (only) return cudaSuccess;
        switch (fp.kp.P) {
#define SE_CASE(PP) case PP: e = fx_spread_P<PP>(fp, b, c0, c1, s); break;
            SE_FOR_EACH_P(SE_CASE)
#undef SE_CASE
            default: e = cudaErrorInvalidValue;
        }
        if (c1 == N) break;
    }
    if (N == 0) mark(ctx, 1);
    if (e != cudaSuccess || only) return e;
    const int M = fp.kp.M;
    const int blocks = (int)std::min(((long long)M * M + 7) / 8, 8LL * 152);
    k_fx_fold<<<blocks, 256, 0, s>>>(b.g64, M + fp.kp.P - 1, fp.kp.P / 2 - 1, fp, b.acc, b.grid);
    return cudaGetLastError();
}

cudaError_t fx_gather(const FxParams& fp, const FxBufs& b, const double* grid, double* phi,
                      double* F, double e_scale, double* E_out, const double* adj, cudaStream_t s) {
    const int N = fp.kp.N;
    const int Mp = fp.kp.M + fp.kp.P - 1;
    const int blocks = (int)std::min(((long long)Mp * Mp + 7) / 8, 8LL * 152);
    k_grid_split<<<blocks, 256, 0, s>>>(grid, fp.kp.M, Mp, fp.kp.P / 2 - 1, fp.gbound,
                                        fp.gbound1, b.acc, b.top, fp.hb, (int2*)b.split);
    cudaError_t e = cudaGetLastError();
    for (int c0 = 0; e == cudaSuccess; c0 += b.cap) {
        const int c1 = (int)std::min<long long>(N, (long long)c0 + b.cap);
        if (N > b.cap) e = scatter(nullptr, nullptr, fp, b, c0, c1, true, s);   // its factors again
        if (e != cudaSuccess) break;
        switch (fp.kp.P) {
#define SE_CASE(PP) \
    case PP: e = fx_gather_P<PP>(fp, b, phi, F, e_scale, E_out, adj, c0, c1, s); break;
            SE_FOR_EACH_P(SE_CASE)
#undef SE_CASE
            default: e = cudaErrorInvalidValue;
        }
        if (c1 == N) break;
    }
    return e;
}

}  // namespace se
