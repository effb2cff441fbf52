// se_fx64.cu -- the double-precision integer spread and gather (se_fx64.cuh):
// dispatch over the support and over ranges of particles.
#include "se_fx64_launch.cuh"

namespace se {

#define SE_FX_EXTERN(P)                                                                           \
    extern template cudaError_t fx_scatter_P<P>(const double*, const double*, const FxParams&,    \
                                                const FxBufs&, int, int, cudaStream_t);           \
    extern template cudaError_t fx_spread_P<P>(const FxParams&, const FxBufs&, int, int,          \
                                               cudaStream_t);                                     \
    extern template cudaError_t fx_gather_P<P>(const FxParams&, const FxBufs&, double*, double*,  \
                                               double, double*, const double*, int, int,          \
                                               cudaStream_t);
SE_P_LIST(SE_FX_EXTERN)

namespace {

// The padded integer grid (units of 2^-grid_bits of the largest charge, times
// c_g) -> FP64: every grid point is the sum of its images.  A warp takes a row
// (x, y).  The integer grid is cleared by a memset afterwards: clearing what was
// read here made the loads wait for the stores (113 us instead of 10 for 119^3
// points).
__global__ void __launch_bounds__(256)
k_fx_fold(const long long* __restrict__ g, int Mp, int p0, const FxParams fp,
          const Acc* __restrict__ acc, double* __restrict__ grid) {
    const double unit = fp.kp.qcg * acc->qunit * pow2i(-grid_bits(acc, fp));
    const int M = fp.kp.M, warps = gridDim.x * (blockDim.x >> 5), lane = threadIdx.x & 31;
    // the images of index i: i + p0, and one more M above or below (P <= M)
    auto other = [&](int i) { return i <= p0 ? i + p0 + M : (i >= M - p0 ? i + p0 - M : -1); };
    for (int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < M * M; r += warps) {
        const int x = r / M, y = r - x * M;
        const int xo = other(x), yo = other(y);
        for (int z = lane; z < M; z += 32) {
            const int zo = other(z);
            long long v = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int px = j & 1 ? xo : x + p0, py = j & 2 ? yo : y + p0;
                if (px < 0 || py < 0) continue;   // uniform over the warp
                const long long* s = g + ((size_t)px * Mp + py) * Mp;
                v += __ldg(s + z + p0);
                if (zo >= 0) v += __ldg(s + zo);
            }
            grid[(size_t)r * M + z] = (double)v * unit;
        }
    }
}

// Largest high word (sign bit cleared) of the grid's values, per block.
__global__ void __launch_bounds__(256)
k_grid_top(const double* __restrict__ grid, long long n, unsigned* __restrict__ top) {
    __shared__ unsigned m;
    if (threadIdx.x == 0) m = 0u;
    __syncthreads();
    unsigned v = 0u;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        v = max(v, (unsigned)__double2hiint(grid[i]) & 0x7fffffffu);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&m, v);
    __syncthreads();
    if (threadIdx.x == 0) top[blockIdx.x] = m;
}

// The grid split in units of 2^(E - hb), every |value| < 2^E, by integer
// operations on the bits, and padded by its periodic images to Mp^3 points,
// Mp = M + P - 1, point (x, y, z) being grid point (x - p0, y - p0, z - p0) mod M.
// Block 0 leaves the biased exponent E + 1022 in top[kFxTopBlocks].
__global__ void __launch_bounds__(256)
k_grid_split(const double* __restrict__ grid, int M, int Mp, int p0, unsigned* __restrict__ top,
             int ntop, int hb, int2* __restrict__ out) {
    __shared__ unsigned m;
    if (threadIdx.x == 0) m = 0u;
    __syncthreads();
    unsigned v = 0u;
    for (int i = threadIdx.x; i < ntop; i += blockDim.x) v = max(v, top[i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&m, v);
    __syncthreads();
    const int etop = max(1, (int)(m >> 20));   // biased exponent of the largest
    if (blockIdx.x == 0 && threadIdx.x == 0) top[kFxTopBlocks] = (unsigned)etop;
    const int warps = gridDim.x * (blockDim.x >> 5), lane = threadIdx.x & 31;
    for (int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < Mp * Mp; r += warps) {
        const int x = r / Mp, y = r - x * Mp;
        const double* src = grid + ((size_t)wrap_index(x - p0, M) * M + wrap_index(y - p0, M)) * M;
        for (int z = lane; z < Mp; z += 32) {
            const long long b = __double_as_longlong(__ldg(src + wrap_index(z - p0, M)));
            const int e = (int)(b >> 52) & 0x7ff;
            const long long mant = (b & 0xfffffffffffffLL) | (e ? 1LL << 52 : 0LL);   // < 2^53
            // |value| = mant 2^(max(e,1) - 1075); hb + 32 bits below 2^E, E = etop - 1022
            const int sh = etop - max(e, 1);
            long long f = hb + 32 >= 53 ? mant << (hb + 32 - 53) : mant >> (53 - hb - 32);
            f = sh < 63 ? f >> sh : 0;
            if (b < 0) f = -f;
            out[(size_t)r * Mp + z] = make_int2((int)((f + (1LL << 31)) >> 32), (int)f >> 2);
        }
    }
}

cudaError_t scatter(const double* xyz, const double* q, const FxParams& fp, const FxBufs& b, int c0,
                    int c1, cudaStream_t s) {
    switch (fp.kp.P) {
#define SE_CASE(PP) case PP: return fx_scatter_P<PP>(xyz, q, fp, b, c0, c1, s);
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
        e = scatter(xyz, q, fp, b, c0, c1, s);
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
    const size_t Mp = (size_t)M + fp.kp.P - 1;
    k_fx_fold<<<blocks, 256, 0, s>>>(b.g64, (int)Mp, fp.kp.P / 2 - 1, fp, b.acc, b.grid);
    e = cudaMemsetAsync(b.g64, 0, Mp * Mp * Mp * sizeof(long long), s);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t fx_gather(const double* xyz, const double* q, const FxParams& fp, const FxBufs& b,
                      const double* grid, double* phi, double* F, double e_scale, double* E_out,
                      const double* adj, cudaStream_t s) {
    const int N = fp.kp.N;
    const long long n = (long long)fp.kp.M * fp.kp.M * fp.kp.M;
    const int ntop = (int)std::min((n + 1023) / 1024, (long long)kFxTopBlocks);
    k_grid_top<<<ntop, 256, 0, s>>>(grid, n, b.top);
    const int Mp = fp.kp.M + fp.kp.P - 1;
    const int blocks = (int)std::min(((long long)Mp * Mp + 7) / 8, 8LL * 152);
    k_grid_split<<<blocks, 256, 0, s>>>(grid, fp.kp.M, Mp, fp.kp.P / 2 - 1, b.top, ntop, fp.hb,
                                        (int2*)b.split);
    cudaError_t e = cudaGetLastError();
    for (int c0 = 0; e == cudaSuccess; c0 += b.cap) {
        const int c1 = (int)std::min<long long>(N, (long long)c0 + b.cap);
        if (N > b.cap) e = scatter(xyz, q, fp, b, c0, c1, s);   // the factors of this range again
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
