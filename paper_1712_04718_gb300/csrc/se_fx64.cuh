// se_fx64.cuh -- double-precision spread and gather (Eq. 3.5, Eq. 3.9 and the
// analytic force of Sec. 3.1) in integer arithmetic.
//
// This GPU retires about 1.7 FP64 operations per clock and SM (the library's own
// probe; two nominally), but 51 multiply-adds of 32-bit integers into 64 bits.  The
// P^3 sums of a particle therefore run on numbers split into two integers,
//     v = hi + lo 2^-30,  hi = round(v), |lo| <= 2^29   (v scaled to at most 2^30),
// whose product is  hi hi' + (hi lo' + lo hi') 2^-30  with lo lo' (below 2^-60
// of the largest product) left out: three multiply-adds, exact, and so are
// their sums.
//
//   k_scatter_fx    particles into tile order, and the window factors of each
//                   (the only FP64 arithmetic per particle: two exponentials,
//                   a reciprocal and two operations a factor, per dimension)
//   k_spread_fx     Eq. 3.5: a weight is rounded to a multiple of 2^-54 to 2^-56
//                   max|q| and added to a 64-bit integer grid, padded so that no
//                   support wraps, with global reductions: integer sums, the same
//                   for every order.  Where that quantum is too coarse (crowded
//                   tiles, a few large charges: grid_bits) the weights are added
//                   as FP64 numbers instead (the last bits then depend on the order)
//   k_fx_fold       that grid -> FP64, its periodic images added
//   k_grid_split    the transformed grid split, padded by its periodic images
//   k_gather_fx     Eq. 3.9 and the forces: y, x and z sums as above, one
//                   conversion to FP64 per particle and result
//
// Measured against FP64 arithmetic (tiles with FP64 shared-memory adds up to P =
// 12 and global FP64 reductions above for the spread, FP64 sums for the gather),
// a whole evaluation: 21 642 atoms, M = 52, P = 8: 478 -> 201 us (spread 220 ->
// 25, gather 136 -> 31); M = 96, P = 24: 2517 -> 1074 us (958 -> 382, 1324 ->
// 405); 1000 charges, M = 32, P = 16: 181 -> 103 us (53 -> 11, 64 -> 18).  Errors of
// potentials against extended precision 7.1e-15 -> 2.9e-15 (water, P = 8), 1.6e-15
// -> 3.6e-16 (1000 charges, P = 24), 9.0e-16 -> 3.8e-16 (1000 charges, P = 16).
//
// Particles are taken in ranges of the tile order, so that the factors
// (56 P bytes a particle) never need more than kFxFactorBytes.
#pragma once
#include <math_constants.h>

#include <algorithm>

#include "se_kernels.cuh"

namespace se {

// Offset of the particle from the centre of its support, as centre_offset,
// without the rounding of x M / L (an ulp of up to M): the product enters
// through an exact FMA and the rounding of M / L is made good.
__device__ __forceinline__ double offset_of(double x, int c, double invh, double invh_lo) {
    return fma(x, invh_lo, fma(x, invh, -(double)c) - 0.5);
}

__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}

// The FP64 number r, |r| <= 2^30, split, by integer operations on its bits.
__device__ __forceinline__ int2 fx_pair(double r) {
    const long long b = __double_as_longlong(r);
    const int sh = ((int)(b >> 52) & 0x7ff) - (1023 + 20);   // r 2^32 = mantissa 2^sh, sh <= 10
    const long long mant = (b & 0xfffffffffffffLL) | (1LL << 52);
    long long f = sh >= 0 ? mant << sh : (sh > -63 ? mant >> -sh : 0);
    if (b < 0) f = -f;
    return make_int2((int)((f + (1LL << 31)) >> 32), (int)f >> 2);
}

// 2^e (0 below the smallest subnormal), without the FP64 pipe.
__device__ __forceinline__ double pow2i(int e) {
    if (e >= -1022) return __hiloint2double((e + 1023) << 20, 0);
    return e >= -1074 ? __longlong_as_double(1LL << (e + 1074)) : 0.0;
}

// Scales below 2^kTinyExp are taken 2^kTinyShift times larger and the results
// made smaller at the end, so that no scale is subnormal.
constexpr int kTinyExp = -850, kTinyShift = 200;

// Bits of the integer grid: a weight of the largest charge is below 2^bits, 56
// but for crowded tiles, so that no grid point can reach 2^63: all tiles together
// give a point at most crowd times the fullest tile's count of such weights
// (tile_crowd, which takes the tiles as they are cut, the narrow last ones too).
// 0: the grid is summed in FP64, because the quantum 2^-bits is coarser than
// 2^-kFxMinBits of the mean charge's largest weight.  FP64 sums keep 53 bits of
// every weight however many meet in a tile and however large the largest charge
// is, but FP64 reductions are slower than integer ones: 21 642 atoms, M = 52,
// P = 8: 64 -> 68 us for all steps of the spread, M = 96, P = 24: 403 -> 664 (and
// 226 and 981 with the FP64 tiles of before).  Relative error of the potentials
// against extended precision, FP64 sums / integers at the bits in brackets: 20 000
// charges of both signs in one place (P = 8) 3e-15 / 1.4e-12 (45), 2 000 1e-15 /
// 2.8e-14 (49), 250 5e-16 / 1.1e-15 (53), 100 6e-16 / 8e-16 (54); one charge of 1e8
// among 5 000 of 1 3e-16 / 1.8e-14 (52 for the large one); a water box 2.4e-15 /
// 3.0e-15 (55).
constexpr int kFxMinBits = 54;
__device__ __forceinline__ int grid_bits(const Acc* acc, const FxParams& fp) {
    const int n = min(fp.kp.N, __float2int_ru(fp.crowd * (float)acc->tile_max));   // saturates
    const int bits = min(56, 63 - (n > 1 ? 32 - __clz(n - 1) : 0));
    return acc->qmean >= __int_as_float((127 + kFxMinBits - bits) << 23) ? bits : 0;
}

// q as +-[1/4, 1/2) times 2^(field - 1021), field the biased exponent (below 1
// for subnormal numbers); q = 0 gives 0.
__device__ __forceinline__ double split_exponent(double q, int* field) {
    int sub = 0;
    if (((__double2hiint(q) >> 20) & 0x7ff) == 0) {
        q *= 0x1p54;
        sub = 54;
    }
    const int hi = __double2hiint(q);
    *field = ((hi >> 20) & 0x7ff) - sub;
    return q == 0.0 ? q : __hiloint2double((hi & 0x800fffff) | (1021 << 20), __double2loint(q));
}

// One thread per particle and dimension (dimension-major, so that a warp has
// one).  fac[r][d][a] = (g hi, g lo, dg hi, dg lo) scaled by 2^30 and 2^(30 - sd):
// the window and its derivative's offset factor dz g, dz = a - (P-1)/2 - u, at
// support point a; xq[r][a] = q / max|q| times the x factor, scaled by
// 2^(grid_bits - 27), or for FP64 sums the charge's significand (split_exponent)
// times the x factor, scaled by 2^30; r = position in tile order - c0.  Only particles with
// c0 <= position < c1 get factors.  dz is split too (hi scaled by 2^26, one lo
// for all a), so that dg costs integer operations only.
// Bound by the FP64 pipe: two exponentials, a reciprocal and two operations a
// factor.
// again: the factors of a further range, or of a range once more, from the sorted
// copies (the caller's arrays are read by the first scatter of a spread only).
template <int P>
__global__ void __launch_bounds__(64)
k_scatter_fx(const double* __restrict__ xyz, const double* __restrict__ q, const FxParams fp,
             const int* __restrict__ slot, const int* __restrict__ tile_of,
             const int* __restrict__ tile_start, double* __restrict__ sorted,
             int* __restrict__ perm, int* __restrict__ cells, int4* __restrict__ fac,
             int2* __restrict__ xq, const Acc* __restrict__ acc, int c0, int c1, bool again) {
    const KParams<double>& kp = fp.kp;
    __shared__ double sE3[P];   // exp(-beta a_c^2) 2^30
    if (threadIdx.x < P) sE3[threadIdx.x] = kp.E3[threadIdx.x] * 1073741824.0;
    __syncthreads();
    const int d = blockIdx.y;
    const int cut = 26 + fp.sd;   // 26 to 30
    const int end = again ? c1 : kp.N;
    for (int i = (again ? c0 : 0) + blockIdx.x * blockDim.x + threadIdx.x; i < end;
         i += gridDim.x * blockDim.x) {
        int dst = i, c;
        double x, qp = 0.0;
        if (again) {   // uniform
            x = sorted[4 * (size_t)dst + d];
            c = cells[4 * (size_t)dst + d];
            if (d == 0) qp = sorted[4 * (size_t)dst + 3];
        } else {
            dst = tile_start[tile_of[i]] + slot[i];
            x = wrap_coord(xyz[3 * (size_t)i + d], kp.L, kp.invL);
            double s;
            c = cell_of(x, kp.invh, kp.M, &s);
            sorted[4 * (size_t)dst + d] = x;
            cells[4 * (size_t)dst + d] = c;
            if (d == 0) {
                qp = q[i];
                sorted[4 * (size_t)dst + 3] = qp;
                perm[dst] = i;
            }
        }
        if (d == 0) {
            const int bits = grid_bits(acc, fp);
            int field;
            if (bits > 0) qp *= acc->qscale * pow2i(bits - 57);
            else qp = split_exponent(qp, &field);
        }
        if (dst < c0 || dst >= c1) continue;
        const double u = offset_of(x, c, kp.invh, fp.invh_lo);
        // from the centre of the support outwards, so that the large factors
        // carry the fewest roundings of the products: support points P/2 + j
        // and P/2 - 1 - j at offsets +-(j + 1/2),
        //   g = exp(-beta u^2 +- 2 beta u (j + 1/2)) E3
        const double B = exp(2.0 * kp.beta * u), Bi = 1.0 / B;
        double pu = exp(kp.beta * u * (1.0 - u)), pd = pu * Bi;
        // dz of point P/2, in units of 2^-26
        const double w = (0.5 - u) * 67108864.0;
        int dzh = __double2int_rn(w);
        const int dzl = __double2int_rn((w - (double)dzh) * 1073741824.0);
        int4* f = fac + ((size_t)(dst - c0) * 3 + d) * P;
        int2* xf = xq + (size_t)(dst - c0) * P;
        auto put = [&](int a, double e, int h) {
            const int2 g = fx_pair(e);
            const long long cr = mad_wide(g.x, dzl, mad_wide(g.y, h, 1LL << 29));
            const long long v = mad_wide(g.x, h, cr >> 30);
            const int dg = (int)((v + (1LL << (cut - 1))) >> cut);
            f[a] = make_int4(g.x, g.y, dg, ((int)v - (int)((unsigned)dg << cut)) << (30 - cut));
            if (d == 0) xf[a] = fx_pair(qp * e);
        };
#pragma unroll 2
        for (int j = 0; j < P / 2; ++j) {
            const int up = P / 2 + j, dn = P / 2 - 1 - j;
            put(up, pu * sE3[up], dzh + (j << 26));
            put(dn, pd * sE3[dn], dzh - ((j + 1) << 26));
            pu *= B;
            pd *= Bi;
        }
    }
}

// Particles of a warp: a lane per z point.
template <int P>
constexpr int kFxGPW = 32 / P;
// rows of the support whose factors a lane of the spread keeps in registers
template <int P>
constexpr int kFxRows = P <= 16 ? P : P / 2;
// rows of the support whose grid values a lane loads at once
template <int P>
constexpr int kFxBatch = P <= 12 ? P : (P % 8 == 0 ? 8 : P / 2);
constexpr int kFxThreads = 128;

// Spread.  The integer grid is padded as the split one (k_gather_fx).  A lane
// holds its z point's factor times the y factors (kFxRows rows at a time) and
// runs over the x planes; the weight xq yz is
//   W = xhi yzhi + (xhi yzlo + xlo yzhi) 2^-30,  |W| < 2^59,
// an integer in units of 2^-3 of the grid's.  Particles come in tile order, but
// nothing depends on it.
// Bound by the reductions: 2.4 lanes per clock and SM at P = 24, with the L1's path
// to the L2 at 89 % and the L2 at 66 % of their rates (issue 41 %).
// For FP64 sums (grid_bits) W, an integer of 2^-60 of the particle's own charge,
// goes as an FP64 number in units of the largest charge's power of two to the
// same grid, as FP64 reductions.
template <int P>
__global__ void __launch_bounds__(kFxThreads)
k_spread_fx(const int4* __restrict__ fac, const int2* __restrict__ xq,
            const int* __restrict__ cells, const double* __restrict__ sorted,
            unsigned long long* __restrict__ g64, const FxParams fp, const Acc* __restrict__ acc,
            int c0, int c1) {
    constexpr int GPW = kFxGPW<P>, BC = kFxRows<P>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gi = lane / P, k = lane - gi * P;
    if (gi >= GPW) return;
    const int Mp = fp.kp.M + P - 1;
    const int per = (kFxThreads / 32) * GPW;
    // W: integer sums
    auto particles = [&](auto W, int ref) {
        constexpr bool kWords = decltype(W)::value;
        for (long long pl = c0 + (long long)blockIdx.x * per + warp * GPW + gi; pl < c1;
             pl += (long long)gridDim.x * per) {
            const int p = (int)pl;
            const int4 cell = *reinterpret_cast<const int4*>(cells + 4 * (size_t)p);
            const int4* fy = fac + ((size_t)(p - c0) * 3 + 1) * P;
            const int2* fx = xq + (size_t)(p - c0) * P;
            const int2 z = *reinterpret_cast<const int2*>(fy + P + k);
            unsigned long long* g0 = g64 + ((size_t)cell.x * Mp + cell.y) * Mp + cell.z + k;
            int shift = 0;
            if constexpr (!kWords) {
                split_exponent(sorted[4 * (size_t)p + 3], &shift);
                shift -= ref + 60;
            }
#pragma unroll 1
            for (int bc = 0; bc < P; bc += BC) {
                int yzh[BC], yzl[BC];
#pragma unroll
                for (int b = 0; b < BC; ++b) {
                    const int2 y = __ldg(reinterpret_cast<const int2*>(fy + bc + b));
                    const long long cr = mad_wide(y.x, z.y, mad_wide(y.y, z.x, 1LL << 29));
                    const long long v = mad_wide(y.x, z.x, cr >> 30);
                    yzh[b] = (int)((v + (1 << 29)) >> 30);
                    yzl[b] = (int)v - (int)((unsigned)yzh[b] << 30);
                }
                unsigned long long* ga = g0 + (size_t)bc * Mp;
#pragma unroll 1
                for (int a = 0; a < P; ++a, ga += (size_t)Mp * Mp) {
                    const int2 x = __ldg(fx + a);
                    unsigned long long* g = ga;
#pragma unroll
                    for (int b = 0; b < BC; ++b, g += Mp) {
                        // the cuts round without a preferred sign (errors of one sign
                        // add up over the weights of a cluster): integer sums: W cut,
                        // plus 4, cut by three bits, mean error (-1/2 + 1/2) / 8;
                        // FP64 sums: W rounded
                        const long long start = kWords ? 4LL << 30 : 1LL << 29;
                        const long long cr = mad_wide(x.x, yzl[b], mad_wide(x.y, yzh[b], start));
                        const long long w = mad_wide(x.x, yzh[b], (long long)(int)(cr >> 30));
                        if constexpr (kWords) {
                            atomicAdd(g, (unsigned long long)(w >> 3));
                        } else {
                            const double v = __ll2double_rn(w);
                            const int hi = __double2hiint(v);
                            if (((hi >> 20) & 0x7ff) + shift > 0)   // not for w = 0: shift <= -60
                                atomicAdd(reinterpret_cast<double*>(g),
                                          __hiloint2double(hi + (int)((unsigned)shift << 20),
                                                           __double2loint(v)));
                        }
                    }
                }
            }
        }
    };
    if (grid_bits(acc, fp) > 0) particles(std::true_type(), 0);   // uniform over the grid
    else particles(std::false_type(), (__double2hiint(acc->qunit) >> 20) & 0x7ff);
}

// A sum of products of split numbers: A + B 2^-30.
struct FxSum {
    long long A, B;
    __device__ __forceinline__ void mac(int2 h, int2 g) {
        A = mad_wide(g.x, h.x, A);
        B = mad_wide(g.x, h.y, B);
        B = mad_wide(g.y, h.x, B);
    }
};
// The sum times 2^-(32 + e), split.  The result is cut by e + 2 bits and the sum's
// own by one before, which takes 2^(e + 1) units away on average; they are added,
// so that errors have no preferred sign: the force's derivative window turns
// errors of one sign into a field of its own (P = 4: field errors of 2.2e-15 of the
// field instead of 9e-16; a water box 4.1e-15 instead of 1.8e-15).
__device__ __forceinline__ int2 fx_top(const FxSum& s, int e) {
    const long long v = (s.A + (s.B >> 30) + (2LL << e)) >> e;
    return make_int2((int)((v + (1LL << 31)) >> 32), (int)v >> 2);
}

// Gather (Eq. 3.9, Sec. 3.1): one lane per z point sums over y, then x, as in
// gather_accum, then the lanes' sums are multiplied by the z factors and added
// over the lanes.  The grid is split and padded (k_grid_split): support point
// (a, b, c) of a particle in cell (cx, cy, cz) is grid[(cx + a) Mp + cy + b) Mp +
// cz + c], Mp = M + P - 1, so that the rows of the support are a constant apart.
// Particles come in tile order, so that the L1 cache serves most of the loads.
// Scales: the grid's hi has hb bits (30 for all but the flattest windows), and
// each of the three sums is at most gs times the largest term, gs a bound of
// the sum of a window's factors; the first two are cut to 32 + e1 and 32 + e2
// bits less, so that every sum stays below 2^63 (fx_params).
// Bound by latency: six of about nine instructions a grid value are the multiply-
// adds, but at P = 24 the issue slots are 46 %, the multiply-add pipe 32 % and the
// L1 52 % busy with 30 warps an SM (128 or 64 registers a thread).
// Consecutive particles share a block, and with it the L1 cache: up to 512
// threads (fewer where the particles are too few for every SM).  Supports 14 and
// 16 keep 16 rows of loads and factors in flight in more than 128 registers
// (P = 16, 1000 charges: 21 us against 37 at 128).
template <int P>
__global__ void __launch_bounds__(P <= 16 ? 256 : 512, P == 14 || P == 16 ? 1 : 2)
k_gather_fx(const int4* __restrict__ fac, const int* __restrict__ cells,
            const double* __restrict__ sorted, const int* __restrict__ perm,
            const int2* __restrict__ grid, const int* __restrict__ top,
            double* __restrict__ phi, double* __restrict__ F, const FxParams fp,
            double* __restrict__ parts, unsigned* ticket, Acc* acc, double e_scale, double* E_out,
            const double* __restrict__ adj, int c0, int c1) {
    constexpr int GPW = kFxGPW<P>, UB = kFxBatch<P>;
    constexpr bool kHold = P <= 12;   // y factors in registers, else loaded again for each x
    const KParams<double>& kp = fp.kp;
    __shared__ double sbuf[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gi = lane / P, k = lane - gi * P;
    const int Mp = kp.M + P - 1;
    // the grid's units 2^(E - hb); the sums are scaled by 2^30 per window and
    // cut by 2^(32 + e1) and 2^(32 + e2); NaN where an input was NaN or infinite
    // or the grid overflowed
    const int ue = top[0] - 1022 - fp.hb - 26 + fp.e1 + fp.e2;
    const bool tiny = ue < kTinyExp;
    const double unit = acc->nonfinite | acc->overflow ? CUDART_NAN
                                                       : pow2i(ue + (tiny ? kTinyShift : 0));
    const double gsc = adj ? __ldg(adj) : 1.0;
    const double u_phi = unit * kp.phi_scale;
    // where the scale was raised, forces and energy are 0 either way
    const double g_phi = tiny ? gsc * pow2i(-kTinyShift) : gsc;
    const double u_F = unit * kp.F_scale * pow2i(fp.sd) * (adj ? -gsc : 1.0);
    double e_loc = 0.0;
    const int per = (blockDim.x >> 5) * GPW;
    for (long long pb = c0 + (long long)blockIdx.x * per + warp * GPW; pb < c1;
         pb += (long long)gridDim.x * per) {
        const int p = (int)pb + gi;
        const bool valid = gi < GPW && p < c1;
        long long v[4] = {0, 0, 0, 0};
        if (valid) {
            const int4* f = fac + (size_t)(p - c0) * 3 * P;
            const int4 cell = *reinterpret_cast<const int4*>(cells + 4 * (size_t)p);
            const int2* row0 = grid + ((size_t)cell.x * Mp + cell.y) * Mp + cell.z + k;
            int2 g[kHold ? P : 1], dg[kHold ? P : 1];
            if constexpr (kHold) {
#pragma unroll
                for (int b = 0; b < P; ++b) {
                    const int4 y = __ldg(f + P + b);
                    g[b] = make_int2(y.x, y.y);
                    dg[b] = make_int2(y.z, y.w);
                }
            }
            FxSum s0 = {0, 0}, sx = {0, 0}, sy = {0, 0};
#pragma unroll 1
            for (int a = 0; a < P; ++a) {
                const int4 xa = __ldg(f + a);
                const int2* row = row0;
                row0 += (size_t)Mp * Mp;
                FxSum t0 = {0, 0}, t1 = {0, 0};
                // loaded again for each x: hoisted out of the loop they spill (P = 18)
                const int4* fy = f + P;
                if constexpr (P > 16) asm volatile("" : "+l"(fy));
#pragma unroll
                for (int b0 = 0; b0 < P; b0 += UB) {
                    int2 w[UB];
#pragma unroll
                    for (int b = 0; b < UB; ++b, row += Mp) w[b] = __ldg(row);
#pragma unroll
                    for (int b = 0; b < UB; ++b) {
                        if constexpr (kHold) {
                            t0.mac(w[b], g[b]);
                            t1.mac(w[b], dg[b]);
                        } else {
                            const int4 y = __ldg(fy + b0 + b);
                            t0.mac(w[b], make_int2(y.x, y.y));
                            t1.mac(w[b], make_int2(y.z, y.w));
                        }
                    }
                }
                const int2 gx = make_int2(xa.x, xa.y), dgx = make_int2(xa.z, xa.w);
                const int2 n0 = fx_top(t0, fp.e1), n1 = fx_top(t1, fp.e1);
                s0.mac(n0, gx);
                sx.mac(n0, dgx);
                sy.mac(n1, gx);
            }
            // z: the lane's share of the four results
            const int4 za = __ldg(f + 2 * P + k);
            const int2 gz = make_int2(za.x, za.y), dgz = make_int2(za.z, za.w);
            const int2 n0 = fx_top(s0, fp.e2), nx = fx_top(sx, fp.e2), ny = fx_top(sy, fp.e2);
            FxSum t[4] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
            t[0].mac(n0, gz);
            t[1].mac(nx, gz);
            t[2].mac(ny, gz);
            t[3].mac(n0, dgz);
#pragma unroll
            for (int c = 0; c < 4; ++c) v[c] = t[c].A + ((t[c].B + (1LL << 29)) >> 30);
        }
#pragma unroll
        for (int o = 1; o < P; o <<= 1) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const long long a = __shfl_down_sync(0xffffffffu, v[c], o);
                if (k + o < P) v[c] += a;
            }
        }
        // result c to lane c of the group: one conversion and two products a lane
        long long mine[(4 + P - 1) / P];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const long long t = __shfl_sync(0xffffffffu, v[c], lane - k);
            if (k == c % P) mine[c / P] = t;
        }
        if (valid) {
            const double qq = sorted[4 * (size_t)p + 3];
            const int orig = perm[p];
#pragma unroll
            for (int j = 0; j < (4 + P - 1) / P; ++j) {
                const int c = k + j * P;
                if (c > 3) break;
                const double w = (double)mine[j] * (c == 0 ? u_phi : u_F);
                if (c == 0) {
                    if (phi) phi[orig] = w * g_phi;
                    e_loc += qq * w;
                } else if (F) {
                    F[3 * (size_t)orig + c - 1] = w * qq;
                }
            }
        }
    }
    const double r = block_sum(e_loc, sbuf);
    if (threadIdx.x == 0) parts[blockIdx.x] = r;
    if (!last_block(ticket)) return;
    const double s = sum_partials(parts, gridDim.x, 1, 0, sbuf);
    if (threadIdx.x == 0) {
        const double e = c0 == 0 ? s : acc->e_gather + s;   // later ranges add to the first
        acc->e_gather = e;
        if (E_out) *E_out = e_scale * e;
        *ticket = 0u;
    }
}

}  // namespace se
