// se_real.cu -- the real-space part of the Ewald sum on the GPU, with cell
// lists: the complement of the SE k-space path for full Ewald energies and
// forces (Sec. 1, Eq. 1.5-1.7, the erfc terms and the self term).
//
// For charges q_n at x_n in the periodic box [0, L)^3, splitting parameter
// xi and cut-off r_c:
//   phi_m = kc [ sum_{n, images; 0 < r < r_c} q_n erfc(xi r) / r  -  2 xi / sqrt(pi) q_m ]
//   F_m   = kc q_m sum_{n, images; r < r_c} q_n (2 xi / sqrt(pi) e^{-xi^2 r^2} + erfc(xi r) / r)
//           (x_m - x_n^image) / r^2
//   E     = 1/2 sum_m q_m phi_m            (real-space energy plus the self energy)
// so that these plus the k-space results of se_evaluate are the whole Ewald
// potential, force and energy.
//
// GPU design: particles are counted into cells of edge >= r_c / K (nc =
// floor(K L / r_c) per dimension, at most 40, nc >= 2K+1, so the (2K+1)^3
// cells around a cell are distinct periodic images and every pair within r_c
// is met exactly once), scanned and scattered into cell order.  One CTA per
// home cell stages its stencil in shared memory with the image shifts
// applied (the cells' ranges fetched in parallel, offsets by a warp scan,
// each staged particle located by binary search; in chunks when they do not
// fit).  In single precision each thread holds three home particles and
// tests every candidate it loads from shared memory against all three (one
// shared load per three distance tests); the candidate loop of a set of home
// particles is split over S adjacent lanes (S a power of two), reduced by
// shuffles.  In double precision one warp takes a home particle: the
// candidates are tested in single precision, the survivors queued and their
// terms evaluated from a table of polynomials (k_rs_pairs64).  Every particle
// sums its own potential and force: no atomics on the outputs.  The energy is
// a deterministic two-level reduction (last block).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <new>

#include "../../include/se.h"
#include "se_internal.h"

namespace {

constexpr int kThreads = 256;
constexpr int kMaxCellsPerDim = 40;     // at most 64 000 cells (one energy partial each)
#ifndef SE_RS_NB_KB
#define SE_RS_NB_KB 32
#endif
constexpr size_t kNbSmem = SE_RS_NB_KB * 1024;   // shared memory for staged neighbours

template <typename T> struct R4 { using type = se::v4_t<T>; };

// Single precision: erfc(x) = erfcx(x) e^{-x^2} with erfcx(x) ~ t P(t),
// t = 1 / (1 + p x), P of degree 8 (the form of Hastings' approximations,
// Abramowitz and Stegun 7.1.26), coefficients fitted by gen_erfcx_fit.py for
// relative accuracy on 0 <= x <= 6 (3.5e-7 evaluated in float32; beyond 6,
// where erfc < 2e-17, within 2e-5).  The e^{-x^2} is the one the force term
// needs anyway, so each pair evaluates one exponential.
constexpr float kErfcxP = 4.50000000e-01f;
__constant__ float kErfcx[9] = {
    2.536794543e-01f,
    2.576121688e-01f,
    1.990700811e-01f,
    3.049189448e-01f,
    -2.398110330e-01f,
    6.246721148e-01f,
    -6.125214100e-01f,
    2.510224283e-01f,
    -3.864272311e-02f};

__device__ __forceinline__ float erfcx_fit(float x) {
    const float t = __fdividef(1.0f, fmaf(kErfcxP, x, 1.0f));   // 2 ulp
    float a = kErfcx[8];
#pragma unroll
    for (int k = 7; k >= 0; --k) a = fmaf(a, t, kErfcx[k]);
    return a * t;
}

// erfc(xi r)/r and the force factor (2 xi/sqrt(pi) e^{-xi^2 r^2} + erfc(xi r)/r)/r^2
// for one pair, given r^2 and 1/r.
__device__ __forceinline__ void pair_terms(float r2, float ir, float xi, float c2xi, float& ec,
                                           float& fr) {
    const float x = xi * (r2 * ir);
    const float e = expf(-x * x);
    ec = erfcx_fit(x) * e * ir;
    fr = (c2xi * e + ec) * ir * ir;
}
__device__ __forceinline__ void pair_terms(double r2, double ir, double xi, double c2xi,
                                           double& ec, double& fr) {
    const double r = r2 * ir;
    ec = erfc(xi * r) * ir;
    fr = (c2xi * exp(-xi * xi * r2) + ec) * ir * ir;
}
__device__ __forceinline__ float floorR(float a) { return floorf(a); }
__device__ __forceinline__ double floorR(double a) { return floor(a); }

// Wrap into [0, L): x - L floor(x / L), then one correction; NaN or anything
// still outside becomes 0.
template <typename T>
__device__ __forceinline__ T wrapR(T x, T L, T invL) {
    if (x >= T(0) && x < L) return x;
    T y = x - L * floorR(x * invL);
    if (y >= L) y -= L;
    if (!(y >= T(0) && y < L)) y = T(0);
    return y;
}

template <typename T>
__device__ __forceinline__ int cellR(T x, T cscale, int nc) {
    int c = (int)(x * cscale);
    return c < 0 ? 0 : (c >= nc ? nc - 1 : c);
}

template <typename T>
__global__ void __launch_bounds__(kThreads)
k_rs_count(const T* __restrict__ xyz, int N, T L, T invL, T cscale, int nc, int* count,
           int* __restrict__ cell_of, int* __restrict__ slot) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int cx = cellR(wrapR(xyz[3 * i], L, invL), cscale, nc);
    const int cy = cellR(wrapR(xyz[3 * i + 1], L, invL), cscale, nc);
    const int cz = cellR(wrapR(xyz[3 * i + 2], L, invL), cscale, nc);
    const int c = (cx * nc + cy) * nc + cz;
    cell_of[i] = c;
    slot[i] = atomicAdd(&count[c], 1);
}

// Exclusive scan of the cell counts into start[0..ncells] by one CTA of 1024
// threads, chunk by chunk with a running carry; the counts are cleared for
// the next evaluation.
__global__ void __launch_bounds__(1024) k_rs_scan(int* count, int* start, int ncells) {
    __shared__ int wsum[32];
    __shared__ int carry_s;
    if (threadIdx.x == 0) carry_s = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int base = 0; base < ncells; base += 1024) {
        const int i = base + threadIdx.x;
        const int v = i < ncells ? count[i] : 0;
        if (i < ncells) count[i] = 0;
        int x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        if (warp == 0) {
            int w = wsum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += y;
            }
            wsum[lane] = w;
        }
        __syncthreads();
        const int carry = carry_s;
        const int incl = x + (warp > 0 ? wsum[warp - 1] : 0);
        if (i < ncells) start[i] = carry + incl - v;
        __syncthreads();
        if (threadIdx.x == 1023) carry_s = carry + incl;
        __syncthreads();
    }
    if (threadIdx.x == 0) start[ncells] = carry_s;
}

template <typename T>
__global__ void __launch_bounds__(kThreads)
k_rs_scatter(const T* __restrict__ xyz, const T* __restrict__ q, int N, T L, T invL,
             const int* __restrict__ cell_of, const int* __restrict__ slot,
             const int* __restrict__ start, typename R4<T>::type* __restrict__ sorted,
             se::f4* __restrict__ sorted_f, int* __restrict__ perm) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int p = start[cell_of[i]] + slot[i];
    typename R4<T>::type v;
    v.x = wrapR(xyz[3 * i], L, invL);
    v.y = wrapR(xyz[3 * i + 1], L, invL);
    v.z = wrapR(xyz[3 * i + 2], L, invL);
    v.w = q[i];
    sorted[p] = v;
    if constexpr (sizeof(T) == 8) {   // the copy that the distance test of k_rs_pairs64 reads
        se::f4 f;                     // in units of L: its squares are in range whatever the units
        f.x = (float)(v.x * invL);
        f.y = (float)(v.y * invL);
        f.z = (float)(v.z * invL);
        f.w = 0.0f;
        sorted_f[p] = f;
    }
    perm[p] = i;
}

__device__ __forceinline__ double block_sum_d(double v, double* sbuf) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sbuf[warp] = v;
    __syncthreads();
    double r = 0.0;
    if (warp == 0) {
        r = lane < (int)(blockDim.x >> 5) ? sbuf[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
    }
    return r;
}

// Stencil of a home cell: the (2K+1)^3 cells within K cells per direction
// (cells of edge >= rc / K, so that every pair within rc has both ends in
// such a pair of cells), each a distinct periodic image since nc >= 2K+1.
constexpr int kMaxStencil = 343;   // K <= 3
#ifndef SE_RS_THREADS
#define SE_RS_THREADS 192
#endif
constexpr int kPairThreads = SE_RS_THREADS;
#ifndef SE_RS_R32
#define SE_RS_R32 3   // home particles per thread, single precision
#endif

// The stencil of home cell (cx, cy, cz): per stencil cell its first sorted
// particle s_b0, the image shift s_sh (per axis 0, 1: -L, 2: +L) and the
// exclusive prefix sums s_off of the counts (s_off[W^3]: all candidates).
// Called by the whole block; ends with a barrier.
__device__ __forceinline__ void stencil_ranges(const int* __restrict__ start, int nc, int K,
                                               int cx, int cy, int cz, int* s_b0, int* s_off,
                                               unsigned char* s_sh) {
    const int W = 2 * K + 1, W3 = W * W * W;
    for (int k = threadIdx.x; k < W3; k += blockDim.x) {
        int nx = cx + k / (W * W) - K, ny = cy + (k / W) % W - K, nz = cz + k % W - K;
        unsigned char sh = 0;
        if (nx < 0) { nx += nc; sh |= 1; } else if (nx >= nc) { nx -= nc; sh |= 2; }
        if (ny < 0) { ny += nc; sh |= 4; } else if (ny >= nc) { ny -= nc; sh |= 8; }
        if (nz < 0) { nz += nc; sh |= 16; } else if (nz >= nc) { nz -= nc; sh |= 32; }
        const int nid = (nx * nc + ny) * nc + nz;
        const int b0 = start[nid];
        s_b0[k] = b0;
        s_off[k + 1] = start[nid + 1] - b0;   // count, scanned below
        s_sh[k] = sh;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int carry = 0;
        if (lane == 0) s_off[0] = 0;
        for (int base = 0; base < W3; base += 32) {
            const int k = base + lane;
            int v = k < W3 ? s_off[k + 1] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += y;
            }
            if (k < W3) s_off[k + 1] = carry + v;
            carry += __shfl_sync(0xffffffffu, v, 31);
        }
    }
    __syncthreads();
}

// The stencil cell k with s_off[k] <= g < s_off[k + 1].
__device__ __forceinline__ int stencil_cell(const int* s_off, int W3, int g) {
    int lo = 0, hi = W3 - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s_off[mid] <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
}

template <typename V, typename T>
__device__ __forceinline__ V image_of(V v, unsigned sh, T L) {
    v.x += (sh & 1) ? -L : ((sh & 2) ? L : T(0));
    v.y += (sh & 4) ? -L : ((sh & 8) ? L : T(0));
    v.z += (sh & 16) ? -L : ((sh & 32) ? L : T(0));
    return v;
}

// Energy of the call from every block's e_loc: per-block partials, summed by
// the last block (which leaves the ticket at zero for the next call).
__device__ __forceinline__ void finish_energy(double e_loc, double* __restrict__ partials,
                                              unsigned* ticket, double* E_out, int accumulate,
                                              double* sbuf) {
    __shared__ bool last;
    const double r = block_sum_d(e_loc, sbuf);
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = r;
        __threadfence();
        const unsigned t = atomicAdd(ticket, 1u);
        last = t == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double e = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) e += partials[b];
    e = block_sum_d(e, sbuf);
    if (threadIdx.x == 0) {
        if (E_out) *E_out = accumulate ? *E_out + 0.5 * e : 0.5 * e;
        *ticket = 0u;
    }
}

// Single precision.
__global__ void __launch_bounds__(kPairThreads)
k_rs_pairs(const se::f4* __restrict__ sorted, const int* __restrict__ start,
           const int* __restrict__ perm, int nc, int K, float L, float rc2, float xi, float c2xi,
           float kc, int cap, float* __restrict__ phi, float* __restrict__ F, int accumulate,
           double* __restrict__ partials, unsigned* ticket, double* E_out) {
    extern __shared__ __align__(32) unsigned char smem_raw[];
    se::f4* nb = reinterpret_cast<se::f4*>(smem_raw);
    __shared__ int s_b0[kMaxStencil], s_off[kMaxStencil + 1];
    __shared__ unsigned char s_sh[kMaxStencil];
    __shared__ double sbuf[32];
    const int cid = blockIdx.x;
    const int cx = cid / (nc * nc), cy = (cid / nc) % nc, cz = cid % nc;
    const int h0 = start[cid], nh = start[cid + 1] - h0;
    const int W = 2 * K + 1, W3 = W * W * W;
    stencil_ranges(start, nc, K, cx, cy, cz, s_b0, s_off, s_sh);
    const int total = s_off[W3];
    // kR home particles per thread, so that every candidate loaded from shared
    // memory is tested against three of them; S lanes per set of kR particles,
    // S the largest power of two up to 32 with 2 S ceil(nh / kR) <= the
    // block's threads
    constexpr int kR = SE_RS_R32;
    const int nset = (nh + kR - 1) / kR;
    int S = 1;
    while (S < 32 && 2 * S * nset <= (int)blockDim.x) S <<= 1;
    const int sets = blockDim.x / S;
    const int per_pass = sets * kR;
    const int s = threadIdx.x % S, set = threadIdx.x / S;
    double e_loc = 0.0;
    for (int pass0 = 0; pass0 < nh; pass0 += per_pass) {
        int li[kR];
        bool act[kR];
        se::f4 me[kR];
        float ph[kR], fx[kR], fy[kR], fz[kR];
#pragma unroll
        for (int r = 0; r < kR; ++r) {
            li[r] = pass0 + set + r * sets;
            act[r] = li[r] < nh;
            if (act[r]) {
                me[r] = sorted[h0 + li[r]];
            } else {   // far from every candidate: no hits
                me[r].x = me[r].y = me[r].z = 1e18f;
                me[r].w = 0.0f;
            }
            ph[r] = fx[r] = fy[r] = fz[r] = 0.0f;
        }
        for (int c0 = 0; c0 < total; c0 += cap) {
            const int filled = min(cap, total - c0);
            __syncthreads();
            for (int t = threadIdx.x; t < filled; t += blockDim.x) {
                const int k = stencil_cell(s_off, W3, c0 + t);
                nb[t] = image_of(sorted[s_b0[k] + c0 + t - s_off[k]], s_sh[k], L);
            }
            __syncthreads();
            if (!act[0]) continue;   // act[r] implies act[0]
            // 32 candidates per lane at a time: distance tests into bit masks,
            // then the erfc terms of the hits only
            for (int jb = 0; jb < filled; jb += 32 * S) {   // uniform over the set
                const int j0 = jb + s;
                unsigned mask[kR];
#pragma unroll
                for (int r = 0; r < kR; ++r) mask[r] = 0u;
#pragma unroll 8
                for (int b = 0; b < 32; ++b) {
                    const int j = j0 + b * S;
                    if (j < filled) {
                        const se::f4 n = nb[j];
#pragma unroll
                        for (int r = 0; r < kR; ++r) {
                            const float dx = me[r].x - n.x, dy = me[r].y - n.y, dz = me[r].z - n.z;
                            const float r2 = dx * dx + dy * dy + dz * dz;
                            if (r2 < rc2 && r2 > 0.0f) mask[r] |= 1u << b;
                        }
                    }
                }
#pragma unroll
                for (int r = 0; r < kR; ++r) {
                    unsigned m = mask[r];
                    while (m) {
                        const int b = __ffs(m) - 1;
                        m &= m - 1u;
                        const se::f4 n = nb[j0 + b * S];
                        const float dx = me[r].x - n.x, dy = me[r].y - n.y, dz = me[r].z - n.z;
                        const float r2 = dx * dx + dy * dy + dz * dz;
                        float ec, fr;
                        pair_terms(r2, rsqrtf(r2), xi, c2xi, ec, fr);
                        ph[r] += n.w * ec;
                        const float f = n.w * fr;
                        fx[r] += f * dx;
                        fy[r] += f * dy;
                        fz[r] += f * dz;
                    }
                }
            }
        }
#pragma unroll
        for (int r = 0; r < kR; ++r) {
            // sum over the S lanes of the set (adjacent lanes, aligned groups)
            for (int o = S >> 1; o > 0; o >>= 1) {
                ph[r] += __shfl_xor_sync(0xffffffffu, ph[r], o);
                fx[r] += __shfl_xor_sync(0xffffffffu, fx[r], o);
                fy[r] += __shfl_xor_sync(0xffffffffu, fy[r], o);
                fz[r] += __shfl_xor_sync(0xffffffffu, fz[r], o);
            }
            if (act[r] && s == 0) {
                const float pm = kc * (ph[r] - c2xi * me[r].w);
                const float fq = kc * me[r].w;
                const int o = perm[h0 + li[r]];
                if (phi) phi[o] = accumulate ? phi[o] + pm : pm;
                if (F) {
                    if (accumulate) {
                        F[3 * o] += fq * fx[r];
                        F[3 * o + 1] += fq * fy[r];
                        F[3 * o + 2] += fq * fz[r];
                    } else {
                        F[3 * o] = fq * fx[r];
                        F[3 * o + 1] = fq * fy[r];
                        F[3 * o + 2] = fq * fz[r];
                    }
                }
                e_loc += (double)me[r].w * (double)pm;
            }
        }
    }
    finish_energy(e_loc, partials, ticket, E_out, accumulate, sbuf);
}

// ---------------------------------------------------------------------------
// Double precision.  This GPU retires about 1.7 FP64 operations per clock and SM
// (the library's own probe; two nominally, a 64th of its FP32 rate), so the kernel
// is bound by the FP64 operations of its pairs and by nothing else (its FP64 pipe
// is 84 % busy); the design spends as few as it can:
//
//  - The distance test, which 73 % of the candidates fail on a water box, is
//    made in FP32, on positions in units of L, with a bound wide enough for
//    every FP32 rounding on the way (rs_run); the pairs that pass are tested again in FP64, as before, so
//    the set of pairs that are summed is the same.
//  - erfc(x)/x and (2/sqrt(pi) e^{-x^2} + erfc(x)/x)/x^2 are both smooth
//    functions of v = x^2 = xi^2 r^2 alone, which needs no square root.  They
//    come from a table of degree-7 polynomials (one row per interval of v,
//    below): 15 operations instead of the 150 or so of rsqrt, exp and erfc.
//  - The second test and the row's index and centre are integer operations
//    on the bits of r^2 and v.
//
// 27 FP64 operations a pair in all.  One warp takes a home particle; its
// lanes test 128 candidates at a time and queue the hits, and every 32 hits
// are evaluated by the 32 lanes, so that all lanes of the FP64 pipe work.
//
// 21 642-atom water box, r_c = 1 nm (420 pairs a particle): 3314 -> 626 us a
// call, of which the 27 operations of its 9.1 M pairs take 470 us at the
// probed rate; the error against 64-bit sums 8.3e-16 -> 8.1e-16.
constexpr int kVMinExp = -5, kVMaxExp = 6;   // the table covers 2^-5 <= v < 2^6
constexpr int kVDeg = 7;
// rows per octave: 64 below v = 16, then 128 and 256 (e^{-v} needs shorter
// intervals there); the interpolation error stays below 1e-16 everywhere
constexpr int kVRows = 64 * (4 - kVMinExp) + 128 + 256;
constexpr int kVRowLen = 2 * (kVDeg + 1);

// Row of v and the centre of its interval, from the high word of v.
__device__ __forceinline__ int vrow(int hi, double* centre) {
    const int over = max(0, (hi >> 20) - (1023 + 3));   // octaves above 2^4
    const int sh = 14 - over;                           // 64, 128 or 256 rows per octave
    const int base = over == 0 ? -((1023 + kVMinExp) << 6)
                   : over == 1 ? 64 * (4 - kVMinExp) - ((1023 + 4) << 7)
                               : 64 * (4 - kVMinExp) + 128 - ((1023 + 5) << 8);
    *centre = __hiloint2double(((hi >> sh) << sh) | (1 << (sh - 1)), 0);
    return (hi >> sh) + base;
}

// The sums of 4 values over the 32 lanes of a warp: 7 additions a lane
// instead of 20.  Lane 8 k of the warp returns the sum of value k.
__device__ __forceinline__ double warp_sum4(double a, double b, double c, double d, int lane) {
    const bool up = lane & 16, up2 = lane & 8;
    double x = up ? c : a, y = up ? d : b;
    x += __shfl_xor_sync(0xffffffffu, up ? a : c, 16);
    y += __shfl_xor_sync(0xffffffffu, up ? b : d, 16);
    double z = up2 ? y : x;
    z += __shfl_xor_sync(0xffffffffu, up2 ? x : y, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    return z;
}

// The pair sums of potential and force are kept in units of s and s^3: xi, as the
// table has them, or 1 where every pair is nearer than the table begins (bare:
// xi r_c below 2^-5/2), so that a small xi r needs no power of itself.
struct PairScales {
    double xi, c2xi, s;   // c2xi = 2 xi / sqrt(pi)
    bool bare;
};

constexpr int kPair64Warps = 6;
// Staged candidates: at most 2048 (96 KB: two CTAs per SM); half a box's mean count
// over, and at least 512 (24 KB: four CTAs, as many as the registers allow), where
// fewer will do (rs_run): sparse cells are many short CTAs (20 000 particles in
// 40^3 cells: 780 us at 2048, 548 at 512; with FP64 arithmetic for every pair 755).
constexpr int kCap64 = 2048, kCap64Min = 512;
constexpr int kTest64 = 128;        // candidates tested per step
constexpr int kQueue64 = kTest64 + 32;

__global__ void __launch_bounds__(32 * kPair64Warps)
k_rs_pairs64(const se::d4* __restrict__ sorted, const se::f4* __restrict__ sorted_f,
             const int* __restrict__ start, const int* __restrict__ perm, int cap, int nc, int K,
             double L, double rc2, float rc2_f, const PairScales sc, double kc, const double2* __restrict__ table,
             double* __restrict__ phi, double* __restrict__ F, int accumulate,
             double* __restrict__ partials, unsigned* ticket, double* E_out) {
    extern __shared__ __align__(32) unsigned char smem_raw[];
    se::d4* nb = reinterpret_cast<se::d4*>(smem_raw);
    se::f4* nf = reinterpret_cast<se::f4*>(smem_raw + cap * sizeof(se::d4));
    __shared__ int s_b0[kMaxStencil], s_off[kMaxStencil + 1];
    __shared__ unsigned char s_sh[kMaxStencil];
    __shared__ unsigned short s_q[kPair64Warps][kQueue64];
    __shared__ double sbuf[32];
    const int cid = blockIdx.x;
    const int cx = cid / (nc * nc), cy = (cid / nc) % nc, cz = cid % nc;
    const int h0 = start[cid], nh = start[cid + 1] - h0;
    const int W = 2 * K + 1, W3 = W * W * W;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (nh > 0) stencil_ranges(start, nc, K, cx, cy, cz, s_b0, s_off, s_sh);   // per block
    const int total = nh > 0 ? s_off[W3] : 0;
    const double xi2 = sc.xi * sc.xi;
    const long long rc2_bits = __double_as_longlong(rc2);
    unsigned short* q = s_q[warp];
    double e_loc = 0.0;
    for (int pass0 = 0; pass0 < nh; pass0 += kPair64Warps) {
        const bool act = pass0 + warp < nh;   // uniform over the warp
        se::d4 me;
        se::f4 mf;
        if (act) {
            me = sorted[h0 + pass0 + warp];
            mf = sorted_f[h0 + pass0 + warp];
        }
        double ph = 0.0, fx = 0.0, fy = 0.0, fz = 0.0;
        auto pair = [&](int j) {
            const se::d4 n = nb[j];
            const double dx = me.x - n.x, dy = me.y - n.y, dz = me.z - n.z;
            const double r2 = dx * dx + dy * dy + dz * dz;
            // r2 < rc2 and r2 > 0, on the bits (non-negative doubles order as integers)
            const long long bits = __double_as_longlong(r2);
            if (bits >= rc2_bits || bits <= 0) return;
            const double v = xi2 * r2;
            const int hi = __double2hiint(v);
            double f, g;
            if (hi >= ((1023 + kVMinExp) << 20) && hi < ((1023 + kVMaxExp) << 20)) {
                double c;
                const double2* row = table + vrow(hi, &c) * (kVRowLen / 2);
                const double t = v - c;   // exact
                double2 w = __ldg(row + kVDeg);   // (f, g) coefficients side by side
                f = w.x;
                g = w.y;
#pragma unroll
                for (int k = kVDeg - 1; k >= 0; --k) {
                    w = __ldg(row + k);
                    f = fma(f, t, w.x);
                    g = fma(g, t, w.y);
                }
            } else {   // very close or very far pairs
                if (sc.bare) pair_terms(r2, rsqrt(r2), sc.xi, sc.c2xi, f, g);
                else pair_terms(v, rsqrt(v), 1.0, 1.1283791670955126, f, g);
            }
            ph += n.w * f;
            const double fq = n.w * g;
            fx += fq * dx;
            fy += fq * dy;
            fz += fq * dz;
        };
        for (int c0 = 0; c0 < total; c0 += cap) {
            const int filled = min(cap, total - c0);
            if (pass0 == 0 || total > cap) {   // one chunk: staged once for all passes
                __syncthreads();
                for (int t = threadIdx.x; t < filled; t += blockDim.x) {
                    const int k = stencil_cell(s_off, W3, c0 + t);
                    const int p = s_b0[k] + c0 + t - s_off[k];
                    nb[t] = image_of(sorted[p], s_sh[k], L);
                    nf[t] = image_of(sorted_f[p], s_sh[k], 1.0f);
                }
                __syncthreads();
            }
            if (!act) continue;
            int nq = 0;
            for (int jb = 0; jb < filled; jb += kTest64) {
                bool hit[kTest64 / 32];
#pragma unroll
                for (int u = 0; u < kTest64 / 32; ++u) {
                    const int j = jb + 32 * u + lane;
                    const se::f4 n = nf[min(j, filled - 1)];
                    const float dx = mf.x - n.x, dy = mf.y - n.y, dz = mf.z - n.z;
                    hit[u] = j < filled && dx * dx + dy * dy + dz * dz < rc2_f;
                }
#pragma unroll
                for (int u = 0; u < kTest64 / 32; ++u) {
                    const unsigned m = __ballot_sync(0xffffffffu, hit[u]);
                    if (hit[u])
                        q[nq + __popc(m & ((1u << lane) - 1u))] = (unsigned short)(jb + 32 * u + lane);
                    nq += __popc(m);
                }
                __syncwarp();
                int done = 0;
                for (; nq - done >= 32; done += 32) pair(q[done + lane]);
                if (done > 0) {   // the rest (under 32) moves to the front
                    const unsigned short rest = q[min(done + lane, kQueue64 - 1)];
                    __syncwarp();
                    nq -= done;
                    if (lane < nq) q[lane] = rest;
                }
                __syncwarp();
            }
            if (lane < nq) pair(q[lane]);
            __syncwarp();   // the queue is rewritten by the next chunk or pass
        }
        if (act) {
            const double sum = warp_sum4(ph, fx, fy, fz, lane);
            const int o = perm[h0 + pass0 + warp], k = lane >> 3;
            if ((lane & 7) == 0) {
                if (k == 0) {
                    const double pm = kc * (sc.s * sum - sc.c2xi * me.w);
                    if (phi) phi[o] = accumulate ? phi[o] + pm : pm;
                    e_loc += me.w * pm;
                } else if (F) {
                    const double f = kc * me.w * (sc.s * sum * sc.s * sc.s);
                    double* dst = F + 3 * (size_t)o + (k - 1);
                    *dst = accumulate ? *dst + f : f;
                }
            }
        }
    }
    finish_energy(e_loc, partials, ticket, E_out, accumulate, sbuf);
}

// The table of k_rs_pairs64: row by row the coefficients, lowest order first
// and the two functions side by side, of
//   f(v) = erfc(sqrt v)/sqrt v   and   g(v) = (2/sqrt(pi) e^{-v} + f(v))/v = -2 f'(v)
// in powers of v - c, c the centre of the row's interval.  f solves
// v f' + f/2 = -e^{-v}/sqrt(pi), so its Taylor coefficients a_n at c follow from
// a_0 = f(c) by
//   a_{n+1} = -(E (-1)^n / n! + (n + 1/2) a_n) / (c (n + 1)),  E = e^{-c}/sqrt(pi)
// (both terms have the sign of a_n's, so nothing cancels), and g's are
// b_n = -2 (n + 1) a_{n+1}.  Each series is cut at degree kVTaylor and
// economised to degree kVDeg by taking out the Chebyshev polynomials of
// the interval from the top down (Lanczos), whose error is 2^{n-1} times
// smaller than the cut Taylor term's.  The leading coefficients
// are formed in long double, so that rounding them is their only error.
// Host work, once per process.
constexpr int kVTaylor = 15;


// a: powers of x = t / h, |x| <= 1, degree kVTaylor -> kVDeg.
void economise(double* a, const double (*T)[kVTaylor + 1]) {
    for (int k = kVTaylor; k > kVDeg; --k) {
        const double top = a[k] / T[k][k];
        for (int i = 0; i <= k; ++i) a[i] -= top * T[k][i];
    }
}

struct VTable {
    double t[kVRows * kVRowLen];
    VTable() {
        double T[kVTaylor + 1][kVTaylor + 1] = {};   // Chebyshev polynomials in powers of x
        T[0][0] = T[1][1] = 1.0;
        for (int k = 2; k <= kVTaylor; ++k)
            for (int i = 0; i <= k; ++i) T[k][i] = (i > 0 ? 2.0 * T[k - 1][i - 1] : 0.0) - T[k - 2][i];
        double* row = t;
        for (int e = kVMinExp; e < kVMaxExp; ++e) {
            const int rows = e < 4 ? 64 : (e == 4 ? 128 : 256);
            const double w = ldexp(1.0 / rows, e), h = 0.5 * w;
            for (int i = 0; i < rows; ++i, row += kVRowLen) {
                const double c = ldexp(1.0, e) + (i + 0.5) * w;
                const long double sc = sqrtl((long double)c);
                const long double E = expl(-(long double)c) / sqrtl(acosl(-1.0L));
                const long double f0 = erfcl(sc) / sc, f1 = -(E + 0.5L * f0) / c;
                double a[kVTaylor + 2], b[kVTaylor + 1];
                a[0] = (double)f0;
                a[1] = (double)f1;
                double fac = 1.0, sgn = -1.0;
                for (int n = 1; n <= kVTaylor; ++n) {
                    fac *= n;
                    a[n + 1] = -((double)E * sgn / fac + (n + 0.5) * a[n]) / (c * (n + 1));
                    sgn = -sgn;
                }
                for (int n = 0; n <= kVTaylor; ++n) b[n] = -2.0 * (n + 1) * a[n + 1];
                double p = 1.0;
                for (int n = 0; n <= kVTaylor; ++n, p *= h) {
                    a[n] *= p;
                    b[n] *= p;
                }
                economise(a, T);
                economise(b, T);
                p = 1.0;
                for (int n = 0; n <= kVDeg; ++n, p *= h) {
                    row[2 * n] = a[n] / p;
                    row[2 * n + 1] = b[n] / p;
                }
            }
        }
    }
};

const VTable& vtable() {
    static const VTable table;
    return table;
}

}  // namespace

struct se_real {
    int64_t N = 0;
    double L = 0, xi = 0, rc = 0, kc = 1.0;
    int prec = SE_FP64;
    cudaStream_t stream = nullptr;
    int nc = 0, ncells = 0, K = 1;   // cells per dimension, stencil reach
    bool ready = false;
    int ready_prec = -1;
    int* count = nullptr;
    int* start = nullptr;
    int* cell_of = nullptr;
    int* slot = nullptr;
    int* perm = nullptr;
    void* sorted = nullptr;
    se::f4* sorted_f = nullptr;      // FP64: the positions / L in FP32
    double2* table = nullptr;        // FP64: the pair functions (vtable)
    double* partials = nullptr;
    unsigned* ticket = nullptr;
};

namespace {

void rs_release(se_real* r) {
    void* b[] = {r->count, r->start, r->cell_of, r->slot, r->perm, r->sorted, r->sorted_f, r->table, r->partials,
                 r->ticket};
    for (void* p : b)
        if (p) cudaFree(p);
    r->count = r->start = r->cell_of = r->slot = r->perm = nullptr;
    r->sorted = nullptr;
    r->sorted_f = nullptr;
    r->table = nullptr;
    r->partials = nullptr;
    r->ticket = nullptr;
    r->ready = false;
}

int rs_alloc(void** p, size_t bytes) {
    return cudaMalloc(p, bytes ? bytes : 16) == cudaSuccess ? SE_OK : SE_ERR_NOMEM;
}

int rs_prepare(se_real* r) {
    if (r->ready && r->ready_prec == r->prec) return SE_OK;
    rs_release(r);
    const size_t N = (size_t)r->N, ts = r->prec == SE_FP64 ? 8 : 4;
    int rc = SE_OK;
    if (rc == SE_OK) rc = rs_alloc((void**)&r->count, (size_t)r->ncells * sizeof(int));
    if (rc == SE_OK) rc = rs_alloc((void**)&r->start, ((size_t)r->ncells + 1) * sizeof(int));
    if (rc == SE_OK) rc = rs_alloc((void**)&r->cell_of, N * sizeof(int));
    if (rc == SE_OK) rc = rs_alloc((void**)&r->slot, N * sizeof(int));
    if (rc == SE_OK) rc = rs_alloc((void**)&r->perm, N * sizeof(int));
    if (rc == SE_OK) rc = rs_alloc(&r->sorted, N * 4 * ts);
    if (rc == SE_OK && r->prec == SE_FP64) {
        rc = rs_alloc((void**)&r->sorted_f, N * sizeof(se::f4));
        const VTable& v = vtable();
        if (rc == SE_OK) rc = rs_alloc((void**)&r->table, sizeof(v.t));
        if (rc == SE_OK &&
            cudaMemcpy(r->table, v.t, sizeof(v.t), cudaMemcpyHostToDevice) != cudaSuccess)
            rc = SE_ERR_CUDA;
    }
    if (rc == SE_OK) rc = rs_alloc((void**)&r->partials, (size_t)r->ncells * sizeof(double));
    if (rc == SE_OK) rc = rs_alloc((void**)&r->ticket, sizeof(unsigned));
    if (rc == SE_OK && (cudaMemset(r->count, 0, (size_t)r->ncells * sizeof(int)) != cudaSuccess ||
                        cudaMemset(r->ticket, 0, sizeof(unsigned)) != cudaSuccess))
        rc = SE_ERR_CUDA;
    if (rc != SE_OK) {
        rs_release(r);
        return rc;
    }
    r->ready = true;
    r->ready_prec = r->prec;
    return SE_OK;
}

template <typename T>
int rs_run(se_real* r, const void* xyz, const void* q, void* F, void* phi, double* E, int acc) {
    using V = typename R4<T>::type;
    const int N = (int)r->N, nc = r->nc;
    const T L = (T)r->L, invL = (T)(1.0 / r->L), cscale = (T)(nc / r->L);
    const int nb = (N + kThreads - 1) / kThreads;
    cudaStream_t s = r->stream;
    k_rs_count<T><<<nb, kThreads, 0, s>>>((const T*)xyz, N, L, invL, cscale, nc, r->count,
                                          r->cell_of, r->slot);
    k_rs_scan<<<1, 1024, 0, s>>>(r->count, r->start, r->ncells);
    k_rs_scatter<T><<<nb, kThreads, 0, s>>>((const T*)xyz, (const T*)q, N, L, invL, r->cell_of,
                                            r->slot, r->start, (V*)r->sorted, r->sorted_f, r->perm);
    if constexpr (sizeof(T) == 8) {
        // The bound of the FP32 distance test, in units of L.  A position
        // rounded to FP32 is off by at most 2^-24, an image of it (the sum
        // with +-1) and a difference of two by at most e = 8 2^-24 in all per
        // axis, so a pair within r_c has an FP32 distance within r_c / L + 2 e;
        // its square is formed with a relative error below 2^-21.
        const double e = 8.0 / 16777216.0, rf = r->rc / r->L + 2.0 * e;
        const float rc2_f = (float)(rf * rf * (1.0 + 1.0 / 1048576.0));
        const bool bare = r->xi * r->rc < 0.17;
        const PairScales sc = {r->xi, 2.0 * r->xi / sqrt(3.14159265358979323846),
                               bare ? 1.0 : r->xi, bare};
        const int W = 2 * r->K + 1;
        const double mean = (double)N * W * W * W / r->ncells;   // candidates of a cell
        const int cap = (int)std::min<double>(kCap64, std::max<double>(kCap64Min, 1.5 * mean));
        const int each = (int)(sizeof(se::d4) + sizeof(se::f4));
        // the limit is the kernel's, not the call's: the same for every object
        if (cudaFuncSetAttribute(k_rs_pairs64, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kCap64 * each) != cudaSuccess)
            return SE_ERR_CUDA;
        k_rs_pairs64<<<r->ncells, 32 * kPair64Warps, cap * each, s>>>(
            (const V*)r->sorted, r->sorted_f, r->start, r->perm, cap, nc, r->K, L, r->rc * r->rc, rc2_f,
            sc, r->kc, r->table, (T*)phi, (T*)F, acc, r->partials, r->ticket, E);
    } else {
        const int cap = (int)(kNbSmem / sizeof(V));
        if (cudaFuncSetAttribute(k_rs_pairs, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kNbSmem) != cudaSuccess)
            return SE_ERR_CUDA;
        const double c2xi = 2.0 * r->xi / sqrt(3.14159265358979323846);
        k_rs_pairs<<<r->ncells, kPairThreads, kNbSmem, s>>>(
            (const V*)r->sorted, r->start, r->perm, nc, r->K, L, (T)(r->rc * r->rc), (T)r->xi,
            (T)c2xi, (T)r->kc, cap, (T*)phi, (T*)F, acc, r->partials, r->ticket, E);
    }
    return cudaGetLastError() == cudaSuccess ? SE_OK : SE_ERR_CUDA;
}

}  // namespace

// Cells per dimension and stencil reach for (L, rc); reach_user 1-3 forces
// K (SE_ERR_UNSUPPORTED if its 2K+1 cells do not fit), 0 chooses.
static int rs_layout(double L, double rc, int reach_user, int* K_out, int* nc_out) {
    if (floor(L / rc) < 3.0) return SE_ERR_UNSUPPORTED;   // r_c > L/3
    // stencil reach K: cells of edge >= rc/K, nc >= 2K+1 distinct images
    // (rc <= L/3 gives floor(2 L / rc) >= 6); K = 2 by default (a 5^3 stencil:
    // fewer candidates per particle than 3^3 cells of edge rc, and 8 times
    // the CTAs; measured 2-5 times faster than K = 1 and 1.2-1.5 times faster
    // than K = 3 on water boxes of 21.6k and 100k atoms), K = 3 when K = 2
    // leaves fewer than 512 cells (CTAs) for the GPU (1000 charges in a 3 nm
    // box: 1.3 times faster than K = 2)
    auto cells_for = [&](int K) {
        return (int)std::min<double>(floor(K * L / rc), kMaxCellsPerDim);
    };
    int K = 2;
    if (reach_user >= 1) K = reach_user;
    else if (cells_for(3) >= 7 && cells_for(2) * cells_for(2) * cells_for(2) < 512)
        K = 3;
    if (cells_for(K) < 2 * K + 1) return SE_ERR_UNSUPPORTED;
    *K_out = K;
    *nc_out = cells_for(K);
    return SE_OK;
}

extern "C" int se_real_create(se_real** out, int64_t N, double L, double xi, double rc) {
    if (!out) return SE_ERR_ARG;
    *out = nullptr;
    if (N < 0 || N >= ((int64_t)1 << 31) || !(L > 0.0) || !isfinite(L) || !(xi > 0.0) ||
        !isfinite(xi) || !(rc > 0.0) || !isfinite(rc))
        return SE_ERR_ARG;
    int K = 0, nc = 0;
    const int st = rs_layout(L, rc, 0, &K, &nc);
    if (st != SE_OK) return st;
    se_real* r = new (std::nothrow) se_real;
    if (!r) return SE_ERR_NOMEM;
    r->N = N;
    r->L = L;
    r->xi = xi;
    r->rc = rc;
    r->K = K;
    r->nc = nc;
    r->ncells = nc * nc * nc;
    *out = r;
    return SE_OK;
}

extern "C" int se_real_set_reach(se_real* r, int K) {
    if (!r || K < 0 || K > 3) return SE_ERR_ARG;
    int Kn = 0, nc = 0;
    const int st = rs_layout(r->L, r->rc, K, &Kn, &nc);
    if (st != SE_OK) return st;
    if (nc * nc * nc != r->ncells) rs_release(r);   // buffers sized by the cell count
    r->K = Kn;
    r->nc = nc;
    r->ncells = nc * nc * nc;
    return SE_OK;
}

extern "C" int se_real_destroy(se_real* r) {
    if (!r) return SE_OK;
    rs_release(r);
    delete r;
    return SE_OK;
}

extern "C" int se_real_set_precision(se_real* r, int prec) {
    if (!r || (prec != SE_FP64 && prec != SE_FP32)) return SE_ERR_ARG;
    r->prec = prec;
    return SE_OK;
}

extern "C" int se_real_set_prefactor(se_real* r, double kc) {
    if (!r || !(kc > 0.0) || !isfinite(kc)) return SE_ERR_ARG;
    r->kc = kc;
    return SE_OK;
}

extern "C" int se_real_set_stream(se_real* r, void* stream) {
    if (!r) return SE_ERR_ARG;
    r->stream = (cudaStream_t)stream;
    return SE_OK;
}

extern "C" int se_real_get_cells(const se_real* r, int* cells_per_dim) {
    if (!r || !cells_per_dim) return SE_ERR_ARG;
    *cells_per_dim = r->nc;
    return SE_OK;
}

extern "C" int se_real_evaluate(se_real* r, const void* xyz, const void* q, void* F, void* phi,
                                double* E, int accumulate) {
    if (!r || (r->N > 0 && (!xyz || !q))) return SE_ERR_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return SE_ERR_CUDA;
    int rc = rs_prepare(r);
    if (rc != SE_OK) return rc;
    if (r->N == 0) {
        if (E && !accumulate && cudaMemsetAsync(E, 0, sizeof(double), r->stream) != cudaSuccess)
            return SE_ERR_CUDA;
        return SE_OK;
    }
    return r->prec == SE_FP64 ? rs_run<double>(r, xyz, q, F, phi, E, accumulate)
                              : rs_run<float>(r, xyz, q, F, phi, E, accumulate);
}
