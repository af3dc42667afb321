// kernels_diag.cu -- FP64 diagnostics (arXiv 2406.16796 Sec. 3.2-3.4 energy
// densities, conversion probabilities and laser centroid; Sec. 2.2 Gauss law).
//
// Deterministic two-stage reduction: a fixed grid of blocks writes one FP64
// partial per quantity per block (fixed tree order inside the block), then one
// block sums the partials in fixed order.  The result depends only on the
// grid size, never on scheduling, so a grid's diagnostics are bit-identical
// however the work around it is arranged.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <mutex>

#include "cells.cuh"
#include "device_common.cuh"

namespace axp {
namespace {

constexpr int kDiagThreads = 256;
constexpr int kQ = 7;  // H_phi, H_g0, H_g1, cross, sum x B1z^2, sum B1z^2, gauss

// ---------------------------------------------------------------------------
// Sums over the grid (the regular entry points).  What bounds it: a literal double
// evaluation spends most of its time on GB300's narrow FP64 pipe (2 operations per
// cycle per SM: 36.7 ms for the 512^3 FP32 box, whose 8 arrays cross HBM in 0.7 ms).
//  * Only the components that can be non-zero are read (template masks).
//  * Constants (1/2, dV, 1/d^2, m^2, 1/dt^2) are applied to the sums, not per cell.
//  * FP64 grids work in double.  FP32 grids do no less, mostly on the FP32 pipe that is 64
//    times wider: each input is a float, so a difference or a product of two is exactly a
//    pair of floats (error-free sums and products after Knuth and Dekker, products by
//    fma), and a thread adds such pairs into three floats with error-free sums (what is
//    dropped is below 2^-70).  The thread's sum becomes a double once, with one rounding where
//    a sum of doubles takes one per term.  The Gauss residual, a sum of scaled differences
//    that cancel, is formed and squared in double, its floats widened by their bits: the FP64
//    pipe is idle otherwise (the E1 and B1 sums there too: 512^3 6.5 -> 8.8 ms).
//    Worst relative error of H_g0, H_g1 and sum_B1z2 against exact sums, 52 states of 300 to
//    2.1M cells: 3.2e-16 (literal doubles 2.5e-16; pairs of floats 2.4e-14).
//  * Floats span less than squares of small fields need, so each group of fields is
//    scaled by a power of two taken from its largest magnitude in the region (max_group:
//    a pass of its own, or part of the pass that forms E^n).  Scaling by a power of
//    two is exact; what then underflows is below 2^-60 of the largest value.
// Measured, a whole record while stepping (us, literal doubles before; cells of 0.05 x 0.07 x 0.06, a
// background along every axis): 512^3 FP32 box 53600 -> 6540; 4096 x 2048 pulse FP32 3970 -> 530, FP64
// 3840 -> 1080 (49 operations per cell on the FP64 pipe, 87% busy).  Pairs of floats took 6170 and 430.
// ---------------------------------------------------------------------------
struct FF {
    float h, l;
};
__device__ __forceinline__ FF two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ FF two_prod(float a, float b)
{
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}

// a float as a double, by its bits: a conversion instruction takes the FP64 pipe.  (Zero, and
// what has no normal exponent, apart.)
__device__ __forceinline__ double as_double(float x)
{
    const int u = __float_as_int(x);
    const unsigned e = (unsigned)u & 0x7f800000u;
    if (e - 1u >= 0x7f800000u - 1u) return x == 0.0f ? 0.0 : (double)x;
    return __hiloint2double(((u >> 3) & (int)0x8fffffff) + (896 << 20), u << 29);
}
__device__ __forceinline__ double as_double(double x) { return x; }

// a thread's running sum of pairs: high and middle words by error-free sums; the last takes
// what those leave over, 2^-48 of the sum and less, in plain float
struct Acc3 {
    float h, m, l;
};
__device__ __forceinline__ void accumulate_low(Acc3 &acc, FF x)  // a term 2^-23 of its sum or less
{
    const FF u = two_sum(acc.m, x.h);
    acc.m = u.h;
    acc.l = __fadd_rn(acc.l, __fadd_rn(u.l, x.l));
}
__device__ __forceinline__ void accumulate(Acc3 &acc, FF x)
{
    const FF s = two_sum(acc.h, x.h);
    acc.h = s.h;
    accumulate_low(acc, two_sum(x.l, s.l));
}

// Sums of 7 quantities over a warp: at each of the first three steps a lane keeps half of
// its values and adds its partner's, so 9 additions take the place of 35 (an FP64
// addition holds its SM sub-partition's unit for 64 cycles).  Lane 4 k holds quantity k.
__device__ __forceinline__ double warp_sums(double v[8], int lane)
{
#pragma unroll
    for (int h = 4, w = 16; h >= 1; h >>= 1, w >>= 1) {
        const bool upper = lane & w;
#pragma unroll
        for (int i = 0; i < h; i++) {
            const double give = upper ? v[i] : v[i + h], keep = upper ? v[i + h] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, w);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    return v[0];
}
// the block's sums into sh[quantity][warp] (then a __syncthreads), and their total over warps
__device__ __forceinline__ void block_sums(double v[8], double sh[8][kDiagThreads / 32])
{
    const int lane = threadIdx.x % 32;
    const double t = warp_sums(v, lane);
    if (lane % 4 == 0) sh[lane / 4][threadIdx.x / 32] = t;
    __syncthreads();
}

// the arithmetic of the sums of values T: Acc a running sum
template <typename T>
struct Ops;
template <>
struct Ops<double> {
    using Acc = double;
    static __device__ __forceinline__ void add_prod(Acc &s, double a, double b) { s = fma(a, b, s); }
    static __device__ __forceinline__ void add_square_of_diff(Acc &s, double a, double b)
    {
        const double d = a - b;
        s = fma(d, d, s);
    }
    static __device__ __forceinline__ void add_sum_times(Acc &s, double a, double b, double c) { s = fma(a + b, c, s); }
    static __device__ __forceinline__ void add_square_times(Acc &s, double a, int k) { s = fma((double)k, a * a, s); }
    static __device__ __forceinline__ double diff(double a, double b) { return a - b; }
    static __device__ __forceinline__ double total(Acc a) { return a; }
    static __device__ __forceinline__ double total(Acc a, Acc b) { return a + b; }
    static __device__ __forceinline__ double scaled(double a, double) { return a; }
};
template <>
struct Ops<float> {
    using Acc = Acc3;
    static __device__ __forceinline__ void add_prod(Acc &s, float a, float b) { accumulate(s, two_prod(a, b)); }
    // (a - b)^2, exact: h^2 + 2 h l + l^2 (l is 0 for neighbours within a factor of 2)
    static __device__ __forceinline__ void add_square_of_diff(Acc &s, float a, float b)
    {
        const FF d = two_sum(a, -b);
        accumulate(s, two_prod(d.h, d.h));
        if (d.l != 0.0f) {
            accumulate_low(s, two_prod(__fadd_rn(d.h, d.h), d.l));
            s.l = __fmaf_rn(d.l, d.l, s.l);
        }
    }
    static __device__ __forceinline__ void add_sum_times(Acc &s, float a, float b, float c)
    {
        const FF d = two_sum(a, b);
        accumulate(s, two_prod(d.h, c));
        if (d.l != 0.0f) accumulate_low(s, two_prod(d.l, c));
    }
    // k a^2; a float holds integers up to 2^24, larger ones come as two
    static __device__ __forceinline__ void add_square_times(Acc &s, float a, int k)
    {
        const FF p = two_prod(a, a);
        const int low = k > (1 << 24) ? k & 0xfff : 0;
        const float k1 = (float)(k - low);
        accumulate(s, two_prod(p.h, k1));
        accumulate_low(s, two_prod(p.l, k1));
        if (low) {
            accumulate(s, two_prod(p.h, (float)low));
            accumulate_low(s, two_prod(p.l, (float)low));
        }
    }
    static __device__ __forceinline__ double diff(float a, float b)
    {
        const FF d = two_sum(a, -b);
        const double x = as_double(d.h);
        return __any_sync(__activemask(), d.l != 0.0f) ? x + as_double(d.l) : x;
    }
    static __device__ __forceinline__ double total(const Acc &a) { return (double)a.h + ((double)a.m + (double)a.l); }
    static __device__ __forceinline__ double total(const Acc &a, const Acc &b)
    {
        return ((double)a.h + (double)b.h) + (((double)a.m + (double)b.m) + ((double)a.l + (double)b.l));
    }
    static __device__ __forceinline__ float scaled(float a, float s) { return __fmul_rn(a, s); }
};

template <typename T>
struct Sums {
    const T *E0[3], *B0[3], *E1[3], *B1[3];
    const T *phi, *phib;               // phi^{n+1/2}; phi^{n-1/2}, or the increment (FP32 split)
    const T *gh[3][2], *gh_old[3][2];  // outflow ghosts of the two levels
    int n[3], per[3], axbc[3][2];
    int lo[3], hi[3];                  // the region summed
    unsigned N;
    T Bext[3], Eext[3];
    int ext;                           // bits: non-zero background components, E (0-2) and B (3-5)
    double d[3], lo0, dt, m2;
    double rd[3], kg, kgb[3];          // 1/d; g/2 times phi^n over what mid_at gives, and that times B_ext
    unsigned *top;      // FP32: largest magnitude of E0/B0, E1/B1, phi (float bits)
    double *partials;
    axp_diag *out;
    int64_t step;
};

constexpr int kSums = 10;  // phi: Dt^2, mid^2, 3 forward differences; E0B0^2; E1B1^2 less B1z; cross; x B1z^2; B1z^2

// a power of two near 1 / (largest magnitude), kept well inside the floats' range
__device__ __forceinline__ float scale_of(double top)
{
    if (!(top > 0.0) || !isfinite(top)) return 1.0f;
    return exp2f((float)min(max(-ilogb(top), -100), 100));
}

// phi^n of a neighbour: phi^n itself in FP32 split, 2 phi^n (the levels' sum) in FP64
template <typename T, int MASK>
__device__ __forceinline__ T mid_at(const Sums<T> &s, int a, int side, const Cell &q)
{
    constexpr bool INCR = sizeof(T) == 4;
    const bool in = side ? q.hu[a] : q.hd[a];
    const int bc = s.axbc[a][side];
    if (in || bc == AXP_BC_REFLECT) {
        const int c = in ? (side ? q.up[a] : q.dn[a]) : q.c;
        return INCR ? s.phi[c] - T(0.5) * s.phib[c] : s.phi[c] + s.phib[c];
    }
    if (bc != AXP_BC_OUTFLOW) return T(0);
    const int pi = ghost_index(s.n, a, q);
    const T sum = s.gh[a][side][pi] + s.gh_old[a][side][pi];
    return INCR ? T(0.5) * sum : sum;
}

// Resident blocks: the 3D form waits on memory more and takes a fourth in spite of a few spills
// (512^3 FP32: 7.3 ms with three, 6.5 with four; 1024 x 512 0.094 and 0.104).
template <typename T>
__host__ __device__ constexpr int diag_blocks_per_sm(int mask) { return sizeof(T) == 4 && mask != 7 ? 3 : 4; }

// EM, BM: the order-0 components present
template <typename T, int MASK, int EM, int BM>
__global__ void __launch_bounds__(kDiagThreads, diag_blocks_per_sm<T>(MASK)) k_diag_sums(Sums<T> s)
{
    using O = Ops<T>;
    constexpr bool INCR = sizeof(T) == 4;
    // scales: of phi, of the order-0 and order-1 fields, and of the order-0 fields with the
    // background (1 in double)
    T sp = T(1), s0 = T(1), s1 = T(1), sx = T(1);
    if (INCR) {
        const double t0 = __uint_as_float(s.top[0]), t1 = __uint_as_float(s.top[1]), tp = __uint_as_float(s.top[2]);
        double ext = 0.0;
        for (int a = 0; a < 3; a++) ext = max(ext, max(fabs((double)s.Bext[a]), fabs((double)s.Eext[a])));
        sp = scale_of(tp);
        s0 = scale_of(t0);
        s1 = scale_of(t1);
        sx = scale_of(max(t0, ext));
    }
    typename O::Acc acc[kSums] = {};
    double gauss = 0.0;        // sum of R^2
    constexpr double half = INCR ? 1.0 : 0.5;  // phi^n over what mid_at gives
    for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < s.N; c += gridDim.x * blockDim.x) {
        Cell q;
        cell_of_index<MASK>(s.n, s.per, c, q);
        bool in = true;
#pragma unroll
        for (int a = 0; a < 3; a++) in = in && q.x[a] >= s.lo[a] && q.x[a] < s.hi[a];
        if (!in) continue;
        const T hi = s.phi[c], b = s.phib[c];
        const T mid = O::scaled(INCR ? hi - T(0.5) * b : hi + b, sp);
        if constexpr (INCR) O::add_prod(acc[0], O::scaled(b, sp), O::scaled(b, sp));
        else O::add_square_of_diff(acc[0], hi, b);
        O::add_prod(acc[1], mid, mid);
        double R = 0.0;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            if (!(MASK >> a & 1)) continue;
            const T up = mid_at<T, MASK>(s, a, 1, q), dn = mid_at<T, MASK>(s, a, 0, q);
            O::add_square_of_diff(acc[2 + a], O::scaled(up, sp), mid);
            // div E1 + g Bbar0 . grad_c phi, term by term along the axis
            double t = O::diff(s.E1[a][c], ldz(s.E1[a], q.dn[a], q.hd[a]));
            if (BM >> a & 1) {
                const int p = (a + 1) % 3, r = (a + 2) % 3;
                const T *B = s.B0[a];
                constexpr bool all = MASK == 7;
                T f = B[c], w = T(1);  // (along an inactive axis the neighbour is the cell itself)
                if (all || (MASK >> p & 1)) {
                    f = f + ldz(B, q.dn[p], q.hd[p]);
                    w = T(0.5);
                }
                if (all || (MASK >> r & 1)) {
                    T h = ldz(B, q.dn[r], q.hd[r]);
                    if (all || (MASK >> p & 1)) h = h + ldz(B, q.dn[p] + (q.dn[r] - q.c), q.hd[p] && q.hd[r]);
                    f = f + h;
                    w = w * T(0.5);
                }
                t = fma(O::diff(up, dn), s.kg * as_double(w * f + s.Bext[a]), t);
            } else if (s.ext >> (3 + a) & 1) {
                t = fma(O::diff(up, dn), s.kgb[a], t);
            }
            R = fma(t, s.rd[a], R);
        }
        gauss = fma(R, R, gauss);
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const T e1 = O::scaled(s.E1[a][c], s1), b1 = O::scaled(s.B1[a][c], s1);
            O::add_prod(acc[6], e1, e1);
            if (a < 2) {
                O::add_prod(acc[6], b1, b1);
            } else {
                O::add_prod(acc[9], b1, b1);
                O::add_square_times(acc[8], b1, q.x[0] + 1);
            }
            if (EM >> a & 1) {
                const T e0 = s.E0[a][c];
                O::add_prod(acc[5], O::scaled(e0, s0), O::scaled(e0, s0));
                O::add_sum_times(acc[7], O::scaled(e0, sx), O::scaled(s.Eext[a], sx), e1);
            } else if (s.ext >> a & 1) {
                O::add_prod(acc[7], O::scaled(s.Eext[a], sx), e1);
            }
            if (BM >> a & 1) {
                const T b0 = s.B0[a][c];
                O::add_prod(acc[5], O::scaled(b0, s0), O::scaled(b0, s0));
                O::add_sum_times(acc[7], O::scaled(b0, sx), O::scaled(s.Bext[a], sx), b1);
            } else if (s.ext >> (3 + a) & 1) {
                O::add_prod(acc[7], O::scaled(s.Bext[a], sx), b1);
            }
        }
    }
    // each thread's sums as doubles, the scales undone; then a fixed tree over the block
    const double up = 1.0 / ((double)sp * (double)sp), u0 = 1.0 / ((double)s0 * (double)s0);
    const double u1 = 1.0 / ((double)s1 * (double)s1), ux = 1.0 / ((double)sx * (double)s1);
    const double dV = s.d[0] * s.d[1] * s.d[2];
    double tot[8];
    tot[7] = 0.0;
    double hphi = O::total(acc[0]) / (s.dt * s.dt) + s.m2 * half * half * O::total(acc[1]);
#pragma unroll
    for (int a = 0; a < 3; a++)
        if (MASK >> a & 1) hphi += half * half * O::total(acc[2 + a]) / (s.d[a] * s.d[a]);
    const double bz2 = O::total(acc[9]) * u1;  // (H_g1: both parts as one sum, rounded once)
    tot[0] = 0.5 * dV * up * hphi;
    tot[1] = 0.5 * dV * u0 * O::total(acc[5]);
    tot[2] = 0.5 * dV * u1 * O::total(acc[6], acc[9]);
    tot[3] = dV * ux * O::total(acc[7]);
    tot[4] = dV * (s.lo0 * bz2 + s.d[0] * u1 * O::total(acc[8]));
    tot[5] = dV * bz2;
    tot[6] = dV * gauss;
    __shared__ double sh[8][kDiagThreads / 32];
    block_sums(tot, sh);
    if (threadIdx.x < kQ) {
        double t = 0.0;
        for (int w = 0; w < kDiagThreads / 32; w++) t += sh[threadIdx.x][w];
        s.partials[(int64_t)blockIdx.x * kQ + threadIdx.x] = t;
    }
}

// largest magnitudes by group, as float bits (of non-negative floats: their order);
// NaN and infinity come out above every finite value
__device__ __forceinline__ unsigned mag(float x) { return __float_as_uint(x) & 0x7fffffffu; }
__device__ __forceinline__ void max_group(unsigned *top, unsigned m0, unsigned m1, unsigned mp)
{
    m0 = __reduce_max_sync(0xffffffffu, m0);
    m1 = __reduce_max_sync(0xffffffffu, m1);
    mp = __reduce_max_sync(0xffffffffu, mp);
    if (threadIdx.x % 32 == 0) {
        if (m0) atomicMax(top, m0);
        if (m1) atomicMax(top + 1, m1);
        if (mp) atomicMax(top + 2, mp);
    }
}
template <typename T>
__device__ __forceinline__ void max_of_cell(const Sums<T> &s, int64_t c, uint32_t mask, bool with_e, unsigned &m0, unsigned &m1,
                                            unsigned &mp)
{
    if constexpr (sizeof(T) == 4) {
        for (int a = 0; a < 3; a++) {
            if (with_e && (mask >> a & 1u)) m0 = max(m0, mag(s.E0[a][c]));
            if (mask >> (3 + a) & 1u) m0 = max(m0, mag(s.B0[a][c]));
            if (with_e) m1 = max(m1, mag(s.E1[a][c]));
            m1 = max(m1, mag(s.B1[a][c]));
        }
        mp = max(mp, max(mag(s.phi[c]), mag(s.phib[c])));
    }
}

// the magnitudes alone, over the region's cells (mask: order-0 components present)
template <typename T>
__global__ void __launch_bounds__(kDiagThreads) k_diag_max(Sums<T> s, uint32_t mask)
{
    unsigned m0 = 0, m1 = 0, mp = 0;
    const unsigned n0 = s.n[0], n1 = s.n[1];
    for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < s.N; c += gridDim.x * blockDim.x) {
        const unsigned r = c / n0, k = r / n1;
        const int x[3] = {(int)(c - r * n0), (int)(r - k * n1), (int)k};
        bool in = true;
#pragma unroll
        for (int a = 0; a < 3; a++) in = in && x[a] >= s.lo[a] && x[a] < s.hi[a];
        if (in) max_of_cell(s, c, mask, true, m0, m1, mp);
    }
    max_group(s.top, m0, m1, mp);
}

// the literal evaluation (fields of a caller, and grids of 2^30 cells or more)
template <typename T, bool INCR>
__global__ void __launch_bounds__(kDiagThreads) k_diag_partial(View<T> v, PhiPair<T, INCR> q, double *partials)
{
    double acc[kQ];
#pragma unroll
    for (int s = 0; s < kQ; s++) acc[s] = 0.0;
    const double dV = (double)v.d[0] * (double)v.d[1] * (double)v.d[2];
    const double m2 = (double)v.m2;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < v.N; c += (int64_t)gridDim.x * blockDim.x) {
        int64_t i, j, k;
        cell_of(c, v.n, &i, &j, &k);
        if (i < v.region_lo[0] || i >= v.region_hi[0] || j < v.region_lo[1] || j >= v.region_hi[1] ||
            k < v.region_lo[2] || k >= v.region_hi[2])
            continue;
        T midT, DtT;
        phi_mid_dt<T, INCR>(v, q, i, j, k, &midT, &DtT);
        const double mid = midT, Dt = DtT;
        double g2 = 0.0, R = 0.0, bg = 0.0;
        // divisions by d and 2d (a multiplication where the reciprocal is exact)
        auto od = [&](double x, int a) { return v.rd[a] != T(0) ? x * (double)v.rd[a] : x / (double)v.d[a]; };
        auto o2d = [&](double x, int a) {
            return v.rd2[a] != T(0) ? x * (double)v.rd2[a] : x / (2.0 * (double)v.d[a]);
        };
        for (int a = 0; a < 3; a++) {
            int64_t u[3];
            unit(a, u);
            const double up = (double)phi_mid<T, INCR>(v, q, i + u[0], j + u[1], k + u[2]);
            const double dn = (double)phi_mid<T, INCR>(v, q, i - u[0], j - u[1], k - u[2]);
            const double fw = od(up - mid, a);
            g2 += fw * fw;
            const T *E1 = v.f[kE1 + a];
            R += od((double)E1[c] - (double)ld(v, E1, i - u[0], j - u[1], k - u[2]), a);
            bg += (double)b0_bar(v, a, i, j, k) * o2d(up - dn, a);
        }
        R += (double)v.g * bg;
        acc[0] += 0.5 * ((Dt * Dt + g2) + m2 * mid * mid) * dV;
        double e0 = 0.0, e1 = 0.0, x = 0.0;
        for (int a = 0; a < 3; a++) {
            const double E0a = v.f[kE0 + a][c], B0a = v.f[kB0 + a][c];
            const double E1a = v.f[kE1 + a][c], B1a = v.f[kB1 + a][c];
            e0 += E0a * E0a + B0a * B0a;
            e1 += E1a * E1a + B1a * B1a;
            x += (E0a + (double)v.Eext[a]) * E1a + (B0a + (double)v.Bext[a]) * B1a;
        }
        acc[1] += 0.5 * e0 * dV;
        acc[2] += 0.5 * e1 * dV;
        acc[3] += x * dV;
        const double xb = (double)v.lo[0] + (double)(i + 1) * (double)v.d[0];
        const double b1z = v.f[kB1 + 2][c];
        const double bz2 = b1z * b1z * dV;
        acc[4] += xb * bz2;
        acc[5] += bz2;
        acc[6] += R * R * dV;
    }
    __shared__ double sh[kQ][kDiagThreads];
#pragma unroll
    for (int s = 0; s < kQ; s++) sh[s][threadIdx.x] = acc[s];
    __syncthreads();
    for (int w = kDiagThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
#pragma unroll
            for (int s = 0; s < kQ; s++) sh[s][threadIdx.x] += sh[s][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < kQ) partials[(int64_t)blockIdx.x * kQ + threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void __launch_bounds__(kDiagThreads) k_diag_final(const double *partials, int nblocks, axp_diag *out,
                                                             int64_t step, double t, unsigned *top)
{
    if (top && threadIdx.x < 3) top[threadIdx.x] = 0;  // for the next record's magnitudes
    __shared__ double part[8][kDiagThreads / 32], sh[kQ];
    double acc[8];
#pragma unroll
    for (int s = 0; s < 8; s++) acc[s] = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += kDiagThreads)
#pragma unroll
        for (int s = 0; s < kQ; s++) acc[s] += partials[(int64_t)b * kQ + s];
    block_sums(acc, part);
    if (threadIdx.x < kQ) {
        double t = 0.0;
        for (int w = 0; w < kDiagThreads / 32; w++) t += part[threadIdx.x][w];
        sh[threadIdx.x] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        axp_diag d;
        d.step = step;
        d.t = t;
        d.H_phi = sh[0];
        d.H_g0 = sh[1];
        d.H_g1 = sh[2];
        d.P_g2a = d.H_g0 > 0 ? d.H_phi / d.H_g0 : 0.0;
        d.P_a2g = d.H_phi > 0 ? d.H_g1 / d.H_phi : 0.0;
        d.W = d.H_phi + sh[3];
        d.sum_xB1z2 = sh[4];
        d.sum_B1z2 = sh[5];
        d.gauss_l2 = sh[6];
        *out = d;
    }
}

}  // namespace

template <typename T>
static Ghosts<T> ghosts_lvl(axp_grid *g, int level)
{
    Ghosts<T> G;
    for (int a = 0; a < 3; a++)
        for (int s = 0; s < 2; s++) {
            const size_t off = g->layout.off_ghost[a][s][g->ghost_level_slot[level]];
            G.p[a][s] = off ? (T *)(g->ws + off) : nullptr;
        }
    return G;
}

template <typename T>
cudaError_t diag_compute(axp_grid *g, axp_diag *dev_dst)
{
    return diag_compute_rows<T>(g, dev_dst, -1, 0, 0);
}

// E^n from the two E levels a single-pass step leaves (Sec. 2.3): both E
// half-steps of the step from n-1/2 read the same X = curl B^n - g J^n, so
// E^n = a E^{n-1/2} + b X and E^{n+1/2} = a E^n + b X, where a, b are the
// half-step's layer coefficients (a = 1, b = h outside the layers; the smallest
// a of the axes at a corner).  Hence E^n = (E^{n+1/2} + a E^{n-1/2}) / (1 + a),
// the mean of the two levels outside the layers.  Written over E^{n-1/2} (the
// other field set); only the E arrays that can be non-zero (the others are zero in
// both sets).
template <typename T>
struct ELevels {
    T *lo[6];        // E^{n-1/2}, overwritten with E^n (order 0 xyz, order 1 xyz)
    const T *hi[6];  // E^{n+1/2}
    const T *a1[3];  // per axis, the one-half-step layer coefficient a (null: no layer along the axis)
    unsigned mask;   // arrays to form
    int lay[3][2];   // cells of absorbing layer at each side
    int64_t n0, n1, n2;
};

template <typename T, typename I>
__global__ void __launch_bounds__(kDiagThreads) k_e_level(ELevels<T> L, Sums<T> s, uint32_t mask)
{
    unsigned m0 = 0, m1 = 0, mp = 0;  // FP32: the region's largest magnitudes on the way
    const I N = (I)L.n0 * (I)L.n1 * (I)L.n2, n0 = (I)L.n0, n1 = (I)L.n1;
    for (I c = (I)blockIdx.x * blockDim.x + threadIdx.x; c < N; c += (I)gridDim.x * blockDim.x) {
        const I r = c / n0, k = r / n1;
        const int x[3] = {(int)(c - r * n0), (int)(r - k * n1), (int)k};
        bool layer = false, in = sizeof(T) == 4 && s.top;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            layer = layer || x[a] < L.lay[a][0] || x[a] >= s.n[a] - L.lay[a][1];
            in = in && x[a] >= s.lo[a] && x[a] < s.hi[a];
        }
        T a1 = T(1), inv = T(0.5);
        if (layer) {
#pragma unroll
            for (int a = 0; a < 3; a++)
                if (L.a1[a]) a1 = min(a1, L.a1[a][x[a]]);
            inv = T(1) / (T(1) + a1);
        }
#pragma unroll
        for (int f = 0; f < 6; f++) {
            if (!(L.mask >> f & 1u)) continue;
            const T hi = L.hi[f][c], lo = L.lo[f][c];
            T e = hi + lo;
            if (layer) e = hi + a1 * lo;
            e = e * inv;
            L.lo[f][c] = e;
            if constexpr (sizeof(T) == 4) {
                if (in && f < 3) m0 = max(m0, mag(e));
                if (in && f >= 3) m1 = max(m1, mag(e));
            }
        }
        if (in) max_of_cell(s, c, mask, false, m0, m1, mp);
    }
    if (sizeof(T) == 4 && s.top) max_group(s.top, m0, m1, mp);
}

template <typename T>
static Sums<T> make_sums(axp_grid *g, const View<T> &v)
{
    Sums<T> s;
    for (int a = 0; a < 3; a++) {
        s.E0[a] = v.f[kE0 + a];
        s.B0[a] = v.f[kB0 + a];
        s.E1[a] = v.f[kE1 + a];
        s.B1[a] = v.f[kB1 + a];
        for (int e = 0; e < 2; e++) {
            s.gh[a][e] = v.gh[a][e][0];
            s.gh_old[a][e] = v.gh[a][e][1];
            s.axbc[a][e] = v.axbc[a][e];
        }
        s.n[a] = (int)v.n[a];
        s.per[a] = v.periodic[a];
        s.lo[a] = v.region_lo[a];
        s.hi[a] = v.region_hi[a];
        s.Bext[a] = v.Bext[a];
        s.Eext[a] = v.Eext[a];
        s.d[a] = (double)v.d[a];
        s.rd[a] = 1.0 / s.d[a];
        s.kgb[a] = (sizeof(T) == 4 ? 0.5 : 0.25) * (double)v.g * (double)v.Bext[a];
        s.ext = (a ? s.ext : 0) | (v.Eext[a] != T(0) ? 1 << a : 0) | (v.Bext[a] != T(0) ? 8 << a : 0);
    }
    s.phi = v.phi_cur;
    s.phib = v.phi_b;
    s.N = (unsigned)v.N;
    s.lo0 = (double)v.lo[0];
    s.dt = (double)v.dt;
    s.kg = (sizeof(T) == 4 ? 0.5 : 0.25) * (double)v.g;
    s.m2 = (double)v.m2;
    s.top = sizeof(T) == 4 ? (unsigned *)(g->ws + g->layout.off_flag) + 8 : nullptr;
    s.partials = (double *)(g->ws + g->layout.off_partials);
    return s;
}

// the kernel for the active axes and the order-0 components present (mask: bits 0-2 E0,
// 3-5 B0)
template <typename T>
static void launch_sums(const Sums<T> &s, uint32_t mask, int nb, cudaStream_t st)
{
    const uint32_t tm = 4u | (3u << 3), te = 3u | (4u << 3);
    const int set = mask == 0 ? 0 : (mask & ~tm) == 0 ? 1 : (mask & ~te) == 0 ? 2 : 3;
#define AXP_SUMS(M)                                                                                        \
    switch (set) {                                                                                         \
    case 0: k_diag_sums<T, M, 0, 0><<<nb, kDiagThreads, 0, st>>>(s); break;                                \
    case 1: k_diag_sums<T, M, 4, 3><<<nb, kDiagThreads, 0, st>>>(s); break;                                \
    case 2: k_diag_sums<T, M, 3, 4><<<nb, kDiagThreads, 0, st>>>(s); break;                                \
    default: k_diag_sums<T, M, 7, 7><<<nb, kDiagThreads, 0, st>>>(s); break;                               \
    }
    if (s.n[2] == 1 && s.n[1] == 1) {
        AXP_SUMS(1)
    } else if (s.n[2] == 1) {
        AXP_SUMS(3)
    } else {
        AXP_SUMS(7)
    }
#undef AXP_SUMS
}

template <typename T>
cudaError_t e_level_from_halves(axp_grid *g, const Sums<T> &s, uint32_t mask)
{
    ELevels<T> L;
    const Workspace &w = g->layout;
    const int oset = 1 - g->fset;
    const int fe[6] = {kE0, kE0 + 1, kE0 + 2, kE1, kE1 + 1, kE1 + 2};
    L.mask = 0;
    for (int f = 0; f < 6; f++) {
        L.lo[f] = (T *)(g->ws + w.off_fields[oset][fe[f]]);
        L.hi[f] = (const T *)(g->ws + w.off_fields[g->fset][fe[f]]);
        if (f >= 3 || (mask >> f & 1u)) L.mask |= 1u << f;  // (injected, driven or from another grid's rows)
    }
    for (int a = 0; a < 3; a++) {
        const bool lay = g->desc.em_bc[a][0] != AXP_BC_PERIODIC && g->desc.pml_cells > 0 && g->desc.pml_sigma_max_dt > 0;
        L.a1[a] = lay ? (const T *)(g->ws + w.off_pml_tab[a]) : nullptr;
        for (int e = 0; e < 2; e++)
            L.lay[a][e] = lay && g->desc.em_bc[a][e] == AXP_BC_PML ? (int)std::min<int64_t>(g->desc.pml_cells, g->desc.n[a]) : 0;
    }
    L.n0 = g->desc.n[0];
    L.n1 = g->desc.n[1];
    L.n2 = g->desc.n[2];
    const int64_t N = L.n0 * L.n1 * L.n2;
    const unsigned nb = (unsigned)std::min<int64_t>((N + kDiagThreads - 1) / kDiagThreads, 152 * 8);
    if (N < (int64_t)1 << 30) k_e_level<T, unsigned><<<nb, kDiagThreads, 0, g->stream>>>(L, s, mask);
    else k_e_level<T, int64_t><<<nb, kDiagThreads, 0, g->stream>>>(L, s, mask);
    g->launches++;
    g->half_prev = false;  // the other set now holds E^n
    return cudaGetLastError();
}

// The sums over the cells whose index along `axis` lies in [lo, hi) as well as in
// the physical region (axis < 0: no restriction).  A slab of a decomposed grid
// sums its owned rows this way; the records' sums add up across slabs.
template <typename T>
cudaError_t diag_compute_rows(axp_grid *g, axp_diag *dev_dst, int axis, int64_t lo, int64_t hi)
{
    // staggered (fused-path) state: reconstruct E^n into the spare field set first,
    // from the two levels of the last single-pass step where the other set holds
    // them, else by the general kernels' inverse half-step
    const bool halves = g->staggered && g->half_prev && g->half_prev_cfg == g->cfg_version;
    // the time-blocked 1D kernel leaves E^n in the current's scratch (J: E0y, E0z, E1x; P: E1y, E1z)
    const bool scratch = g->staggered && g->en_scratch && g->en_scratch_cfg == g->cfg_version;
    const bool wide = (int64_t)g->desc.n[0] * g->desc.n[1] * g->desc.n[2] >= (int64_t)1 << 30;  // (64-bit indexes)
    const uint32_t mask = order0_present(g);
    if (g->staggered && !halves && !scratch) {
        const cudaError_t e = exit_staggered<T>(g, false);
        if (e != cudaSuccess) return e;
    }
    View<T> v = g->staggered && !scratch ? make_view_eset<T>(g, 1 - g->fset) : make_view<T>(g);
    if (scratch) {
        const Workspace &w = g->layout;
        const size_t off[5] = {w.off_J[0], w.off_J[1], w.off_J[2], w.off_P[0], w.off_P[1]};
        const int f[5] = {kE0 + 1, kE0 + 2, kE1, kE1 + 1, kE1 + 2};
        for (int q = 0; q < 5; q++) v.f[f[q]] = (T *)(g->ws + off[q]);
    }
    if (axis >= 0) {
        if (lo > v.region_lo[axis]) v.region_lo[axis] = (int)lo;
        if (hi < v.region_hi[axis]) v.region_hi[axis] = (int)hi;
    }
    Sums<T> s = make_sums<T>(g, v);
    if (wide) s.top = nullptr;
    if (halves) {
        const cudaError_t e = e_level_from_halves<T>(g, s, mask);
        if (e != cudaSuccess) return e;
    } else if (s.top) {
        const unsigned grid = std::min<unsigned>((s.N + kDiagThreads - 1) / kDiagThreads, 152 * 8);
        k_diag_max<T><<<grid, kDiagThreads, 0, g->stream>>>(s, mask);
        g->launches++;
    }
    double *partials = s.partials;
    // one wave of blocks: a wave and a part of the next costs two
    const int nb = wide ? g->layout.diag_blocks : std::min(g->layout.diag_blocks, 152 * diag_blocks_per_sm<T>(g->desc.n[2] > 1 ? 7 : 3));
    if (wide) {
        PhiPair<T, sizeof(T) == 4> q{v.phi_cur, v.phi_b, ghosts_lvl<T>(g, 0), ghosts_lvl<T>(g, 1)};
        k_diag_partial<T, sizeof(T) == 4><<<nb, kDiagThreads, 0, g->stream>>>(v, q, partials);
    } else {
        launch_sums<T>(s, mask, nb, g->stream);
    }
    k_diag_final<<<1, kDiagThreads, 0, g->stream>>>(partials, nb, dev_dst, g->step, (double)g->step * g->desc.dt, s.top);
    g->launches += 2;
    return cudaGetLastError();
}

template cudaError_t diag_compute<double>(axp_grid *, axp_diag *);
template cudaError_t diag_compute<float>(axp_grid *, axp_diag *);
template cudaError_t diag_compute_rows<double>(axp_grid *, axp_diag *, int, int64_t, int64_t);
template cudaError_t diag_compute_rows<float>(axp_grid *, axp_diag *, int, int64_t, int64_t);

// ---------------------------------------------------------------------------
// Diagnostics for callers that cannot allocate device memory.
//
// The per-block partial sums and the result record live in file-scope static
// device arrays instead of a workspace, so this entry point needs no
// allocation at all.  Every GPU that loads the library holds these arrays
// (kNoallocBlocks x 7 doubles + one record, about 230 KB) until the process
// exits.  The arrays are shared by every call: each call rewrites all the
// partials it uses and the result record, so nothing carries over between
// calls, but calls that overlap on the GPU (other host threads or streams)
// race on the shared arrays.
// ---------------------------------------------------------------------------
namespace {

constexpr int kNoallocBlocks = 4096;         // partial sums: one block of 256 threads ...
constexpr int kNoallocCellsPerBlock = 2048;  // ... covers 2048 cells (8 per thread)
constexpr int64_t kNoallocMaxCells = (int64_t)kNoallocBlocks * kNoallocCellsPerBlock;  // 8,388,608
constexpr int kNoallocMaxDevices = 64;

static __device__ __align__(256) double g_noalloc_partials[kNoallocBlocks * kQ];
static __device__ __align__(256) axp_diag g_noalloc_result;

std::mutex g_noalloc_mutex;
double *g_noalloc_partials_addr[kNoallocMaxDevices];
axp_diag *g_noalloc_result_addr[kNoallocMaxDevices];

// Device addresses of the static arrays for the current device.  In host code
// the array names are host-side stand-ins, never device addresses, so the
// real addresses are looked up once per device with that device current.
cudaError_t noalloc_setup(int dev, double **partials, axp_diag **result)
{
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_partials_addr[dev]) {
        void *p = nullptr, *r = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_partials);
        if (e != cudaSuccess) return e;
        e = cudaGetSymbolAddress(&r, g_noalloc_result);
        if (e != cudaSuccess) return e;
        g_noalloc_partials_addr[dev] = (double *)p;
        g_noalloc_result_addr[dev] = (axp_diag *)r;
    }
    *partials = g_noalloc_partials_addr[dev];
    *result = g_noalloc_result_addr[dev];
    return cudaSuccess;
}

}  // namespace
}  // namespace axp

extern "C" axp_status axp_diagnostics_noalloc(const axp_grid_desc *desc, const double *const dev_fields[14],
                                              const double B_ext[3], const double E_ext[3], int64_t step,
                                              void *cuda_stream, axp_diag *host_out)
{
    using namespace axp;
    if (!desc || !dev_fields || !B_ext || !E_ext || !host_out) return AXP_E_INVAL;
    for (int f = 0; f < 14; f++)
        if (!dev_fields[f]) return AXP_E_INVAL;
    size_t ws = 0;
    const axp_status st = axp_workspace_bytes(desc, &ws);  // host-side validation only
    if (st != AXP_OK) return st;
    if (desc->precision != AXP_FP64) {
        fprintf(stderr, "axp_diagnostics_noalloc: only FP64 fields are accepted\n");
        return AXP_E_INVAL;
    }
    for (int a = 0; a < 3; a++)
        for (int s = 0; s < 2; s++)
            if (desc->axion_bc[a][s] == AXP_BC_OUTFLOW) {
                fprintf(stderr, "axp_diagnostics_noalloc: outflow faces need ghost planes; use axp_compute_diagnostics\n");
                return AXP_E_INVAL;
            }
    const int64_t N = desc->n[0] * desc->n[1] * desc->n[2];
    if (N > kNoallocMaxCells) {
        fprintf(stderr, "axp_diagnostics_noalloc: %lld cells exceed the maximum of %lld\n", (long long)N,
                (long long)kNoallocMaxCells);
        return AXP_E_INVAL;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoallocMaxDevices) return AXP_E_CUDA;
    double *partials = nullptr;
    axp_diag *result = nullptr;
    if (noalloc_setup(dev, &partials, &result) != cudaSuccess) return AXP_E_CUDA;

    View<double> v;
    memset(&v, 0, sizeof(v));
    for (int f = 0; f < kFields; f++) v.f[f] = const_cast<double *>(dev_fields[f]);
    v.phi_cur = const_cast<double *>(dev_fields[12]);
    v.phi_b = const_cast<double *>(dev_fields[13]);
    for (int a = 0; a < 3; a++) {
        v.n[a] = desc->n[a];
        v.d[a] = desc->d[a];
        v.lo[a] = desc->lo[a];
        v.Bext[a] = B_ext[a];
        v.Eext[a] = E_ext[a];
        v.periodic[a] = desc->em_bc[a][0] == AXP_BC_PERIODIC;
        for (int s = 0; s < 2; s++) v.axbc[a][s] = desc->axion_bc[a][s];
        int rlo = 0, rhi = (int)desc->n[a];
        if (desc->n[a] > 1 && !v.periodic[a]) {
            if (desc->em_bc[a][0] == AXP_BC_PML || desc->axion_bc[a][0] == AXP_BC_PML) rlo = desc->pml_cells;
            if (desc->em_bc[a][1] == AXP_BC_PML || desc->axion_bc[a][1] == AXP_BC_PML) rhi = (int)desc->n[a] - desc->pml_cells;
        }
        v.region_lo[a] = rlo;
        v.region_hi[a] = rhi;
    }
    v.N = N;
    v.dt = desc->dt;
    v.h = desc->dt / 2.0;
    v.g = desc->g;
    v.m2 = desc->m * desc->m;
    set_reciprocals(v);
    PhiPair<double, false> q;
    memset(&q, 0, sizeof(q));
    q.hi = v.phi_cur;
    q.b = v.phi_b;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    int nb = (int)((N + kNoallocCellsPerBlock - 1) / kNoallocCellsPerBlock);
    if (nb < 1) nb = 1;
    k_diag_partial<double, false><<<nb, kDiagThreads, 0, stream>>>(v, q, partials);
    k_diag_final<<<1, kDiagThreads, 0, stream>>>(partials, nb, result, step, (double)step * desc->dt, nullptr);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(host_out, result, sizeof(axp_diag), cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) {
        fprintf(stderr, "axp: CUDA error %s\n", cudaGetErrorString(e));
        return AXP_E_CUDA;
    }
    const double vals[] = {host_out->H_phi, host_out->H_g0, host_out->H_g1, host_out->W, host_out->gauss_l2};
    for (double x : vals)
        if (!std::isfinite(x)) return AXP_E_NONFINITE;
    return AXP_OK;
}

