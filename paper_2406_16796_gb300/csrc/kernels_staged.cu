// kernels_staged.cu -- the multi-pass step with folded arithmetic (arXiv 2406.16796
// Sec. 2.3-2.4), for the grids that no specialised single-pass kernel takes:
// outflow sides, a uniform E, FP64 3D, macroparticles, lasers outside the TM set.
//
// What bounds it: on GB300 an FP64 step is bound by the FP64 pipe (2 operations
// per cycle per SM), so each quantity is formed once and every constant is folded;
// an FP32 step by memory and launch latency.  The literal kernels
// (kernels_general.cu) take 8 launches and several hundred FP64 operations per 3D cell
// (their divisions included); these take 4 launches and 187:
//   B      B^{n+1} of both orders; B0^{n+1/2} is kept in scratch
//   phi    S and phi^{n+3/2}; E0^{n+1} (to scratch) and E0^{n+3/2}
//   P      the axion current's P at the cell centres
//   J      J, E1^{n+1} and E1^{n+3/2}
// With macroparticles the B pass is two half passes around the push and the E0
// update a pass of its own.  One thread per cell, neighbours through L1/L2 by
// offsets that already hold the wrap, the closure of non-periodic sides as
// predicated loads: no branch over cells but the absorbing layer's.
//
// Only active axes and order-0 components that can be non-zero are computed (template
// arguments).  Field sets alternate: the step reads one and writes the other.
//
// The E half-steps of one step and of the next read the same X = curl B - g J, so
// both are taken at once, but as two updates by the same increment: a run cut into
// several calls then gives the bits of the uncut one.  Multiply-adds are written
// out and the unit is compiled without contraction, for the same reason.
//
// Measured on one GB300 (us per step, before: the literal or the generic kernel):
//   2D TM laser, outflow axion sides, FP64, 1024 x 512       686 -> 115
//   3D laser, absorbing x sides, FP64, 160 x 96 x 96        1922 -> 547
//   2D laser polarised in the plane, FP32 split, 1024 x 512  130 -> 33
//   2D TM laser, absorbing sides, FP64, 400 x 400            160 -> 42 (the 2D kernel)
// ncu: the FP64 passes keep the FP64 pipe 73 to 84% busy while an SM is active on the two larger
// grids (93 operations per cell of the 1024 x 512 one, 187 of the 3D one), 63 to 66% at 400 x 400,
// where a pass is less than one wave of blocks
// (profiles/k_stage_warp_line_records_counters.md).
#include <algorithm>

#include "cells.cuh"
#include "device_common.cuh"

namespace axp {
namespace {

constexpr int kThreads = 128;  // (256: 3% slower on 1024 x 512, 8% on 400 x 400)

template <typename T>
struct Stage {
    const T *Ein[6], *Bin[6];  // E^{n+1/2}, B^n (order 0 xyz, order 1 xyz)
    T *Eout[6], *Bout[6];
    T *Bh[3];  // scratch: B0^{n+1/2}
    T *Eh[3];  // scratch: E0^{n+1}
    T *P[3], *J[3];
    const T *phi, *phib;  // phi^{n+1/2}; phi^{n-1/2} (FP64) or the increment (FP32 split)
    T *phi_out, *phib_out;
    const T *jp[2][3];                  // macroparticle currents (null without)
    // outflow ghosts: phi^{n+1/2}, phi^{n-1/2}, phi^{n+3/2} written, and (gh_hi) the later
    // level the P pass reads
    const T *gh[3][2], *gh_old[3][2], *gh_hi[3][2];
    T *gh_new[3][2];
    const T *tab[3];                    // layer coefficients per axis (null: no layer)
    const T *sig_ax[3];
    int n[3], per[3], axbc[3][2];
    int lay[3][2];  // cells of absorbing layer at each side
    int N;
    int uniform_e;
    T hd[3];              // h/d
    T inv_h, h;
    T hg2;                // h g / 2: J is used as the sum of two P
    T lap_c[3], dt2g, m2dt2, dt, dt2, inv_dt2, inv_dt, q4d[3], of_r[3];
    T Bext[3], Eext[3];
    int src_x;            // x index of the soft source's E cells (-1: none)
    const T *src_w[2];
    T src_e, src_b;       // h tau of the electric and of the magnetic sheet
    int last;             // the step ends at integer time (only the first E half-step)
};

// Programmatic dependent launch: a pass is set up while the one before it ends, and
// waits here before its first access to memory another pass writes.  No earlier
// trigger is given: blocks of the next pass that come in while this one still runs
// land on the SMs that are free first and leave them unevenly loaded (256 x 128 FP64:
// 41 us per step with a trigger at the start, 18 without).
__device__ __forceinline__ void wait_for_previous_pass()
{
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
}
template <typename... KArgs, typename... Args>
void launch_pass(void (*kern)(KArgs...), int blocks, cudaStream_t st, const Args &...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);  // (errors: the caller's cudaGetLastError)
}

// this thread's cell
template <int MASK, typename T>
__device__ __forceinline__ bool cell_at(const Stage<T> &s, Cell &q)
{
    const unsigned c = blockIdx.x * (unsigned)kThreads + threadIdx.x;
    if (c >= (unsigned)s.N) return false;
    cell_of_index<MASK>(s.n, s.per, c, q);
    return true;
}

// h (curl F)_a with differences towards `up` (forward) or from `dn` (backward):
// hb (dF_c along b) - hc (dF_b along c), without the terms of inactive axes and
// of components that are zero (CM: mask of the components present).
template <int MASK, int CM, bool FWD, typename T>
__device__ __forceinline__ T curl_h(const Stage<T> &s, const T *const F[3], int a, const Cell &q)
{
    const int b = (a + 1) % 3, c = (a + 2) % 3;
    const bool t1 = (MASK >> b & 1) && (CM >> c & 1), t2 = (MASK >> c & 1) && (CM >> b & 1);
    T d1 = T(0), d2 = T(0);
    if (t1) d1 = FWD ? ldz(F[c], q.up[b], q.hu[b]) - F[c][q.c] : F[c][q.c] - ldz(F[c], q.dn[b], q.hd[b]);
    if (t2) d2 = FWD ? ldz(F[b], q.up[c], q.hu[c]) - F[b][q.c] : F[b][q.c] - ldz(F[b], q.dn[c], q.hd[c]);
    if (t1 && t2) return fma(s.hd[b], d1, -(s.hd[c] * d2));
    if (t1) return s.hd[b] * d1;
    if (t2) return -(s.hd[c] * d2);
    return T(0);
}

// The absorbing layer at a cell: a half-step is F <- a F + r (h X) (a = r = 1 outside
// the layers); both decrease with sigma, so a corner takes the smallest.  Whether a
// cell lies in a layer is decided on integers (a comparison of doubles takes the FP64
// pipe), and a warp with any layer cell takes the IN body for all its cells: with
// a = r = 1 it rounds as the plain one, and two bodies run in turn by a divided warp
// cost more (3D laser 160 x 96 x 96: 658 against 538 us per step).
template <typename T, bool IN>
struct Layer {
    T a, r;
    bool in;
    __device__ __forceinline__ T half_step(T F, T hX) const { return IN ? fma(a, F, r * hX) : F + hX; }
};
template <int MASK, typename T>
__device__ __forceinline__ bool in_layer(const Stage<T> &s, const Cell &q)
{
    bool in = false;
#pragma unroll
    for (int a = 0; a < 3; a++)
        if (MASK >> a & 1) in = in || q.x[a] < s.lay[a][0] || q.x[a] >= s.n[a] - s.lay[a][1];
    return in;
}
// whether any of the warp's cells (those of an incomplete last warp) lies in a layer
template <int MASK, typename T>
__device__ __forceinline__ bool warp_in_layer(const Stage<T> &s, const Cell &q)
{
    return __any_sync(__activemask(), in_layer<MASK>(s, q));
}
template <int MASK, bool IN, typename T>
__device__ __forceinline__ Layer<T, IN> layer_at(const Stage<T> &s, const Cell &q)
{
    Layer<T, IN> L{T(1), T(1), false};
    if (!IN || !in_layer<MASK>(s, q)) return L;
    L.in = true;
    T b = s.h;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        if (!(MASK >> a & 1) || !s.tab[a]) continue;
        L.a = min(L.a, s.tab[a][q.x[a]]);
        b = min(b, s.tab[a][s.n[a] + q.x[a]]);
    }
    L.r = b * s.inv_h;
    return L;
}

// MODE 0: the full B step (B0^{n+1/2} to scratch); 1 and 2: one half-step from Bin
// to Bout (with macroparticles; the second in place).
template <typename T, int MASK, int EM, int BM, int MODE, bool IN>
__device__ __forceinline__ void b_pass(const Stage<T> &s, const Cell &q)
{
    const Layer<T, IN> L = layer_at<MASK, IN>(s, q);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        if (!(BM >> a & 1)) continue;
        T hX = -curl_h<MASK, EM, true>(s, s.Ein, a, q);
        if (a > 0 && q.x[0] == s.src_x - 1) {
            const int jk = q.x[1] + s.n[1] * q.x[2];
            hX = a == 1 ? fma(-s.src_w[1][jk], s.src_b, hX) : fma(s.src_w[0][jk], s.src_b, hX);
        }
        const T Bh = L.half_step(s.Bin[a][q.c], hX);
        if (MODE == 0) {
            s.Bh[a][q.c] = Bh;
            s.Bout[a][q.c] = L.half_step(Bh, hX);
        } else {
            s.Bout[a][q.c] = Bh;
        }
    }
    const T *const E1[3] = {s.Ein[3], s.Ein[4], s.Ein[5]};
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const T hX = -curl_h<MASK, 7, true>(s, E1, a, q), B = s.Bin[3 + a][q.c];
        T r;
        if (MODE > 0) r = L.half_step(B, hX);
        else if (IN && L.in) r = L.half_step(L.half_step(B, hX), hX);
        else r = fma(T(2), hX, B);
        s.Bout[3 + a][q.c] = r;
    }
}
template <typename T, int MASK, int EM, int BM, int MODE>
__global__ void __launch_bounds__(kThreads) k_stage_b(Stage<T> s)
{
    Cell q;
    const bool mine = cell_at<MASK>(s, q);
    wait_for_previous_pass();
    if (!mine) return;
    if (warp_in_layer<MASK>(s, q)) b_pass<T, MASK, EM, BM, MODE, true>(s, q);
    else b_pass<T, MASK, EM, BM, MODE, false>(s, q);
}

// 2-point average of E0_a at the cell centre plus the background
template <int MASK, int EM, typename T>
__device__ __forceinline__ T ebar(const Stage<T> &s, const T *const E[3], int a, const Cell &q)
{
    if (!(EM >> a & 1)) return s.Eext[a];
    const T f = E[a][q.c];
    if (!(MASK >> a & 1)) return s.uniform_e ? f + s.Eext[a] : f;
    return fma(T(0.5), f + ldz(E[a], q.dn[a], q.hd[a]), s.Eext[a]);
}

// 4-point average of B0_a at the cell centre plus the background
template <int MASK, int BM, typename T>
__device__ __forceinline__ T bbar(const Stage<T> &s, const T *const B[3], int a, const Cell &q)
{
    if (!(BM >> a & 1)) return s.Bext[a];
    const int b = (a + 1) % 3, c = (a + 2) % 3;
    const bool mb = MASK >> b & 1, mc = MASK >> c & 1;
    T f = B[a][q.c], w = T(1);
    if (mb) {
        f = f + ldz(B[a], q.dn[b], q.hd[b]);
        w = T(0.5);
    }
    if (mc) {
        T g = ldz(B[a], q.dn[c], q.hd[c]);
        if (mb) g = g + ldz(B[a], q.dn[b] + (q.dn[c] - q.c), q.hd[b] && q.hd[c]);
        f = f + g;
        w = w * T(0.5);
    }
    return fma(w, f, s.Bext[a]);
}

// Neighbour of an axion level along axis a: inside the grid, by the boundary beyond it
// (periodic wrap, reflect: the cell itself, outflow: the ghost plane, PML: 0).
template <typename T>
__device__ __forceinline__ T phi_nb(const Stage<T> &s, const T *__restrict__ F, const T *const gh[3][2], int a, int side,
                                    const Cell &q)
{
    if (side ? q.hu[a] : q.hd[a]) return F[side ? q.up[a] : q.dn[a]];
    const int bc = s.axbc[a][side];
    if (bc == AXP_BC_REFLECT) return F[q.c];
    if (bc != AXP_BC_OUTFLOW) return T(0);
    return gh[a][side][ghost_index(s.n, a, q)];
}

// The outflow ghost next to cell q on one face, at the new level (Sec. 2.4 item 3): the
// one-way wave equation and the wave equation at the ghost, solved for phi^{cur} half
// a cell further out (V) and phi^{new} at the ghost.  The source at the ghost cell, which
// sees zero fields outside the grid plus the background: along the face normal E0 of
// the last cell (high side) meets B_ext, across it E_ext meets B0 averaged with zeros.
template <typename T, int MASK, int EM, int BM>
__device__ void outflow_ghost(const Stage<T> &s, const T *const Bs[3], int ax, int side, T p0, const Cell &q)
{
    T S = T(0);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        T e = s.Eext[a], b = s.Bext[a];
        if (a == ax) {
            if (side && (EM >> a & 1)) e = fma(T(0.5), s.Ein[a][q.c], e);
        } else if (side && (BM >> a & 1)) {
            const int o = 3 - a - ax;  // the third axis
            b = fma(T(0.25), Bs[a][q.c] + ldz(Bs[a], q.dn[o], q.hd[o]), b);
        }
        S = fma(e, b, S);
    }
    const int pi = ghost_index(s.n, ax, q);
    const T gc = s.gh[ax][side][pi], go = s.gh_old[ax][side][pi], r = s.of_r[ax];
    T rhs = fma(T(2), go - gc, fma(s.m2dt2, gc, -(s.dt2g * S)));
    rhs = fma(r, p0, rhs) - r * r * fma(T(-2), gc, p0);
    const T V = rhs / fma(r, r, r);
    s.gh_new[ax][side][pi] = fma(r, p0 - V, go);
}

// E0 from E0^{n+1/2}: E0^{n+1} to scratch and, unless the step ends at integer time,
// E0^{n+3/2} to the output set.
template <typename T, int MASK, int EM, int BM, bool IN>
__device__ __forceinline__ void e0_update(const Stage<T> &s, const Cell &q)
{
    const Layer<T, IN> L = layer_at<MASK, IN>(s, q);
    const T *const B0[3] = {s.Bout[0], s.Bout[1], s.Bout[2]};
#pragma unroll
    for (int a = 0; a < 3; a++) {
        if (!(EM >> a & 1)) continue;
        T hX = curl_h<MASK, BM, false>(s, B0, a, q);
        if (a > 0 && q.x[0] == s.src_x) hX = fma(s.src_w[a - 1][q.x[1] + s.n[1] * q.x[2]], s.src_e, hX);
        if (s.jp[0][a]) hX = fma(-s.h, s.jp[0][a][q.c], hX);
        const T E = L.half_step(s.Ein[a][q.c], hX);
        s.Eh[a][q.c] = E;
        s.Eout[a][q.c] = s.last ? E : L.half_step(E, hX);
    }
}

// PHI: the axion leapfrog with its source; E0: the order-0 E update.  Bs: where
// B0^{n+1/2} lies (the B pass's scratch, or Bout between the half passes).
template <typename T, int MASK, int EM, int BM, bool PHI, bool E0>
__global__ void __launch_bounds__(kThreads) k_stage_phi(Stage<T> s, const T *bs0, const T *bs1, const T *bs2)
{
    constexpr bool INCR = sizeof(T) == 4;
    Cell q;
    const bool mine = cell_at<MASK>(s, q);
    wait_for_previous_pass();
    if (!mine) return;
    if (PHI) {
        const T *const Bs[3] = {bs0, bs1, bs2};
        T S = T(0);
#pragma unroll
        for (int a = 0; a < 3; a++)
            if ((EM >> a & 1) || s.uniform_e) S = fma(ebar<MASK, EM>(s, s.Ein, a, q), bbar<MASK, BM>(s, Bs, a, q), S);
        const T ph = s.phi[q.c], old = s.phib[q.c];
        T lap = s.dt2g * S;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            if (!(MASK >> a & 1)) continue;
            const T up = phi_nb(s, s.phi, s.gh, a, 1, q), dn = phi_nb(s, s.phi, s.gh, a, 0, q);
            // FP32 split: from neighbour differences, which do not round against 2 phi
            lap = fma(s.lap_c[a], INCR ? (up - ph) + (dn - ph) : fma(T(-2), ph, up + dn), lap);
        }
        lap = fma(-s.m2dt2, ph, lap);
        T nw;  // phi^{n+3/2}, or its increment in FP32 split
        if (in_layer<MASK>(s, q)) {
            // (lap - (sigma dt)^2 phi -+ (1 - sigma dt) old) / (1 + sigma dt) from the tables
            // c1 = dt^2 / (1 + sigma dt) and c2 = (1 - sigma dt) / (1 + sigma dt)
            T sd = T(0), c1 = s.dt2, c2 = T(1);
#pragma unroll
            for (int a = 0; a < 3; a++) {
                if (!(MASK >> a & 1) || !s.tab[a]) continue;
                sd = max(sd, s.sig_ax[a][q.x[a]]);
                c1 = min(c1, s.tab[a][4 * s.n[a] + q.x[a]]);
                c2 = min(c2, s.tab[a][5 * s.n[a] + q.x[a]]);
            }
            sd = sd * s.dt;
            lap = fma(-(sd * sd), ph, lap);
            if (!INCR) lap = fma(T(2), ph, lap);
            nw = fma(INCR ? c2 : -c2, old, c1 * s.inv_dt2 * lap);
        } else {
            // (2 phi apart from the mass and the Laplacian: folded into one coefficient, its
            // rounding acts as a mass and grows with the square of the steps)
            nw = INCR ? lap + old : fma(T(2), ph, -old) + lap;
        }
        s.phi_out[q.c] = INCR ? ph + nw : nw;
        if (INCR) s.phib_out[q.c] = nw;
        // the ghosts beyond outflow faces belong to the cells next to them
#pragma unroll
        for (int a = 0; a < 3; a++) {
            if (!(MASK >> a & 1)) continue;
            if (!q.hd[a] && s.axbc[a][0] == AXP_BC_OUTFLOW) outflow_ghost<T, MASK, EM, BM>(s, Bs, a, 0, ph, q);
            if (!q.hu[a] && s.axbc[a][1] == AXP_BC_OUTFLOW) outflow_ghost<T, MASK, EM, BM>(s, Bs, a, 1, ph, q);
        }
    }
    if (E0) {
        if (warp_in_layer<MASK>(s, q)) e0_update<T, MASK, EM, BM, true>(s, q);
        else e0_update<T, MASK, EM, BM, false>(s, q);
    }
}

// P = (D_t phi) Bbar0 - Ebar0 x grad_c phi^{n+1} at the cell centres, from E0^{n+1}
// (e0..e2) and B0^{n+1} (b0..b2); hi/lo: the axion levels around n+1 (lo the
// increment in FP32 split).
template <typename T, int MASK, int EM, int BM>
__global__ void __launch_bounds__(kThreads) k_stage_p(Stage<T> s, const T *e0, const T *e1, const T *e2, const T *b0,
                                                      const T *b1, const T *b2, const T *hi, const T *lo)
{
    constexpr bool INCR = sizeof(T) == 4;
    Cell q;
    const bool mine = cell_at<MASK>(s, q);
    wait_for_previous_pass();
    if (!mine) return;
    const T *const E[3] = {e0, e1, e2};
    const T *const B[3] = {b0, b1, b2};
    T g[3], e[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        g[a] = T(0);
        e[a] = ebar<MASK, EM>(s, E, a, q);
        if (!(MASK >> a & 1)) continue;
        // 2 phi^{n+1} at the two neighbours: the sum of the levels (ghost planes hold
        // levels, also in FP32 split, where the arrays hold phi and its increment)
        T two[2];
#pragma unroll
        for (int side = 0; side < 2; side++) {
            const bool in = side ? q.hu[a] : q.hd[a];
            const T h = phi_nb(s, hi, s.gh_hi, a, side, q), l = phi_nb(s, lo, s.gh, a, side, q);
            const bool incr = INCR && (in || s.axbc[a][side] == AXP_BC_REFLECT);
            two[side] = incr ? fma(T(2), h, -l) : h + l;
        }
        g[a] = s.q4d[a] * (two[1] - two[0]);
    }
    const T l = lo[q.c];
    const T Dt = (INCR ? l : hi[q.c] - l) * s.inv_dt;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const int b = (a + 1) % 3, c = (a + 2) % 3;
        T p = Dt * bbar<MASK, BM>(s, B, a, q);
        if ((MASK >> c & 1) && ((EM >> b & 1) || s.uniform_e)) p = fma(-e[b], g[c], p);
        if ((MASK >> b & 1) && ((EM >> c & 1) || s.uniform_e)) p = fma(e[c], g[b], p);
        s.P[a][q.c] = p;
    }
}

// Inverse of a half-step: the field a half-step earlier, given h X.
template <typename T, bool IN>
__device__ __forceinline__ T half_back(const Layer<T, IN> &L, T F, T hX)
{
    return IN ? fma(-L.r, hX, F) / L.a : F - hX;
}

// E0^n from E0^{n+1/2} (Eout may be Ein)
template <typename T, int MASK, int EM, int BM, bool IN>
__device__ __forceinline__ void e0_back(const Stage<T> &s, const Cell &q)
{
    const Layer<T, IN> L = layer_at<MASK, IN>(s, q);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        if (!(EM >> a & 1)) continue;
        T hX = curl_h<MASK, BM, false>(s, s.Bin, a, q);
        if (a > 0 && q.x[0] == s.src_x) hX = fma(s.src_w[a - 1][q.x[1] + s.n[1] * q.x[2]], s.src_e, hX);
        s.Eout[a][q.c] = half_back(L, s.Ein[a][q.c], hX);
    }
}
template <typename T, int MASK, int EM, int BM>
__global__ void __launch_bounds__(kThreads) k_stage_e0_back(Stage<T> s)
{
    Cell q;
    const bool mine = cell_at<MASK>(s, q);
    wait_for_previous_pass();
    if (!mine) return;
    if (in_layer<MASK>(s, q)) e0_back<T, MASK, EM, BM, true>(s, q);
    else e0_back<T, MASK, EM, BM, false>(s, q);
}

template <typename T, int MASK, bool IN>
__device__ __forceinline__ void e1_back(const Stage<T> &s, const T J2[3], const Cell &q)
{
    const Layer<T, IN> L = layer_at<MASK, IN>(s, q);
    const T *const B1[3] = {s.Bin[3], s.Bin[4], s.Bin[5]};
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const T hX = fma(-s.hg2, J2[a], curl_h<MASK, 7, false>(s, B1, a, q));
        s.Eout[3 + a][q.c] = half_back(L, s.Ein[3 + a][q.c], hX);
    }
}

template <typename T, int MASK, bool IN>
__device__ __forceinline__ void e1_update(const Stage<T> &s, const T J2[3], const Cell &q)
{
    const Layer<T, IN> L = layer_at<MASK, IN>(s, q);
    const T *const B1[3] = {s.Bout[3], s.Bout[4], s.Bout[5]};
#pragma unroll
    for (int a = 0; a < 3; a++) {
        T hX = fma(-s.hg2, J2[a], curl_h<MASK, 7, false>(s, B1, a, q));
        if (s.jp[1][a]) hX = fma(-s.h, s.jp[1][a][q.c], hX);
        T E = L.half_step(s.Ein[3 + a][q.c], hX);
        if (!s.last) E = L.half_step(E, hX);
        s.Eout[3 + a][q.c] = E;
    }
}
// J = (P(c) + P(c + a)) / 2 and the order-1 E update.  Beyond the
// last cell of a non-periodic axis P follows the ghost rules: 0 at a PML side without
// a uniform E, else evaluated in place (one cell per row or plane).
// WHAT 0: the step's update; 1: J alone, into its cache; 2: J and E1^n from E1^{n+1/2}
template <typename T, int MASK, int WHAT>
__global__ void __launch_bounds__(kThreads) k_stage_j(Stage<T> s, View<T> v, PhiPair<T, sizeof(T) == 4> pq)
{
    Cell q;
    const bool mine = cell_at<MASK>(s, q);
    wait_for_previous_pass();
    if (!mine) return;
    T J2[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const T p0 = s.P[a][q.c];
        T p1 = p0;
        if (MASK >> a & 1) {
            if (q.hu[a]) p1 = s.P[a][q.up[a]];
            else if (s.axbc[a][1] == AXP_BC_PML && !s.uniform_e) p1 = T(0);
            else
                p1 = p_comp<T, sizeof(T) == 4>(v, pq, a, q.x[0] + (a == 0), q.x[1] + (a == 1), q.x[2] + (a == 2));
        }
        J2[a] = p0 + p1;
        if (WHAT || s.last) s.J[a][q.c] = T(0.5) * J2[a];
    }
    if (WHAT == 1) return;
    if (WHAT == 2) {
        if (in_layer<MASK>(s, q)) e1_back<T, MASK, true>(s, J2, q);
        else e1_back<T, MASK, false>(s, J2, q);
        return;
    }
    if (warp_in_layer<MASK>(s, q)) e1_update<T, MASK, true>(s, J2, q);
    else e1_update<T, MASK, false>(s, J2, q);
}

// The first E half-step of a run that starts at integer time, in place, with the J
// of the present state (the same increments as the step's own half-steps).
template <typename T, int MASK, int EM, int BM, bool IN>
__device__ __forceinline__ void e_half_pass(const Stage<T> &s, const Cell &q)
{
    const Layer<T, IN> L = layer_at<MASK, IN>(s, q);
    const T *const B1[3] = {s.Bin[3], s.Bin[4], s.Bin[5]};
#pragma unroll
    for (int a = 0; a < 3; a++) {
        if (EM >> a & 1) {
            T hX = curl_h<MASK, BM, false>(s, s.Bin, a, q);
            if (a > 0 && q.x[0] == s.src_x) hX = fma(s.src_w[a - 1][q.x[1] + s.n[1] * q.x[2]], s.src_e, hX);
            if (s.jp[0][a]) hX = fma(-s.h, s.jp[0][a][q.c], hX);
            T *E = const_cast<T *>(s.Ein[a]);
            E[q.c] = L.half_step(E[q.c], hX);
        }
        T hX = fma(-s.hg2, T(2) * s.J[a][q.c], curl_h<MASK, 7, false>(s, B1, a, q));
        if (s.jp[1][a]) hX = fma(-s.h, s.jp[1][a][q.c], hX);
        T *E = const_cast<T *>(s.Ein[3 + a]);
        E[q.c] = L.half_step(E[q.c], hX);
    }
}
template <typename T, int MASK, int EM, int BM>
__global__ void __launch_bounds__(kThreads) k_stage_e_half(Stage<T> s)
{
    Cell q;
    const bool mine = cell_at<MASK>(s, q);
    wait_for_previous_pass();
    if (!mine) return;
    if (warp_in_layer<MASK>(s, q)) e_half_pass<T, MASK, EM, BM, true>(s, q);
    else e_half_pass<T, MASK, EM, BM, false>(s, q);
}

template <typename T>
Stage<T> make_stage(axp_grid *g)
{
    Stage<T> s;
    const axp_grid_desc &d = g->desc;
    const Workspace &w = g->layout;
    const int in = g->fset, out = 1 - g->fset;
    auto at = [&](size_t off) { return (T *)(g->ws + off); };
    for (int q = 0; q < 6; q++) {
        const int fe = q < 3 ? kE0 + q : kE1 + (q - 3), fb = q < 3 ? kB0 + q : kB1 + (q - 3);
        s.Ein[q] = at(w.off_fields[in][fe]);
        s.Bin[q] = at(w.off_fields[in][fb]);
        s.Eout[q] = at(w.off_fields[out][fe]);
        s.Bout[q] = at(w.off_fields[out][fb]);
    }
    s.phi = at(w.off_phi[g->phi_cur_slot]);
    s.phib = at(w.off_phi[g->phi_b_slot]);
    s.phi_out = at(w.off_phi[g->phi_next_slot]);
    s.phib_out = sizeof(T) == 4 ? at(w.off_phi[g->phi_next_b_slot]) : nullptr;
    const double h = d.dt / 2.0;
    for (int a = 0; a < 3; a++) {
        s.Bh[a] = s.P[a] = at(w.off_P[a]);
        s.Eh[a] = s.J[a] = at(w.off_J[a]);
        for (int o = 0; o < 2; o++)
            s.jp[o][a] = g->parts && sizeof(T) == sizeof(double) ? (const T *)g->parts->j[o][a] : nullptr;
        bool layer = false;
        for (int e = 0; e < 2; e++) {
            const size_t *lev = w.off_ghost[a][e];
            const bool of = d.axion_bc[a][e] == AXP_BC_OUTFLOW;
            s.gh[a][e] = of ? at(lev[g->ghost_level_slot[0]]) : nullptr;
            s.gh_old[a][e] = of ? at(lev[g->ghost_level_slot[1]]) : nullptr;
            s.gh_new[a][e] = of ? at(lev[g->ghost_level_slot[2]]) : nullptr;
            s.gh_hi[a][e] = s.gh_new[a][e];
            s.axbc[a][e] = d.axion_bc[a][e];
            const bool pml = (d.em_bc[a][e] == AXP_BC_PML || d.axion_bc[a][e] == AXP_BC_PML) && d.pml_sigma_max_dt > 0;
            s.lay[a][e] = pml ? (int)std::min<int64_t>(d.pml_cells, d.n[a]) : 0;
            if (s.lay[a][e] > 0) layer = true;
        }
        s.tab[a] = layer ? at(w.off_pml_tab[a]) : nullptr;
        s.of_r[a] = (T)(d.dt / d.d[a]);
        s.sig_ax[a] = at(w.off_sig_ax[a]);
        s.n[a] = (int)d.n[a];
        s.per[a] = d.em_bc[a][0] == AXP_BC_PERIODIC;
        s.hd[a] = (T)(h / d.d[a]);
        s.lap_c[a] = d.n[a] > 1 ? (T)(d.dt * d.dt / (d.d[a] * d.d[a])) : T(0);
        s.q4d[a] = (T)(0.25 / d.d[a]);
        s.Bext[a] = (T)g->B_ext[a];
        s.Eext[a] = (T)g->E_ext[a];
    }
    s.N = (int)(d.n[0] * d.n[1] * d.n[2]);
    s.h = (T)h;
    s.inv_h = (T)(1.0 / h);
    s.hg2 = (T)(0.5 * h * d.g);
    s.dt2g = (T)(d.dt * d.dt * d.g);
    s.m2dt2 = (T)(d.dt * d.dt * d.m * d.m);
    s.uniform_e = g->E_ext[0] != 0.0 || g->E_ext[1] != 0.0 || g->E_ext[2] != 0.0;
    s.dt = (T)d.dt;
    s.dt2 = (T)(d.dt * d.dt);
    s.inv_dt2 = (T)(1.0 / (d.dt * d.dt));
    s.inv_dt = (T)(1.0 / d.dt);
    s.src_x = -1;
    s.src_w[0] = at(w.off_src[0]);
    s.src_w[1] = at(w.off_src[1]);
    s.src_e = s.src_b = T(0);
    if (g->src_on) s.src_x = (int)g->src.plane;
    s.last = 0;
    return s;
}

// Launches of one configuration: active axes MASK, order-0 components EM and BM.
template <typename T, int MASK, int EM, int BM>
struct Passes {
    static constexpr int kE = EM;
    static int blocks(const Stage<T> &s) { return (s.N + kThreads - 1) / kThreads; }
    static void b(const Stage<T> &s, int mode, cudaStream_t st)
    {
        if (mode == 0) launch_pass(k_stage_b<T, MASK, EM, BM, 0>, blocks(s), st, s);
        else if (mode == 1) launch_pass(k_stage_b<T, MASK, EM, BM, 1>, blocks(s), st, s);
        else launch_pass(k_stage_b<T, MASK, EM, BM, 2>, blocks(s), st, s);
    }
    // part 1: the axion, 2: E0, 3: both
    static void phi(const Stage<T> &s, T *const bs[3], int part, cudaStream_t st)
    {
        if (part == 3) launch_pass(k_stage_phi<T, MASK, EM, BM, true, true>, blocks(s), st, s, bs[0], bs[1], bs[2]);
        else if (part == 1) launch_pass(k_stage_phi<T, MASK, EM, BM, true, false>, blocks(s), st, s, bs[0], bs[1], bs[2]);
        else launch_pass(k_stage_phi<T, MASK, EM, BM, false, true>, blocks(s), st, s, bs[0], bs[1], bs[2]);
    }
    static void p(const Stage<T> &s, const T *const e[3], const T *const b[3], const T *hi, const T *lo, cudaStream_t st)
    {
        launch_pass(k_stage_p<T, MASK, EM, BM>, blocks(s), st, s, e[0], e[1], e[2], b[0], b[1], b[2], hi, lo);
    }
    static void j(const Stage<T> &s, const View<T> &v, const PhiPair<T, sizeof(T) == 4> &pq, int what, cudaStream_t st)
    {
        if (what == 0) launch_pass(k_stage_j<T, MASK, 0>, blocks(s), st, s, v, pq);
        else if (what == 1) launch_pass(k_stage_j<T, MASK, 1>, blocks(s), st, s, v, pq);
        else launch_pass(k_stage_j<T, MASK, 2>, blocks(s), st, s, v, pq);
    }
    static void e0_back(const Stage<T> &s, cudaStream_t st)
    {
        if (EM) launch_pass(k_stage_e0_back<T, MASK, EM, BM>, blocks(s), st, s);
    }
    static void e_half(const Stage<T> &s, cudaStream_t st)
    {
        launch_pass(k_stage_e_half<T, MASK, EM, BM>, blocks(s), st, s);
    }
};

// Ghost planes of an axion level as the boundary-aware accessors take them.
template <typename T>
Ghosts<T> ghost_planes(axp_grid *g, int level)
{
    Ghosts<T> G;
    for (int a = 0; a < 3; a++)
        for (int e = 0; e < 2; e++) {
            const size_t off = g->layout.off_ghost[a][e][g->ghost_level_slot[level]];
            G.p[a][e] = off ? (T *)(g->ws + off) : nullptr;
        }
    return G;
}

// P and J of the state around integer time n (E0^n in e, the axion levels n+1/2 and
// n-1/2), and what the J pass does with them
template <typename T, typename Q>
void current_at_n(axp_grid *g, Stage<T> s, const T *const e[3], int what)
{
    for (int a = 0; a < 3; a++)
        for (int f = 0; f < 2; f++) {
            s.gh_hi[a][f] = s.gh[a][f];
            s.gh[a][f] = s.gh_old[a][f];
        }
    View<T> v = make_view<T>(g);
    for (int a = 0; a < 3; a++) v.f[kE0 + a] = const_cast<T *>(e[a]);
    const T *const b[3] = {s.Bin[0], s.Bin[1], s.Bin[2]};
    Q::p(s, e, b, s.phi, s.phib, g->stream);
    PhiPair<T, sizeof(T) == 4> pq{s.phi, s.phib, ghost_planes<T>(g, 0), ghost_planes<T>(g, 1)};
    Q::j(s, v, pq, what, g->stream);
    g->launches += 2;
}

// E^n -> E^{n+1/2} in place
template <typename T, typename Q>
void first_half(axp_grid *g)
{
    Stage<T> s = make_stage<T>(g);
    if (!g->J_valid) current_at_n<T, Q>(g, s, s.Ein, 1);
    if (g->src_on) s.src_e = (T)(g->desc.dt / 2.0 * source_wave(g, source_x_b(g), time_n(g, g->step)));
    Q::e_half(s, g->stream);
    g->launches++;
}

// E^{n+1/2} -> E^n into field set `oset`
template <typename T, typename Q>
void back_half(axp_grid *g, int oset)
{
    Stage<T> s = make_stage<T>(g);
    for (int f = 0; f < 6; f++) s.Eout[f] = (T *)(g->ws + g->layout.off_fields[oset][f < 3 ? kE0 + f : kE1 + f - 3]);
    if (g->src_on) s.src_e = (T)(g->desc.dt / 2.0 * source_wave(g, source_x_b(g), time_n(g, g->step)));
    Q::e0_back(s, g->stream);
    if (Q::kE) g->launches++;
    const T *const e[3] = {s.Eout[0], s.Eout[1], s.Eout[2]};
    current_at_n<T, Q>(g, s, e, 2);
}

template <typename T, typename Q>
cudaError_t run_staged(axp_grid *g, int64_t nsteps)
{
    const axp_grid_desc &d = g->desc;
    const bool stag = g->staggered;  // the single-pass kernels' state: E stays half a step ahead
    const bool parts = g->parts != nullptr;
    bool ahead = stag;  // E at n+1/2
    cudaError_t e = cudaSuccess;
    for (int64_t it = 0; it < nsteps; it++) {
        const bool record = d.diag_every > 0 && (g->step + 1) % d.diag_every == 0;
        if (!ahead) {
            first_half<T, Q>(g);
            ahead = true;
        }
        Stage<T> s = make_stage<T>(g);
        s.last = !stag && (it + 1 == nsteps || record);
        if (g->src_on) {
            s.src_b = (T)(d.dt / 2.0 * source_wave(g, source_x_e(g), time_half(g, g->step)));
            s.src_e = (T)(d.dt / 2.0 * source_wave(g, source_x_b(g), time_n(g, g->step + 1)));
        }
        if constexpr (sizeof(T) == sizeof(double)) {
            if (parts) {
                Q::b(s, 1, g->stream);
                View<double> v = make_view<double>(g);
                for (int a = 0; a < 3; a++) {
                    v.f[kB0 + a] = s.Bout[a];
                    v.f[kB1 + a] = s.Bout[3 + a];
                }
                if ((e = particles_push(g, v)) != cudaSuccess) return e;
                Q::phi(s, s.Bout, 1, g->stream);
                Stage<double> s2 = s;
                for (int f = 0; f < 6; f++) s2.Bin[f] = s.Bout[f];
                Q::b(s2, 2, g->stream);
                Q::phi(s, s.Bh, 2, g->stream);
                g->launches += 4;
            }
        }
        if (!parts) {
            Q::b(s, 0, g->stream);
            Q::phi(s, s.Bh, 3, g->stream);
            g->launches += 2;
        }
        const T *hi = s.phi_out, *lo = sizeof(T) == 4 ? s.phib_out : s.phi;
        const T *const b[3] = {s.Bout[0], s.Bout[1], s.Bout[2]};
        const T *eh[3];
        View<T> v = make_view<T>(g);
        for (int a = 0; a < 3; a++) {
            eh[a] = (Q::kE >> a & 1) ? s.Eh[a] : s.Eout[a];  // (an inactive array is zero in both sets)
            v.f[kE0 + a] = const_cast<T *>(eh[a]);
            v.f[kB0 + a] = s.Bout[a];
        }
        if (s.last) {  // E0^{n+1} lies in the output set too, and J takes the scratch
            for (int a = 0; a < 3; a++) {
                eh[a] = s.Eout[a];
                v.f[kE0 + a] = s.Eout[a];
            }
        }
        Q::p(s, eh, b, hi, lo, g->stream);
        PhiPair<T, sizeof(T) == 4> pq{hi, lo, ghost_planes<T>(g, 2), ghost_planes<T>(g, 0)};
        Q::j(s, v, pq, 0, g->stream);
        g->launches += 2;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        rotate_roles(g);
        const int s0 = g->ghost_level_slot[0], s1 = g->ghost_level_slot[1], s2 = g->ghost_level_slot[2];
        g->ghost_level_slot[0] = s2;
        g->ghost_level_slot[1] = s0;
        g->ghost_level_slot[2] = s1;
        g->step++;
        g->J_valid = s.last != 0;
        ahead = !s.last;
        if (stag) {
            g->half_prev = true;  // the other set holds the last step's E^{n-1/2}
            g->half_prev_cfg = g->cfg_version;
        }
        if (record) {
            if ((e = diag_compute<T>(g, ring_slot(g, g->ring_written))) != cudaSuccess) return e;
            g->ring_written++;
        }
    }
    return cudaGetLastError();
}

// f(Passes of the grid's active axes and the order-0 components m)
template <typename T, typename F>
auto with_passes(const axp_grid *g, uint32_t m, F &&f)
{
    const int64_t *n = g->desc.n;
    auto in = [&](uint32_t set) { return (m & ~set) == 0; };
    const uint32_t tm = 4u | (3u << 3), te = 3u | (4u << 3);  // (E0z; B0x, B0y) and (E0x, E0y; B0z)
    if (n[1] == 1 && n[2] == 1) {
        if (m == 0) return f(Passes<T, 1, 0, 0>{});
        if (in(tm)) return f(Passes<T, 1, 4, 3>{});
        if (in(te)) return f(Passes<T, 1, 3, 4>{});
        return f(Passes<T, 1, 7, 7>{});
    }
    if (n[2] == 1) {
        if (m == 0) return f(Passes<T, 3, 0, 0>{});
        if (in(tm)) return f(Passes<T, 3, 4, 3>{});
        if (in(te)) return f(Passes<T, 3, 3, 4>{});
        return f(Passes<T, 3, 7, 7>{});
    }
    if (m == 0) return f(Passes<T, 7, 0, 0>{});
    return f(Passes<T, 7, 7, 7>{});
}

}  // namespace

// 32-bit cell indexes, and at least one active axis (a single cell keeps the general kernels)
bool staged_supported(const axp_grid *g)
{
    const int64_t *n = g->desc.n;
    return n[0] * n[1] * n[2] < ((int64_t)1 << 30) && n[0] > 1;
}

template <typename T>
cudaError_t staged_step(axp_grid *g, int64_t nsteps, uint32_t order0)
{
    return with_passes<T>(g, order0, [&](auto q) { return run_staged<T, decltype(q)>(g, nsteps); });
}

template <typename T>
cudaError_t staged_enter(axp_grid *g)
{
    with_passes<T>(g, order0_present(g), [&](auto q) { first_half<T, decltype(q)>(g); });
    return cudaGetLastError();
}

template <typename T>
cudaError_t staged_exit(axp_grid *g, int oset)
{
    with_passes<T>(g, order0_present(g), [&](auto q) { back_half<T, decltype(q)>(g, oset); });
    return cudaGetLastError();
}

template cudaError_t staged_step<double>(axp_grid *, int64_t, uint32_t);
template cudaError_t staged_step<float>(axp_grid *, int64_t, uint32_t);
template cudaError_t staged_enter<double>(axp_grid *);
template cudaError_t staged_enter<float>(axp_grid *);
template cudaError_t staged_exit<double>(axp_grid *, int);
template cudaError_t staged_exit<float>(axp_grid *, int);

}  // namespace axp
