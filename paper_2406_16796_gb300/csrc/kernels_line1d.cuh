// kernels_line1d.cuh -- time-blocked step for 1D grids (arXiv 2406.16796 Sec. 2.3; the
// 1D conversion workload): FP64 and FP32 split, periodic along x or with absorbing layers.
//
// A 1D grid of a few thousand cells is far too small to fill the GPU: launched
// one step at a time its steps cost launch and synchronisation latency, not
// arithmetic.  Here one cooperative launch (a plain one where no wait is met) runs a
// whole run of steps.  Each
// block owns `seg` consecutive cells and holds them, with `halo` cells on each
// side, in shared memory; it advances that window `tblock` steps on its own,
// writes its owned cells to the other buffer set and meets the other blocks at
// a grid-wide wait (bounded in polls and in time) before it reads its next
// window.  A step's dependency cone is one cell wide and the axion current
// widens it by two, so the owned cells stay exact while halo >= tblock + 2
// (kept at tblock + 3); outside the window the closure is zero.
//
// The state and the update are those of the single-pass kernels: E at n+1/2,
// B at n, phi at n+1/2 and n-1/2.  Along x only the y and z components curl;
// E_x of order 1 changes through the axion current alone, B_x and E0_x not at
// all.  Per step, one barrier after each stage:
//   1. B^{n+1/2}, B^{n+1} = B^n - h curl E^{n+1/2} (twice)
//   2. S^{n+1/2} = g Ebar0 . Bbar0 (E0^{n+1/2}, B0^{n+1/2}); phi^{n+3/2};
//      2 phi^{n+1}, dt D_t phi^{n+1}; E0^{n+1} = E0^{n+1/2} + h curl B0^{n+1}
//   3. P^{n+1} = (D_t phi) Bbar0 - Ebar0 x grad_c phi at cell centres
//   4. J^{n+1} (face average of P along x); E1^{n+3/2} = E1^{n+1/2}
//      + 2h (curl B1^{n+1} - g J^{n+1}); E0^{n+3/2} = 2 E0^{n+1} - E0^{n+1/2}
// with the averages of Sec. 2.3 reduced to 1D (a 4-point mean over cells that
// coincide along y and z is the 2-point mean along x).
//
// Absorbing layers (LAYER): windows that reach a layer or the grid's end take a body
// that asks each cell where it lies; a cell outside the layers takes the plain update's
// own operations, so its bits do not depend on the window it is computed in.  Cells
// beyond the grid hold zeros (the closure of E and B and the PML ghost of phi): their
// coefficients are zero.
//
// FP32 split holds phi^{n+1/2} and its increment, and takes the generic single-pass kernel's
// operations in their order (rounding differences of a few 1e-5 would come from any other
// over a few hundred steps): its bits where the cell size is a power of two (other sizes round
// 1/dx once more) and no damped quotient is below 1e-30.  Its step is bound by the barriers' latency (about 0.55 us), not by a pipe,
// so its windows are blocked over more steps (line_block).
//
// Measured, us per step (one launch per step before): 2048 cells with absorbing ends
// FP32 5.2 -> 1.3, FP64 16.8 -> 2.7; 4096 periodic FP32 2.9 -> 0.63;
// 65536 with absorbing ends FP32 7.0 -> 3.2, FP64 36 -> 11.0.  Periodic FP64 (blocked before too):
// 4096 cells 1.80 -> 1.71, 65536 10.9 -> 10.4 with three of 29 FP64 operations of the longer
// half taken out of a step (an FP64 instruction takes a warp 64 to 76 cycles, whatever its lanes).
#pragma once

#include "kernels_fused.cuh"

namespace axp {
namespace line1d {

// Four warps: each SM sub-partition has its own FP64 unit, which takes about 64
// cycles per warp instruction, so a warp issues at most a quarter of the SM's
// FP64 rate.  The window's cells are covered by two warps and each stage's work
// on a cell is split into two halves of independent outputs: warps 0-1 take one
// half and warps 2-3 (the other two sub-partitions) the other.
// FP32: eight warps, so that a pass covers 128 cells.
template <typename T>
__host__ __device__ constexpr int threads_of() { return sizeof(T) == 8 ? 128 : 256; }
template <typename T>
__host__ __device__ constexpr int lanes_of() { return threads_of<T>() / 2; }  // cells a pass of one half covers
constexpr int kArrays = 28;              // window arrays (listed in k_line1d)
constexpr int kLayerArrays = 7;          // and the layer's coefficients
// A window's largest shared memory: 1000 cells of a periodic FP64 grid (218.75 of the 227 KB a
// block may have), 789 cells with layers (their own arrays on top: 216 KB); twice that in FP32.
constexpr int kWindowBytes = 1000 * kArrays * (int)sizeof(double);
constexpr int kLayerWindow = 789;
static_assert(kLayerWindow * (kArrays + kLayerArrays) * (int)sizeof(double) <= kWindowBytes, "layered windows fit");
template <typename T>
__host__ __device__ constexpr int max_window(bool layer)
{
    return (layer ? kLayerWindow : 1000) * (int)(sizeof(double) / sizeof(T));
}
constexpr unsigned kSpinLimit = 1u << 26;        // polls of a grid-wide wait before it gives up ...
constexpr unsigned long long kWaitNs = 1000000000ull;  // ... or one second, whichever comes first

template <typename T>
struct Args {
    const T *E[2][6], *B[2][6];  // buffer sets: order-0 xyz, order-1 xyz (E^{n+1/2}, B^n)
    T *Ew[2][6], *Bw[2][6];      // the same arrays, written
    T *phi[2][2];                     // per set: phi^{n+1/2}; phi^{n-1/2} (FP64) or the increment
    int64_t n;                        // cells
    int64_t nsteps;
    int tblock, halo, seg;
    // step constants
    T cB;           // h/dx: one B or E0 half-step per difference
    T c2B;          // 2h/dx: the two half-steps of E1 (and of B1) per difference
    T h2g;          // 2hg (FP64: 2hg/dt): the current's term in E1's two half-steps
    T hgx;          // FP64: half of it, for the face sum of P_x
    // FP64: phi^{n+3/2} = lap_0 phi + lap_c (phi+ + phi-) - phi^{n-1/2} + dt2g S/g;
    // FP32: the increment grows by lap_0 phi + lap_c (second difference) + dt2g S/g
    T lap_0, lap_c, dt2g;
    T inv_dt, q4dx;        // 1/dt; dt/(4 dx) for dt times the central gradient of 2 phi^{n+1}
    T Bext[3];
    // absorbing layers: their cells at either end, the coefficient tables of the grid
    // (a, b, a^2, b (1 + a), c1, c2: n each), sigma of the axion, 1/h, 1/dt^2, dt
    int lay[2];
    const T *tab, *sig, *sig_em;
    T inv_h, inv_dt2, dt;
    T h, idx, hidx, idx2, g, m2, dt2;  // FP32: h, 1/dx, 1/(2 dx), 1/dx^2, g, m^2, dt^2
    unsigned *ctr;  // grid-wait arrivals (zeroed before the launch)
    int *err;       // 1 once a wait gave up
    T *En[5];  // E at the integer time the launch ends at: E0 y z, E1 x y z
    int absent;     // failure-detection test: this block leaves before its first wait (-1: none)
};

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Grid-wide wait on an arrival counter, bounded: after kSpinLimit polls, a
// second, or once another block has given up, it records the failure and
// returns false.
__device__ __forceinline__ bool grid_wait(unsigned *ctr, unsigned target, int *err)
{
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(ctr, 1u);
        ok = 1;
        unsigned spins = 0;
        const unsigned long long t0 = global_ns();
        while (*(volatile unsigned *)ctr < target) {
            if (++spins > kSpinLimit || *(volatile int *)err || global_ns() - t0 > kWaitNs) {
                atomicExch(err, 1);
                ok = 0;
                break;
            }
            __nanosleep(64);
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

template <typename T, bool LAYER>
__global__ void __launch_bounds__(threads_of<T>()) k_line1d(Args<T> A)
{
    // (a plain launch may be set up while the kernel before it ends, and waits here for that
    // kernel's memory)
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    constexpr bool INCR = sizeof(T) == 4;
    constexpr int LANES = lanes_of<T>();
    extern __shared__ __align__(16) unsigned char l1_raw[];
    T *l1_sm = reinterpret_cast<T *>(l1_raw);
    const int64_t N = A.n;
    const int64_t s0 = (int64_t)blockIdx.x * A.seg;
    const int own = (int)(min(N, s0 + A.seg) - s0);
    const int H = A.halo, W = own + 2 * H, Wm = A.seg + 2 * A.halo;
    const int tid = threadIdx.x, nt = blockDim.x;
    // window arrays: E (6), B (6), phi^{n+1/2}, phi^{n-1/2} (FP32: the next phi), B0^{n+1/2}
    // y z, E0^{n+1} y z, 2 phi^{n+1}, dt D_t phi^{n+1}, P (3), Bbar0^{n+1} y z (with B_ext),
    // two values that stay fixed over a window's steps (E0x and B0x do not change in 1D, no
    // curl along x: Bbar0_x = B0x + B_ext,x and the source's term Ebar0_x Bbar0_x), and
    // FP32's increment (FP64: phi+ + phi- for the next step).  FP64 holds dt P: D_t phi and the
    // gradient then take no product of their own
    auto arr = [&](int q) { return l1_sm + (size_t)q * Wm; };
    T *E[6], *B[6];
    for (int q = 0; q < 6; q++) {
        E[q] = arr(q);
        B[q] = arr(6 + q);
    }
    T *cur = arr(12), *old = arr(13), *Bhy = arr(14), *Bhz = arr(15), *Eny = arr(16), *Enz = arr(17);
    T *SM = arr(18), *DF = arr(19), *Px = arr(20), *PY = arr(21), *PZ = arr(22), *BY = arr(23), *BZ = arr(24);
    T *BXT = arr(25), *SX = arr(26), *inc = INCR ? arr(27) : arr(13), *SP = arr(27);
    // the layer's a, r = b/h, and for the axion 1/(1 + sigma dt), (1 - sigma dt)/(1 + sigma dt), (sigma dt)^2
    T *La = arr(28), *Lr = arr(29), *Lc1 = arr(30), *Lc2 = arr(31), *Lss = arr(32);
    // FP32: La 1 - sigma h/2 (of either sign: sigma h may exceed 2), Ld and Lr the divisor
    // 1 + sigma h/2 and its reciprocal (0 beyond the grid, which marks those cells); for the axion Lc2 1 - sigma dt, Le and Lc1 the divisor 1 + sigma dt and its
    // reciprocal, Lss sigma^2
    T *Ld = arr(33), *Le = arr(34);
    const int half = tid / LANES, lane = tid % LANES;  // (a warp-uniform half)
    // values beyond the window's ends: the zero closure
    auto at = [&](const T *a, int w) { return (w >= 0 && w < W) ? a[w] : T(0); };
    const T Bx = A.Bext[0], By = A.Bext[1], Bz = A.Bext[2];
    // window cells [wl, wh) lie in the grid outside the layers
    const int64_t wl = LAYER ? A.lay[0] - (s0 - H) : 0, wh = LAYER ? N - A.lay[1] - (s0 - H) : W;
    const bool layered = LAYER && (wl > 0 || wh < W);  // this window's body
    auto in_layer = [&](int w) { return LAYER && layered && (w < wl || w >= wh); };
    if (LAYER && layered) {
        for (int w = tid; w < W; w += nt) {
            const int64_t gi = s0 - H + w;
            const bool in = gi >= 0 && gi < N;
            if (INCR) {
                const T se = in ? A.sig_em[gi] : T(0), sa = in ? A.sig[gi] : T(0);
                La[w] = T(1) - se * A.h / T(2);
                Ld[w] = in ? T(1) + se * A.h / T(2) : T(0);
                Lr[w] = in ? T(1) / Ld[w] : T(0);
                Lc2[w] = T(1) - sa * A.dt;
                Le[w] = T(1) + sa * A.dt;
                Lc1[w] = T(1) / Le[w];
                Lss[w] = sa * sa;
                // the stages pass over the cells beyond the grid: what neighbours read there is 0
                if (!in) old[w] = Bhy[w] = Bhz[w] = SM[w] = DF[w] = T(0);
                continue;
            }
            La[w] = in ? A.tab[gi] : T(0);
            Lr[w] = in ? A.tab[N + gi] * A.inv_h : T(0);
            Lc1[w] = in ? A.tab[4 * N + gi] * A.inv_dt2 : T(0);
            Lc2[w] = in ? A.tab[5 * N + gi] : T(0);
            const T sd = in ? A.sig[gi] * A.dt : T(0);
            Lss[w] = sd * sd;
        }
    }

    int par = 0;
    unsigned waits = 0;
    // E1^{n+1} of a damped cell at the launch's last step, for a record: taken between the two
    // half-steps (undoing the second would divide by 1 - sigma h/2, which may be zero)
    auto keep = [&](int q, int w, T v) {
        if (w >= H && w < H + own) A.En[q][s0 + (w - H)] = v;
    };
    for (int64_t done = 0; done < A.nsteps; done += A.tblock) {
        const int steps = (int)min((int64_t)A.tblock, A.nsteps - done);
        const int last = done + steps >= A.nsteps ? steps - 1 : -1;  // the launch's last step
        for (int w = tid; w < W; w += nt) {
            int64_t gi = s0 - H + w;
            const bool in = !LAYER || (gi >= 0 && gi < N);
            if (!LAYER) {
                gi %= N;
                if (gi < 0) gi += N;
            }
#pragma unroll
            for (int q = 0; q < 6; q++) {
                E[q][w] = in ? A.E[par][q][gi] : T(0);
                B[q][w] = in ? A.B[par][q][gi] : T(0);
            }
            cur[w] = in ? A.phi[par][0][gi] : T(0);
            inc[w] = in ? A.phi[par][1][gi] : T(0);
        }
        __syncthreads();
        for (int w = tid; w < W; w += nt) {
            const T ex = T(0.5) * (E[0][w] + at(E[0], w - 1));
            const T bx = B[0][w] + Bx;
            BXT[w] = bx;
            SX[w] = ex * bx;
            if (!INCR) SP[w] = at(cur, w + 1) + at(cur, w - 1);
        }
        __syncthreads();
        for (int st = 0; st < (INCR ? 0 : steps); st++) {
            const bool fin = LAYER && st == last;
            // 1. B^{n+1/2} and B^{n+1}: (curl E)_y = -D_x E_z, (curl E)_z = D_x E_y (forward)
            for (int w = lane; w < W; w += LANES) {
                if (half == 0) {
                    const T d0z = at(E[2], w + 1) - E[2][w], d1z = at(E[5], w + 1) - E[5][w];
                    if (in_layer(w)) {
                        const T a = La[w], x0 = Lr[w] * (A.cB * d0z), x1 = Lr[w] * (A.cB * d1z);
                        const T hy = fma(a, B[1][w], x0);
                        Bhy[w] = hy;
                        B[1][w] = fma(a, hy, x0);
                        B[4][w] = fma(a, fma(a, B[4][w], x1), x1);
                        B[3][w] = a * (a * B[3][w]);
                    } else {
                        const T hy = fma(A.cB, d0z, B[1][w]);
                        Bhy[w] = hy;
                        B[1][w] = fma(A.cB, d0z, hy);
                        B[4][w] = fma(A.c2B, d1z, B[4][w]);
                    }
                } else {
                    const T d0y = at(E[1], w + 1) - E[1][w], d1y = at(E[4], w + 1) - E[4][w];
                    if (in_layer(w)) {
                        const T a = La[w], x0 = Lr[w] * (-A.cB * d0y), x1 = Lr[w] * (-A.cB * d1y);
                        const T hz = fma(a, B[2][w], x0);
                        Bhz[w] = hz;
                        B[2][w] = fma(a, hz, x0);
                        B[5][w] = fma(a, fma(a, B[5][w], x1), x1);
                    } else {
                        const T hz = fma(-A.cB, d0y, B[2][w]);
                        Bhz[w] = hz;
                        B[2][w] = fma(-A.cB, d0y, hz);
                        B[5][w] = fma(-A.c2B, d1y, B[5][w]);
                    }
                }
            }
            __syncthreads();
            // 2. source, phi^{n+3/2}, 2 phi^{n+1}, dt D_t phi^{n+1} | E0^{n+1}, Bbar0^{n+1} y z
            for (int w = lane; w < W; w += LANES) {
                if (half == 0) {
                    const T by = fma(T(0.5), Bhy[w] + at(Bhy, w - 1), By);
                    const T bz = fma(T(0.5), Bhz[w] + at(Bhz, w - 1), Bz);
                    const T S = fma(E[2][w], bz, fma(E[1][w], by, SX[w]));  // S/g
                    const T ph = cur[w];
                    {
                        T nw;
                        if (in_layer(w)) {
                            nw = A.lap_0 * ph;
                            nw = fma(A.lap_c, SP[w], nw);
                            nw = fma(A.dt2g, S, nw);
                            nw = fma(-Lc2[w], old[w], Lc1[w] * fma(-Lss[w], ph, nw));
                        } else {
                            nw = fma(A.lap_0, ph, -old[w]);
                            nw = fma(A.lap_c, SP[w], nw);
                            nw = fma(A.dt2g, S, nw);
                        }
                        old[w] = nw;  // phi^{n+3/2} over phi^{n-1/2} (read by this cell only)
                        SM[w] = nw + ph;
                        DF[w] = nw - ph;
                    }
                } else {
                    // (curl B0)_y = -D_x B0z, (curl B0)_z = D_x B0y (backward)
                    const T dz = B[2][w] - at(B[2], w - 1), dy = B[1][w] - at(B[1], w - 1);
                    if (in_layer(w)) {
                        Eny[w] = fma(La[w], E[1][w], Lr[w] * (-A.cB * dz));
                        Enz[w] = fma(La[w], E[2][w], Lr[w] * (A.cB * dy));
                    } else {
                        Eny[w] = fma(-A.cB, dz, E[1][w]);
                        Enz[w] = fma(A.cB, dy, E[2][w]);
                    }
                    BY[w] = fma(T(0.5), B[1][w] + at(B[1], w - 1), By);
                    BZ[w] = fma(T(0.5), B[2][w] + at(B[2], w - 1), Bz);
                }
            }
            __syncthreads();
            // 3. dt P^{n+1} at the cell centres
            for (int w = lane; w < W; w += LANES) {
                const T Dt = DF[w];
                const T dphi = (at(SM, w + 1) - at(SM, w - 1)) * A.q4dx;
                if (half == 0) {
                    PY[w] = fma(-Enz[w], dphi, Dt * BY[w]);
                    SP[w] = at(old, w + 1) + at(old, w - 1);  // of phi^{n+3/2}
                } else {
                    Px[w] = Dt * BXT[w];
                    PZ[w] = fma(Eny[w], dphi, Dt * BZ[w]);
                }
            }
            __syncthreads();
            // 4. J^{n+1}; E1^{n+3/2}; E0^{n+3/2}
            for (int w = lane; w < W; w += LANES) {
                if (half == 0) {
                    const T Jx = Px[w] + at(Px, w + 1), dz = B[5][w] - at(B[5], w - 1);
                    if (in_layer(w)) {
                        // two half-steps: a^2 E + (1 + a) r h X
                        const T a = La[w], r2 = T(0.5) * Lr[w];
                        const T xx = r2 * (-A.hgx * Jx), xy = r2 * fma(-A.c2B, dz, -A.h2g * PY[w]);
                        const T mx = fma(a, E[3][w], xx), my = fma(a, E[4][w], xy);
                        E[3][w] = fma(a, mx, xx);
                        E[4][w] = fma(a, my, xy);
                        if (fin) {
                            keep(2, w, mx);
                            keep(3, w, my);
                        }
                    } else {
                        E[3][w] = fma(-A.hgx, Jx, E[3][w]);
                        E[4][w] = fma(-A.c2B, dz, fma(-A.h2g, PY[w], E[4][w]));
                    }
                } else {
                    const T dy = B[4][w] - at(B[4], w - 1);
                    if (in_layer(w)) {
                        const T a = La[w], xz = T(0.5) * Lr[w] * fma(A.c2B, dy, -A.h2g * PZ[w]);
                        const T mz = fma(a, E[5][w], xz);
                        E[5][w] = fma(a, mz, xz);
                        if (fin) keep(4, w, mz);
                        E[1][w] = fma(T(1) + a, Eny[w], -a * E[1][w]);
                        E[2][w] = fma(T(1) + a, Enz[w], -a * E[2][w]);
                    } else {
                        E[5][w] = fma(A.c2B, dy, fma(-A.h2g, PZ[w], E[5][w]));
                        E[1][w] = fma(T(2), Eny[w], -E[1][w]);
                        E[2][w] = fma(T(2), Enz[w], -E[2][w]);
                    }
                }
            }
            T *t = cur;
            cur = old;
            old = t;
            inc = old;
            __syncthreads();
        }
        // FP32 split.  One half-step, damped in a layer.  x / d as the correctly rounded quotient
        // from the correctly rounded reciprocal r of d (Markstein's theorem: q = x r, then
        // q + (x - q d) r): the plain division of every damped cell and stage doubled the step
        // of a grid with absorbing ends (2.2 us against 1.3).
        // Below about 1e-30 the residual underflows and the quotient's last bit may differ: dividing
        // there costs 9% of a pulse's whole call, whose far tails are that small.
        auto over = [](T x, T d, T r) {
            const T q = x * r;
            return fma(fma(-q, d, x), r, q);
        };
        // (which product of the damped form is rounded is the generic kernel's choice, for its bits)
        auto half_b = [&](T F, T X, bool lay, int w) {
            return lay ? over(fma(La[w], F, A.h * X), Ld[w], Lr[w]) : fma(A.h, X, F);
        };
        auto half_e = [&](T F, T X, bool lay, int w) {
            return lay ? over(fma(A.h, X, La[w] * F), Ld[w], Lr[w]) : fma(A.h, X, F);
        };
        for (int st = 0; st < (INCR ? steps : 0); st++) {
            const bool fin = LAYER && st == last;
            for (int w = lane; w < W; w += LANES) {
                bool lay = in_layer(w);
                if (lay && Ld[w] == T(0)) continue;
                lay = lay && Ld[w] != T(1);
                if (half == 0) {
                    const T c0 = -((at(E[2], w + 1) - E[2][w]) * A.idx), c1 = -((at(E[5], w + 1) - E[5][w]) * A.idx);
                    const T hy = half_b(B[1][w], -c0, lay, w);
                    Bhy[w] = hy;
                    B[1][w] = half_b(hy, -c0, lay, w);
                    B[4][w] = half_b(half_b(B[4][w], -c1, lay, w), -c1, lay, w);
                    if (lay) B[3][w] = half_b(half_b(B[3][w], T(0), lay, w), T(0), lay, w);
                } else {
                    const T c0 = (at(E[1], w + 1) - E[1][w]) * A.idx, c1 = (at(E[4], w + 1) - E[4][w]) * A.idx;
                    const T hz = half_b(B[2][w], -c0, lay, w);
                    Bhz[w] = hz;
                    B[2][w] = half_b(hz, -c0, lay, w);
                    B[5][w] = half_b(half_b(B[5][w], -c1, lay, w), -c1, lay, w);
                }
            }
            __syncthreads();
            for (int w = lane; w < W; w += LANES) {
                bool lay = in_layer(w);
                const bool dead = lay && Ld[w] == T(0);
                if (half == 0) {
                    if (dead) continue;
                    const T by = fma(T(0.5), Bhy[w] + at(Bhy, w - 1), By);
                    const T bz = fma(T(0.5), Bhz[w] + at(Bhz, w - 1), Bz);
                    const T S = fma(E[2][w], bz, fma(E[1][w], by, SX[w]));  // S/g
                    const T ph = cur[w], pb = inc[w];
                    const T sp = (at(cur, w + 1) - ph) + (at(cur, w - 1) - ph);
                    T pin;
                    if (!lay || Lss[w] == T(0)) {
                        pin = fma(A.dt2g, S, fma(A.lap_c, sp, fma(A.lap_0, ph, pb)));
                    } else {
                        const T Y = fma(-Lss[w], ph, fma(A.g, S, -(A.m2 * ph)) + sp * A.idx2);
                        pin = over(fma(A.dt2, Y, Lc2[w] * pb), Le[w], Lc1[w]);
                    }
                    inc[w] = pin;
                    old[w] = ph + pin;
                    SM[w] = fma(T(0.5), pin, ph);  // phi^{n+1}
                    DF[w] = pin * A.inv_dt;
                } else {
                    lay = lay && Ld[w] != T(1);
                    const T cy = -((B[2][w] - at(B[2], w - 1)) * A.idx), cz = (B[1][w] - at(B[1], w - 1)) * A.idx;
                    Eny[w] = dead ? T(0) : half_e(E[1][w], cy, lay, w);
                    Enz[w] = dead ? T(0) : half_e(E[2][w], cz, lay, w);
                    BY[w] = fma(T(0.5), B[1][w] + at(B[1], w - 1), By);
                    BZ[w] = fma(T(0.5), B[2][w] + at(B[2], w - 1), Bz);
                }
            }
            __syncthreads();
            for (int w = lane; w < W; w += LANES) {
                const T Dt = DF[w], dphi = (at(SM, w + 1) - at(SM, w - 1)) * A.hidx;
                if (half == 0) {
                    PY[w] = fma(-Enz[w], dphi, Dt * BY[w]);
                } else {
                    Px[w] = Dt * BXT[w];
                    PZ[w] = fma(Eny[w], dphi, Dt * BZ[w]);
                }
            }
            __syncthreads();
            for (int w = lane; w < W; w += LANES) {
                bool lay = in_layer(w);
                if (lay && Ld[w] == T(0)) continue;
                lay = lay && Ld[w] != T(1);
                if (half == 0) {
                    const T X = -A.g * (T(0.5) * (Px[w] + at(Px, w + 1)));
                    const T Y = fma(-A.g, PY[w], -((B[5][w] - at(B[5], w - 1)) * A.idx));
                    const T mx = half_e(E[3][w], X, lay, w), my = half_e(E[4][w], Y, lay, w);
                    E[3][w] = half_e(mx, X, lay, w);
                    E[4][w] = half_e(my, Y, lay, w);
                    if (lay && fin) {
                        keep(2, w, mx);
                        keep(3, w, my);
                    }
                } else {
                    const T Z = fma(-A.g, PZ[w], (B[4][w] - at(B[4], w - 1)) * A.idx);
                    const T mz = half_e(E[5][w], Z, lay, w);
                    E[5][w] = half_e(mz, Z, lay, w);
                    if (lay && fin) keep(4, w, mz);
                    E[1][w] = half_e(Eny[w], -((B[2][w] - at(B[2], w - 1)) * A.idx), lay, w);
                    E[2][w] = half_e(Enz[w], (B[1][w] - at(B[1], w - 1)) * A.idx, lay, w);
                }
            }
            T *t = cur;
            cur = old;
            old = t;
            __syncthreads();
        }
        for (int w = H + tid; w < H + own; w += nt) {
            const int64_t gi = s0 + (w - H);
#pragma unroll
            for (int q = 0; q < 6; q++) {
                A.Ew[1 - par][q][gi] = E[q][w];
                A.Bw[1 - par][q][gi] = B[q][w];
            }
            A.phi[1 - par][0][gi] = cur[w];
            A.phi[1 - par][1][gi] = inc[w];
            if (done + A.tblock >= A.nsteps) {
                // E^{n+1} of the last step, for a record taken here: E0 as the step formed it,
                // E1 less the second of its two half-steps (a damped cell's: kept above)
                A.En[0][gi] = Eny[w];
                A.En[1][gi] = Enz[w];
                if constexpr (LAYER)
                    if (in_layer(w) && !(INCR && Ld[w] == T(1))) continue;
                const T Jx = T(0.5) * (Px[w] + at(Px, w + 1));
                const T hx = T(-0.5) * A.h2g * Jx, hy = fma(-A.cB, B[5][w] - at(B[5], w - 1), T(-0.5) * A.h2g * PY[w]);
                const T hz = fma(A.cB, B[4][w] - at(B[4], w - 1), T(-0.5) * A.h2g * PZ[w]);
                A.En[2][gi] = E[3][w] - hx;
                A.En[3][gi] = E[4][w] - hy;
                A.En[4][gi] = E[5][w] - hz;
            }
        }
        par ^= 1;
        if (done + A.tblock < A.nsteps) {
            if ((int)blockIdx.x == A.absent) return;  // never arrives: the others' waits run out
            waits++;
            if (!grid_wait(A.ctr, waits * gridDim.x, A.err)) return;
        }
    }
}

}  // namespace line1d
}  // namespace axp
