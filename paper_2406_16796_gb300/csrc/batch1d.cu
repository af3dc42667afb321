// batch1d.cu -- batches of 1D conversion runs in one persistent, time-blocked
// launch (arXiv 2406.16796 Sec. 2.3 scheme; Sec. 3.2 set-up), FP32 split.
//
// Each instance: periodic box of nx cells, CW laser E0y/B0z along x, uniform
// background (0, By, Bz), axion and order-1 fields initially zero.  In 1D the
// fields that can become non-zero are E0y, B0z (laser), E1y, E1z, B1y, B1z and
// phi; with the leapfrog-staggered E (as in the single-grid fused kernels) one
// step is
//   1. B^{n+1} = B^n - 2h curl E^{n+1/2}            (B0z, B1y, B1z)
//   2. S = E0y By; pi^{n+1}, phi^{n+3/2}, phi^{n+1}; E0y^{n+1} = E0y + h curl B0^{n+1}
//   3. P_y = D_t phi By, P_z = D_t phi (Bbar0z + Bz) + E0y^{n+1} d_x phi^{n+1}
//      (face averages along the invariant y, z are identities, so J = P);
//      E1^{n+3/2} = E1^{n+1/2} + 2h (curl B1^{n+1} - g J);  E0y^{n+3/2} = E0y^{n+1} + h curl B0^{n+1}
//
// Work items are (instance, segment).  A CTA loads its item's cells into
// registers -- each thread K consecutive cells of the whole instance (periodic
// wrap) when it fits, else of a segment plus a halo of 3 cells per step --
// advances T steps there, and writes the valid cells to the other of two
// global state buffers.  Only the cells at the ends of a thread's run are
// exchanged, through shared memory, once per stage.  Each
// cell's arithmetic is the same whatever the segmentation, the block length or
// the other instances in the batch, so results are bit-identical alone and in
// the mix.  Work items are taken from an atomic queue by a persistent grid;
// steps remaining per instance live on the device, so consecutive launches
// need no host round trip and can be captured in a CUDA graph.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <type_traits>
#include <vector>

#include "axp_internal.h"

namespace axp {
namespace {

constexpr int kArr = 6 + 2;   // E0y B0z E1y E1z B1y B1z phi pi (global, per buffer)
constexpr int kK = 8;         // consecutive cells per thread (held in registers)
constexpr int kMaxThreads = 512;  // a work item spans at most kK * kMaxThreads cells

struct Slot {
    int64_t off;        // first cell of this instance in every pool array
    int64_t remaining;  // steps still to do
    int64_t done;       // steps done
    int32_t nx;
    int32_t parity;     // buffer holding the present state
    int32_t active;     // admitted
    int32_t pad;
    float h, idx, hidx, cx, c0, dt2g, inv_dt, g, By, Bz;
    double dx, dt, m, gd, Byd, Bzd;
};

struct Item {
    int32_t slot;
    int32_t x0;   // first core cell
    int32_t len;  // core cells
    int32_t whole;  // 1: the item is the whole instance (periodic wrap in shared memory)
};

struct Dev {
    float *pool;   // [2 buffers][kArr][max_cells]
    int64_t max_cells;
    Slot *slots;
    Item *items;
    int32_t *counter;
    int32_t nitems;
};

__device__ __forceinline__ float *arr(const Dev &D, int buf, int a, int64_t off)
{
    return D.pool + ((int64_t)(buf * kArr + a) * D.max_cells + off);
}

// a[j] for a run-time j without indexing the register array (which would move
// it to local memory)
__device__ __forceinline__ float pick(const float (&a)[kK], int j)
{
    float v = a[0];
#pragma unroll
    for (int k = 1; k < kK; k++) v = k == j ? a[k] : v;
    return v;
}

// Packed FP32 pairs (the sm_100 pair pipe): one instruction for two cells, the
// same IEEE operation on each lane as the scalar form, so a cell's bits do not
// depend on which form advanced it.
__device__ __forceinline__ float2 p2(float s) { return make_float2(s, s); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
// a - b as a + b (-1): one rounding, the subtraction's bits
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// One launch: every work item advances min(budget, remaining) steps.
//
// Thread t holds cells [t K, t K + K) of the item (of n cells) in registers.
// Per stage it needs one cell beyond each end of its run; the threads publish
// their first and last cells' values in shared memory and read their
// neighbours' after a barrier (the instance's last thread and thread 0 are
// neighbours when the item is the whole periodic instance; a segment's end
// cells see themselves, as the halo absorbs what that spoils).
__global__ void __launch_bounds__(kMaxThreads) k_batch_block(Dev D, int budget, int halo_per_step)
{
    __shared__ float fE0[kMaxThreads], fE1y[kMaxThreads], fE1z[kMaxThreads];  // first cells
    __shared__ float lB0[kMaxThreads], lB1y[kMaxThreads], lB1z[kMaxThreads];  // last cells
    __shared__ float fMID[kMaxThreads], lMID[kMaxThreads];
    __shared__ float fPH[2][kMaxThreads], lPH[2][kMaxThreads];  // by step parity
    __shared__ int s_item;
    const int t = threadIdx.x;
    for (;;) {
        if (t == 0) s_item = atomicAdd(D.counter, 1);
        __syncthreads();
        const int it = s_item;
        __syncthreads();
        if (it >= D.nitems) return;
        const Item I = D.items[it];
        const Slot S = D.slots[I.slot];
        const int64_t rem = S.remaining;
        const int T = (int)(rem < budget ? rem : budget);
        if (!S.active || T <= 0) continue;
        const int nx = S.nx;
        const bool wrapc = I.whole != 0;
        const int H = wrapc ? 0 : halo_per_step * T;
        const int n = wrapc ? nx : I.len + 2 * H;
        const int c0 = t * kK;
        const int cnt = max(0, min(kK, n - c0));  // cells this thread holds
        const int lastT = (n - 1) / kK;           // thread holding cell n - 1
        const int tl = t > 0 ? t - 1 : (wrapc ? lastT : -1);  // left neighbour thread (-1: none)
        const int tr = t < lastT ? t + 1 : (wrapc ? 0 : -1);  // right neighbour thread
        const int in = S.parity, out = S.parity ^ 1;
        float E0[kK], B0[kK], E1y[kK], E1z[kK], B1y[kK], B1z[kK], PH[kK], PI[kK], MID[kK];
#pragma unroll
        for (int j = 0; j < kK; j++) {
            E0[j] = B0[j] = E1y[j] = E1z[j] = B1y[j] = B1z[j] = PH[j] = PI[j] = MID[j] = 0.0f;
            if (j < cnt) {
                int gx = wrapc ? c0 + j : I.x0 - H + c0 + j;  // periodic wrap in the instance
                gx %= nx;
                if (gx < 0) gx += nx;
                const int64_t o = S.off + gx;
                E0[j] = arr(D, in, 0, o)[0];
                B0[j] = arr(D, in, 1, o)[0];
                E1y[j] = arr(D, in, 2, o)[0];
                E1z[j] = arr(D, in, 3, o)[0];
                B1y[j] = arr(D, in, 4, o)[0];
                B1z[j] = arr(D, in, 5, o)[0];
                PH[j] = arr(D, in, 6, o)[0];
                PI[j] = arr(D, in, 7, o)[0];
            }
        }
        const int jl = cnt > 0 ? cnt - 1 : 0;  // this thread's last cell
        // the first cells' E and the end cells' phi for the first step
        fE0[t] = E0[0];
        fE1y[t] = E1y[0];
        fE1z[t] = E1z[0];
        fPH[0][t] = PH[0];
        lPH[0][t] = pick(PH, jl);
        __syncthreads();
        const float h = S.h, idx = S.idx, hidx = S.hidx, cx = S.cx, c0m = S.c0, dt2g = S.dt2g, inv_dt = S.inv_dt;
        const float g = S.g, By = S.By, Bz = S.Bz;
        const float hx = h * idx, h2x = 2.0f * hx, h2g = 2.0f * h * g;  // folded step constants
        // The stage bodies, for a thread holding K cells (F: the run is full, so
        // the tests on the run's length are known at compile time) or fewer.
        auto stage1 = [&](auto fullc) {  // B^{n+1}: needs E at i + 1
            constexpr bool F = decltype(fullc)::value;
            const int cn = F ? kK : cnt, jlast = F ? kK - 1 : jl;
            const float rE0 = tr >= 0 ? fE0[tr] : pick(E0, jlast), rE1y = tr >= 0 ? fE1y[tr] : pick(E1y, jlast);
            const float rE1z = tr >= 0 ? fE1z[tr] : pick(E1z, jlast);
#pragma unroll
            for (int j = 0; j < kK; j++) {
                const float e0p = j + 1 < cn ? E0[j + 1] : rE0;
                const float e1zp = j + 1 < cn ? E1z[j + 1] : rE1z;
                const float e1yp = j + 1 < cn ? E1y[j + 1] : rE1y;
                // B^{n+1} = B^n - 2h curl E^{n+1/2}, one multiply-add per difference:
                // (curl E0)_z = D_x E0y, (curl E1)_y = -D_x E1z, (curl E1)_z = D_x E1y
                B0[j] = fmaf(-h2x, e0p - E0[j], B0[j]);
                B1y[j] = fmaf(h2x, e1zp - E1z[j], B1y[j]);
                B1z[j] = fmaf(-h2x, e1yp - E1y[j], B1z[j]);
            }
            lB0[t] = pick(B0, jlast);
            lB1y[t] = pick(B1y, jlast);
            lB1z[t] = pick(B1z, jlast);
        };
        auto stage2 = [&](auto fullc, int pb) {  // axion; E0y^{n+1}: needs phi at i +- 1, B0 at i - 1
            constexpr bool F = decltype(fullc)::value;
            const int cn = F ? kK : cnt, jlast = F ? kK - 1 : jl;
            const float lph = tl >= 0 ? lPH[pb][tl] : PH[0], rph = tr >= 0 ? fPH[pb][tr] : pick(PH, jlast);
            float prevB0 = tl >= 0 ? lB0[tl] : B0[0];
#pragma unroll
            for (int j = 0; j < kK; j++) {
                const float php = j + 1 < cn ? PH[j + 1] : rph;
                const float phm = j > 0 ? PH[j - 1] : lph;
                const float Sg = E0[j] * By;  // Ebar0 . Bbar0 / g: E0y with the background along y
                const float ph = PH[j];
                // second difference from neighbour differences and the mass term kept
                // apart (c0 = -(m dt)^2), so neither rounds against 2*phi
                const float pin = fmaf(dt2g, Sg, fmaf(cx, (php - ph) + (phm - ph), fmaf(c0m, ph, PI[j])));
                PI[j] = pin;
                MID[j] = fmaf(0.5f, pin, ph);
                E0[j] = fmaf(-hx, B0[j] - prevB0, E0[j]);  // + h (curl B0)_y, (curl B0)_y = -D_x B0z
                prevB0 = B0[j];
            }
            fMID[t] = MID[0];
            lMID[t] = pick(MID, jlast);
        };
        auto stage3 = [&](auto fullc, int pb) {  // current and E updates: MID at i +- 1, B at i - 1
            constexpr bool F = decltype(fullc)::value;
            const int cn = F ? kK : cnt, jlast = F ? kK - 1 : jl;
            const float lmid = tl >= 0 ? lMID[tl] : MID[0], rmid = tr >= 0 ? fMID[tr] : pick(MID, jlast);
            float pB0 = tl >= 0 ? lB0[tl] : B0[0];
            float pB1z = tl >= 0 ? lB1z[tl] : B1z[0];
            float pB1y = tl >= 0 ? lB1y[tl] : B1y[0];
#pragma unroll
            for (int j = 0; j < kK; j++) {
                const float midp = j + 1 < cn ? MID[j + 1] : rmid;
                const float midm = j > 0 ? MID[j - 1] : lmid;
                const float Dt = PI[j] * inv_dt;
                const float Py = Dt * By;
                const float bz = fmaf(0.5f, B0[j] + pB0, Bz);
                const float Pz = fmaf(E0[j], (midp - midm) * hidx, Dt * bz);
                // E1^{n+3/2} = E1^{n+1/2} + 2h (curl B1 - g J), (curl B1)_y = -D_x B1z,
                // (curl B1)_z = D_x B1y; E0y^{n+3/2} = E0y^{n+1} + h (curl B0)_y
                E1y[j] = fmaf(-h2x, B1z[j] - pB1z, fmaf(-h2g, Py, E1y[j]));
                E1z[j] = fmaf(h2x, B1y[j] - pB1y, fmaf(-h2g, Pz, E1z[j]));
                E0[j] = fmaf(-hx, B0[j] - pB0, E0[j]);
                pB0 = B0[j];
                pB1z = B1z[j];
                pB1y = B1y[j];
            }
#pragma unroll
            for (int j = 0; j < kK; j++) PH[j] += PI[j];  // phi^{n+3/2} = phi^{n+1/2} + pi^{n+1}
            fE0[t] = E0[0];
            fE1y[t] = E1y[0];
            fE1z[t] = E1z[0];
            fPH[pb ^ 1][t] = PH[0];
            lPH[pb ^ 1][t] = pick(PH, jlast);
        };
        // Threads past the item's last cell only keep the barriers: no thread that
        // holds cells has them as neighbours (the item's last thread clamps or wraps).
        // The pair path runs a whole warp's threads or none of them: its barriers are
        // other instructions than the scalar path's, and all threads of a warp must
        // meet at the same barrier instruction.  (Threads holding K cells in a warp
        // with a partial or idle thread take the scalar path, to the same bits.)
#ifdef AXP_BATCH_SCALAR
        const bool full = false, idle = cnt == 0;
#else
        const bool full = __all_sync(0xffffffffu, cnt == kK), idle = cnt == 0;
#endif
        using Part = std::integral_constant<bool, false>;
        if (full) {
            // A full run of K cells advances on the pair pipe.  Pair q holds cells
            // (q, q + K/2), so the neighbour of pair q is pair q +- 1, and only the
            // run's end pairs take one cell from a neighbouring thread.
            constexpr int Q = kK / 2;
            float2 pE0[Q], pB0[Q], pE1y[Q], pE1z[Q], pB1y[Q], pB1z[Q], pPH[Q], pPI[Q], pMID[Q];
#pragma unroll
            for (int q = 0; q < Q; q++) {
                pE0[q] = make_float2(E0[q], E0[q + Q]);
                pB0[q] = make_float2(B0[q], B0[q + Q]);
                pE1y[q] = make_float2(E1y[q], E1y[q + Q]);
                pE1z[q] = make_float2(E1z[q], E1z[q + Q]);
                pB1y[q] = make_float2(B1y[q], B1y[q + Q]);
                pB1z[q] = make_float2(B1z[q], B1z[q + Q]);
                pPH[q] = make_float2(PH[q], PH[q + Q]);
                pPI[q] = make_float2(PI[q], PI[q + Q]);
                pMID[q] = make_float2(0.f, 0.f);
            }
            // cells i + 1 and i - 1 of pair q, given the neighbouring threads' end cells
            auto right = [&](const float2 (&a)[Q], int q, float r) {
                return q + 1 < Q ? a[q + 1] : make_float2(a[0].y, r);
            };
            auto left = [&](const float2 (&a)[Q], int q, float l) {
                return q > 0 ? a[q - 1] : make_float2(l, a[Q - 1].x);
            };
            const float2 mh2x = p2(-h2x), ph2x = p2(h2x), mhx = p2(-hx), mh2g = p2(-h2g);
            for (int st = 0; st < T; st++) {
                const int pb = st & 1;
                {  // stage 1: B^{n+1}
                    const float rE0 = tr >= 0 ? fE0[tr] : pE0[Q - 1].y, rE1y = tr >= 0 ? fE1y[tr] : pE1y[Q - 1].y;
                    const float rE1z = tr >= 0 ? fE1z[tr] : pE1z[Q - 1].y;
                    float2 n0[Q], n1y[Q], n1z[Q];
#pragma unroll
                    for (int q = 0; q < Q; q++) {
                        n0[q] = fma2(mh2x, sub2(right(pE0, q, rE0), pE0[q]), pB0[q]);
                        n1y[q] = fma2(ph2x, sub2(right(pE1z, q, rE1z), pE1z[q]), pB1y[q]);
                        n1z[q] = fma2(mh2x, sub2(right(pE1y, q, rE1y), pE1y[q]), pB1z[q]);
                    }
#pragma unroll
                    for (int q = 0; q < Q; q++) {
                        pB0[q] = n0[q];
                        pB1y[q] = n1y[q];
                        pB1z[q] = n1z[q];
                    }
                    lB0[t] = pB0[Q - 1].y;
                    lB1y[t] = pB1y[Q - 1].y;
                    lB1z[t] = pB1z[Q - 1].y;
                }
                __syncthreads();
                {  // stage 2: axion; E0y^{n+1}
                    const float lph = tl >= 0 ? lPH[pb][tl] : pPH[0].x, rph = tr >= 0 ? fPH[pb][tr] : pPH[Q - 1].y;
                    const float lB = tl >= 0 ? lB0[tl] : pB0[0].x;
                    float2 pin[Q], e0n[Q];
#pragma unroll
                    for (int q = 0; q < Q; q++) {
                        const float2 ph = pPH[q];
                        const float2 d2 = add2(sub2(right(pPH, q, rph), ph), sub2(left(pPH, q, lph), ph));
                        pin[q] = fma2(p2(dt2g), mul2(pE0[q], p2(By)), fma2(p2(cx), d2, fma2(p2(c0m), ph, pPI[q])));
                        e0n[q] = fma2(mhx, sub2(pB0[q], left(pB0, q, lB)), pE0[q]);
                    }
#pragma unroll
                    for (int q = 0; q < Q; q++) {
                        pPI[q] = pin[q];
                        pMID[q] = fma2(p2(0.5f), pin[q], pPH[q]);
                        pE0[q] = e0n[q];
                    }
                    fMID[t] = pMID[0].x;
                    lMID[t] = pMID[Q - 1].y;
                }
                __syncthreads();
                {  // stage 3: current, E updates
                    const float lmid = tl >= 0 ? lMID[tl] : pMID[0].x, rmid = tr >= 0 ? fMID[tr] : pMID[Q - 1].y;
                    const float lB = tl >= 0 ? lB0[tl] : pB0[0].x, lBz1 = tl >= 0 ? lB1z[tl] : pB1z[0].x;
                    const float lBy1 = tl >= 0 ? lB1y[tl] : pB1y[0].x;
                    float2 e1y[Q], e1z[Q], e0[Q];
#pragma unroll
                    for (int q = 0; q < Q; q++) {
                        const float2 Dt = mul2(pPI[q], p2(inv_dt));
                        const float2 Py = mul2(Dt, p2(By));
                        const float2 bz = fma2(p2(0.5f), add2(pB0[q], left(pB0, q, lB)), p2(Bz));
                        const float2 dm = mul2(sub2(right(pMID, q, rmid), left(pMID, q, lmid)), p2(hidx));
                        const float2 Pz = fma2(pE0[q], dm, mul2(Dt, bz));
                        e1y[q] = fma2(mh2x, sub2(pB1z[q], left(pB1z, q, lBz1)), fma2(mh2g, Py, pE1y[q]));
                        e1z[q] = fma2(ph2x, sub2(pB1y[q], left(pB1y, q, lBy1)), fma2(mh2g, Pz, pE1z[q]));
                        e0[q] = fma2(mhx, sub2(pB0[q], left(pB0, q, lB)), pE0[q]);
                    }
#pragma unroll
                    for (int q = 0; q < Q; q++) {
                        pE1y[q] = e1y[q];
                        pE1z[q] = e1z[q];
                        pE0[q] = e0[q];
                        pPH[q] = add2(pPH[q], pPI[q]);
                    }
                    fE0[t] = pE0[0].x;
                    fE1y[t] = pE1y[0].x;
                    fE1z[t] = pE1z[0].x;
                    fPH[pb ^ 1][t] = pPH[0].x;
                    lPH[pb ^ 1][t] = pPH[Q - 1].y;
                }
                __syncthreads();
            }
#pragma unroll
            for (int q = 0; q < Q; q++) {
                E0[q] = pE0[q].x, E0[q + Q] = pE0[q].y;
                B0[q] = pB0[q].x, B0[q + Q] = pB0[q].y;
                E1y[q] = pE1y[q].x, E1y[q + Q] = pE1y[q].y;
                E1z[q] = pE1z[q].x, E1z[q + Q] = pE1z[q].y;
                B1y[q] = pB1y[q].x, B1y[q + Q] = pB1y[q].y;
                B1z[q] = pB1z[q].x, B1z[q + Q] = pB1z[q].y;
                PH[q] = pPH[q].x, PH[q + Q] = pPH[q].y;
                PI[q] = pPI[q].x, PI[q + Q] = pPI[q].y;
            }
        } else {
            for (int st = 0; st < T; st++) {
                const int pb = st & 1;
                if (!idle) stage1(Part{});
                __syncthreads();
                if (!idle) stage2(Part{}, pb);
                __syncthreads();
                if (!idle) stage3(Part{}, pb);
                __syncthreads();
            }
        }
        // write the valid core cells to the other buffer
#pragma unroll
        for (int j = 0; j < kK; j++) {
            const int i = c0 + j;  // local cell
            const int lo = wrapc ? 0 : H, hi = wrapc ? nx : H + I.len;
            if (j < cnt && i >= lo && i < hi) {
                const int gx = wrapc ? i : I.x0 + (i - H);
                const int64_t o = S.off + gx;
                arr(D, out, 0, o)[0] = E0[j];
                arr(D, out, 1, o)[0] = B0[j];
                arr(D, out, 2, o)[0] = E1y[j];
                arr(D, out, 3, o)[0] = E1z[j];
                arr(D, out, 4, o)[0] = B1y[j];
                arr(D, out, 5, o)[0] = B1z[j];
                arr(D, out, 6, o)[0] = PH[j];
                arr(D, out, 7, o)[0] = PI[j];
            }
        }
        __syncthreads();
    }
}

// After each launch: charge the steps, flip the buffers, reset the queue.
__global__ void k_batch_account(Dev D, int nslots, int budget)
{
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < nslots; s += gridDim.x * blockDim.x) {
        Slot &S = D.slots[s];
        if (!S.active) continue;
        const int64_t T = S.remaining < budget ? S.remaining : budget;
        if (T <= 0) continue;
        S.remaining -= T;
        S.done += T;
        S.parity ^= 1;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *D.counter = 0;
}

// Initial state of one instance in buffer 0: the CW eigenmode laser at t = 0
// (E0y = A cos(k x_E), B0z = discrete curl of F = (A / cos(theta/2)) sin(k x)/K),
// then E0y moved to t = +dt/2 (E0y^{1/2} = E0y^0 + h (curl B0^0)_y); zero elsewhere.
__global__ void k_batch_init(Dev D, int slot, double A, double k)
{
    const Slot S = D.slots[slot];
    const int nx = S.nx;
    const double dx = S.dx, dt = S.dt;
    const double K = (2.0 / dx) * sin(k * dx / 2.0);
    const double sh = dt * K / 2.0;
    const double ch = sqrt(1.0 - sh * sh);
    const double Fs = A / (ch * K);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nx; i += gridDim.x * blockDim.x) {
        // F_y at the E_y samples (cell centres), periodic
        auto F = [&](int c) {
            c %= nx;
            if (c < 0) c += nx;
            return Fs * sin(k * ((double)c + 0.5) * dx);
        };
        const double bz_i = (F(i + 1) - F(i)) / dx;      // B0z(i) = D_x F_y
        const double bz_m = (F(i) - F(i - 1)) / dx;      // B0z(i-1)
        const double e0 = A * cos(k * ((double)i + 0.5) * dx);
        const double e_half = e0 + (dt / 2.0) * (-(bz_i - bz_m) / dx);
        const int64_t o = S.off + i;
        arr(D, 0, 0, o)[0] = (float)e_half;
        arr(D, 0, 1, o)[0] = (float)bz_i;
        for (int a = 2; a < kArr; a++) arr(D, 0, a, o)[0] = 0.0f;
    }
}

// FP64 diagnostics of instances at their present (integer) time, with E taken back from
// n+1/2 to n.
// One block per kDiagCells cells of a listed slot: large slots are spread over the chip (one
// block per slot left a 65536-cell slot 2.4 ms on one SM), and the FP64 pipe, which bounds the
// sums, gets each product once, with every constant on the sums (no division per cell):
// 512 slots, 7.9M cells: 4.8 -> 1.7 ms a call.  The segments and the order of every sum depend on
// the slot's size alone, so a record does not depend on the list it is asked for in.
constexpr int kDiagCells = 4096, kDiagSums = 8;

__global__ void __launch_bounds__(256) k_batch_diag(Dev D, const int *slots, const int *first, int n, double *partials)
{
    int lo = 0, hi = n;  // the entry with first[lo] <= block < first[lo + 1]
    while (hi - lo > 1) {
        const int mid = (lo + hi) / 2;
        if (first[mid] <= (int)blockIdx.x) lo = mid;
        else hi = mid;
    }
    const Slot S = D.slots[slots[lo]];
    const int nx = S.nx, buf = S.parity;
    const int c0 = ((int)blockIdx.x - first[lo]) * kDiagCells, c1 = min(nx, c0 + kDiagCells);
    const float *E0 = arr(D, buf, 0, S.off), *B0 = arr(D, buf, 1, S.off), *E1y = arr(D, buf, 2, S.off);
    const float *E1z = arr(D, buf, 3, S.off), *B1y = arr(D, buf, 4, S.off), *B1z = arr(D, buf, 5, S.off);
    const float *PH = arr(D, buf, 6, S.off), *PI = arr(D, buf, 7, S.off);
    const double h = S.dt / 2.0, hx = h / S.dx, hg = h * S.gd, hgt = hg / S.dt, hgyt = hgt * S.Byd, hg2x = hg / (2.0 * S.dx);
    const double By = S.Byd, Bz = S.Bzd;
    // PI^2, (d phi)^2, phi^2 | E0^2 + B0^2 | E1^2 + B1y^2 | E0.E1 + ... | (i + 1) B1z^2, B1z^2
    double acc[kDiagSums] = {0, 0, 0, 0, 0, 0, 0, 0};
    auto mid = [&](int c) { return fma(-0.5, (double)PI[c], (double)PH[c]); };
    for (int i = c0 + (int)threadIdx.x; i < c1; i += 256) {
        const int im = i > 0 ? i - 1 : nx - 1, ip = i + 1 < nx ? i + 1 : 0;
        const double pi = PI[i], ph = mid(i), up = mid(ip), dn = mid(im);
        acc[0] = fma(pi, pi, acc[0]);
        acc[1] = fma(up - ph, up - ph, acc[1]);
        acc[2] = fma(ph, ph, acc[2]);
        // E^n = E^{n+1/2} - h (curl B - g J): (curl B0)_y = -D_x B0z; P_y = D_t phi By,
        // P_z = D_t phi (Bbar0z + Bz) + E0y^n d_x phi^n
        const double b0 = B0[i], b0m = B0[im], b1y = B1y[i], b1z = B1z[i];
        const double e0 = fma(hx, b0 - b0m, (double)E0[i]);
        const double e1y = fma(hx, b1z - (double)B1z[im], fma(hgyt, pi, (double)E1y[i]));
        const double e1z = fma(-hx, b1y - (double)B1y[im],
                               fma(hgt * pi, fma(0.5, b0 + b0m, Bz), fma(hg2x * e0, up - dn, (double)E1z[i])));
        acc[3] = fma(e0, e0, fma(b0, b0, acc[3]));
        acc[4] = fma(e1y, e1y, fma(e1z, e1z, fma(b1y, b1y, acc[4])));
        acc[5] = fma(e0, e1y, fma(By, b1y, fma(b0 + Bz, b1z, acc[5])));
        const double bz2 = b1z * b1z;
        acc[6] = fma((double)(i + 1), bz2, acc[6]);
        acc[7] += bz2;
    }
    __shared__ double sh[kDiagSums][8];
#pragma unroll
    for (int q = 0; q < kDiagSums; q++) {
#pragma unroll
        for (int w = 16; w > 0; w >>= 1) acc[q] += __shfl_down_sync(0xffffffffu, acc[q], w);
        if (threadIdx.x % 32 == 0) sh[q][threadIdx.x / 32] = acc[q];
    }
    __syncthreads();
    if (threadIdx.x < kDiagSums) {
        double t = 0.0;
        for (int w = 0; w < 8; w++) t += sh[threadIdx.x][w];
        partials[(int64_t)blockIdx.x * kDiagSums + threadIdx.x] = t;
    }
}

// the record of one listed slot from its segments' sums, in their order
__global__ void __launch_bounds__(32) k_batch_record(Dev D, const int *slots, const int *first, const double *partials,
                                                     axp_diag *out)
{
    __shared__ double sum[kDiagSums];
    const int q = (int)blockIdx.x;
    if (threadIdx.x < kDiagSums) {
        double t = 0.0;
        for (int b = first[q]; b < first[q + 1]; b++) t += partials[(int64_t)b * kDiagSums + threadIdx.x];
        sum[threadIdx.x] = t;
    }
    __syncwarp();
    if (threadIdx.x == 0) {
        const Slot S = D.slots[slots[q]];
        const double dx = S.dx, dt = S.dt, dV = dx * dx * dx;
        axp_diag d;
        d.step = S.done;
        d.t = (double)S.done * dt;
        d.H_phi = 0.5 * (sum[0] / (dt * dt) + sum[1] / (dx * dx) + S.m * S.m * sum[2]) * dV;
        d.H_g0 = 0.5 * sum[3] * dV;
        d.H_g1 = 0.5 * (sum[4] + sum[7]) * dV;
        d.P_g2a = d.H_g0 > 0 ? d.H_phi / d.H_g0 : 0.0;
        d.P_a2g = d.H_phi > 0 ? d.H_g1 / d.H_phi : 0.0;
        d.W = d.H_phi + sum[5] * dV;
        d.sum_xB1z2 = sum[6] * dx * dV;
        d.sum_B1z2 = sum[7] * dV;
        d.gauss_l2 = 0.0;  // div E1 and B_ext,x d_x phi vanish identically in this 1D set-up
        out[q] = d;
    }
}

constexpr size_t kAlign = 256;
size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

// Read-out of one array of one slot, in pieces of at most kReadCells: gathered into a scratch
// on the device (where the slot's present buffer is known), copied into pinned memory of the
// batch and widened from there into the caller's.  One launch, one copy and one
// synchronisation where there were two copies and two synchronisations.  The caller's pages
// are touched by the host only: a copy straight into fresh pageable memory takes the GPU's
// page faults (512 reads of 15.5k cells: 54 ms that way, 16-20 ms before, 12.5-17 ms now).
constexpr int64_t kReadCells = 1 << 17;

__global__ void __launch_bounds__(256) k_batch_gather(Dev D, int slot, int which, int64_t first, int n, float *dst)
{
    const Slot S = D.slots[slot];
    const float *src = arr(D, S.parity, which, S.off) + first;
    for (int i = (int)(blockIdx.x * blockDim.x + threadIdx.x); i < n; i += (int)(gridDim.x * blockDim.x)) dst[i] = src[i];
}

struct Layout {
    size_t pool, slots, items, counter, diag, partials, read, total;
};

// segments the sums have room for: every slot's at once
size_t diag_segments(int32_t max_instances, int64_t max_cells)
{
    return (size_t)max_instances + (size_t)max_cells / kDiagCells;
}

Layout layout(int32_t max_instances, int64_t max_cells)
{
    Layout L;
    size_t off = 0;
    L.pool = off;
    off += align_up((size_t)2 * kArr * max_cells * sizeof(float));
    L.slots = off;
    off += align_up((size_t)max_instances * sizeof(Slot));
    L.items = off;
    // an instance of nx cells makes at most nx / 64 + 1 items (segments are >= 64 cells)
    off += align_up(((size_t)max_instances + (size_t)max_cells / 64 + 1) * sizeof(Item));
    L.counter = off;
    off += kAlign;
    // one record per slot, then the list of slots asked for and where their segments begin,
    // then the segments' sums
    L.diag = off;
    off += align_up((size_t)max_instances * (sizeof(axp_diag) + 2 * sizeof(int)) + sizeof(int));
    L.partials = off;
    off += align_up(diag_segments(max_instances, max_cells) * kDiagSums * sizeof(double));
    L.read = off;
    off += align_up((size_t)std::min(max_cells, kReadCells) * sizeof(float));
    L.total = off;
    return L;
}

axp_status cuda_st(cudaError_t e)
{
    if (e == cudaSuccess) return AXP_OK;
    fprintf(stderr, "axp batch: CUDA error %s\n", cudaGetErrorString(e));
    return AXP_E_CUDA;
}

}  // namespace
}  // namespace axp

using namespace axp;

struct axp_batch {
    int32_t max_instances;
    int64_t max_cells;
    char *ws;
    cudaStream_t stream;
    Layout L;
    Dev D;
    std::vector<Slot> slots;                         // host mirror
    std::vector<std::pair<int64_t, int64_t>> free;  // free cell ranges (offset, length), sorted
    bool dirty;
    int32_t block_steps, segment_cells, threads;
    int sms;
    int64_t launches;
    // CUDA graph of one axp_batch_run call, reused while the call's step count,
    // the tiling and the work table stay the same
    bool use_graph;
    cudaGraphExec_t graph;
    int64_t graph_steps;
    float *host;  // pinned, of the first axp_batch_read_state on
};

extern "C" {

axp_status axp_batch_workspace_bytes(int32_t max_instances, int64_t max_cells, size_t *bytes)
{
    if (!bytes || max_instances < 1 || max_cells < 8 || max_cells > ((int64_t)1 << 31)) return AXP_E_INVAL;
    *bytes = layout(max_instances, max_cells).total;
    return AXP_OK;
}

axp_status axp_batch_create(int32_t max_instances, int64_t max_cells, void *dev_workspace, size_t bytes,
                            void *cuda_stream, axp_batch **out)
{
    if (!out || !dev_workspace || max_instances < 1 || max_cells < 8 || max_cells > ((int64_t)1 << 31))
        return AXP_E_INVAL;
    if ((uintptr_t)dev_workspace % kAlign) return AXP_E_INVAL;
    *out = nullptr;
    const Layout L = layout(max_instances, max_cells);
    if (bytes < L.total) return AXP_E_NOMEM;
    axp_batch *b = new (std::nothrow) axp_batch();
    if (!b) return AXP_E_NOMEM;
    b->max_instances = max_instances;
    b->max_cells = max_cells;
    b->ws = (char *)dev_workspace;
    b->stream = (cudaStream_t)cuda_stream;
    b->L = L;
    b->D.pool = (float *)(b->ws + L.pool);
    b->D.max_cells = max_cells;
    b->D.slots = (Slot *)(b->ws + L.slots);
    b->D.items = (Item *)(b->ws + L.items);
    b->D.counter = (int32_t *)(b->ws + L.counter);
    b->D.nitems = 0;
    b->slots.assign(max_instances, Slot());
    std::memset(b->slots.data(), 0, sizeof(Slot) * max_instances);
    b->free.push_back({0, max_cells});
    b->dirty = true;
    // default tiling: a segment and its halo fill a 256-thread block, two blocks per SM
    b->block_steps = 32;
    b->segment_cells = 8 * 256 - 6 * 32;
    b->threads = 256;
    b->use_graph = false;
    b->graph = nullptr;
    b->graph_steps = -1;
    b->host = nullptr;
    int dev = 0;
    cudaGetDevice(&dev);
    b->sms = 152;
    cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaMemsetAsync(b->ws + L.slots, 0, L.total - L.slots, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) {
        delete b;
        return cuda_st(e);
    }
    *out = b;
    return AXP_OK;
}

axp_status axp_batch_destroy(axp_batch *b)
{
    if (!b) return AXP_E_INVAL;
    // the caller frees the workspace after this returns: let queued work finish
    cudaStreamSynchronize(b->stream);
    if (b->graph) cudaGraphExecDestroy(b->graph);
    if (b->host) cudaFreeHost(b->host);
    delete b;
    return AXP_OK;
}

axp_status axp_batch_add(axp_batch *b, const axp_batch_instance *in, int32_t *slot)
{
    axp::TraceRange trace_("axp_batch_add");
    if (!b || !in || !slot) return AXP_E_INVAL;
    if (in->nx < 8 || in->nx > (1 << 30) || !(in->dx > 0) || !(in->dt > 0) || in->steps < 0 || !std::isfinite(in->g) ||
        !std::isfinite(in->m) || !std::isfinite(in->By) || !std::isfinite(in->Bz) || !std::isfinite(in->amplitude) ||
        !std::isfinite(in->k))
        return AXP_E_INVAL;
    if (in->dt > in->dx || in->dt * in->dt * (4.0 / (in->dx * in->dx) + in->m * in->m) > 4.0) return AXP_E_UNSTABLE;
    int s = -1;
    for (int i = 0; i < b->max_instances; i++)
        if (!b->slots[i].active) {
            s = i;
            break;
        }
    if (s < 0) return AXP_E_NOMEM;
    int64_t off = -1;
    for (auto &r : b->free)
        if (r.second >= in->nx) {
            off = r.first;
            r.first += in->nx;
            r.second -= in->nx;
            break;
        }
    if (off < 0) return AXP_E_NOMEM;
    b->free.erase(std::remove_if(b->free.begin(), b->free.end(), [](const std::pair<int64_t, int64_t> &r) {
                      return r.second == 0;
                  }),
                  b->free.end());
    Slot S;
    std::memset(&S, 0, sizeof(S));
    S.off = off;
    S.remaining = in->steps;
    S.done = 0;
    S.nx = (int32_t)in->nx;
    S.parity = 0;
    S.active = 1;
    const double dx = in->dx, dt = in->dt;
    S.h = (float)(dt / 2.0);
    S.idx = (float)(1.0 / dx);
    S.hidx = (float)(0.5 / dx);
    S.cx = (float)(dt * dt / (dx * dx));
    S.c0 = (float)(-dt * dt * in->m * in->m);
    S.dt2g = (float)(dt * dt * in->g);
    S.inv_dt = (float)(1.0 / dt);
    S.g = (float)in->g;
    S.By = (float)in->By;
    S.Bz = (float)in->Bz;
    S.dx = dx;
    S.dt = dt;
    S.m = in->m;
    S.gd = in->g;
    S.Byd = in->By;
    S.Bzd = in->Bz;
    b->slots[s] = S;
    cudaError_t e = cudaMemcpyAsync(b->D.slots + s, &b->slots[s], sizeof(Slot), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess) {
        const int blocks = (int)std::min<int64_t>((in->nx + 255) / 256, 1024);
        k_batch_init<<<blocks, 256, 0, b->stream>>>(b->D, s, in->amplitude, in->k);
        e = cudaGetLastError();
    }
    // the host copy of the slot must stay valid until the copy above has run
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return cuda_st(e);
    b->dirty = true;
    *slot = s;
    return AXP_OK;
}

static void drop_graph(axp_batch *b)
{
    if (b->graph) cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
    b->graph_steps = -1;
}

axp_status axp_batch_remove(axp_batch *b, int32_t slot)
{
    if (!b || slot < 0 || slot >= b->max_instances || !b->slots[slot].active) return AXP_E_INVAL;
    Slot &S = b->slots[slot];
    b->free.push_back({S.off, S.nx});
    std::sort(b->free.begin(), b->free.end());
    std::vector<std::pair<int64_t, int64_t>> merged;
    for (auto &r : b->free) {
        if (!merged.empty() && merged.back().first + merged.back().second == r.first) merged.back().second += r.second;
        else merged.push_back(r);
    }
    b->free.swap(merged);
    S.active = 0;
    cudaError_t e = cudaMemcpyAsync(&b->D.slots[slot].active, &S.active, sizeof(int32_t), cudaMemcpyHostToDevice,
                                    b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    b->dirty = true;
    return cuda_st(e);
}

static axp_status rebuild_items(axp_batch *b)
{
    const int cap = kK * b->threads;  // cells a work item holds
    const int halo = 3 * b->block_steps;
    int seg = b->segment_cells;
    if (seg + 2 * halo > cap) seg = cap - 2 * halo;
    if (seg < 64) return AXP_E_INVAL;
    std::vector<Item> items;
    for (int s = 0; s < b->max_instances; s++) {
        const Slot &S = b->slots[s];
        if (!S.active) continue;
        if (S.nx <= cap) {
            items.push_back({s, 0, S.nx, 1});
        } else {
            for (int x0 = 0; x0 < S.nx; x0 += seg) items.push_back({s, x0, std::min(seg, S.nx - x0), 0});
        }
    }
    // largest items first for the persistent queue
    std::stable_sort(items.begin(), items.end(), [](const Item &a, const Item &c) { return a.len > c.len; });
    cudaError_t e = cudaSuccess;
    if (!items.empty())
        e = cudaMemcpyAsync(b->D.items, items.data(), items.size() * sizeof(Item), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return cuda_st(e);
    b->D.nitems = (int32_t)items.size();
    b->dirty = false;
    return AXP_OK;
}

static cudaError_t enqueue_run(axp_batch *b, int64_t nsteps)
{
    const int halo = 3;  // cells of halo per step on each side of a segment
    int occ = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_batch_block, b->threads, 0) != cudaSuccess || occ < 1)
        occ = 1;
    const int grid = std::min<int>(b->sms * occ, std::max<int>(1, b->D.nitems));
    for (int64_t done = 0; done < nsteps; done += b->block_steps) {
        const int budget = (int)std::min<int64_t>(b->block_steps, nsteps - done);
        k_batch_block<<<grid, b->threads, 0, b->stream>>>(b->D, budget, halo);
        k_batch_account<<<(b->max_instances + 255) / 256, 256, 0, b->stream>>>(b->D, b->max_instances, budget);
        b->launches += 2;
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

axp_status axp_batch_run(axp_batch *b, int64_t nsteps)
{
    axp::TraceRange trace_("axp_batch_run");
    if (!b || nsteps < 0) return AXP_E_INVAL;
    if (nsteps == 0) return AXP_OK;
    if (b->dirty) {
        drop_graph(b);
        const axp_status st = rebuild_items(b);
        if (st != AXP_OK) return st;
    }
    if (b->D.nitems == 0) return AXP_OK;
    if (!b->use_graph || b->stream == nullptr) return cuda_st(enqueue_run(b, nsteps));
    if (!b->graph || b->graph_steps != nsteps) {
        drop_graph(b);
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return cuda_st(e);
        const int64_t l0 = b->launches;
        e = enqueue_run(b, nsteps);
        const cudaError_t e2 = cudaStreamEndCapture(b->stream, &g);
        b->launches = l0;
        if (e != cudaSuccess || e2 != cudaSuccess) {
            if (g) cudaGraphDestroy(g);
            return cuda_st(e != cudaSuccess ? e : e2);
        }
        e = cudaGraphInstantiate(&b->graph, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) {
            b->graph = nullptr;
            return cuda_st(e);
        }
        b->graph_steps = nsteps;
    }
    b->launches += 2 * ((nsteps + b->block_steps - 1) / b->block_steps);
    return cuda_st(cudaGraphLaunch(b->graph, b->stream));
}

axp_status axp_batch_use_graphs(axp_batch *b, int32_t enable)
{
    if (!b) return AXP_E_INVAL;
    if (!enable) drop_graph(b);
    b->use_graph = enable != 0;
    return AXP_OK;
}

axp_status axp_batch_launch_count(const axp_batch *b, int64_t *count)
{
    if (!b || !count) return AXP_E_INVAL;
    *count = b->launches;
    return AXP_OK;
}

axp_status axp_batch_progress(axp_batch *b, int64_t *steps_done, int32_t max_slots)
{
    if (!b || !steps_done || max_slots < 0) return AXP_E_INVAL;
    std::vector<Slot> tmp(b->max_instances);
    cudaError_t e = cudaMemcpyAsync(tmp.data(), b->D.slots, sizeof(Slot) * b->max_instances, cudaMemcpyDeviceToHost,
                                    b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return cuda_st(e);
    for (int s = 0; s < std::min<int32_t>(max_slots, b->max_instances); s++)
        steps_done[s] = b->slots[s].active ? tmp[s].done : -1;
    return AXP_OK;
}

axp_status axp_batch_results(axp_batch *b, const int32_t *slots, int32_t n, axp_diag *out)
{
    axp::TraceRange trace_("axp_batch_results");
    if (!b || !slots || !out || n < 1 || n > b->max_instances) return AXP_E_INVAL;
    for (int32_t q = 0; q < n; q++)
        if (slots[q] < 0 || slots[q] >= b->max_instances || !b->slots[slots[q]].active) return AXP_E_INVAL;
    axp_diag *dev = (axp_diag *)(b->ws + b->L.diag);
    int *dev_slots = (int *)(dev + b->max_instances), *dev_first = dev_slots + b->max_instances;
    double *partials = (double *)(b->ws + b->L.partials);
    const size_t room = diag_segments(b->max_instances, b->max_cells);
    cudaError_t e = cudaMemcpyAsync(dev_slots, slots, (size_t)n * sizeof(int), cudaMemcpyHostToDevice, b->stream);
    std::vector<int> first(n + 1);
    // every slot once fits in one go; a list that repeats slots may take several
    for (int32_t q0 = 0; q0 < n && e == cudaSuccess;) {
        int32_t q1 = q0;
        size_t total = 0;
        while (q1 < n) {
            const size_t seg = ((size_t)b->slots[slots[q1]].nx + kDiagCells - 1) / kDiagCells;
            if (q1 > q0 && total + seg > room) break;
            first[q1 - q0] = (int)total;
            total += seg;
            q1++;
        }
        first[q1 - q0] = (int)total;
        const int m = q1 - q0;
        e = cudaMemcpyAsync(dev_first, first.data(), (size_t)(m + 1) * sizeof(int), cudaMemcpyHostToDevice, b->stream);
        if (e != cudaSuccess) break;
        k_batch_diag<<<(unsigned)total, 256, 0, b->stream>>>(b->D, dev_slots + q0, dev_first, m, partials);
        k_batch_record<<<m, 32, 0, b->stream>>>(b->D, dev_slots + q0, dev_first, partials, dev + q0);
        b->launches += 2;
        e = cudaGetLastError();
        q0 = q1;
        if (q0 < n && e == cudaSuccess) e = cudaStreamSynchronize(b->stream);  // (before `first` is written again)
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(out, dev, (size_t)n * sizeof(axp_diag), cudaMemcpyDeviceToHost, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return cuda_st(e);
    for (int32_t q = 0; q < n; q++)
        if (!std::isfinite(out[q].H_phi) || !std::isfinite(out[q].H_g0) || !std::isfinite(out[q].H_g1))
            return AXP_E_NONFINITE;
    return AXP_OK;
}

axp_status axp_batch_result(axp_batch *b, int32_t slot, axp_diag *out) { return axp_batch_results(b, &slot, 1, out); }

axp_status axp_batch_read_state(axp_batch *b, int32_t slot, int32_t which, double *host_dst, size_t bytes)
{
    if (!b || !host_dst || slot < 0 || slot >= b->max_instances || !b->slots[slot].active || which < 0 || which >= kArr)
        return AXP_E_INVAL;
    const int64_t nx = b->slots[slot].nx;
    if (bytes != (size_t)nx * sizeof(double)) return AXP_E_INVAL;
    float *scratch = (float *)(b->ws + b->L.read);
    const int64_t piece = std::min(b->max_cells, kReadCells);
    cudaError_t e = cudaSuccess;
    if (!b->host && (e = cudaMallocHost((void **)&b->host, (size_t)piece * sizeof(float))) != cudaSuccess) {
        b->host = nullptr;
        return cuda_st(e);
    }
    for (int64_t c = 0; c < nx; c += piece) {
        const int n = (int)std::min(piece, nx - c);
        k_batch_gather<<<std::min((n + 255) / 256, 152 * 8), 256, 0, b->stream>>>(b->D, slot, which, c, n, scratch);
        e = cudaGetLastError();
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(b->host, scratch, (size_t)n * sizeof(float), cudaMemcpyDeviceToHost, b->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
        if (e != cudaSuccess) return cuda_st(e);
        for (int i = 0; i < n; i++) host_dst[c + i] = b->host[i];
    }
    return AXP_OK;
}

axp_status axp_batch_set_tiling(axp_batch *b, int32_t block_steps, int32_t segment_cells, int32_t threads)
{
    if (!b || block_steps < 1 || block_steps > 256 || threads < 64 || threads > kMaxThreads || threads % 32)
        return AXP_E_INVAL;
    if (segment_cells < 64 || segment_cells + 6 * block_steps > kK * threads) return AXP_E_INVAL;
    b->block_steps = block_steps;
    b->segment_cells = segment_cells;
    b->threads = threads;
    b->dirty = true;
    drop_graph(b);
    return AXP_OK;
}

axp_status axp_batch_get_tiling(const axp_batch *b, int32_t *block_steps, int32_t *segment_cells, int32_t *threads)
{
    if (!b || !block_steps || !segment_cells || !threads) return AXP_E_INVAL;
    *block_steps = b->block_steps;
    *segment_cells = b->segment_cells;
    *threads = b->threads;
    return AXP_OK;
}

}  // extern "C"
