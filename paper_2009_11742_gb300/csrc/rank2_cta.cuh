// One-CTA kernel for the rank-2 leapfrog of small models (FP32, Kp <= 128).
//
// Both operators of a model this small (2 x 64 KB at Kp = 128) fit in the
// registers of one CTA, so a column block needs no cluster: the block's V and
// S live in the CTA's shared memory, a half-step (Sec. 3.1, velocity first)
// reads one of them and updates the other in place, and one __syncthreads
// ends it.  The split kernel spends two cluster barriers with remote stores
// on every step, about 2.2 us whatever the size.
//
// 256 threads.  Thread (row group, chunk j) holds 4 KI rows (KI = Kp / 64) of
// Avs and of Asv at k = 64 i + 4 j + t: the split kernel's k stripes, and the
// sums, the reduction over the 16 chunk lanes, the epilogue and the receiver
// traces are the split kernel's too, so every column comes out bit for bit as
// there.  8 rows a thread at Kp = 128 instead of 4 (512 threads) halve the
// operand reads and the reductions: 0.43 us a step against 0.87 (M = 16).
// Columns go through in groups of CB (1, 2 or 4); a block of one group keeps
// its elements and carries in registers.  The forcing of the next kCtaTab
// steps is tabulated by all threads at once.
//
// Bound: latency (operand reads, the 4-deep reduction, the Kahan chain, the
// barrier) while a block holds few columns, FMA issue above.  us a step, this
// kernel / split kernel / one-block kernel:
//     Kp = 64:  M = 16 0.31 / 1.98 / 2.36,  M = 500 0.50 / 2.00 / 2.40,  M = 4000 3.2 / 6.0 / 7.1
//     Kp = 128: M = 16 0.43 / 2.10 / 2.71,  M = 500 1.26 / 2.99 / 3.85,  M = 4000 7.9 / 12.8 / 16.9
// so it is the plan for every M there.  At Kp = 192 the two operators no
// longer fit the registers (288 of them a thread).
#pragma once

#include <cuda_runtime.h>

#include "dev_common.cuh"
#include "rank2_simt.cuh"
#include "rank2_split.cuh"
#include "rom_internal.h"

namespace romk {

constexpr int kCtaTab = 32;   // steps of forcing tabulated at a time
constexpr int kCtaPad = 8;    // column stride Kp + 8: the epilogue's 8 rows x 4 columns on distinct banks

// A thread's RT x CB sums are reduced NV at a time over the 16 chunk lanes, in
// NG groups of NV / CB rows.
template <int RT, int CB>
struct CtaTile {
    static constexpr int NV = RT * CB < 16 ? RT * CB : 16;
    static constexpr int NG = RT * CB / NV;
};

struct CtaSmem {
    size_t V, S, cV, cS, C, f, Tpre, total;
};

// nC: receiver rows staged in shared memory (0: read from global memory).
__host__ __device__ inline CtaSmem cta_smem_layout(int Wa, int Kp, int nC) {
    CtaSmem s{};
    const size_t st = (size_t)Wa * (Kp + kCtaPad) * sizeof(float);
    size_t o = 0;
    s.V = o;    o += align16(st);
    s.S = o;    o += align16(st);
    s.cV = o;   o += align16(st);
    s.cS = o;   o += align16(st);
    s.C = o;    o += align16((size_t)nC * Kp * sizeof(float));
    s.f = o;    o += align16((size_t)kCtaTab * Wa * sizeof(float));
    s.Tpre = o; o += align16((size_t)2 * Wa * sizeof(double));
    s.total = o;
    return s;
}

// RT rows of one operator per thread.
template <int KI, int RT>
__device__ __forceinline__ void cta_load_op(float (&op)[RT][4 * KI], const float* __restrict__ A, int row, int j) {
#pragma unroll
    for (int r = 0; r < RT; ++r) {
#pragma unroll
        for (int i = 0; i < KI; ++i) {
            float x[4];
            load4_ro(A + (size_t)(row + r) * 64 * KI + 64 * i + 4 * j, x);
#pragma unroll
            for (int t = 0; t < 4; ++t) op[r][4 * i + t] = x[t];
        }
    }
}

// Y += dt (op . X [+ g f^T] [+ Xref]) over the block's columns.  With CB < 4
// the block is one column group, so a lane's element and carry stay in y0 and
// carry0; otherwise they are in Y and comp.
template <int KI, int RT, int CB, bool FORCED, bool XR>
__device__ __forceinline__ void cta_half(const float (&op)[RT][4 * KI], const float* __restrict__ X,
                                         float* __restrict__ Y, float* __restrict__ comp, float& y0, float& carry0,
                                         const float (&g)[CtaTile<RT, CB>::NG], const float* __restrict__ f,
                                         const float dt, const int Wa, const int row, const int j,
                                         const float* __restrict__ Xref, const int Krows, const int ncol) {
    constexpr int ST = 64 * KI + kCtaPad;
    constexpr int NV = CtaTile<RT, CB>::NV, NG = CtaTile<RT, CB>::NG;
    constexpr bool ONE = CB < 4;
    const int slot = rs16_slot<NV>(j);
    const int rl = row + slot / CB, cl = slot % CB;
    for (int c0 = 0; c0 < (ONE ? 1 : Wa); c0 += CB) {
        const int c = c0 + cl;
        float xr[NG];
        if constexpr (XR) {
#pragma unroll
            for (int h = 0; h < NG; ++h) {
                const int rw = rl + h * (NV / CB);
                xr[h] = Xref && c < ncol && rw < Krows ? Xref[(size_t)c * Krows + rw] : 0.f;
            }
        }
        float acc[RT][CB];
#pragma unroll
        for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int cc = 0; cc < CB; ++cc) acc[r][cc] = 0.f;
#pragma unroll
        for (int i = 0; i < KI; ++i) {
            float x[CB][4];
#pragma unroll
            for (int cc = 0; cc < CB; ++cc) load4(X + (c0 + cc) * ST + 64 * i + 4 * j, x[cc]);
#pragma unroll
            for (int t = 0; t < 4; ++t)
#pragma unroll
                for (int cc = 0; cc < CB; ++cc)
#pragma unroll
                    for (int r = 0; r < RT; ++r) acc[r][cc] = __fmaf_rn(op[r][4 * i + t], x[cc][t], acc[r][cc]);
        }
#pragma unroll
        for (int h = 0; h < NG; ++h) {
            float* yp = Y + c * ST + rl + h * (NV / CB);
            float* cp = comp + c * ST + rl + h * (NV / CB);
            const float yo = ONE ? y0 : *yp;
            float carry = ONE ? carry0 : *cp;
            float v[NV];
#pragma unroll
            for (int k = 0; k < NV; ++k) v[k] = acc[h * (NV / CB) + k / CB][k % CB];
            int vi;
            bool active;
            float inc = reduce_scatter16<float, NV>(v, j, vi, active);
            if constexpr (FORCED) inc = __fmaf_rn(g[h], f[c], inc);
            if constexpr (XR) inc = inc + xr[h];
            inc = inc * dt;
            const float y = kahan_add(yo, inc, carry);
            if constexpr (ONE) {
                y0 = y;
                carry0 = carry;
                if (active) *yp = y;
            } else {
                *yp = y;
                *cp = carry;
            }
        }
    }
}

// Receiver traces of the block's ncol columns (ST apart) in tiles of 4 receivers
// x 4 columns, of a one-column block in tiles of 8 receivers (Kp = 128, us a step
// with 4 x 4 / 8 x 1: 1000 receivers, read from global memory, on every step
// 16.4 / 6.9, 64 receivers 1.35 / 0.81).
template <int ST, int CB>
__device__ __forceinline__ void cta_traces(const float* C, const float* V, int Kp, int R, int ncol, int warp, int lane,
                                           float* out) {
    constexpr int kWarps = kThreads / 32;
    if constexpr (CB == 1) {
        for (int j0 = 8 * warp; j0 < R; j0 += 8 * kWarps)
            trace_tile<8, 1, float>(C, Kp, j0, R, 1, lane, out, R,
                                    [&](int, int kq, float (&x)[4]) { load4(V + 4 * kq, x); });
    } else {
        const int tcn = (ncol + 3) >> 2, ntile = ((R + 3) >> 2) * tcn;
        for (int t = warp; t < ntile; t += kWarps) {
            const int tj = t / tcn, c0 = 4 * (t - tj * tcn), nc = ncol - c0;
            trace_tile<4, 4, float>(
                C, Kp, 4 * tj, R, nc, lane, out + (size_t)c0 * R, R,
                [&](int c, int kq, float (&x)[4]) { load4(V + (c0 + min(c, nc - 1)) * ST + 4 * kq, x); });
        }
    }
}

template <int KI, int CB, bool XR>
__global__ void __launch_bounds__(kThreads, 1) rank2_cta_kernel(const Rank2Args a) {
    constexpr int NT = kThreads, Kp = 64 * KI, ST = Kp + kCtaPad;
    constexpr int RT = 4 * KI;                      // rows per thread
    constexpr int NV = CtaTile<RT, CB>::NV, NG = CtaTile<RT, CB>::NG;
    const int Wa = a.Wa, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j = lane & 15, row = (warp * 2 + (lane >> 4)) * RT;
    const int c0 = (int)blockIdx.x * a.Wv;          // first column of the block
    const int ncol = min(a.Wv, a.M - c0);
    const int gc0 = a.col_base + c0;
    const float dt = (float)a.dt;
    extern __shared__ __align__(16) unsigned char smem[];
    const int nC = a.c_global || !a.traces ? 0 : a.R;
    const CtaSmem L = cta_smem_layout(Wa, Kp, nC);
    float* V = reinterpret_cast<float*>(smem + L.V);      // [Wa][ST]
    float* S = reinterpret_cast<float*>(smem + L.S);
    float* cV = reinterpret_cast<float*>(smem + L.cV);
    float* cS = reinterpret_cast<float*>(smem + L.cS);
    float* Cs = reinterpret_cast<float*>(smem + L.C);     // [R][Kp]
    float* ftab = reinterpret_cast<float*>(smem + L.f);   // [kCtaTab][Wa]
    double* Tpre = reinterpret_cast<double*>(smem + L.Tpre);  // [Wa][-1.5 T, pi / T]
    float* Vg = static_cast<float*>(a.V);
    float* Sg = static_cast<float*>(a.S);
    float* cVg = static_cast<float*>(a.compV);
    float* cSg = static_cast<float*>(a.compS);
    for (int idx = tid; idx < Wa * Kp; idx += NT) {
        const int c = idx / Kp, k = idx % Kp;
        const bool okv = c < ncol && k < a.Kv, oks = c < ncol && k < a.Ks;
        const size_t iv = (size_t)(gc0 + c) * a.Kv + k, is = (size_t)(gc0 + c) * a.Ks + k;
        V[c * ST + k] = okv ? Vg[iv] : 0.f;
        S[c * ST + k] = oks ? Sg[is] : 0.f;
        cV[c * ST + k] = okv && cVg ? cVg[iv] : 0.f;
        cS[c * ST + k] = oks && cSg ? cSg[is] : 0.f;
    }
    const float* Cg = static_cast<const float*>(a.C_p);
    for (int idx = tid; idx < nC * Kp; idx += NT) Cs[idx] = Cg[idx];
    const float* Crows = nC > 0 ? Cs : Cg;
    const float* Tper = static_cast<const float*>(a.Tper);
    for (int c = tid; c < Wa; c += NT) {
        const double T = Tper && c < ncol ? (double)Tper[gc0 + c] : 1.0;
        Tpre[2 * c] = -1.5 * T;
        Tpre[2 * c + 1] = 3.14159265358979323846 / T;
    }
    float opA[RT][4 * KI], opB[RT][4 * KI];
    cta_load_op<KI, RT>(opA, static_cast<const float*>(a.Avs_rm), row, j);
    cta_load_op<KI, RT>(opB, static_cast<const float*>(a.Asv_rm), row, j);
    const int slot = rs16_slot<NV>(j), own = row + slot / CB;  // this lane's first row
    float g[NG];
#pragma unroll
    for (int h = 0; h < NG; ++h) g[h] = static_cast<const float*>(a.g_p)[own + h * (NV / CB)];
    const float* Xv = XR && a.Xv ? static_cast<const float*>(a.Xv) + (size_t)gc0 * a.Kv : nullptr;
    const float* Xs = XR && a.Xs ? static_cast<const float*>(a.Xs) + (size_t)gc0 * a.Ks : nullptr;
    float* traces = static_cast<float*>(a.traces);
    const float* ftg = static_cast<const float*>(a.ftab);
    __syncthreads();
    const int e0 = (slot % CB) * ST + own;          // its element when CB < 4
    float yV = V[e0], kV = cV[e0], yS = S[e0], kS = cS[e0];
    int rec = 0, to_rec = a.r;                      // steps until the next record
    for (int n = 0; n < a.nsteps; ++n) {
        const int nt = n % kCtaTab;
        if (nt == 0) {
            // the last readers of the table are behind the barrier that ended step n - 1
            for (int idx = tid; idx < kCtaTab * Wa; idx += NT) {
                const int s = idx / Wa, c = idx - s * Wa;
                float f = 0.f;
                if (n + s < a.nsteps && c < ncol) {
                    if (ftg) f = ftg[(size_t)(n + s) * a.Mtot + gc0 + c];
                    else if (Tper) f = wavelet_eval_pre(a.wavelet, a.n0 + n + s, a.dt, Tpre[2 * c], Tpre[2 * c + 1]);
                }
                ftab[idx] = f;
            }
            __syncthreads();
        }
        cta_half<KI, RT, CB, true, XR>(opA, S, V, cV, yV, kV, g, ftab + nt * Wa, dt, Wa, row, j, Xv, a.Kv, ncol);
        __syncthreads();
        cta_half<KI, RT, CB, false, XR>(opB, V, S, cS, yS, kS, g, nullptr, dt, Wa, row, j, Xs, a.Ks, ncol);
        if (traces && --to_rec == 0) {
            cta_traces<ST, CB>(Crows, V, Kp, a.R, ncol, warp, lane, traces + ((size_t)rec * a.Mtot + gc0) * a.R);
            to_rec = a.r;
            ++rec;
        }
        __syncthreads();
    }
    if (CB < 4) {
        cV[e0] = kV;                                // (the lanes that share an element hold the same value)
        cS[e0] = kS;
        __syncthreads();
    }
    int bad = 0;
    for (int idx = tid; idx < ncol * Kp; idx += NT) {
        const int c = idx / Kp, k = idx % Kp;
        if (k < a.Kv) {
            const size_t i = (size_t)(gc0 + c) * a.Kv + k;
            Vg[i] = V[c * ST + k];
            if (cVg) cVg[i] = cV[c * ST + k];
            bad |= !is_finite(V[c * ST + k]);
        }
        if (k < a.Ks) {
            const size_t i = (size_t)(gc0 + c) * a.Ks + k;
            Sg[i] = S[c * ST + k];
            if (cSg) cSg[i] = cS[c * ST + k];
            bad |= !is_finite(S[c * ST + k]);
        }
    }
    bad = __syncthreads_or(bad);
    if (bad && tid == 0 && a.status) atomicCAS(a.status, 0, 6 /* ROM_E_NONFINITE */);
}

}  // namespace romk
