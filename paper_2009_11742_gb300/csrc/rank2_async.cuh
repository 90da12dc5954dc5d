// One-block cluster kernel with asynchronous exchange: the rank-2 leapfrog of
// few columns per cluster (FP32, Kp <= 512; FP64, Kp <= 256).
//
// The schedule is the one-block kernel's (rank2_simt.cuh): a cluster of
// Kp / 32 CTAs owns a column block, CTA `rank` owns rows [32 rank, 32 rank + 32)
// of V and S, holds those rows of both operators in registers and full copies
// of the block's V and S in shared memory.  There a half-step ended with a
// block barrier, a loop of remote stores over the peers and a cluster barrier,
// 1.1 us or more of waiting per half-step whatever the work.  Here a warp
// sends its 4 rows of a column group to every CTA (its own too) with
// st.async as soon as it has them, which counts the bytes on the receiver's
// mbarrier of that group; a warp waits for a group's operand on that mbarrier
// alone.  No barrier stands in the step.  The columns go through in groups of
// CB, so with several groups one group's exchange runs behind another's
// products.
//
// Order.  A CTA's copy of V is overwritten by V^{n+2} only after its sender
// has received S^{n+1} from every warp of the cluster, and a warp sends its
// S^{n+1} only after it has read V^{n+1} (products, traces); the same holds
// with V and S exchanged.  So one buffer each suffices, an mbarrier's phase
// n + 1 receives no bytes before its phase n was waited for by every warp, and
// the rows a warp adds to are overwritten by its own stores alone.  Every wait
// is bounded; one that runs out stops the CTA at the next refill of the
// forcing table, reports ROM_E_TIMEOUT, and the final drain retires the bytes
// that will not come, so that no store is in flight when a CTA exits.
//
// Sums, reductions and epilogue are the split kernel's and the one-block
// kernel's, value for value: thread (row pair, chunk j) sums k = 64 i + 4 j + t,
// the 16 chunk lanes meet in the same butterfly.
//
// Bound: the exchange and the chain of a half-step (operand reads, products,
// reduction, update) while a cluster has few columns in FP32, shared-memory
// reads and FMA issue with more; FP64 by the SMs' two FP64 lanes (16 product,
// 4 reduction and 2 epilogue operations a thread and half-step at Kp = 128).
// us a step, before (one-block kernel, two-block kernel for FP32 with M > 1)
// and now: rank-1 FP32 K = 256 2.52 -> 0.90, K = 512 2.88 -> 1.30; FP32 K = 512
// M = 14 4.02 -> 1.90, M = 28 4.02 -> 2.37; FP64 K = 64 M = 16 4.75 -> 2.86,
// K = 128 M = 16 5.84 -> 3.87, M = 512 46.5 -> 40.2, K = 256 M = 512 175.8 -> 161.3
// (all with a few traces).
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "cluster_mbar.cuh"
#include "dev_common.cuh"
#include "rank2_simt.cuh"
#include "rank2_split.cuh"
#include "rom_internal.h"

namespace romk {

constexpr int kAsyncTab = 32;     // steps of forcing tabulated at a time
constexpr int kAsyncMaxCs = 16;   // CTAs per cluster, at most

struct AsyncSmem {
    size_t V, S, cV, cS, C, f, Tpre, g, mbar, sent, flag, total;
};

// W columns in G groups; nC receiver rows staged in shared memory.
template <typename T>
__host__ __device__ inline AsyncSmem async_smem_layout(int W, int G, int Kp, int nC) {
    AsyncSmem s{};
    const size_t carry = sizeof(T) == 4 ? align16((size_t)W * kRowsPerCta * sizeof(float)) : 0;
    size_t o = 0;
    s.V = o;    o += align16((size_t)W * Kp * sizeof(T));
    s.S = o;    o += align16((size_t)W * Kp * sizeof(T));
    s.cV = o;   o += carry;
    s.cS = o;   o += carry;
    s.C = o;    o += align16((size_t)nC * Kp * sizeof(T));
    s.f = o;    o += align16((size_t)kAsyncTab * W * sizeof(T));
    s.Tpre = o; o += sizeof(T) == 4 ? align16((size_t)2 * W * sizeof(double)) : 0;
    s.g = o;    o += align16((size_t)kRowsPerCta * sizeof(T));
    s.mbar = o; o += align16((size_t)2 * G * sizeof(unsigned long long));  // [V, S][G]
    // armed phases [2][G], bytes sent [2][G], bytes each CTA sent here [cs][2][G]
    s.sent = o; o += align16((size_t)(2 + kAsyncMaxCs) * 2 * G * sizeof(unsigned));
    s.flag = o; o += 16;
    s.total = o;
    return s;
}

// The lane offset (bits 2 and 1) that holds column cc of a group after the
// reduce-scatter of 2 CB values; row r of the warp's four is at 8 r + offset.
template <int CB>
__device__ __forceinline__ int async_col_lane(int cc) {
    return CB == 4 ? 4 * (cc >> 1) + 2 * (cc & 1) : (CB == 2 ? 4 * cc : 0);
}

// The warp's 4 rows of the group's CB columns to every CTA of the cluster:
// lane l carries unit (l mod U) ^ z of the piece to peers l / U, l / U + 32 / U, ...;
// dst and bar are own addresses (the piece, the group's mbarrier), dpeer the
// distance of those peers' windows.
template <int CB, int NP>
__device__ __forceinline__ void async_send(float y, unsigned dst, unsigned bar, int z, const unsigned (&dpeer)[NP],
                                           int lane, int npeer) {
    constexpr int U = CB;
    const int p = lane & (U - 1), o = async_col_lane<CB>(p ^ z);
    float v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) v[r] = __shfl_sync(0xffffffffu, y, 8 * r + o);
#pragma unroll
    for (int m = 0; m < NP; ++m)
        if (lane / U + m * (32 / U) < npeer)
            asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                         ::"r"(dst + 16u * p + dpeer[m]), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]),
                         "r"(bar + dpeer[m])
                         : "memory");
}
template <int CB, int NP>
__device__ __forceinline__ void async_send(double y, unsigned dst, unsigned bar, int z, const unsigned (&dpeer)[NP],
                                           int lane, int npeer) {
    constexpr int U = 2 * CB;
    const int p = lane & (U - 1), u = p ^ z, o = 16 * (u & 1) + async_col_lane<CB>(u >> 1);
    const double a = __shfl_sync(0xffffffffu, y, o), b = __shfl_sync(0xffffffffu, y, o + 8);
#pragma unroll
    for (int m = 0; m < NP; ++m)
        if (lane / U + m * (32 / U) < npeer)
            asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];"
                         ::"r"(dst + 16u * p + dpeer[m]), "l"(__double_as_longlong(a)),
                         "l"(__double_as_longlong(b)), "r"(bar + dpeer[m])
                         : "memory");
}

// op . X of the thread's two rows and CB columns, reduced over the 16 chunk
// lanes; vi is the value (row CB + column) this lane is left with.
template <typename T, int KI, int CB>
__device__ __forceinline__ T async_product(const T (&op)[2][4 * KI], const T* X, int j, int& vi, bool& active) {
    T acc[2][CB];
#pragma unroll
    for (int cc = 0; cc < CB; ++cc) acc[0][cc] = acc[1][cc] = T(0);
#pragma unroll
    for (int i = 0; i < KI; ++i) {
        T x[CB][4];
#pragma unroll
        for (int cc = 0; cc < CB; ++cc) AsyncLayout<T, CB>::load(X + 64 * CB * i, cc, j, x[cc]);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int cc = 0; cc < CB; ++cc) {
                acc[0][cc] = fmadd(op[0][4 * i + q], x[cc][q], acc[0][cc]);
                acc[1][cc] = fmadd(op[1][4 * i + q], x[cc][q], acc[1][cc]);
            }
    }
    T v[2 * CB];
#pragma unroll
    for (int cc = 0; cc < CB; ++cc) {
        v[cc] = acc[0][cc];
        v[CB + cc] = acc[1][cc];
    }
    return reduce_scatter16<T, 2 * CB>(v, j, vi, active);
}

__device__ __forceinline__ float state_add(float y, float inc, float& carry) { return kahan_add(y, inc, carry); }
__device__ __forceinline__ double state_add(double y, double inc, float&) { return y + inc; }

// Source signal of step n (FP32: from the column's -1.5 T and pi / T).
__device__ __forceinline__ float async_wavelet(const Rank2Args& a, int n, const double* pre, float) {
    return wavelet_eval_pre(a.wavelet, a.n0 + n, a.dt, pre[0], pre[1]);
}
__device__ __forceinline__ double async_wavelet(const Rank2Args& a, int n, const double*, double T) {
    return wavelet_eval(a.wavelet, a.n0 + n, a.dt, T);
}

// Receiver traces of the first nc columns of group X for this CTA's nj rows of
// C: one dot product per warp at a time, or with many of them (in FP32 with 4
// columns: more than warps; MANY) a tile of 4 receivers x CB columns (the same
// values: lanes sum the same stripes and meet in the same order).
template <typename T, int CB, bool MANY>
__device__ __forceinline__ void async_traces(const T* C, const T* X, int Kp, int nj, int nc, int warp, int lane,
                                             T* out, int R) {
    using Lay = AsyncLayout<T, CB>;
    constexpr int kWarps = kThreads / 32;
    if (MANY || (sizeof(T) == 4 && CB == 4 && nj * nc > kWarps)) {
        for (int j0 = 4 * warp; j0 < nj; j0 += 4 * kWarps) trace_group<T, CB>(C, X, Kp, j0, nj, nc, lane, out, R);
        return;
    }
    for (int pr = warp; pr < nj * nc; pr += kWarps) {
        const int jj = pr / nc, c = pr - jj * nc;
        T acc = T(0);
        for (int k = 4 * lane; k < Kp; k += 128) {
            T cx[4], vx[4];
            load4(C + (size_t)jj * Kp + k, cx);
            Lay::load(X, c, k >> 2, vx);
#pragma unroll
            for (int q = 0; q < 4; ++q) acc = fmadd(cx[q], vx[q], acc);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) out[(size_t)c * R + jj] = acc;
    }
}

// MANY: the form for many receivers (async_many).  An instance of its own, since
// the other trace code alone makes the compiler lay out the whole step
// differently (K = 192, 28 columns, no traces: 0.86 -> 0.92 us a step).
template <typename T, int KI, int CB, bool MANY>
__global__ void __launch_bounds__(kThreads, 1) rank2_async_kernel(const Rank2Args a) {
    using Lay = AsyncLayout<T, CB>;
    constexpr int Kp = 64 * KI, NV = 2 * CB;
    constexpr int kGroup = Kp * CB;                                     // elements of a group's V or S
    constexpr int NP = (2 * KI * Lay::U + 31) / 32;                     // peers a lane sends to
    constexpr unsigned kGroupBytes = (unsigned)(kGroup * sizeof(T));    // one group's V or S
    constexpr unsigned kWarpBytes = (unsigned)(4 * CB * sizeof(T));     // a warp's part of it
    cg::cluster_group cluster = cg::this_cluster();
    const int cs = (int)cluster.num_blocks(), crank = (int)cluster.block_rank();
    const int W = a.Wa, G = W / CB, N = a.nsteps;
    const int col0 = (int)(blockIdx.x / cs) * a.Wv;
    const int ncol = min(a.Wv, a.M - col0), gc0 = a.col_base + col0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, j = lane & 15;
    const int row0 = crank * kRowsPerCta;
    const T dt = (T)a.dt;
    extern __shared__ __align__(16) unsigned char smem[];
    const int nC = a.c_global || !a.traces ? 0 : a.rpc;
    const AsyncSmem L = async_smem_layout<T>(W, G, Kp, nC);
    T* Vf = reinterpret_cast<T*>(smem + L.V);             // [G] groups (AsyncLayout)
    T* Sf = reinterpret_cast<T*>(smem + L.S);
    float* cV = reinterpret_cast<float*>(smem + L.cV);    // [W][32] carries of the own rows (FP32)
    float* cS = reinterpret_cast<float*>(smem + L.cS);
    T* Cs = reinterpret_cast<T*>(smem + L.C);             // [rpc][Kp]
    T* ftab = reinterpret_cast<T*>(smem + L.f);           // [kAsyncTab][W]
    double* Tpre = reinterpret_cast<double*>(smem + L.Tpre);  // [W][-1.5 T, pi / T] (FP32)
    T* gown = reinterpret_cast<T*>(smem + L.g);           // [32]
    unsigned long long* mbar = reinterpret_cast<unsigned long long*>(smem + L.mbar);
    unsigned* armed = reinterpret_cast<unsigned*>(smem + L.sent);  // [2 G]
    unsigned* sent_out = armed + 2 * G;                            // [2 G]
    unsigned* sent_in = sent_out + 2 * G;                          // [cs][2 G]
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L.flag);

    T* Vg = static_cast<T*>(a.V);
    T* Sg = static_cast<T*>(a.S);
    float* cVg = static_cast<float*>(a.compV);
    float* cSg = static_cast<float*>(a.compS);
    for (int idx = tid; idx < W * Kp; idx += kThreads) {
        const int c = idx / Kp, k = idx % Kp;
        const int e = (c / CB) * kGroup + Lay::at(c % CB, k);
        Vf[e] = c < ncol && k < a.Kv ? Vg[(size_t)(gc0 + c) * a.Kv + k] : T(0);
        Sf[e] = c < ncol && k < a.Ks ? Sg[(size_t)(gc0 + c) * a.Ks + k] : T(0);
    }
    if constexpr (sizeof(T) == 4) {
        for (int idx = tid; idx < W * kRowsPerCta; idx += kThreads) {
            const int c = idx / kRowsPerCta, row = row0 + idx % kRowsPerCta;
            cV[idx] = cVg && c < ncol && row < a.Kv ? cVg[(size_t)(gc0 + c) * a.Kv + row] : 0.f;
            cS[idx] = cSg && c < ncol && row < a.Ks ? cSg[(size_t)(gc0 + c) * a.Ks + row] : 0.f;
        }
    }
    // this CTA's receivers [jr0, jr0 + nj)
    const int jr0 = crank * a.rpc, nj = a.traces ? max(0, min(a.rpc, a.R - jr0)) : 0;
    const T* Cg = static_cast<const T*>(a.C_p) + (size_t)jr0 * Kp;
    for (int idx = tid; idx < (nC > 0 ? nj * Kp : 0); idx += kThreads) Cs[idx] = Cg[idx];
    const T* Crows = nC > 0 ? Cs : Cg;
    if (tid < kRowsPerCta) gown[tid] = static_cast<const T*>(a.g_p)[row0 + tid];
    const T* Tper = static_cast<const T*>(a.Tper);
    if constexpr (sizeof(T) == 4) {
        for (int c = tid; c < W; c += kThreads) {
            const double T0 = Tper && c < ncol ? (double)Tper[gc0 + c] : 1.0;
            Tpre[2 * c] = -1.5 * T0;
            Tpre[2 * c + 1] = 3.14159265358979323846 / T0;
        }
    }
    if (tid == 0) {
        *abort_flag = 0;
        for (int i = 0; i < 2 * G; ++i) {
            mbar_init(&mbar[i], 1u);
            armed[i] = 1u;
            sent_out[i] = 0u;
        }
        fence_mbar_init_cluster();
        for (int i = 0; i < 2 * G; ++i) mbar_arrive_expect_tx(&mbar[i], kGroupBytes);
    }
    T opA[2][4 * KI], opB[2][4 * KI];
    const int rp = warp * 2 + (lane >> 4);
    load_op_rows<T, KI>(opA, static_cast<const T*>(a.Avs_rm), Kp, row0 + 2 * rp, j);
    load_op_rows<T, KI>(opB, static_cast<const T*>(a.Asv_rm), Kp, row0 + 2 * rp, j);
    // the value this lane is left with: own row rl, column cl of a group
    const int slot = rs16_slot<NV>(j), rl = 2 * rp + slot / CB, cl = slot % CB;
    const int own = Lay::at(cl, row0 + rl);               // its element in a group
    // the warp's piece of a group's V and S, and where the peers' windows lie
    const int kqw = (row0 >> 2) + warp, zw = Lay::swz(kqw);
    const unsigned base = smem_addr(smem), piece = (unsigned)(kqw * Lay::U * 16);
    const unsigned mV = base + (unsigned)L.V + piece, mS = base + (unsigned)L.S + piece, mB = smem_addr(mbar);
    unsigned dpeer[NP];
#pragma unroll
    for (int m = 0; m < NP; ++m) {
        const int peer = lane / Lay::U + m * (32 / Lay::U);
        dpeer[m] = cluster_addr(base, peer < cs ? peer : crank) - base;
    }
    const T* ftg = static_cast<const T*>(a.ftab);
    T* traces = static_cast<T*>(a.traces);
    const T* Xv = static_cast<const T*>(a.Xv);
    const T* Xs = static_cast<const T*>(a.Xs);
    // every CTA's buffers and mbarriers are there before a peer writes to them
    cluster.sync();

    const int npeer = a.debug_skip_push && crank == 0 ? 0 : cs;  // fault injection: this CTA sends nothing
    // a wait of the whole warp; false when it ran out here or in another warp
    auto wait = [&](int b, unsigned parity) {
        const bool ok = mbar_wait_bounded(&mbar[b], parity, a.spin_limit, abort_flag);
        return __all_sync(0xffffffffu, ok) != 0;
    };
    // this warp's sends: nV steps of V in the groups below gV, one less from there on; S alike
    int nV = 0, nS = 0, gV = G, gS = G;
    bool dead = false;
    int rec = 0, to_rec = a.r;
    for (int nb = 0; nb < N; nb += kAsyncTab) {
        // (the barrier also keeps the last table until every warp has read it)
        if (__syncthreads_or(dead)) break;
        for (int idx = tid; idx < kAsyncTab * W; idx += kThreads) {
            const int s = idx / W, c = idx - s * W;
            T f = T(0);
            if (nb + s < N && c < ncol) {
                if (ftg) f = ftg[(size_t)(nb + s) * a.Mtot + gc0 + c];
                else if (Tper) f = async_wavelet(a, nb + s, Tpre + 2 * c, Tper[gc0 + c]);
            }
            ftab[idx] = f;
        }
        __syncthreads();
        const int ne = min(N, nb + kAsyncTab);
        for (int n = nb; n < ne && !dead; ++n) {
            // ---- V += dt (Avs S + g f^T [+ Xv])
            for (int g = 0; g < G; ++g) {
                const int c = g * CB + cl;
                float* cp = cV + c * kRowsPerCta + rl;
                const T y0 = Vf[g * kGroup + own], gr = gown[rl], f = ftab[(n - nb) * W + c];
                float carry = sizeof(T) == 4 ? *cp : 0.f;
                T xr = T(0);
                if (Xv && c < ncol && row0 + rl < a.Kv) xr = Xv[(size_t)(gc0 + c) * a.Kv + row0 + rl];
                if (n > 0) {
                    if (!wait(G + g, (unsigned)((n - 1) & 1))) {
                        dead = true;
                        nV = n + 1, gV = g, nS = n;
                        break;
                    }
                    if (tid == 0) {
                        mbar_arrive_expect_tx(&mbar[G + g], kGroupBytes);
                        armed[G + g] += 1u;
                    }
                }
                int vi;
                bool active;
                T inc = async_product<T, KI, CB>(opA, Sf + g * kGroup, j, vi, active);
                inc = fmadd(gr, f, inc);
                if (Xv) inc = inc + xr;
                inc = inc * dt;
                const T y = state_add(y0, inc, carry);
                if (sizeof(T) == 4 && active) *cp = carry;
                async_send<CB>(y, mV + (unsigned)g * kGroupBytes, mB + 8u * (unsigned)g, zw, dpeer, lane, npeer);
            }
            if (dead) break;
            // ---- S += dt (Asv V [+ Xs]) with the new V, and its traces
            const bool record = traces && --to_rec == 0;
            for (int g = 0; g < G; ++g) {
                const int c = g * CB + cl;
                float* cp = cS + c * kRowsPerCta + rl;
                const T y0 = Sf[g * kGroup + own];
                float carry = sizeof(T) == 4 ? *cp : 0.f;
                T xr = T(0);
                if (Xs && c < ncol && row0 + rl < a.Ks) xr = Xs[(size_t)(gc0 + c) * a.Ks + row0 + rl];
                if (!wait(g, (unsigned)(n & 1))) {
                    dead = true;
                    nV = n + 1, nS = n + 1, gS = g;
                    break;
                }
                if (tid == 0 && n + 1 < N) {
                    mbar_arrive_expect_tx(&mbar[g], kGroupBytes);
                    armed[g] += 1u;
                }
                int vi;
                bool active;
                const T* Vc = Vf + g * kGroup;
                T inc = async_product<T, KI, CB>(opB, Vc, j, vi, active);
                if (Xs) inc = inc + xr;
                inc = inc * dt;
                const T y = state_add(y0, inc, carry);
                if (sizeof(T) == 4 && active) *cp = carry;
                if (record)  // before this warp's S lets V be overwritten
                    async_traces<T, CB, MANY>(Crows, Vc, Kp, nj, min(CB, ncol - g * CB), warp, lane,
                                    traces + ((size_t)rec * a.Mtot + gc0 + g * CB) * a.R + jr0, a.R);
                __syncwarp();
                async_send<CB>(y, mS + (unsigned)g * kGroupBytes, mB + 8u * (unsigned)(G + g), zw, dpeer, lane, npeer);
            }
            if (record) {
                to_rec = a.r;
                ++rec;
            }
        }
        if (!dead) nV = nS = ne;
    }
    // the last S has arrived, too
    if (!dead && nS == N)
        for (int g = 0; g < G && !dead; ++g) dead = !wait(G + g, (unsigned)((N - 1) & 1));
    if (dead && lane == 0) *abort_flag = 1;
    // ---- drain (see the split kernel): every CTA tells every other how many
    // bytes it sent per mbarrier, and each retires on the phase armed last those
    // that will not come; after a complete run nothing is outstanding.
    if (lane == 0 && npeer > 0) {
        for (int g = 0; g < G; ++g) {
            atomicAdd(&sent_out[g], kWarpBytes * (unsigned)(nV - (g >= gV ? 1 : 0)));
            atomicAdd(&sent_out[G + g], kWarpBytes * (unsigned)(nS - (g >= gS ? 1 : 0)));
        }
    }
    __syncthreads();
    for (int idx = tid; idx < cs * 2 * G; idx += kThreads) {
        const int d = idx / (2 * G), b = idx - d * 2 * G;
        asm volatile("st.shared::cluster.u32 [%0], %1;"
                     ::"r"(cluster_addr(smem_addr(sent_in + crank * 2 * G + b), d)), "r"(sent_out[b])
                     : "memory");
    }
    cluster.sync();
    if (tid == 0) {
        bool late = false;
        for (int b = 0; b < 2 * G; ++b) {
            unsigned got = 0u;
            for (int d = 0; d < cs; ++d) got += sent_in[d * 2 * G + b];
            const unsigned expect = armed[b] * kGroupBytes;
            if (expect != got) mbar_complete_tx(&mbar[b], expect - got);
            const unsigned parity = (armed[b] - 1u) & 1u;
            const long long t0 = clock64();
            while (!mbar_try_wait(&mbar[b], parity)) {
                if (clock64() - t0 > 4000000000LL) {
                    late = true;
                    break;
                }
            }
        }
        if ((late || *abort_flag) && a.status) atomicCAS(a.status, 0, 5 /* ROM_E_TIMEOUT */);
    }
    __syncthreads();
    // ---- write back this CTA's rows and carries
    int bad = 0;
    for (int idx = tid; idx < ncol * kRowsPerCta; idx += kThreads) {
        const int c = idx / kRowsPerCta, row = row0 + idx % kRowsPerCta;
        const int e = (c / CB) * kGroup + Lay::at(c % CB, row);
        if (row < a.Kv) {
            const T x = Vf[e];
            Vg[(size_t)(gc0 + c) * a.Kv + row] = x;
            if (sizeof(T) == 4 && cVg) cVg[(size_t)(gc0 + c) * a.Kv + row] = cV[idx];
            bad |= !is_finite(x);
        }
        if (row < a.Ks) {
            const T x = Sf[e];
            Sg[(size_t)(gc0 + c) * a.Ks + row] = x;
            if (sizeof(T) == 4 && cSg) cSg[(size_t)(gc0 + c) * a.Ks + row] = cS[idx];
            bad |= !is_finite(x);
        }
    }
    bad = __syncthreads_or(bad);
    if (bad && tid == 0 && a.status) atomicCAS(a.status, 0, 6 /* ROM_E_NONFINITE */);
}

}  // namespace romk
