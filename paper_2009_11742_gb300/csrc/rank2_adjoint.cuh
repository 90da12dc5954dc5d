// Reverse-time adjoint of the rank-2 leapfrog for the receiver-trace misfit
//     L = sum_{n=1..N} sum_m || C V_m^n - ystar_m^n ||^2 .
// The paper has no adjoint; this is the exact reverse of the forward step
// V^{n+1} = V^n + dt (Avs S^n + g f_n^T), S^{n+1} = S^n + dt Asv V^{n+1}
// (Sec. 3.1).  With lamV, lamS the adjoints of (V, S), reverse step n
// (n = N-1 .. 0) is
//     half A:  lamV <- lamV + 2 C^T r^{n+1} + dt Asv^T lamS      (= a_V^n)
//              dL/dT_m += dt g^T a_V^n[:, m] df/dT(t_n; T_m)
//     half B:  lamS <- lamS + dt Avs^T a_V^n
// with r^n = C V^n - ystar^n, starting from lamV = lamS = 0; after n = 0,
// lamV = dL/dV^0 and lamS = dL/dS^0.
//
// The kernel is the one-block cluster kernel of rank2_simt.cuh run backwards
// in time with the transposed operators (the column-major copies of Asv and
// Avs are the row-major Asv^T and Avs^T).  FP32: resident in registers up to
// Kp = 512 (one 32-row tile per CTA), and for 512 < Kp <= 1024 read from L2
// for each of the CTA's two 32-row tiles every half-step, as the forward
// kernel does there; the adjoint state is Kahan-compensated.  FP64 (the
// check path, Kp <= 512, one tile per CTA): resident up to Kp = 256 and
// read from L2 per half-step above, plain sums, as the FP64 forward kernel.
// Half A's epilogue adds the rank-R source 2 C^T r^{n+1}, read precomputed
// for the launch's range of steps (adj_source_kernel) and copied one step
// ahead.  A deterministic per-CTA column reduction accumulates the period
// gradient.  The split-role kernel below (FP32, Kp <= 512) is the faster
// form there.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "dev_common.cuh"
#include "rank2_simt.cuh"
#include "rank2_split.cuh"
#include "rom_internal.h"

namespace romk {

// Steps of df/dT tabulated at a time (shared memory, kAdjTab x Wa values).
constexpr int kAdjTab = 64;

struct AdjSmem {
    size_t Vf, Sf, cV, cS, src, g, T, gT, dfT, total;
};

// nrt: 32-row tiles owned per CTA (1 for Kp <= 512, 2 above); T the element
// type (the carries are FP32 and only the FP32 path has them).  The source
// term arrives precomputed (src: two step buffers of Wa x own rows), so the
// layout does not depend on R.
template <typename T>
__host__ __device__ inline AdjSmem adj_smem_layout(int Wa, int Kp, int R, int nrt = 1) {
    (void)R;
    AdjSmem s{};
    const size_t own = (size_t)nrt * kRowsPerCta;
    const size_t ncarry = sizeof(T) == 4 ? (size_t)Wa * own : 0;
    size_t o = 0;
    s.Vf = o;   o += align16((size_t)Wa * Kp * sizeof(T));
    s.Sf = o;   o += align16((size_t)Wa * Kp * sizeof(T));
    s.cV = o;   o += align16(ncarry * sizeof(float));
    s.cS = o;   o += align16(ncarry * sizeof(float));
    s.src = o;  o += align16(2 * (size_t)Wa * own * sizeof(T));
    s.g = o;    o += align16(own * sizeof(T));
    s.T = o;    o += align16((size_t)Wa * sizeof(T));
    s.gT = o;   o += align16((size_t)Wa * sizeof(T));
    s.dfT = o;  o += align16((size_t)kAdjTab * Wa * sizeof(T));
    s.total = o;
    return s;
}

// Half A of a reverse step on one 32-row tile of the CTA (rows row0 ..):
//   Y_own += dt (op . X) + 2 C_own^T r   (Kahan-compensated in FP32),
// with C_own^T r read precomputed from asrc ([Wa][sstride], the tile's rows).
template <typename T, int KI, int CB>
__device__ __forceinline__ void adj_half_a(const T (&op)[2][4 * KI], const T* __restrict__ X,
                                           T* __restrict__ Y, float* __restrict__ comp,
                                           const T* __restrict__ asrc, const int sstride, const T dt,
                                           const int Wa, const int Kp, const int row0, const int rp,
                                           const int j) {
    for (int c0 = 0; c0 < Wa; c0 += CB) {
        T acc[2][CB];
#pragma unroll
        for (int cc = 0; cc < CB; ++cc) { acc[0][cc] = T(0); acc[1][cc] = T(0); }
#pragma unroll
        for (int i = 0; i < KI; ++i) {
            T x[CB][4];
#pragma unroll
            for (int cc = 0; cc < CB; ++cc) load4(X + (size_t)(c0 + cc) * Kp + 64 * i + 4 * j, x[cc]);
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
        for (int cc = 0; cc < CB; ++cc) { v[cc] = acc[0][cc]; v[CB + cc] = acc[1][cc]; }
        int vi;
        bool active;
        const T tot = reduce_scatter16<T, 2 * CB>(v, j, vi, active);
        if (active) {
            const int rl = 2 * rp + vi / CB;
            const int c = c0 + vi % CB;
            const T inc = fmadd(tot, dt, T(2) * asrc[c * sstride + rl]);
            T* yp = Y + (size_t)c * Kp + row0 + rl;
            if constexpr (sizeof(T) == 4) {
                *yp = kahan_add(*yp, inc, comp[c * kRowsPerCta + rl]);
            } else {
                *yp = *yp + inc;
            }
        }
    }
}

// Half A in the 4-row, 32-lane form of the work-list kernel (FP32 with the
// operators streamed from L2): warp w holds rows 4w .. 4w + 3 of the tile,
// lane l the k values 128 i + 4 l + q (k < Kp); the epilogue adds
// 2 C_own^T r, read precomputed from asrc ([Wa][sstride], the tile's rows).
template <int KQ>
__device__ __forceinline__ void wl_adj_half_a(const float (&op)[4][4 * KQ], const float* __restrict__ X,
                                              float* __restrict__ Y, float* __restrict__ comp,
                                              const float* __restrict__ asrc, const int sstride,
                                              const float dt, const int Wa, const int Kp, const int row0,
                                              const int warp, const int lane) {
    constexpr int CB = 8;
    for (int c0 = 0; c0 < Wa; c0 += CB) {
        float acc[4][CB];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int cc = 0; cc < CB; ++cc) acc[r][cc] = 0.f;
#pragma unroll
        for (int i = 0; i < KQ; ++i) {
            if (128 * i + 4 * lane >= Kp) continue;
            float x[CB][4];
#pragma unroll
            for (int cc = 0; cc < CB; ++cc) load4(X + (size_t)(c0 + cc) * Kp + 128 * i + 4 * lane, x[cc]);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int cc = 0; cc < CB; ++cc)
#pragma unroll
                    for (int r = 0; r < 4; ++r) acc[r][cc] = __fmaf_rn(op[r][4 * i + q], x[cc][q], acc[r][cc]);
        }
        float v[4 * CB];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int cc = 0; cc < CB; ++cc) v[r * CB + cc] = acc[r][cc];
        int vi;
        const float tot = reduce_scatter32(v, lane, vi);
        const int rl = 4 * warp + vi / CB;
        const int c = c0 + vi % CB;
        const float inc = __fmaf_rn(tot, dt, 2.f * asrc[c * sstride + rl]);
        float* yp = Y + (size_t)c * Kp + row0 + rl;
        *yp = kahan_add(*yp, inc, comp[c * kRowsPerCta + rl]);
    }
}

// KI = Kp / 64.  FP32 (GEN, KI <= 16): both halves run in the 4-row form;
// for KI <= 8 each CTA owns one 32-row tile and keeps its rows of both
// transposed operators in registers, above that the Kp / 32 row tiles are
// dealt out to the cluster's CTAs (the first Kp/32 mod cs take one more;
// a.nrt is the most any CTA owns) and the operators are streamed per tile.
// FP64 (KI <= 8): the 2-row form, one tile per CTA, resident for KI <= 4.
template <typename T, int KI, int CB>
__global__ void __launch_bounds__(kThreads, 1) rank2_adjoint_kernel(const AdjArgsT<T> a) {
    constexpr bool F32 = sizeof(T) == 4;
    static_assert(F32 ? KI <= 16 : KI <= 8, "unsupported size");
    constexpr bool GEN = F32;
    static_assert(!GEN || CB == 8, "the 4-row form runs 8-column groups");
    constexpr bool RES = F32 ? KI <= 8 : KI <= 4;
    constexpr int KQ = (KI + 1) / 2;  // GEN: k groups of 128
    cg::cluster_group cluster = cg::this_cluster();
    const int cs = (int)cluster.num_blocks();
    const int crank = (int)cluster.block_rank();
    const int blk = blockIdx.x / cs;
    const int col0 = blk * a.Wv;
    const int ncol = min(a.Wv, a.M - col0);
    const int Wa = a.Wa, Kp = a.Kp, R = a.R;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j = lane & 15;
    const int rp = warp * 2 + (lane >> 4);
    // row tiles: the layout holds NRT per CTA, this CTA owns nrt_own from row0
    const int NRT = GEN ? a.nrt : 1;
    const int OWN = NRT * kRowsPerCta;
    int nrt_own = NRT, row0 = crank * OWN;
    if (GEN) {
        const int tiles = Kp / kRowsPerCta, base = tiles / cs, rem = tiles % cs;
        nrt_own = base + (crank < rem ? 1 : 0);
        row0 = (crank * base + (crank < rem ? crank : rem)) * kRowsPerCta;
    }
    const int own_rows = nrt_own * kRowsPerCta;
    const T dt = (T)a.dt;

    extern __shared__ __align__(16) unsigned char smem[];
    const AdjSmem L = adj_smem_layout<T>(Wa, Kp, R, NRT);
    T* Vf = reinterpret_cast<T*>(smem + L.Vf);
    T* Sf = reinterpret_cast<T*>(smem + L.Sf);
    float* cV = reinterpret_cast<float*>(smem + L.cV);
    float* cS = reinterpret_cast<float*>(smem + L.cS);
    T* srcS = reinterpret_cast<T*>(smem + L.src);   // [2][Wa][OWN]: C^T r, by step parity
    T* gown = reinterpret_cast<T*>(smem + L.g);
    T* Tcol = reinterpret_cast<T*>(smem + L.T);
    T* gTacc = reinterpret_cast<T*>(smem + L.gT);
    T* dfT = reinterpret_cast<T*>(smem + L.dfT);    // [kAdjTab][Wa]: df/dT of the chunk

    for (int idx = tid; idx < Wa * Kp; idx += kThreads) {
        const int c = idx / Kp, k = idx % Kp;
        Vf[idx] = (c < ncol && k < a.Kv) ? a.lamV[(size_t)(col0 + c) * a.Kv + k] : T(0);
        Sf[idx] = (c < ncol && k < a.Ks) ? a.lamS[(size_t)(col0 + c) * a.Ks + k] : T(0);
    }
    // carries (FP32): [row tile][column][32 rows]
    for (int idx = tid; idx < (F32 ? nrt_own * Wa * kRowsPerCta : 0); idx += kThreads) {
        const int rt = idx / (Wa * kRowsPerCta);
        const int rem = idx - rt * Wa * kRowsPerCta;
        const int c = rem / kRowsPerCta, rl = rem % kRowsPerCta, row = row0 + rt * kRowsPerCta + rl;
        cV[idx] = (c < ncol && row < a.Kv) ? a.compV[(size_t)(col0 + c) * a.Kv + row] : 0.f;
        cS[idx] = (c < ncol && row < a.Ks) ? a.compS[(size_t)(col0 + c) * a.Ks + row] : 0.f;
    }
    for (int ro = tid; ro < OWN; ro += kThreads) gown[ro] = ro < own_rows ? a.g_p[row0 + ro] : T(0);
    for (int c = tid; c < Wa; c += kThreads) {
        Tcol[c] = (c < ncol) ? a.Tper[col0 + c] : T(1);
        gTacc[c] = (c < ncol) ? a.gTpart[(size_t)crank * a.M + col0 + c] : T(0);
    }
    T opA[GEN ? 1 : 2][GEN ? 1 : 4 * KI], opB[GEN ? 1 : 2][GEN ? 1 : 4 * KI];
    float opQA[GEN ? 4 : 1][GEN ? 4 * KQ : 1], opQB[GEN ? 4 : 1][GEN ? 4 * KQ : 1];
    if constexpr (GEN) {
        if (RES && nrt_own > 0) {
            wl_load_op<KQ>(opQA, a.opA_rm, Kp, row0 + 4 * warp, lane);
            wl_load_op<KQ>(opQB, a.opB_rm, Kp, row0 + 4 * warp, lane);
        }
    } else if (RES) {
        load_op_rows<T, KI>(opA, a.opA_rm, Kp, row0 + 2 * rp, j);
        load_op_rows<T, KI>(opB, a.opB_rm, Kp, row0 + 2 * rp, j);
    }
    // the own rows' C^T r of reverse step n (precomputed for the range) into
    // step buffer pb, 16 bytes (E rows) per copy, zero for absent columns and rows
    constexpr int E = 16 / (int)sizeof(T);
    auto prefetch_src = [&](int n, int pb) {
        T* dst = srcS + (size_t)pb * Wa * OWN;
        for (int idx = tid; idx < Wa * (OWN / E); idx += kThreads) {
            const int c = idx / (OWN / E), ro = E * (idx % (OWN / E));
            const bool ok = c < ncol && ro < own_rows;
            const T* gsrc = ok ? a.src + ((size_t)(n - a.n_lo) * a.M + col0 + c) * Kp + row0 + ro
                               : a.src;  // a valid address for the zero fill
            cp_async16(dst + (size_t)c * OWN + ro, gsrc, ok ? 16 : 0);
        }
    };
    if (a.n_hi > a.n_lo) prefetch_src(a.n_hi - 1, 0);
    cluster.sync();

    for (int n = a.n_hi - 1; n >= a.n_lo; --n) {
        // df/dT(t_n; T_c) for the next kAdjTab steps, all threads at once: the
        // evaluation (FP64 time arithmetic) stays off the per-step critical
        // path.  The previous chunk's last readers passed the cluster barrier
        // at the end of the previous step; the barrier after the residual
        // below publishes the new entries.
        const int done = a.n_hi - 1 - n;
        if (done % kAdjTab == 0) {
            for (int idx = tid; idx < kAdjTab * ncol; idx += kThreads) {
                const int i = idx / ncol, c = idx % ncol;
                if (n - i >= a.n_lo)
                    dfT[i * Wa + c] = wavelet_dT_eval<T>(a.wavelet, (long long)a.n0 + n - i, a.dt, Tcol[c]);
            }
        }
        const T* dfn = dfT + (done % kAdjTab) * Wa;
        // this step's C^T r, copied one step earlier into buffer done & 1; the
        // next step's copies go to the other buffer, whose last readers passed
        // the cluster barriers of the previous step
        cp_async_wait_all();
        __syncthreads();
        if (n > a.n_lo) prefetch_src(n - 1, (done + 1) & 1);
        // ---- half A: lamV <- lamV + 2 C^T r^{n+1} + dt Asv^T lamS
        for (int rt = 0; rt < nrt_own; ++rt) {
            const int rowt = row0 + rt * kRowsPerCta;
            if constexpr (GEN) {
                if (!RES) wl_load_op<KQ>(opQA, a.opA_rm, Kp, rowt + 4 * warp, lane);
                wl_adj_half_a<KQ>(opQA, Sf, Vf, cV + rt * Wa * kRowsPerCta,
                                  srcS + (size_t)(done & 1) * Wa * OWN + rt * kRowsPerCta, OWN, dt, Wa, Kp,
                                  rowt, warp, lane);
            } else {
                if (!RES) load_op_rows<T, KI>(opA, a.opA_rm, Kp, rowt + 2 * rp, j);
                adj_half_a<T, KI, CB>(opA, Sf, Vf, cV + rt * Wa * kRowsPerCta,
                                      srcS + (size_t)(done & 1) * Wa * OWN + rt * kRowsPerCta, OWN, dt, Wa, Kp,
                                      rowt, rp, j);
            }
        }
        __syncthreads();
        // period gradient: dt (g_own . a_V[:, c]) df/dT(t_n; T_c), fixed reduction order
        for (int c = warp; c < ncol; c += kThreads / 32) {
            T s = T(0);
            if (nrt_own > 0) s = gown[lane] * Vf[(size_t)c * Kp + row0 + lane];
            for (int rt = 1; rt < nrt_own; ++rt)
                s = fmadd(gown[rt * kRowsPerCta + lane], Vf[(size_t)c * Kp + row0 + rt * kRowsPerCta + lane], s);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) gTacc[c] = fmadd(dt * s, dfn[c], gTacc[c]);
        }
        push_own_rows<T>(cluster, Vf, Wa, Kp, row0, cs, crank, nrt_own);
        cluster.sync();
        // ---- half B: lamS <- lamS + dt Avs^T a_V
        for (int rt = 0; rt < nrt_own; ++rt) {
            const int rowt = row0 + rt * kRowsPerCta;
            if constexpr (GEN) {
                if (!RES) wl_load_op<KQ>(opQB, a.opB_rm, Kp, rowt + 4 * warp, lane);
                wl_half_step<KQ, false>(opQB, Vf, Sf, cS + rt * Wa * kRowsPerCta, gown, gown, dt, Wa, Kp, rowt,
                                        warp, lane);
            } else {
                if (!RES) load_op_rows<T, KI>(opB, a.opB_rm, Kp, rowt + 2 * rp, j);
                half_step<T, KI, CB, false>(opB, Vf, Sf, cS + rt * Wa * kRowsPerCta, gown, gown, dt, Wa,
                                            Kp, rowt, rp, j);
            }
        }
        __syncthreads();
        push_own_rows<T>(cluster, Sf, Wa, Kp, row0, cs, crank, nrt_own);
        cluster.sync();
    }

    int bad = 0;
    for (int idx = tid; idx < ncol * own_rows; idx += kThreads) {
        const int c = idx / own_rows, ro = idx % own_rows, row = row0 + ro;
        const int ci = (ro / kRowsPerCta) * Wa * kRowsPerCta + c * kRowsPerCta + ro % kRowsPerCta;
        if (row < a.Kv) {
            const T x = Vf[(size_t)c * Kp + row];
            a.lamV[(size_t)(col0 + c) * a.Kv + row] = x;
            if (F32) a.compV[(size_t)(col0 + c) * a.Kv + row] = cV[ci];
            bad |= !is_finite(x);
        }
        if (row < a.Ks) {
            const T x = Sf[(size_t)c * Kp + row];
            a.lamS[(size_t)(col0 + c) * a.Ks + row] = x;
            if (F32) a.compS[(size_t)(col0 + c) * a.Ks + row] = cS[ci];
            bad |= !is_finite(x);
        }
    }
    for (int c = tid; c < ncol; c += kThreads) a.gTpart[(size_t)crank * a.M + col0 + c] = gTacc[c];
    bad = __syncthreads_or(bad);
    if (bad && tid == 0 && a.status) atomicCAS(a.status, 0, 6 /* ROM_E_NONFINITE */);
}

// ---- split-role reverse kernel (FP32, Kp <= 512).  The reverse step has the
// forward step's shape: half A updates lamV from lamS, half B updates lamS from
// the new lamV.  So the forward split kernel's schedule and exchange
// (rank2_split.cuh) carry over: V-role CTAs hold their 64 rows of Asv^T in
// registers and own those rows of lamV, S-role CTAs do the same with Avs^T and
// lamS, both take the columns in groups of 4, and a group's rows travel by
// st.async, counted on the receiver's mbarrier of the group.  Time runs
// backwards: reverse step k is step n = n_hi - 1 - k.  The V role's update adds
// 2 C^T r, which does not depend on the adjoint state: adj_source_kernel forms
// it for the launch's range of steps beforehand, and a lane fetches its element
// one group ahead.  The S role, whose operand copy holds the new lamV, adds its
// slab's share of the period gradient to a per-CTA partial: a warp takes the
// columns c = warp (mod 8), before its rows of lamS let lamV be overwritten.
// K = 512, M = 128, 256 steps with checkpoints every 64, whole gradient: 5.53 ms
// with a cluster barrier a phase here, 5.03 now.
struct AdjSplitSmem {
    size_t X, own, comp, g, T, gT, dfT, mbar, sent, flag, total;
};

__host__ __device__ inline AdjSplitSmem adj_split_smem_layout(int Wa, int Kp) {
    AdjSplitSmem s{};
    const size_t W = 2 * (size_t)Wa, G = W / kSplitCB, H = (size_t)Kp / kSplitRows;
    size_t o = 0;
    s.X = o;    o += align16(W * Kp * sizeof(float));
    s.own = o;  o += align16(W * kSplitRows * sizeof(float));
    s.comp = o; o += align16(W * kSplitRows * sizeof(float));
    s.g = o;    o += align16((size_t)kSplitRows * sizeof(float));
    s.T = o;    o += align16(W * sizeof(float));
    s.gT = o;   o += align16(W * sizeof(float));
    s.dfT = o;  o += align16((size_t)kAdjTab * W * sizeof(float));
    s.mbar = o; o += align16(G * sizeof(unsigned long long));
    s.sent = o; o += align16((1 + H) * G * sizeof(unsigned));
    s.flag = o; o += 16;
    s.total = o;
    return s;
}

template <int KI>
__global__ void __launch_bounds__(kThreads, 1) rank2_adjoint_split_kernel(const AdjArgsT<float> a) {
    using Lay = AsyncLayout<float, kSplitCB>;
    constexpr int CB = kSplitCB, Kp = 64 * KI, H = KI, cs = 2 * KI;
    constexpr int kGroup = Kp * CB;
    constexpr unsigned kGroupBytes = SplitLink<KI>::kGroupBytes;
    cg::cluster_group cluster = cg::this_cluster();
    const int crank = (int)cluster.block_rank();
    const bool vrole = crank < H;
    const int sl = vrole ? crank : crank - H;  // row slab
    const int row0 = sl * kSplitRows;
    const int peer0 = vrole ? H : 0;           // first CTA of the other role
    const int clu = blockIdx.x / cs;
    const int W = 2 * a.Wa, Gmax = W / CB, M = a.M;
    const int gc0 = 2 * clu * a.Wv, ncol = max(0, min(2 * a.Wv, M - gc0));
    const int G = (ncol + CB - 1) / CB;
    const int N = ncol > 0 ? a.n_hi - a.n_lo : 0;  // reverse steps of this range
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j = lane & 15;
    const int q = warp * 2 + (lane >> 4);      // row quad
    const float dt = (float)a.dt;

    extern __shared__ __align__(16) unsigned char smem[];
    const AdjSplitSmem L = adj_split_smem_layout(a.Wa, Kp);
    float* X = reinterpret_cast<float*>(smem + L.X);         // [G] groups of the operand
    float* own = reinterpret_cast<float*>(smem + L.own);     // [G][warp][lane]: the lane's element of the group
    float* comp = reinterpret_cast<float*>(smem + L.comp);   // its carry
    float* gown = reinterpret_cast<float*>(smem + L.g);      // [64]
    float* Tcol = reinterpret_cast<float*>(smem + L.T);      // [W]
    float* gTacc = reinterpret_cast<float*>(smem + L.gT);    // [W] period-gradient partials
    float* dfT = reinterpret_cast<float*>(smem + L.dfT);     // [kAdjTab][W] df/dT
    unsigned long long* mbar = reinterpret_cast<unsigned long long*>(smem + L.mbar);  // [G]
    unsigned* sent_out = reinterpret_cast<unsigned*>(smem + L.sent);  // [G]
    unsigned* sent_in = sent_out + Gmax;                              // [H][G]
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L.flag);

    const int Kown = vrole ? a.Kv : a.Ks;
    float* own_g = vrole ? a.lamV : a.lamS;
    float* comp_g = vrole ? a.compV : a.compS;
    // operand: V role = the full lamS; the S role's arrives with the first V-role sends
    for (int idx = tid; idx < (vrole ? G * kGroup : 0); idx += kThreads) {
        const int c = idx / Kp, k = idx - c * Kp;
        X[(c / CB) * kGroup + Lay::at(c % CB, k)] =
            c < ncol && k < a.Ks ? a.lamS[(size_t)(gc0 + c) * a.Ks + k] : 0.f;
    }
    auto e_row = [&](int e) { return row0 + 8 * ((e >> 5) % kSplitWarps) + 4 * ((e >> 4) & 1) + ((e >> 2) & 3); };
    auto e_col = [&](int e) { return CB * (e / kThreads) + (e & 3); };
    for (int e = tid; e < G * kThreads; e += kThreads) {
        const int c = e_col(e), row = e_row(e);
        const bool ok = c < ncol && row < Kown;
        own[e] = ok ? own_g[(size_t)(gc0 + c) * Kown + row] : 0.f;
        comp[e] = ok ? comp_g[(size_t)(gc0 + c) * Kown + row] : 0.f;
    }
    if (tid < kSplitRows) gown[tid] = a.g_p[row0 + tid];  // the S role's gradient slab
    for (int c = tid; c < W; c += kThreads) {
        Tcol[c] = c < ncol ? a.Tper[gc0 + c] : 1.f;
        gTacc[c] = c < ncol ? a.gTpart[(size_t)crank * M + gc0 + c] : 0.f;
    }
    if (tid == 0) {
        *abort_flag = 0;
        for (int i = 0; i < Gmax; ++i) {
            sent_out[i] = 0u;
            mbar_init(&mbar[i], 1u);
        }
        fence_mbar_init_cluster();
        for (int i = 0; i < Gmax; ++i) mbar_arrive_expect_tx(&mbar[i], kGroupBytes);
    }
    float op[4][4 * KI];
    load_op_quad<KI>(op, vrole ? a.opA_rm : a.opB_rm, Kp, row0 + 4 * q, j);
    const bool sends = !(a.debug_skip_push && crank == 0);  // fault injection: this CTA sends nothing
    const SplitLink<KI> link(smem_addr(smem), (unsigned)L.X, (unsigned)L.mbar, row0, warp, lane, peer0, sends ? H : 0);
    // this lane's element of C^T r at step n (every row of src is Kp wide)
    const int own_row = row0 + 4 * q + (j >> 2);
    auto source = [&](int k, int g) {
        const int c = CB * g + (j & 3);
        return vrole && k < N && c < ncol
                   ? __ldcg(a.src + ((size_t)(a.n_hi - 1 - k - a.n_lo) * M + gc0 + c) * Kp + own_row) : 0.f;
    };
    // every CTA's buffers and mbarriers are there before a peer writes to them
    cluster.sync();

    auto wait = [&](int g, unsigned parity) {
        const bool ok = mbar_wait_bounded(&mbar[g], parity, a.spin_limit, abort_flag);
        return __all_sync(0xffffffffu, ok) != 0;
    };
    // this warp's sends: nsent steps of the groups below gsent, one less from there on
    int nsent = 0, gsent = G;
    bool dead = false, ready = false;
    float src_next = source(0, 0);
    for (int kb = 0; kb < N; kb += kAdjTab) {
        // (the barrier also keeps the last table until every warp has read it)
        if (__syncthreads_or(dead)) break;
        if (!vrole) {
            for (int idx = tid; idx < kAdjTab * W; idx += kThreads) {
                const int i = idx / W, c = idx - i * W, n = a.n_hi - 1 - kb - i;
                dfT[idx] = n >= a.n_lo && c < ncol
                               ? wavelet_dT_eval<float>(a.wavelet, (long long)a.n0 + n, a.dt, Tcol[c]) : 0.f;
            }
        }
        __syncthreads();
        const int ke = min(N, kb + kAdjTab);
        for (int k = kb; k < ke && !dead; ++k) {
            // operand: lamS after k steps, phase k - 1 (V role), the new lamV, phase k (S role)
            const int ph = vrole ? k - 1 : k;
            for (int g = 0; g < G; ++g) {
                const float* Xg = X + g * kGroup;
                float* yp = own + g * kThreads + tid;
                float* cp = comp + g * kThreads + tid;
                const float y0 = *yp, src = src_next;
                float carry = *cp;
                src_next = g + 1 < G ? source(k, g + 1) : source(k + 1, 0);
                if (ph >= 0) {
                    if (!ready && !wait(g, (unsigned)(ph & 1))) {
                        dead = true;
                        nsent = k + 1, gsent = g;
                        break;
                    }
                    if (tid == 0 && ph + 1 < N) mbar_arrive_expect_tx(&mbar[g], kGroupBytes);
                }
                SplitAcc<KI> acc;
                acc.products(op, Xg, j);
                {
                    // has the next group's operand arrived? (asked ahead, as forwards)
                    const bool wrap = g + 1 == G;
                    const int ph2 = wrap ? ph + 1 : ph;
                    ready = __all_sync(0xffffffffu, ph2 >= 0 && ph2 < N && mbar_test_wait(&mbar[wrap ? 0 : g + 1], ph2 & 1));
                }
                const float tot = acc.reduce(j);
                // half A: lamV += dt Asv^T lamS + 2 C^T r;  half B: lamS += dt Avs^T lamV
                const float inc = vrole ? __fmaf_rn(tot, dt, 2.f * src) : tot * dt;
                const float y = kahan_add(y0, inc, carry);
                *yp = y;
                *cp = carry;
                if (!vrole) {
                    // period gradient of the step over this slab's rows of the same new
                    // lamV: dt (g_slab . a_V[:, c]) df/dT(t_n; T_c), fixed order
                    const int c4 = (warp - CB * g) & (kSplitWarps - 1);  // column c of the group with c = warp (mod 8)
                    if (c4 < CB && CB * g + c4 < ncol) {
                        const int c = CB * g + c4;
                        float sg = gown[lane] * Xg[Lay::at(c4, row0 + lane)];
                        sg = __fmaf_rn(gown[lane + 32], Xg[Lay::at(c4, row0 + lane + 32)], sg);
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) sg += __shfl_xor_sync(0xffffffffu, sg, o);
                        if (lane == 0) gTacc[c] = __fmaf_rn(dt * sg, dfT[(k - kb) * W + c], gTacc[c]);
                    }
                    __syncwarp();
                }
                link.send(g, y);
            }
        }
        if (!dead) nsent = ke;
    }
    // the V role has received the last lamS, too
    if (vrole && !dead && nsent == N && N > 0)
        for (int g = 0; g < G && !dead; ++g) dead = !wait(g, (unsigned)((N - 1) & 1));
    if (dead && lane == 0) *abort_flag = 1;
    split_drain<KI>(cluster, mbar, sent_out, sent_in, Gmax, G, N, vrole, sl, peer0, nsent, gsent, sends, abort_flag,
                    a.status);

    // ---- write back the owned rows, carries and the period-gradient partials
    int bad = 0;
    for (int e = tid; e < G * kThreads; e += kThreads) {
        const int c = e_col(e), row = e_row(e);
        if (c < ncol && row < Kown) {
            own_g[(size_t)(gc0 + c) * Kown + row] = own[e];
            comp_g[(size_t)(gc0 + c) * Kown + row] = comp[e];
            bad |= !is_finite(own[e]);
        }
    }
    for (int c = tid; c < ncol; c += kThreads) a.gTpart[(size_t)crank * M + gc0 + c] = gTacc[c];
    bad = __syncthreads_or(bad);
    if (bad && tid == 0 && a.status) atomicCAS(a.status, 0, 6 /* ROM_E_NONFINITE */);
}

}  // namespace romk
