// Streaming companion kernel of the two-block FP32 split kernel.
//
// The split kernel (rank2_split.cuh) keeps both K x K operators in the
// registers of a 2K/32-CTA cluster (16 CTAs at K = 512).  Clusters that large
// fit only where a GPU processing cluster has that many free SMs, so some SMs
// stay idle.  This kernel runs beside it on those SMs and advances a few of
// the M realizations (columns are independent, Sec. 2.4) with the same
// velocity-first leapfrog (Sec. 3.1):
//
//   V += dt (Avs S + g f_n^T),   S += dt Asv V   (the new V).
//
// A cluster of CSZ (2 or 4) CTAs owns up to 4 columns (one column group);
// CTA c owns rows [c Kp / CSZ, (c + 1) Kp / CSZ) of V and of S and keeps the
// full V and S of its columns in shared memory.  The operators do not fit on
// so few SMs, so every half-step streams the CTA's rows of Avs (or Asv) from
// L2 in stages of 64 rows x 64 k: each thread loads its 4 rows x 4 k of a
// stage straight into a ring of registers that holds a whole 64-row pass
// (Kp / 64 stages), refilling each slot with the next pass's stage as soon as
// it is used, so a pass worth of loads is always in flight, across
// half-steps too (the operator does not depend on the state).  The
// arithmetic is the split kernel's, in the same order: thread (row quad q,
// k lane j) accumulates 4 rows x 4 columns over k = 64 i + 4 j + t with k
// ascending, and the same 16-lane butterfly reduce-scatter and fused
// epilogue (forcing g f^T, Kahan-compensated FP32 update) follow; receiver
// traces y = C V (Sec. 4.5.2) use the split kernel's receiver slabs and warp
// tiles.  So every column comes out bit for bit as the split kernel
// computes it.
//
// Exchange: a warp sends the 8 rows x 4 columns of a pass to every CTA of the
// cluster (its own too) with st.async, one instruction, counted on the
// receiver's mbarrier of V or S; a warp waits there for its operand and no
// barrier stands in the step (the order is rank2_async.cuh's; a CTA's warps
// beyond its rows neither send nor wait).  Every wait is bounded.  K = 512,
// clusters of 4 6.49 us a step (clusters of 2:
// 11.8), 8.3 (13.5) with a block barrier, copies to the peers and a cluster
// barrier each half-step.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "cluster_mbar.cuh"
#include "dev_common.cuh"
#include "rank2_simt.cuh"
#include "rank2_split.cuh"
#include "rom_internal.h"

namespace romk {

constexpr int kStrThreads = kThreads;             // 256: thread (row quad q, k lane j)
constexpr int kStrRows = kSplitRows;              // 64 rows per pass (16 row quads)
constexpr int kStrKC = 64;                        // k extent of one stage
constexpr int kStrCols = kSplitCB;                // 4 columns per cluster (one column group)

constexpr int kStrTab = 32;                       // steps of forcing tabulated at a time

struct StreamSmem {
    size_t Vf, Sf, cV, cS, f, Tpre, g, mbar, sent, flag, total;
};

// Shared-memory layout for Kp padded rows and a CSZ-CTA cluster.
__host__ __device__ inline StreamSmem stream_smem_layout(int Kp, int csz) {
    StreamSmem s{};
    const size_t nr = (size_t)Kp / csz;
    size_t o = 0;
    s.Vf = o;    o += align16((size_t)kStrCols * Kp * sizeof(float));
    s.Sf = o;    o += align16((size_t)kStrCols * Kp * sizeof(float));
    s.cV = o;    o += align16((size_t)kStrCols * nr * sizeof(float));
    s.cS = o;    o += align16((size_t)kStrCols * nr * sizeof(float));
    s.f = o;     o += align16((size_t)kStrTab * kStrCols * sizeof(float));
    s.Tpre = o;  o += align16((size_t)kStrCols * 2 * sizeof(double));
    s.g = o;     o += align16(nr * sizeof(float));
    s.mbar = o;  o += 16;                          // [V, S]
    s.sent = o;  o += align16((size_t)(2 + 2 * csz) * sizeof(unsigned));  // bytes sent [2], sent here [CSZ][2]
    s.flag = o;  o += 16;
    s.total = o;
    return s;
}

// KI = Kp / 64 (Kp <= 512); CSZ CTAs per cluster; Kp / CSZ a multiple of 16
// (a last pass of fewer than 64 rows leaves the row quads beyond the CTA's
// rows idle: they load nothing and write nothing).
template <int KI, int CSZ>
__global__ void __launch_bounds__(kStrThreads, 1) rank2_stream_kernel(const Rank2Args a) {
    using Lay = AsyncLayout<float, kStrCols>;
    constexpr int Kp = 64 * KI;
    constexpr int NR = Kp / CSZ;               // rows owned per CTA
    constexpr int NP = (NR + kStrRows - 1) / kStrRows;  // 64-row passes per half-step
    constexpr int NKS = Kp / kStrKC;           // k stages per pass (= KI)
    constexpr int NW = NR / 8 < kStrThreads / 32 ? NR / 8 : kStrThreads / 32;  // warps with rows
    static_assert(NR % 16 == 0, "owned rows must be whole 16-row groups");
    constexpr int CB = kStrCols;
    constexpr unsigned kBytes = (unsigned)(Kp * CB * sizeof(float));  // V or S of the columns
    constexpr unsigned kPassBytes = 8 * CB * sizeof(float);           // a warp's part of a pass
    cg::cluster_group cluster = cg::this_cluster();
    const int crank = (int)cluster.block_rank();
    const int clu = blockIdx.x / CSZ;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int j = lane & 15;
    const int q = warp * 2 + (lane >> 4);      // row quad within a pass
    const int r0 = crank * NR;
    const int col0 = a.col_base + clu * a.Wv;
    const int ncol = min(a.Wv, a.M - clu * a.Wv);
    const float dt = (float)a.dt;

    extern __shared__ __align__(16) unsigned char smem[];
    const StreamSmem L = stream_smem_layout(Kp, CSZ);
    float* Vf = reinterpret_cast<float*>(smem + L.Vf);       // full V of the columns (AsyncLayout)
    float* Sf = reinterpret_cast<float*>(smem + L.Sf);       // full S
    float* cV = reinterpret_cast<float*>(smem + L.cV);       // [NR][4] Kahan carries, own rows
    float* cS = reinterpret_cast<float*>(smem + L.cS);
    float* ftab = reinterpret_cast<float*>(smem + L.f);      // [kStrTab][4]
    double* Tpre = reinterpret_cast<double*>(smem + L.Tpre); // [4][-1.5 T, pi / T]
    float* gown = reinterpret_cast<float*>(smem + L.g);      // [NR] source rows
    unsigned long long* mbar = reinterpret_cast<unsigned long long*>(smem + L.mbar);
    unsigned* sent_out = reinterpret_cast<unsigned*>(smem + L.sent);
    unsigned* sent_in = sent_out + 2;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L.flag);

    float* Vg = static_cast<float*>(a.V);
    float* Sg = static_cast<float*>(a.S);
    float* cVg = static_cast<float*>(a.compV);
    float* cSg = static_cast<float*>(a.compS);
    for (int idx = tid; idx < kStrCols * Kp; idx += kStrThreads) {
        const int c = idx / Kp, k = idx % Kp, e = Lay::at(c, k);
        const bool okc = c < ncol;
        Vf[e] = (okc && k < a.Kv) ? Vg[(size_t)(col0 + c) * a.Kv + k] : 0.f;
        Sf[e] = (okc && k < a.Ks) ? Sg[(size_t)(col0 + c) * a.Ks + k] : 0.f;
    }
    for (int idx = tid; idx < kStrCols * NR; idx += kStrThreads) {
        const int c = idx / NR, rl = idx % NR, row = r0 + rl;
        const bool okc = c < ncol;
        cV[rl * CB + c] = (okc && cVg && row < a.Kv) ? cVg[(size_t)(col0 + c) * a.Kv + row] : 0.f;
        cS[rl * CB + c] = (okc && cSg && row < a.Ks) ? cSg[(size_t)(col0 + c) * a.Ks + row] : 0.f;
    }
    for (int rl = tid; rl < NR; rl += kStrThreads) gown[rl] = static_cast<const float*>(a.g_p)[r0 + rl];
    if (tid < kStrCols) {
        const float T = (a.Tper && tid < ncol) ? static_cast<const float*>(a.Tper)[col0 + tid] : 1.f;
        Tpre[2 * tid] = -1.5 * (double)T;
        Tpre[2 * tid + 1] = 3.14159265358979323846 / (double)T;
    }
    if (tid == 0) {
        *abort_flag = 0;
        sent_out[0] = sent_out[1] = 0u;
        mbar_init(&mbar[0], 1u);
        mbar_init(&mbar[1], 1u);
        fence_mbar_init_cluster();
        mbar_arrive_expect_tx(&mbar[0], kBytes);
        mbar_arrive_expect_tx(&mbar[1], kBytes);
    }
    // sends: 8 lanes a peer, lane p of them its unit p (the rows of quad p / 4 of
    // the warp's two, column (p mod 4) ^ swz; quads of later passes swizzle alike)
    const int p8 = lane & 7, kqs = (r0 >> 2) + 2 * warp + (p8 >> 2);
    const int src_lane = 16 * (p8 >> 2) + ((p8 & 3) ^ Lay::swz(kqs));
    const int peer = lane >> 3;
    const int npeer = a.debug_skip_push && crank == 0 ? 0 : CSZ;  // fault injection: this CTA sends nothing
    const unsigned base = smem_addr(smem);
    const unsigned dpeer = cluster_addr(base, peer < CSZ ? peer : 0) - base;
    const unsigned piece = (unsigned)(kqs * Lay::U + (p8 & 3)) * 16u;
    const int own = Lay::at(j & 3, r0 + 4 * q + (j >> 2));  // this lane's element of a pass (the first)
    // every CTA is initialised before any peer sends to it
    cluster.sync();

    const int N = a.nsteps;
    const float* Avs = static_cast<const float*>(a.Avs_rm);
    const float* Asv = static_cast<const float*>(a.Asv_rm);
    const float* ftg = static_cast<const float*>(a.ftab);
    const float* Tper = static_cast<const float*>(a.Tper);
    // Stage (half h, pass p, k stage ks): this thread's part is rows
    // r0 + 64 p + 4 q .. + 3 of the half's operator at k = 64 ks + 4 j .. + 3.
    // A ring of NKS stages lives in registers: slot ks holds the current
    // pass's stage ks and is refilled with the next pass's stage ks (the
    // next half's first pass after the last one) as soon as it is used, so a
    // pass worth of loads is always in flight, across half-steps too.
    const size_t lane_off = (size_t)(r0 + 4 * q) * Kp + 4 * j;
    // this thread's row quad exists in pass p (only a partial last pass,
    // NR not a multiple of 64, leaves quads out, two of a warp together)
    constexpr bool WHOLE = NR % kStrRows == 0;
    auto quad_in = [&](int p) { return WHOLE || kStrRows * p + 4 * q < NR; };
    float4 ring[NKS][4];
    if (!WHOLE) {  // quads absent from the first pass never load theirs
#pragma unroll
        for (int ks = 0; ks < NKS; ++ks)
#pragma unroll
            for (int r = 0; r < 4; ++r) ring[ks][r] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (N > 0 && quad_in(0)) {
        const float* src = Avs + lane_off;
#pragma unroll
        for (int ks = 0; ks < NKS; ++ks)
#pragma unroll
            for (int r = 0; r < 4; ++r)
                ring[ks][r] = __ldcg(reinterpret_cast<const float4*>(src + (size_t)r * Kp + ks * kStrKC));
    }

    float* traces = static_cast<float*>(a.traces);
    const float* Cp = static_cast<const float*>(a.C_p);
    const int H = Kp / 64;                            // the split kernel's receiver slabs
    const int rpc = (a.R + H - 1) / H;
    int halves = 0;  // half-steps whose rows this warp has sent
    bool dead = false;
    int rec = 0, to_rec = a.r;
    for (int nb = 0; nb < N; nb += kStrTab) {
        // (the barrier also keeps the last table until every warp has read it)
        if (__syncthreads_or(dead)) break;
        if (tid < kStrTab * CB) {
            const int st = tid / CB, c = tid % CB;
            float f = 0.f;
            if (nb + st < N && c < ncol) {
                if (ftg) f = ftg[(size_t)(nb + st) * a.Mtot + col0 + c];
                else if (Tper)
                    f = wavelet_eval_pre(a.wavelet, (long long)a.n0 + nb + st, a.dt, Tpre[2 * c], Tpre[2 * c + 1]);
            }
            ftab[tid] = f;
        }
        __syncthreads();
        const int ne = min(N, nb + kStrTab);
        for (int n = nb; n < ne && !dead && warp < NW; ++n) {
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                const float* X = h ? Vf : Sf;             // operand of this half
                const float* Y = h ? Sf : Vf;             // state updated in its own rows
                float* cY = h ? cS : cV;
                // operand: S^n, phase n - 1 of its mbarrier (S^0 is local); V^{n+1}, phase n
                const int ph = h ? n : n - 1;
                if (ph >= 0) {
                    const bool ok = mbar_wait_bounded(&mbar[h ^ 1], (unsigned)(ph & 1), a.spin_limit, abort_flag);
                    if (!__all_sync(0xffffffffu, ok)) {
                        dead = true;
                        halves = 2 * n + h;
                        break;
                    }
                    if (tid == 0 && ph + 1 < N) mbar_arrive_expect_tx(&mbar[h ^ 1], kBytes);
                }
                // receiver traces of V^{n+1}, before this warp's S lets V be
                // overwritten: the split kernel's receiver slabs crank, crank +
                // CSZ, ..., each with the same warp tiles
                if (h && traces && --to_rec == 0) {
                    for (int sl = crank; sl < H; sl += CSZ) {
                        const int nj = min(rpc, a.R - sl * rpc);
                        for (int j0 = 4 * warp; j0 < nj; j0 += 4 * NW)
                            trace_group<float, CB>(Cp + (size_t)sl * rpc * Kp, Vf, Kp, j0, nj, ncol, lane,
                                                   traces + ((size_t)rec * a.Mtot + col0) * a.R + sl * rpc, a.R);
                    }
                    to_rec = a.r;
                    ++rec;
                    __syncwarp();
                }
#pragma unroll 1
                for (int p = 0; p < NP; ++p) {
                    // the pass whose stages refill the ring
                    const bool last = p + 1 == NP;
                    const bool has_next = !(last && h == 1 && n + 1 == N) && quad_in(last ? 0 : p + 1);
                    const float* nsrc = (last ? (h ? Avs : Asv) : (h ? Asv : Avs)) +
                                        (size_t)(last ? 0 : (p + 1) * kStrRows) * Kp + lane_off;
                    if (!quad_in(p)) {  // the whole warp: only its next pass's loads
                        if (has_next) {
#pragma unroll
                            for (int ks = 0; ks < NKS; ++ks)
#pragma unroll
                                for (int r = 0; r < 4; ++r)
                                    ring[ks][r] =
                                        __ldcg(reinterpret_cast<const float4*>(nsrc + (size_t)r * Kp + ks * kStrKC));
                        }
                        continue;
                    }
                    // this lane's element: row 4 q + j / 4 of the pass, column j mod 4
                    const float y0 = Y[own + p * kStrRows * CB];
                    float carry = cY[p * kStrRows * CB + tid];
                    float acc[4][CB];
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int cc = 0; cc < CB; ++cc) acc[r][cc] = 0.f;
#pragma unroll
                    for (int ks = 0; ks < NKS; ++ks) {
                        float op[4][4];
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            op[r][0] = ring[ks][r].x;
                            op[r][1] = ring[ks][r].y;
                            op[r][2] = ring[ks][r].z;
                            op[r][3] = ring[ks][r].w;
                        }
                        if (has_next) {
#pragma unroll
                            for (int r = 0; r < 4; ++r)
                                ring[ks][r] =
                                    __ldcg(reinterpret_cast<const float4*>(nsrc + (size_t)r * Kp + ks * kStrKC));
                        }
                        float x[CB][4];
#pragma unroll
                        for (int cc = 0; cc < CB; ++cc) Lay::load(X + 64 * CB * ks, cc, j, x[cc]);
                        // the split kernel's FMA order: k ascending within the lane's stripe
#pragma unroll
                        for (int t = 0; t < 4; ++t)
#pragma unroll
                            for (int cc = 0; cc < CB; ++cc)
#pragma unroll
                                for (int r = 0; r < 4; ++r)
                                    acc[r][cc] = __fmaf_rn(op[r][t], x[cc][t], acc[r][cc]);
                    }
                    // reduce-scatter over the 16 k lanes (value j) and the fused epilogue
                    float v[4 * CB];
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int cc = 0; cc < CB; ++cc) v[r * CB + cc] = acc[r][cc];
                    int vi;
                    bool active;
                    float inc = reduce_scatter16<float, 4 * CB>(v, j, vi, active);
                    if (h == 0)
                        inc = __fmaf_rn(gown[p * kStrRows + 4 * q + (j >> 2)], ftab[(n - nb) * CB + (j & 3)], inc);
                    inc = inc * dt;
                    const float y = kahan_add(y0, inc, carry);
                    cY[p * kStrRows * CB + tid] = carry;
                    float u[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) u[r] = __shfl_sync(0xffffffffu, y, src_lane + 4 * r);
                    if (peer < npeer)
                        asm volatile(
                            "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                            ::"r"(base + (unsigned)(h ? L.Sf : L.Vf) + piece + (unsigned)(p * (kStrRows / 4) * Lay::U * 16) +
                                  dpeer),
                              "f"(u[0]), "f"(u[1]), "f"(u[2]), "f"(u[3]),
                              "r"(smem_addr(&mbar[h]) + dpeer)
                            : "memory");
                }
            }
        }
        if (!dead && warp < NW) halves = 2 * ne;
    }
    // the last S has arrived, too
    if (!dead && N > 0 && warp < NW)
        dead = !__all_sync(0xffffffffu, mbar_wait_bounded(&mbar[1], (unsigned)((N - 1) & 1), a.spin_limit, abort_flag));
    if (dead && lane == 0) *abort_flag = 1;
    // ---- drain, as in the split kernel
    if (lane == 0 && npeer > 0) {
        int np = 0;  // this warp's passes per half-step
        for (int p = 0; p < NP; ++p) np += quad_in(p) ? 1 : 0;
        atomicAdd(&sent_out[0], kPassBytes * (unsigned)(np * ((halves + 1) / 2)));
        atomicAdd(&sent_out[1], kPassBytes * (unsigned)(np * (halves / 2)));
    }
    __syncthreads();
    if (tid < 2 * CSZ) {
        asm volatile("st.shared::cluster.u32 [%0], %1;"
                     ::"r"(cluster_addr(smem_addr(sent_in + 2 * crank + (tid & 1)), tid >> 1)), "r"(sent_out[tid & 1])
                     : "memory");
    }
    cluster.sync();
    if (tid == 0 && N > 0) {
        bool late = false;
        for (int h = 0; h < 2; ++h) {
            unsigned got = 0u;
            for (int d = 0; d < CSZ; ++d) got += sent_in[2 * d + h];
            // phases this thread armed: one at the start, one after each wait but the last
            const int arms = min(N, max(1, h ? (halves + 1) / 2 : halves / 2 + 1));
            const unsigned expect = (unsigned)arms * kBytes;
            if (expect != got) mbar_complete_tx(&mbar[h], expect - got);
            const long long t0 = clock64();
            while (!mbar_try_wait(&mbar[h], (unsigned)(arms - 1) & 1u)) {
                if (clock64() - t0 > 4000000000LL) {
                    late = true;
                    break;
                }
            }
        }
        if ((late || *abort_flag) && a.status) atomicCAS(a.status, 0, 5 /* ROM_E_TIMEOUT */);
    }
    __syncthreads();
    // ---- write back the own rows and carries
    int bad = 0;
    for (int idx = tid; idx < ncol * NR; idx += kStrThreads) {
        const int c = idx / NR, rl = idx % NR, row = r0 + rl, e = Lay::at(c, row);
        if (row < a.Kv) {
            Vg[(size_t)(col0 + c) * a.Kv + row] = Vf[e];
            if (cVg) cVg[(size_t)(col0 + c) * a.Kv + row] = cV[rl * CB + c];
            bad |= !is_finite(Vf[e]);
        }
        if (row < a.Ks) {
            Sg[(size_t)(col0 + c) * a.Ks + row] = Sf[e];
            if (cSg) cSg[(size_t)(col0 + c) * a.Ks + row] = cS[rl * CB + c];
            bad |= !is_finite(Sf[e]);
        }
    }
    bad = __syncthreads_or(bad);
    if (bad && tid == 0 && a.status) atomicCAS(a.status, 0, 6 /* ROM_E_NONFINITE */);
}

}  // namespace romk
