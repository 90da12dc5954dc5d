// Split-role cluster kernel for the rank-2 leapfrog (FP32, Kp <= 512).
//
// Sec. 3.1's leapfrog makes every half-step depend on the previous one, so
// columns (independent realizations, Sec. 2.4) are what keeps a cluster busy.
// A cluster owns two column blocks of Wv columns and has 2H CTAs (H = Kp / 64):
//
//   V role, CTA s < H:  V^{n+1} = V^n + dt (Avs S^n + g f_n^T)
//   S role, CTA H + s:  S^{n+1} = S^n + dt Asv V^{n+1}
//
// on rows [64 s, 64 s + 64), which it owns for all columns, with its operator
// rows in registers and the full operand of the block (S for the V role, V for
// the S role) in shared memory.  Both roles take the columns in groups of 4, in
// the same order, step after step: while the S role has one group, the V role
// has another.
//
// Exchange.  A warp that has a group's 8 rows x 4 columns sends them to every
// CTA of the other role with st.async, which counts the bytes on the
// receiver's mbarrier of the group; a warp waits for a group's operand on that
// mbarrier alone and no barrier stands in the step, so that one group's
// exchange, reduction and update run behind other groups' products.  The
// operand layout (AsyncLayout) makes the warp's 8 x 4 piece 128 contiguous
// bytes: two packets a peer.  Whether the next group has arrived is asked before
// the reduction, whose latency hides the answer's.  With remote stores of 32
// contiguous bytes and a cluster barrier a phase a step took, us before / now:
// K = 512, 8 columns a cluster 3.90 / 2.60, 16 5.60 / 4.07, 32 9.4 / 8.05;
// K = 256, 8 columns 2.54 / 1.59.
//
// Bound: the register file.  At 8 warps an SM the products alone, without loads,
// reduction, update or exchange, take 1500 cycles a group where FMA issue
// allows 1024 (of three operands none repeats often enough; packed FMAs are no
// faster), 6.3 us of the 8.05; the exchange and the waits are 1.0 us of it.
//
// Order.  S^{n+1} of a group overwrites S^n in a V-role CTA only after its
// sender has received V^{n+1} of the group from every warp of the V role, and
// a warp sends that after it has read S^n; the S role's copy likewise (traces
// are taken before the send).  So one buffer suffices, and an mbarrier's next
// phase receives no byte before every warp has waited for the last one.  Every
// wait is bounded; one that runs out stops the CTA at the next refill of the
// forcing table, reports ROM_E_TIMEOUT, and the drain retires the bytes that
// will not come, so that no store is in flight when a CTA exits.
//
// Register tiling: thread (row quad q, chunk j) holds Avs/Asv rows 4q..4q+3 at
// k = 64 i + 4 j + t (i < KI, t < 4): every 16-byte shared load of the operand
// feeds 16 FMAs.  A butterfly reduce-scatter over the 16 chunk lanes leaves
// each lane one (row, column) sum for the fused epilogue: the source signal
// g f_n^T (Sec. 2.2, 3.2, tabulated 32 steps at a time), the
// Kahan-compensated update, the send.  Receiver traces y = C V (Sec. 4.5.2)
// are computed by the S role, which holds the full new V, a tile of 4
// receivers x 4 columns per warp, dealt out in turn over groups and tiles.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "cluster_mbar.cuh"
#include "dev_common.cuh"
#include "rank2_simt.cuh"
#include "rom_internal.h"

namespace romk {

constexpr int kSplitRows = 64;   // rows of one operator per CTA
constexpr int kSplitCB = 4;      // columns per register group
constexpr int kSplitBlock = 2;   // a block's columns are a multiple of this: two blocks hold whole groups
constexpr int kSplitWarps = kThreads / 32;
constexpr int kSplitTab = 32;    // steps of forcing tabulated at a time

struct SplitSmem {
    size_t X, own, comp, C, f, Tpre, mbar, sent, flag, total;
};

// Wa columns per block, two blocks.
__host__ __device__ inline SplitSmem split_smem_layout(int Wa, int Kp, int rpc) {
    SplitSmem s{};
    const size_t W = 2 * (size_t)Wa, G = W / kSplitCB, H = (size_t)Kp / kSplitRows;
    size_t o = 0;
    s.X = o;    o += align16(W * Kp * sizeof(float));
    s.own = o;  o += align16(W * kSplitRows * sizeof(float));
    s.comp = o; o += align16(W * kSplitRows * sizeof(float));
    s.C = o;    o += align16((size_t)rpc * Kp * sizeof(float));
    s.f = o;    o += align16(kSplitTab * W * sizeof(float));
    s.Tpre = o; o += align16(2 * W * sizeof(double));
    s.mbar = o; o += align16(G * sizeof(unsigned long long));
    // bytes sent [G], bytes each CTA of the other role sent here [H][G]
    s.sent = o; o += align16((1 + H) * G * sizeof(unsigned));
    s.flag = o; o += 16;
    s.total = o;
    return s;
}

// Shared-memory layout of a group's CB columns of V or S: the four rows of a
// row quad kq of all columns together, as U 16-byte units (FP32: one per
// column; FP64: two), so that a warp's four rows are one contiguous piece,
// whose stores to one peer travel together (up to 64 bytes a packet; of
// single 16-byte stores a CTA of a 16-CTA cluster takes one in 2.5 cycles or
// more, which at four columns was most of the half-step).  Unit u stands at
// place u ^ swz(kq), which keeps reads of one unit over consecutive quads free
// of bank conflicts.
template <typename T, int CB>
struct AsyncLayout {
    static constexpr int U = CB * (int)sizeof(T) / 4;
    static __device__ __forceinline__ int swz(int kq) { return U > 1 ? (kq / (8 / U)) & (U - 1) : 0; }
    // element (row k, column c of the group)
    static __device__ __forceinline__ int at(int c, int k) {
        const int kq = k >> 2;
        if (sizeof(T) == 4) return (kq * U + (c ^ swz(kq))) * 4 + (k & 3);
        return (kq * U + ((2 * c + ((k >> 1) & 1)) ^ swz(kq))) * 2 + (k & 1);
    }
    // rows 4 kq .. 4 kq + 3 of column c
    static __device__ __forceinline__ void load(const T* X, int c, int kq, T (&x)[4]) {
        const int z = swz(kq);
        if constexpr (sizeof(T) == 4) {
            load4(X + (kq * U + (c ^ z)) * 4, x);
        } else {
            const double2 p = *reinterpret_cast<const double2*>(X + (kq * U + ((2 * c) ^ z)) * 2);
            const double2 q = *reinterpret_cast<const double2*>(X + (kq * U + ((2 * c + 1) ^ z)) * 2);
            x[0] = p.x; x[1] = p.y; x[2] = q.x; x[3] = q.y;
        }
    }
};

template <int KI>
__device__ __forceinline__ void load_op_quad(float (&op)[4][4 * KI], const float* __restrict__ A,
                                             int Kp, int row, int j) {
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) {
#pragma unroll
        for (int i = 0; i < KI; ++i) {
            float x[4];
            load4_ro(A + (size_t)(row + rr) * Kp + 64 * i + 4 * j, x);
#pragma unroll
            for (int t = 0; t < 4; ++t) op[rr][4 * i + t] = x[t];
        }
    }
}

// Sums of NV values (a power of two, at most 16) over the 32 lanes: entry
// lane / (32 / NV) is returned.  Lanes with bit `o` set keep the upper half of
// what is left, the others the lower, each adding its partner's copy; the last
// stages add what the remaining lanes hold of one entry.  The order is that of a
// butterfly over each value, so the bits are, too.
template <typename T, int NV>
__device__ __forceinline__ T reduce_scatter32(T (&v)[NV], int lane) {
    int o = 16;
#pragma unroll
    for (int H = NV / 2; H > 0; H >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const T send = up ? v[i] : v[i + H];
            const T keep = up ? v[i + H] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (int q = 16 / NV; q > 0; q >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], q);
    return v[0];
}

// Receiver traces y = C V^{n+1} (Sec. 4.5.2) of receivers j0 .. j0 + RT - 1 (of
// the nj rows of C, Kp wide) for the first nc of CT columns, by one warp:
// out[c R + jj].  Each lane sums 4-wide stripes of k into RT CT independent
// accumulators; load(c, kq, x) gives rows 4 kq .. 4 kq + 3 of column c.
template <int RT, int CT, typename T, typename Load>
__device__ __forceinline__ void trace_tile(const T* C, int Kp, int j0, int nj, int nc, int lane, T* out, int R,
                                           const Load& load) {
    T acc[RT * CT];
#pragma unroll
    for (int i = 0; i < RT * CT; ++i) acc[i] = T(0);
#pragma unroll 1
    for (int k = 4 * lane; k < Kp; k += 128) {
        T cv[RT][4], xv[CT][4];
#pragma unroll
        for (int u = 0; u < RT; ++u) load4(C + (size_t)min(j0 + u, nj - 1) * Kp + k, cv[u]);
#pragma unroll
        for (int w = 0; w < CT; ++w) load(w, k >> 2, xv[w]);
#pragma unroll
        for (int u = 0; u < RT; ++u)
#pragma unroll
            for (int w = 0; w < CT; ++w)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[CT * u + w] = fmadd(cv[u][q], xv[w][q], acc[CT * u + w]);
    }
    const T y = reduce_scatter32<T, RT * CT>(acc, lane);
    constexpr int LPE = 32 / (RT * CT);  // lanes an entry
    const int e = lane / LPE, jj = j0 + e / CT, c = e % CT;
    if (lane % LPE == 0 && jj < nj && c < nc) out[(size_t)c * R + jj] = y;
}

// The same for 4 receivers and the first nc of a group's CB columns X on the
// exchange layout.
template <typename T, int CB>
__device__ __forceinline__ void trace_group(const T* C, const T* X, int Kp, int j0, int nj, int nc, int lane, T* out,
                                            int R) {
    trace_tile<4, CB, T>(C, Kp, j0, nj, nc, lane, out, R,
                         [&](int c, int kq, T (&x)[4]) { AsyncLayout<T, CB>::load(X, c, kq, x); });
}

// The products of the thread's 4 rows with a group's 4 columns, reduced over the
// 16 chunk lanes: lane chunk j is left with row j / 4, column j mod 4.
template <int KI>
struct SplitAcc {
    float a[4][kSplitCB];
    __device__ __forceinline__ void products(const float (&op)[4][4 * KI], const float* Xg, int j) {
        constexpr int CB = kSplitCB;
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int cc = 0; cc < CB; ++cc) a[r][cc] = 0.f;
#pragma unroll
        for (int i = 0; i < KI; ++i) {
            float x[CB][4];
#pragma unroll
            for (int cc = 0; cc < CB; ++cc) AsyncLayout<float, CB>::load(Xg + 64 * CB * i, cc, j, x[cc]);
#pragma unroll
            for (int t = 0; t < 4; ++t)
#pragma unroll
                for (int cc = 0; cc < CB; ++cc)
#pragma unroll
                    for (int r = 0; r < 4; ++r) a[r][cc] = __fmaf_rn(op[r][4 * i + t], x[cc][t], a[r][cc]);
        }
    }
    __device__ __forceinline__ float reduce(int j) {
        float v[4 * kSplitCB];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int cc = 0; cc < kSplitCB; ++cc) v[r * kSplitCB + cc] = a[r][cc];
        int vi;
        bool active;
        return reduce_scatter16<float, 4 * kSplitCB>(v, j, vi, active);
    }
};

// A warp's way to the other role: 8 lanes a peer carry its 8 x 4 piece of a
// group, lane p of them unit p (the rows of quad p / 4, column (p mod 4) ^ swz).
template <int KI>
struct SplitLink {
    static constexpr int H = KI, NP = (H + 3) / 4;  // peers, peers a lane sends to
    static constexpr unsigned kGroupBytes = 64u * KI * kSplitCB * sizeof(float);
    static constexpr unsigned kWarpBytes = 8 * kSplitCB * sizeof(float);
    unsigned mX, mB, dpeer[NP];  // own addresses of the piece and the mbarriers, distance of the peers' windows
    int src_lane, peer, npeer;
    __device__ __forceinline__ SplitLink(unsigned base, unsigned xoff, unsigned boff, int row0, int warp, int lane,
                                         int peer0, int npeer_)
        : peer(lane >> 3), npeer(npeer_) {
        using Lay = AsyncLayout<float, kSplitCB>;
        const int p8 = lane & 7, kqs = (row0 >> 2) + 2 * warp + (p8 >> 2);
        src_lane = 16 * (p8 >> 2) + ((p8 & 3) ^ Lay::swz(kqs));
        mX = base + xoff + (unsigned)(kqs * Lay::U + (p8 & 3)) * 16u;
        mB = base + boff;
#pragma unroll
        for (int m = 0; m < NP; ++m) {
            const int d = peer + 4 * m;
            dpeer[m] = cluster_addr(base, peer0 + (d < H ? d : 0)) - base;
        }
    }
    __device__ __forceinline__ void send(int g, float y) const {
        float u[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) u[r] = __shfl_sync(0xffffffffu, y, src_lane + 4 * r);
#pragma unroll
        for (int m = 0; m < NP; ++m)
            if (peer + 4 * m < npeer)
                asm volatile(
                    "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                    ::"r"(mX + (unsigned)g * kGroupBytes + dpeer[m]), "f"(u[0]), "f"(u[1]), "f"(u[2]), "f"(u[3]),
                      "r"(mB + 8u * (unsigned)g + dpeer[m])
                    : "memory");
    }
};

// The end of a split-role run.  Every CTA (a timeout or not, so the barriers
// stay cluster-uniform) tells each consumer how many bytes it sent per group;
// past the barrier no CTA issues another store.  A consumer then retires, on
// the phase armed last, the bytes that will not come, so that the phase
// completes when every byte sent has landed, and waits for it (bounded).
// After a complete run nothing is outstanding.  nsent, gsent: the calling
// warp has sent nsent steps of the groups below gsent, one less from there on.
template <int KI>
__device__ __forceinline__ void split_drain(cg::cluster_group& cluster, unsigned long long* mbar, unsigned* sent_out,
                                            unsigned* sent_in, int Gmax, int G, int N, bool vrole, int s, int peer0,
                                            int nsent, int gsent, bool sends, volatile int* abort_flag,
                                            int* status) {
    constexpr int H = KI;
    using Link = SplitLink<KI>;
    const int tid = threadIdx.x;
    if ((tid & 31) == 0 && sends)
        for (int g = 0; g < G; ++g)
            atomicAdd(&sent_out[g], Link::kWarpBytes * (unsigned)(nsent - (g >= gsent ? 1 : 0)));
    __syncthreads();
    for (int idx = tid; idx < H * G; idx += kThreads) {
        const int d = idx / G, g = idx - d * G;
        asm volatile("st.shared::cluster.u32 [%0], %1;"
                     ::"r"(cluster_addr(smem_addr(sent_in + s * Gmax + g), peer0 + d)), "r"(sent_out[g])
                     : "memory");
    }
    cluster.sync();
    if (tid == 0) {
        bool late = false;
        for (int g = 0; g < (N > 0 ? G : 0); ++g) {
            unsigned got = 0u;
            for (int d = 0; d < H; ++d) got += sent_in[d * Gmax + g];
            // phases this thread armed: one at the start, one after each wait but the last
            const int done = nsent - (g >= gsent ? 1 : 0), arms = min(N, max(1, vrole ? done : done + 1));
            const unsigned expect = (unsigned)arms * Link::kGroupBytes;
            if (expect != got) mbar_complete_tx(&mbar[g], expect - got);
            const long long t0 = clock64();
            while (!mbar_try_wait(&mbar[g], (unsigned)(arms - 1) & 1u)) {
                if (clock64() - t0 > 4000000000LL) {
                    late = true;
                    break;
                }
            }
        }
        if ((late || *abort_flag) && status) atomicCAS(status, 0, 5 /* ROM_E_TIMEOUT */);
    }
    __syncthreads();
}

// MODE: 0 plain; 1 adds the reduced reference state (a.Xv / a.Xs); 2 is the
// rank-3 grouped launch (operator table a.group).  A template parameter, so
// that each instance compiles to exactly the code its runs need.
template <int KI, int MODE>
__global__ void __launch_bounds__(kThreads, 1) rank2_split_kernel(const Rank2Args a) {
    using Lay = AsyncLayout<float, kSplitCB>;
    constexpr int CB = kSplitCB, Kp = 64 * KI, H = KI, cs = 2 * KI;
    constexpr int kGroup = Kp * CB;                                  // elements of a group's operand
    constexpr unsigned kGroupBytes = SplitLink<KI>::kGroupBytes;
    cg::cluster_group cluster = cg::this_cluster();
    const int crank = (int)cluster.block_rank();
    // rank-3 grouped launch: operator `job` of the table, cluster `clu` of it
    const int job = MODE == 2 ? (int)(blockIdx.x / cs) / a.group_cpj : 0;
    const int clu = MODE == 2 ? (int)(blockIdx.x / cs) % a.group_cpj : (int)(blockIdx.x / cs);
    const GroupOp* gop = MODE == 2 ? a.group + job : nullptr;
    const bool vrole = crank < H;
    const int s = vrole ? crank : crank - H;  // row slab
    const int row0 = s * kSplitRows;
    const int peer0 = vrole ? H : 0;          // first CTA of the other role
    const int W = 2 * a.Wa, Gmax = W / CB;
    const int ncol = max(0, min(2 * a.Wv, a.M - 2 * clu * a.Wv));
    const int gc0 = a.col_base + (MODE == 2 ? job * a.M : 0) + 2 * clu * a.Wv;
    const int G = (ncol + CB - 1) / CB, N = ncol > 0 ? a.nsteps : 0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j = lane & 15;
    const int q = warp * 2 + (lane >> 4);     // row quad
    const float dt = (float)a.dt;

    extern __shared__ __align__(16) unsigned char smem[];
    const SplitSmem L = split_smem_layout(a.Wa, Kp, a.rpc);
    float* X = reinterpret_cast<float*>(smem + L.X);        // [G] groups of the operand
    float* own = reinterpret_cast<float*>(smem + L.own);    // [G][warp][lane]: the lane's element of the group
    float* comp = reinterpret_cast<float*>(smem + L.comp);  // its carry
    float* Cown = reinterpret_cast<float*>(smem + L.C);     // [rpc][Kp]
    float* ftab = reinterpret_cast<float*>(smem + L.f);     // [kSplitTab][W]
    double* Tpre = reinterpret_cast<double*>(smem + L.Tpre);  // [W][-1.5 T, pi / T]
    unsigned long long* mbar = reinterpret_cast<unsigned long long*>(smem + L.mbar);  // [G]
    unsigned* sent_out = reinterpret_cast<unsigned*>(smem + L.sent);  // [G]
    unsigned* sent_in = sent_out + Gmax;                           // [H][G]
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L.flag);

    const int Kown = vrole ? a.Kv : a.Ks;             // rows of the owned state
    float* own_g = static_cast<float*>(vrole ? a.V : a.S);
    float* comp_g = static_cast<float*>(vrole ? a.compV : a.compS);
    const float* Sin = static_cast<const float*>(a.S);

    // ---- initial state.  V role: operand = full S^0, own = V^0 rows.
    //      S role: operand is filled by the first V sends; own = S^0 rows.
    for (int idx = tid; idx < (vrole ? G * kGroup : 0); idx += kThreads) {
        const int c = idx / Kp, k = idx - c * Kp;
        X[(c / CB) * kGroup + Lay::at(c % CB, k)] =
            c < ncol && k < a.Ks ? Sin[(size_t)(gc0 + c) * a.Ks + k] : 0.f;
    }
    // element e = [g][warp][lane] of own is row / column:
    auto e_row = [&](int e) { return row0 + 8 * ((e >> 5) % kSplitWarps) + 4 * ((e >> 4) & 1) + ((e >> 2) & 3); };
    auto e_col = [&](int e) { return CB * (e / kThreads) + (e & 3); };
    for (int e = tid; e < G * kThreads; e += kThreads) {
        const int c = e_col(e), row = e_row(e);
        const bool ok = c < ncol && row < Kown;
        own[e] = ok ? own_g[(size_t)(gc0 + c) * Kown + row] : 0.f;
        comp[e] = ok && comp_g ? comp_g[(size_t)(gc0 + c) * Kown + row] : 0.f;
    }
    const float* Cp = static_cast<const float*>(MODE == 2 ? gop->C_p : a.C_p);
    float* traces = vrole ? nullptr : static_cast<float*>(a.traces);
    const int nj = traces ? max(0, min(a.rpc, a.R - s * a.rpc)) : 0;  // this CTA's receivers
    for (int idx = tid; idx < nj * Kp; idx += kThreads) Cown[idx] = Cp[(size_t)s * a.rpc * Kp + idx];
    for (int c = tid; c < W; c += kThreads) {
        const double T = a.Tper && c < ncol ? (double)static_cast<const float*>(a.Tper)[gc0 + c] : 1.0;
        Tpre[2 * c] = -1.5 * T;
        Tpre[2 * c + 1] = 3.14159265358979323846 / T;
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
    load_op_quad<KI>(op, static_cast<const float*>(vrole ? (MODE == 2 ? gop->Avs_rm : a.Avs_rm)
                                                         : (MODE == 2 ? gop->Asv_rm : a.Asv_rm)),
                     Kp, row0 + 4 * q, j);
    // this lane's element of a group: row 4 q + j / 4 of the slab, column j mod 4
    const float gr = vrole ? static_cast<const float*>(MODE == 2 ? gop->g_p : a.g_p)[row0 + 4 * q + (j >> 2)] : 0.f;
    const int own_row = row0 + 4 * q + (j >> 2);
    const bool sends = !(a.debug_skip_push && crank == 0);  // fault injection: this CTA sends nothing
    const SplitLink<KI> link(smem_addr(smem), (unsigned)L.X, (unsigned)L.mbar, row0, warp, lane, peer0, sends ? H : 0);
    const float* Xrole = static_cast<const float*>(vrole ? a.Xv : a.Xs);
    const float* ftg = static_cast<const float*>(a.ftab);
    // every CTA's buffers and mbarriers are there before a peer writes to them
    cluster.sync();

    // a wait of the whole warp; false when it ran out here or in another warp
    auto wait = [&](int g, unsigned parity) {
        const bool ok = mbar_wait_bounded(&mbar[g], parity, a.spin_limit, abort_flag);
        return __all_sync(0xffffffffu, ok) != 0;
    };
    // this warp's sends: nsent steps of the groups below gsent, one less from there on
    int nsent = 0, gsent = G;
    bool dead = false, ready = false;
    int rec = 0, to_rec = a.r;
    for (int nb = 0; nb < N; nb += kSplitTab) {
        // (the barrier also keeps the last table until every warp has read it)
        if (__syncthreads_or(dead)) break;
        if (vrole) {
            for (int idx = tid; idx < kSplitTab * W; idx += kThreads) {
                const int st = idx / W, c = idx - st * W;
                float f = 0.f;
                if (nb + st < N && c < ncol) {
                    if (ftg) f = ftg[(size_t)(nb + st) * a.Mtot + gc0 + c];
                    else if (a.Tper)
                        f = wavelet_eval_pre(a.wavelet, (long long)a.n0 + nb + st, a.dt, Tpre[2 * c], Tpre[2 * c + 1]);
                }
                ftab[idx] = f;
            }
        }
        __syncthreads();
        const int ne = min(N, nb + kSplitTab);
        for (int n = nb; n < ne && !dead; ++n) {
            const bool record = traces && --to_rec == 0;
            // operand: S^n, phase n - 1 (V role; S^0 is local), V^{n+1}, phase n (S role)
            const int ph = vrole ? n - 1 : n;
            for (int g = 0; g < G; ++g) {
                const float* Xg = X + g * kGroup;
                float* yp = own + g * kThreads + tid;
                float* cp = comp + g * kThreads + tid;
                const float y0 = *yp;
                float carry = *cp;
                const float f = vrole ? ftab[(n - nb) * W + CB * g + (j & 3)] : 0.f;
                float xr = 0.f;
                if constexpr (MODE == 1) {
                    // Xrole is null for a role whose part of the term is not given
                    const int c = CB * g + (j & 3);
                    if (Xrole && c < ncol && own_row < Kown) xr = Xrole[(size_t)(gc0 + c) * Kown + own_row];
                }
                if (ph >= 0) {
                    if (!ready && !wait(g, (unsigned)(ph & 1))) {
                        dead = true;
                        nsent = n + 1, gsent = g;
                        break;
                    }
                    if (tid == 0 && ph + 1 < N) mbar_arrive_expect_tx(&mbar[g], kGroupBytes);
                }
                SplitAcc<KI> acc;
                acc.products(op, Xg, j);
                // has the next group's operand arrived?  Asked here, the answer
                // is there when the reduction and the update are done.
                {
                    const bool wrap = g + 1 == G;
                    const int ph2 = wrap ? ph + 1 : ph;
                    ready = __all_sync(0xffffffffu, ph2 >= 0 && ph2 < N && mbar_test_wait(&mbar[wrap ? 0 : g + 1], ph2 & 1));
                }
                float inc = acc.reduce(j);
                if (vrole) inc = __fmaf_rn(gr, f, inc);
                if constexpr (MODE == 1) inc = inc + xr;
                inc = inc * dt;
                const float y = kahan_add(y0, inc, carry);
                *yp = y;
                *cp = carry;
                if (record) {  // before this warp's S lets V be overwritten
                    const int nt = (nj + 3) >> 2;
                    for (int t = (warp + kSplitWarps - g * nt % kSplitWarps) % kSplitWarps; t < nt; t += kSplitWarps)
                        trace_group<float, CB>(Cown, Xg, Kp, 4 * t, nj, min(CB, ncol - CB * g), lane,
                                               traces + ((size_t)rec * a.Mtot + gc0 + CB * g) * a.R + s * a.rpc, a.R);
                    __syncwarp();
                }
                link.send(g, y);
            }
            if (record) {
                to_rec = a.r;
                ++rec;
            }
        }
        if (!dead) nsent = ne;
    }
    // the V role has received the last S, too
    if (vrole && !dead && nsent == N && N > 0)
        for (int g = 0; g < G && !dead; ++g) dead = !wait(g, (unsigned)((N - 1) & 1));
    if (dead && lane == 0) *abort_flag = 1;
    split_drain<KI>(cluster, mbar, sent_out, sent_in, Gmax, G, N, vrole, s, peer0, nsent, gsent, sends, abort_flag,
                    a.status);

    // ---- write back the owned rows and carries
    int bad = 0;
    for (int e = tid; e < G * kThreads; e += kThreads) {
        const int c = e_col(e), row = e_row(e);
        if (c < ncol && row < Kown) {
            own_g[(size_t)(gc0 + c) * Kown + row] = own[e];
            if (comp_g) comp_g[(size_t)(gc0 + c) * Kown + row] = comp[e];
            bad |= !is_finite(own[e]);
        }
    }
    bad = __syncthreads_or(bad);
    if (bad && tid == 0 && a.status) atomicCAS(a.status, 0, 6 /* ROM_E_NONFINITE */);
}

}  // namespace romk
