// Rank-2 full-order model (FOM) of the paper's test case on the GPU: the
// axisymmetric elastic shear-wave system of Sec. 3, Eq. (fom_asym), in
// velocity-stress form, advanced by the velocity-first leapfrog for M forcing
// realizations at once (the rank-2 FOM of Eq. (shwave_ode_tensor)).
//
// Discretization: second-order staggered grid in flux form on
// r_cmb <= r <= r_earth, 0 <= theta <= pi, Nr x Nt intervals:
//     v        at (r_{i+1/2}, theta_j),       i in [0, Nr), j in [1, Nt)
//     sigma_rp at (r_i, theta_j),             i in [1, Nr), j in [1, Nt)
//     sigma_tp at (r_{i+1/2}, theta_{j+1/2}), i in [0, Nr), j in [1, Nt - 1)
//     rho v_t      = r^-3 (r^3 sigma_rp)_r + (r sin^2)^-1 (sin^2 sigma_tp)_theta + f
//     (sigma_rp)_t = mu r (v / r)_r,  (sigma_tp)_t = mu (sin / r)(v / sin)_theta
// with v = 0 on the axis and sigma_rp = 0 on the axis and on both free
// surfaces (Sec. 3), and sigma_tp = 0 at the two half points next to the axis
// (v / sin(theta) extrapolated to the axis with zero slope).  Each velocity
// row has at most four non-zeros and each stress row two.
//
// Layout: unknown-major, M realizations contiguous per unknown:
//     V[k * M + m], k = i (Nt - 1) + (j - 1);  S1[k * M + m], k = (i - 1)(Nt - 1) + (j - 1);
//     S2[k * M + m], k = i (Nt - 2) + (j - 1).
// A warp reads whole M-vectors of its stencil neighbours, so every access
// is coalesced and the stencil's reuse stays in L1/L2.
//
// Two forms.  The fused form (default) marches blocks through the grid and
// advances one or two steps per pass over the state (fom_march_kernel).  The
// two-pass form runs a velocity kernel, the point source, the receiver
// record, a stress kernel and a one-thread tick of the device step counter
// per step, in place.  Both evaluate the stencils through the functions
// below, so their values agree bit for bit.
#include <cuda_runtime.h>
#include <math.h>

#include <initializer_list>
#include <map>
#include <mutex>
#include <new>
#include <utility>
#include <tuple>
#include <vector>

#include "dev_common.cuh"
#include "rom_internal.h"

namespace romk {

constexpr int kFomThreads = 256;
constexpr int kFomGraphSteps = 64;

struct FomCtl {
    long long step, nsteps, n0;
};

// Per-row factors of the stencils (all divided out of the inner loop).
template <typename T>
struct FomTables {
    const T* cr_p;   // [Nr]  r_{i+1}^3 / (rho r_{i+1/2}^3 dr), 0 at i = Nr - 1
    const T* cr_m;   // [Nr]  r_i^3 / (rho r_{i+1/2}^3 dr), 0 at i = 0
    const T* inv_rh; // [Nr]  1 / r_{i+1/2}
    const T* pt_p;   // [Nt]  sin^2 theta_{j+1/2} / (rho sin^2 theta_j dth), 0 at j = Nt - 1
    const T* pt_m;   // [Nt]  sin^2 theta_{j-1/2} / (rho sin^2 theta_j dth), 0 at j = 1
    const T* q_u;    // [Nr]  mu r_i / (r_{i+1/2} dr)
    const T* q_d;    // [Nr]  mu r_i / (r_{i-1/2} dr)
    const T* w_p;    // [Nt]  mu sin theta_{j+1/2} / (sin theta_{j+1} dth)
    const T* w_m;    // [Nt]  mu sin theta_{j+1/2} / (sin theta_j dth)
};

template <typename T>
struct FomArgs {
    FomTables<T> tb;
    T* V;
    T* S1;
    T* S2;
    const T* Tper;   // M periods, or null
    const int* recv; // nrecv velocity unknowns, or null
    T* traces;       // records of nrecv x M, or null
    const FomCtl* ctl;
    int Nr, Nt, M, src, nrecv, r, wavelet;
    double dt, rho;
};

// One pass of the fused form: the state of step n = base + off is read from
// the `o` buffers, that of step n + 1 (or n + 2) written to the `n` buffers;
// base and n0 come from ctl (a pass of the graph) or are off and n0 alone.
template <typename T>
struct FomPass {
    FomTables<T> tb;
    const T* Vo;
    const T* S1o;
    const T* S2o;
    T* Vn;
    T* S1n;
    T* S2n;
    const T* Tper;
    const int* recv;
    T* traces;
    const FomCtl* ctl;
    long long off, n0;
    int Nr, Nt, M, nrecv, r, wavelet;
    int Mt;             // realizations of the run (M: of the buffers, padded)
    int src_i, src_j;   // the source's grid point
    int seg_rows;       // radial rows per block
    int nmarch;         // blocks that march; those beyond record receivers
    double dt, rho;
};

// Vector of VW consecutive realizations (16-byte loads when VW > 1).
template <typename T, int VW> struct FomVec;
template <> struct FomVec<float, 1> { using type = float; };
template <> struct FomVec<float, 4> { using type = float4; };
template <> struct FomVec<double, 1> { using type = double; };
template <> struct FomVec<double, 2> { using type = double2; };

template <typename T, int VW>
__device__ __forceinline__ void fom_load(const T* p, T (&x)[VW]) {
    const typename FomVec<T, VW>::type v = *reinterpret_cast<const typename FomVec<T, VW>::type*>(p);
    const T* e = reinterpret_cast<const T*>(&v);
#pragma unroll
    for (int q = 0; q < VW; ++q) x[q] = e[q];
}
template <typename T, int VW>
__device__ __forceinline__ void fom_store(T* p, const T (&x)[VW]) {
    typename FomVec<T, VW>::type v;
    T* e = reinterpret_cast<T*>(&v);
#pragma unroll
    for (int q = 0; q < VW; ++q) e[q] = x[q];
    *reinterpret_cast<typename FomVec<T, VW>::type*>(p) = v;
}

// The stencils, with every operation written out so that each caller (an
// owner or a halo recomputing it, one or two steps a pass, either form)
// rounds the same way.
__device__ __forceinline__ float fom_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fom_fma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fom_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double fom_mul(double a, double b) { return __dmul_rn(a, b); }
template <typename T>
__device__ __forceinline__ T fom_vel(T v, T dt, T cp, T s1u, T cm, T s1d, T ir, T pp, T s2r, T pm, T s2l) {
    const T radial = fom_fma(cp, s1u, -fom_mul(cm, s1d));
    const T polar = fom_fma(pp, s2r, -fom_mul(pm, s2l));
    return fom_fma(dt, fom_fma(ir, polar, radial), v);
}
// s += c (a x - b y): sigma_rp with c = dt, sigma_tp with c = dt / r.
template <typename T>
__device__ __forceinline__ T fom_str(T s, T c, T a, T x, T b, T y) {
    return fom_fma(c, fom_fma(a, x, -fom_mul(b, y)), s);
}
template <typename T>
__device__ __forceinline__ T fom_src(T v, T csrc, int wavelet, long long n, double dt, T Tm) {
    return fom_fma(csrc, (T)wavelet_eval(wavelet, n, dt, Tm), v);
}

// Thread layout of the two passes: persistent blocks stride over tiles of
// (radial index i, blockDim.y polar points j); in a tile threadIdx.y picks j
// and threadIdx.x runs over the realizations in groups of VW (a warp reads
// whole M-vectors with 16-byte loads).  The step word is read once per block.
template <typename T, int VW>
__global__ void __launch_bounds__(kFomThreads) fom_velocity_kernel(const FomArgs<T> a) {
    const long long n = a.ctl->step;
    if (n >= a.ctl->nsteps) return;
    const int Nt1 = a.Nt - 1, Nt2 = a.Nt - 2, M = a.M;
    const T dt = (T)a.dt;
    const int gx = (Nt1 + blockDim.y - 1) / blockDim.y;
    const long long tiles = (long long)a.Nr * gx;
    const T* __restrict__ S1 = a.S1;
    const T* __restrict__ S2 = a.S2;
    T* __restrict__ Vv = a.V;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int i = (int)(t / gx);
        const int j = (int)(t - (long long)i * gx) * blockDim.y + threadIdx.y + 1;
        if (j >= a.Nt) continue;
        const T cp = a.tb.cr_p[i], cm = a.tb.cr_m[i], ir = a.tb.inv_rh[i];
        const T pp = a.tb.pt_p[j], pm = a.tb.pt_m[j];
        const bool hp = i + 1 < a.Nr, hm = i >= 1, h2p = j <= Nt2, h2m = j >= 2;
        const size_t kv = (size_t)i * Nt1 + (j - 1);
        // stencil neighbours (the pointers of absent ones are never read)
        const T* s1p = S1 + (hp ? kv : 0) * M;                                  // sigma_rp (i + 1, j)
        const T* s1m = S1 + (hm ? (size_t)(i - 1) * Nt1 + (j - 1) : 0) * M;     // sigma_rp (i, j)
        const T* s2p = S2 + (h2p ? (size_t)i * Nt2 + (j - 1) : 0) * M;          // sigma_tp (i + 1/2, j + 1/2)
        const T* s2m = S2 + (h2m ? (size_t)i * Nt2 + (j - 2) : 0) * M;          // sigma_tp (i + 1/2, j - 1/2)
        T* v = Vv + kv * M;
        for (int m = threadIdx.x * VW; m < M; m += blockDim.x * VW) {
            T x1p[VW], x1m[VW], x2p[VW], x2m[VW], y[VW];
#pragma unroll
            for (int q = 0; q < VW; ++q) x1p[q] = x1m[q] = x2p[q] = x2m[q] = T(0);
            if (hp) fom_load<T, VW>(s1p + m, x1p);
            if (hm) fom_load<T, VW>(s1m + m, x1m);
            if (h2p) fom_load<T, VW>(s2p + m, x2p);
            if (h2m) fom_load<T, VW>(s2m + m, x2m);
            fom_load<T, VW>(v + m, y);
#pragma unroll
            for (int q = 0; q < VW; ++q)
                y[q] = fom_vel(y[q], dt, cp, x1p[q], cm, x1m[q], ir, pp, x2p[q], pm, x2m[q]);
            fom_store<T, VW>(v + m, y);
        }
    }
}

// The point source of the step, after the velocity pass (one row):
// v[src] += (dt / rho) f(t_n; T_m).
template <typename T>
__global__ void __launch_bounds__(kFomThreads) fom_source_kernel(const FomArgs<T> a) {
    const long long n = a.ctl->step;
    if (n >= a.ctl->nsteps) return;
    const T c = (T)(a.dt / a.rho);
    T* v = a.V + (size_t)a.src * a.M;
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < a.M; m += gridDim.x * blockDim.x)
        v[m] = fom_src(v[m], c, a.wavelet, a.ctl->n0 + n, a.dt, a.Tper[m]);
}

template <typename T>
__global__ void __launch_bounds__(kFomThreads) fom_record_kernel(const FomArgs<T> a) {
    const long long n = a.ctl->step;
    if (n >= a.ctl->nsteps || ((n + 1) % a.r) != 0) return;
    const long long rec = (n + 1) / a.r - 1;
    const int tot = a.nrecv * a.M;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < tot; idx += gridDim.x * blockDim.x) {
        const int kk = idx / a.M, m = idx - kk * a.M;
        a.traces[(rec * a.nrecv + kk) * a.M + m] = a.V[(long long)a.recv[kk] * a.M + m];
    }
}

// Receiver records of a pass: V^n as it was found (the record of step n - 1)
// and, of a pass over two steps, V^{n+1}, which the march keeps on chip, from
// the old state by the same arithmetic.
template <typename T, int NS>
__device__ __forceinline__ void fom_march_record(const FomPass<T>& a, long long n, long long n0) {
    const bool rec0 = n > 0 && n % a.r == 0;
    const bool rec1 = NS == 2 && (n + 1) % a.r == 0;
    if (!rec0 && !rec1) return;
    const int Nt1 = a.Nt - 1, Nt2 = a.Nt - 2, M = a.M, Mt = a.Mt;
    const T dt = (T)a.dt;
    const long long tot = (long long)a.nrecv * Mt;
    const long long nthr = (long long)(gridDim.x - a.nmarch) * kFomThreads;
    const int tid = (int)(threadIdx.y * blockDim.x + threadIdx.x);
    for (long long idx = (long long)(blockIdx.x - a.nmarch) * kFomThreads + tid; idx < tot; idx += nthr) {
        const int kk = (int)(idx / Mt), m = (int)(idx - (long long)kk * Mt);
        const long long u = a.recv[kk];
        const T v = a.Vo[u * M + m];
        if (rec0) a.traces[(n / a.r - 1) * tot + idx] = v;
        if (rec1) {
            const int i = (int)(u / Nt1), j = (int)(u - (long long)i * Nt1) + 1;
            const T s1u = i + 1 < a.Nr ? a.S1o[((size_t)i * Nt1 + (j - 1)) * M + m] : T(0);
            const T s1d = i >= 1 ? a.S1o[((size_t)(i - 1) * Nt1 + (j - 1)) * M + m] : T(0);
            const T s2r = j <= Nt2 ? a.S2o[((size_t)i * Nt2 + (j - 1)) * M + m] : T(0);
            const T s2l = j >= 2 ? a.S2o[((size_t)i * Nt2 + (j - 2)) * M + m] : T(0);
            T vn = fom_vel(v, dt, a.tb.cr_p[i], s1u, a.tb.cr_m[i], s1d, a.tb.inv_rh[i], a.tb.pt_p[j], s2r,
                           a.tb.pt_m[j], s2l);
            if (a.Tper && i == a.src_i && j == a.src_j)
                vn = fom_src(vn, (T)(a.dt / a.rho), a.wavelet, n0 + n, a.dt, a.Tper[m]);
            a.traces[((n + 1) / a.r - 1) * tot + idx] = vn;
        }
    }
}

// Rows in flight per thread (512 x 2048, M = 32: 62.8 us a step with 3, 63.2
// with 4), and resident blocks per SM (two-step pass: 128 registers a thread;
// 3 blocks of 80 spill: 123 us).
template <int NS>
__host__ __device__ constexpr int fom_stages() { return NS == 2 ? 3 : 2; }
template <int NS>
__host__ __device__ constexpr int fom_occupancy() { return NS == 2 ? 2 : 4; }
constexpr int kFomMaxSeg = 128;  // radial rows per block, at most

// Asynchronous copy of B bytes to shared memory, zeros beyond src_bytes.
template <int B, typename T>
__device__ __forceinline__ void fom_cp_async(T* dst, const T* src, int src_bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "n"(B), "r"(src_bytes)
                 : "memory");
}

// One pass of the fused form over NS = 1 or 2 steps.  Reads the old state
// from one buffer set and writes the new one to the other, so that
// neighbouring blocks never see each other's writes.  A block takes a strip
// of polar columns times a segment of seg_rows radial rows and marches
// outward in r; thread row ty holds one column, threadIdx.x the realizations
// in groups of VW.  The lower sigma_rp face and the previous row's new
// velocity stay in registers; a row's new velocity goes through shared memory
// to the column's neighbours.  Two steps run one row apart: once step n has
// row i, its sigma_rp face i, and with them every input of step n + 1 at row
// i - 1, is there.  Nothing of step n + 1's input touches memory.
//  * Columns: strip s owns j in [s TJ + 1, s TJ + TJ].  NS = 1 needs one halo
//    column on the right (sigma_tp takes the next column's new velocity).
//    NS = 2 needs two there and one on the left, whose sigma_tp of step n the
//    neighbour recomputes from the velocity in shared memory.
//  * Rows: NS = 1 starts one row early to have the velocity below its first
//    sigma_rp, NS = 2 two rows early, and reads one row past its end.
// Halo values are computed by the owners' arithmetic (forcing included), so
// they equal the owners' values bit for bit.
// A thread's next rows are copied ahead into its own shared-memory slots, and
// the row factors are staged there: with both read from global memory in the
// loop a two-step pass was bound by their latency (96 us a step below).
// Bound: memory.  NS = 1 moves 8 M bytes per unknown and step in FP32, NS = 2
// half of that: 512 x 2048 grid, M = 32, 142 us a step with one step a pass
// (85 % of the HBM copy rate), 61 us with two (98 %); M = 1, which stays in
// L2, 25.4 and 5.8 us.  FP64 (NS = 1) is bound by the FP64 units, for which
// the halo's extra work would be a loss.
template <typename T, int VW, int NS>
__global__ void __launch_bounds__(kFomThreads, fom_occupancy<NS>()) fom_march_kernel(const FomPass<T> a) {
    // the next pass's blocks may take their places as this pass's leave them;
    // like these, they read nothing that a pass writes before the wait below
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if ((int)blockIdx.x >= a.nmarch) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        fom_march_record<T, NS>(a, a.off + (a.ctl ? a.ctl->step : 0), a.ctl ? a.ctl->n0 : a.n0);
        return;
    }
    constexpr int LH = NS - 1;                    // halo columns on the left
    constexpr int STAGES = fom_stages<NS>();
    constexpr int B = VW * (int)sizeof(T);
    const int Nt1 = a.Nt - 1, Nt2 = a.Nt - 2, M = a.M, Nr = a.Nr;
    const int by = (int)blockDim.y;
    const int TJ = by - (2 * NS - 1);
    const int nstrip = (Nt1 + TJ - 1) / TJ;
    const int strip = (int)blockIdx.x % nstrip, seg = (int)blockIdx.x / nstrip;
    const int ia = seg * a.seg_rows;
    const int ib = min(Nr, ia + a.seg_rows);
    const int ty = threadIdx.y, tx = threadIdx.x;
    const int j = strip * TJ + 1 - LH + ty;       // polar index of this thread's column
    const bool act = j >= 1 && j <= Nt1;          // a velocity column
    const bool own = act && ty >= LH && ty < LH + TJ;
    const bool has_s2 = act && j <= Nt2, has_l = act && j >= 2;
    const T dt = (T)a.dt;
    const T pp = act ? a.tb.pt_p[j] : T(0), pm = act ? a.tb.pt_m[j] : T(0);
    const T wp = has_s2 ? a.tb.w_p[j] : T(0), wm = has_s2 ? a.tb.w_m[j] : T(0);
    const T wpl = NS == 2 && has_l ? a.tb.w_p[j - 1] : T(0), wml = NS == 2 && has_l ? a.tb.w_m[j - 1] : T(0);
    const bool src_col = a.Tper && act && j == a.src_j;
    extern __shared__ __align__(16) unsigned char fom_smem[];
    // [row parity][step][thread][VW] new velocity
    T* row = reinterpret_cast<T*>(fom_smem);
    constexpr int rstep = kFomThreads * VW;
    T* slots = row + 2 * NS * rstep;              // [STAGES][V, S1, S2 right, S2 left][thread][VW]
    T* rtab = slots + STAGES * 4 * rstep;         // [row i0 - 1 ..][cr_p, cr_m, 1/r, dt/r, q_u, q_d, -, -]
    const int self = (ty * (int)blockDim.x + tx) * VW;
    const int right = (min(ty + 1, by - 1) * (int)blockDim.x + tx) * VW;
    const int left = (max(ty - 1, 0) * (int)blockDim.x + tx) * VW;
    const int i0 = max(0, ia - NS);
    const int iend = NS == 2 ? ib : ib - 1;       // last row of step n (row Nr is all zeros)
    for (int k = ty * (int)blockDim.x + tx; k < iend - i0 + 2; k += kFomThreads) {
        const int i = i0 - 1 + k;
        const bool in = i >= 0 && i < Nr;         // zero factors outside the grid
        T* e = rtab + 8 * k;
        const T ir = in ? a.tb.inv_rh[i] : T(0);
        e[0] = in ? a.tb.cr_p[i] : T(0);
        e[1] = in ? a.tb.cr_m[i] : T(0);
        e[2] = ir;
        e[3] = fom_mul(dt, ir);
        e[4] = in ? a.tb.q_u[i] : T(0);
        e[5] = in ? a.tb.q_d[i] : T(0);
    }
    // the last pass has ended and its writes are visible
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const long long n = a.off + (a.ctl ? a.ctl->step : 0);
    const long long n0 = a.ctl ? a.ctl->n0 : a.n0;
    const int chunk = (int)blockDim.x * VW;
    const size_t rv = (size_t)Nt1 * M, r2 = (size_t)Nt2 * M;  // elements per row
    for (int mb = 0; mb < M; mb += chunk) {       // same trip count in every thread
        const int m0 = mb + tx * VW;
        const bool lane = act && m0 < M;
        const bool put = own && m0 < M, put2 = put && has_s2;
        // addresses of inactive lanes stay on a valid element
        const int jc = act ? j : 1, mc = m0 < M ? m0 : 0;
        const size_t ov = (size_t)(jc - 1) * M + mc, o2 = (size_t)(min(jc, Nt2) - 1) * M + mc;
        T s1d[VW], vp[VW];                        // step n: sigma_rp face i, new velocity of row i - 1
        T t1d[VW], t2r[VW], t2l[VW], wprev[VW];   // step n + 1: face i - 1, sigma_tp of row i - 1, velocity of i - 2
#pragma unroll
        for (int q = 0; q < VW; ++q) s1d[q] = vp[q] = t1d[q] = t2r[q] = t2l[q] = wprev[q] = T(0);
        if (lane && i0 >= 1) fom_load<T, VW>(a.S1o + (size_t)(i0 - 1) * rv + ov, s1d);
        // rows are copied STAGES - 1 ahead into the thread's own slots
        const T* gv = a.Vo + (size_t)i0 * rv + ov;
        const T* g1 = a.S1o + (size_t)i0 * rv + ov;
        const T* g2 = a.S2o + (size_t)i0 * r2 + o2;
        const T* g2l = has_l ? a.S2o + (size_t)i0 * r2 + (size_t)(jc - 2) * M + mc : g2;
        const int bv = lane ? B : 0, b2r = lane && has_s2 ? B : 0, b2l = lane && has_l ? B : 0;
        int inext = i0, snext = 0, scur = 0;
        auto fetch = [&]() {
            if (inext <= iend) {
                T* d = slots + snext * 4 * rstep + self;
                const bool in = inext < Nr, face = inext + 1 < Nr;
                fom_cp_async<B>(d, in ? gv : a.Vo, in ? bv : 0);
                fom_cp_async<B>(d + rstep, face ? g1 : a.Vo, face ? bv : 0);
                fom_cp_async<B>(d + 2 * rstep, in ? g2 : a.Vo, in ? b2r : 0);
                fom_cp_async<B>(d + 3 * rstep, in ? g2l : a.Vo, in ? b2l : 0);
                gv += rv;
                g1 += rv;
                g2 += r2;
                g2l += r2;
                snext = snext + 1 == STAGES ? 0 : snext + 1;
            }
            ++inext;
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
#pragma unroll
        for (int k = 0; k < STAGES - 1; ++k) fetch();
        // outputs of row i (NS = 1) or i - 1 (NS = 2)
        T* hv = a.Vn + (size_t)i0 * rv + ov - (NS - 1) * rv;
        T* h1 = a.S1n + (size_t)i0 * rv + ov - NS * rv;
        T* h2 = a.S2n + (size_t)i0 * r2 + o2 - (NS - 1) * r2;
        __syncthreads();                          // rtab is there; the last chunk's rows are read
        for (int i = i0; i <= iend; ++i) {
            T* rb = row + (i & 1) * NS * rstep;
            fetch();
            asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 1) : "memory");
            const T* d = slots + scur * 4 * rstep + self;
            scur = scur + 1 == STAGES ? 0 : scur + 1;
            T vo[VW], s1u[VW], s2r[VW], s2l[VW], vn[VW], s1n[VW], w[VW];
            fom_load<T, VW>(d, vo);
            fom_load<T, VW>(d + rstep, s1u);
            fom_load<T, VW>(d + 2 * rstep, s2r);
            fom_load<T, VW>(d + 3 * rstep, s2l);
            const T* e = rtab + 8 * (i - i0 + 1);
            const T c = e[3];
#pragma unroll
            for (int q = 0; q < VW; ++q)
                vn[q] = fom_vel(vo[q], dt, e[0], s1u[q], e[1], s1d[q], e[2], pp, s2r[q], pm, s2l[q]);
            if (src_col && i == a.src_i && m0 < M) {
#pragma unroll
                for (int q = 0; q < VW; ++q)
                    vn[q] = fom_src(vn[q], (T)(a.dt / a.rho), a.wavelet, n0 + n, a.dt, a.Tper[min(m0 + q, a.Mt - 1)]);
            }
            fom_store<T, VW>(rb + self, vn);
            // the face below row i (of the first row: not used, or face 0, whose factors are 0)
#pragma unroll
            for (int q = 0; q < VW; ++q) s1n[q] = fom_str(s1d[q], dt, e[4], vn[q], e[5], vp[q]);
            if (NS == 2) {
                // step n + 1 at row i - 1 (the first rows' values are not used)
#pragma unroll
                for (int q = 0; q < VW; ++q)
                    w[q] = fom_vel(vp[q], dt, e[-8], s1n[q], e[-7], t1d[q], e[-6], pp, t2r[q], pm, t2l[q]);
                if (src_col && i - 1 == a.src_i && m0 < M) {
#pragma unroll
                    for (int q = 0; q < VW; ++q)
                        w[q] = fom_src(w[q], (T)(a.dt / a.rho), a.wavelet, n0 + n + 1, a.dt, a.Tper[min(m0 + q, a.Mt - 1)]);
                }
                fom_store<T, VW>(rb + rstep + self, w);
            }
            __syncthreads();                      // rows are double-buffered by parity: one barrier a row
            T vr[VW];
            fom_load<T, VW>(rb + right, vr);
            if (NS == 1) {
                if (i >= ia) {
                    if (put) fom_store<T, VW>(hv, vn);
                    if (put && i >= 1) fom_store<T, VW>(h1, s1n);
                    if (put2) {
#pragma unroll
                        for (int q = 0; q < VW; ++q) s2r[q] = fom_str(s2r[q], c, wp, vr[q], wm, vn[q]);
                        fom_store<T, VW>(h2, s2r);
                    }
                }
            } else {
                if (i > ia) {
                    if (put) fom_store<T, VW>(hv, w);
                    if (put && i >= 2) {
                        T s1[VW];
#pragma unroll
                        for (int q = 0; q < VW; ++q) s1[q] = fom_str(t1d[q], dt, e[-4], w[q], e[-3], wprev[q]);
                        fom_store<T, VW>(h1, s1);
                    }
                    if (put2) {
                        T wr[VW];
                        fom_load<T, VW>(rb + rstep + right, wr);
#pragma unroll
                        for (int q = 0; q < VW; ++q) wr[q] = fom_str(t2r[q], e[-5], wp, wr[q], wm, w[q]);
                        fom_store<T, VW>(h2, wr);
                    }
                }
                // sigma_tp of row i after step n, this column's and the left one's
                T vl[VW];
                fom_load<T, VW>(rb + left, vl);
#pragma unroll
                for (int q = 0; q < VW; ++q) {
                    t2r[q] = fom_str(s2r[q], c, wp, vr[q], wm, vn[q]);
                    t2l[q] = fom_str(s2l[q], c, wpl, vn[q], wml, vl[q]);
                    t1d[q] = s1n[q];
                    wprev[q] = w[q];
                }
            }
            hv += rv;
            h1 += rv;
            h2 += r2;
#pragma unroll
            for (int q = 0; q < VW; ++q) {
                s1d[q] = s1u[q];
                vp[q] = vn[q];
            }
        }
    }
}

template <typename T, int VW>
__global__ void __launch_bounds__(kFomThreads) fom_stress_kernel(const FomArgs<T> a) {
    const long long n = a.ctl->step;
    if (n >= a.ctl->nsteps) return;
    const int Nt1 = a.Nt - 1, Nt2 = a.Nt - 2, M = a.M;
    const T dt = (T)a.dt;
    const int gx = (Nt1 + blockDim.y - 1) / blockDim.y;
    const long long tiles1 = (long long)(a.Nr - 1) * gx;   // sigma_rp: i in [1, Nr)
    const long long tiles = tiles1 + (long long)a.Nr * gx;  // then sigma_tp: i in [0, Nr)
    const T* __restrict__ Vv = a.V;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        if (t < tiles1) {
            // sigma_rp (i, j), i in [1, Nr), j in [1, Nt)
            const int i = (int)(t / gx) + 1;
            const int j = (int)(t - (long long)(i - 1) * gx) * blockDim.y + threadIdx.y + 1;
            if (j >= a.Nt) continue;
            const T qu = a.tb.q_u[i], qd = a.tb.q_d[i];
            const T* vu = Vv + ((size_t)i * Nt1 + (j - 1)) * M;        // v (i + 1/2, j)
            const T* vd = Vv + ((size_t)(i - 1) * Nt1 + (j - 1)) * M;  // v (i - 1/2, j)
            T* s = a.S1 + ((size_t)(i - 1) * Nt1 + (j - 1)) * M;
            for (int m = threadIdx.x * VW; m < M; m += blockDim.x * VW) {
                T xu[VW], xd[VW], y[VW];
                fom_load<T, VW>(vu + m, xu);
                fom_load<T, VW>(vd + m, xd);
                fom_load<T, VW>(s + m, y);
#pragma unroll
                for (int q = 0; q < VW; ++q) y[q] = fom_str(y[q], dt, qu, xu[q], qd, xd[q]);
                fom_store<T, VW>(s + m, y);
            }
        } else {
            // sigma_tp (i + 1/2, j + 1/2), i in [0, Nr), j in [1, Nt - 1)
            const long long t2 = t - tiles1;
            const int i = (int)(t2 / gx);
            const int j = (int)(t2 - (long long)i * gx) * blockDim.y + threadIdx.y + 1;
            if (j >= a.Nt - 1) continue;
            const T ir = a.tb.inv_rh[i], wp = a.tb.w_p[j], wm = a.tb.w_m[j];
            const T* vr = Vv + ((size_t)i * Nt1 + j) * M;              // v (i + 1/2, j + 1)
            const T* vl = Vv + ((size_t)i * Nt1 + (j - 1)) * M;        // v (i + 1/2, j)
            T* s = a.S2 + ((size_t)i * Nt2 + (j - 1)) * M;
            for (int m = threadIdx.x * VW; m < M; m += blockDim.x * VW) {
                T xr[VW], xl[VW], y[VW];
                fom_load<T, VW>(vr + m, xr);
                fom_load<T, VW>(vl + m, xl);
                fom_load<T, VW>(s + m, y);
#pragma unroll
                for (int q = 0; q < VW; ++q) y[q] = fom_str(y[q], fom_mul(dt, ir), wp, xr[q], wm, xl[q]);
                fom_store<T, VW>(s + m, y);
            }
        }
    }
}

__global__ void fom_tick_kernel(FomCtl* ctl) {
    if (ctl->step < ctl->nsteps) ctl->step = ctl->step + 1;
}

__global__ void fom_advance_kernel(FomCtl* ctl, int steps) { ctl->step = ctl->step + steps; }

// Record of the final velocity of a fused run.
template <typename T>
__global__ void __launch_bounds__(kFomThreads) fom_last_record_kernel(const T* __restrict__ V,
                                                                      const int* __restrict__ recv, int nrecv,
                                                                      int M, int Mt, T* __restrict__ out) {
    const long long tot = (long long)nrecv * Mt;
    for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < tot;
         idx += (long long)gridDim.x * blockDim.x) {
        const int kk = (int)(idx / Mt), m = (int)(idx - (long long)kk * Mt);
        out[idx] = V[(long long)recv[kk] * M + m];
    }
}

// Rows of M values to rows of Mp >= M (zeros beyond) or back, n rows.
template <bool IN>
__global__ void __launch_bounds__(kFomThreads) fom_pad_kernel(const float* __restrict__ src, long long n, int M,
                                                              int Mp, float* __restrict__ dst) {
    const int w = IN ? Mp : M;
    const long long tot = n * w;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < tot;
         i += (long long)gridDim.x * blockDim.x) {
        const long long k = i / w;
        const int m = (int)(i - k * w);
        dst[i] = m < M ? src[k * (IN ? M : Mp) + m] : 0.f;
    }
}

__global__ void fom_set_kernel(FomCtl* ctl, long long nsteps, long long n0) {
    ctl->step = 0;
    ctl->nsteps = nsteps;
    ctl->n0 = n0;
}

}  // namespace romk

using namespace romk;

struct rom_fom_s {
    int Nr = 0, Nt = 0;
    double r_cmb = 0, r_earth = 0, rho = 0, vs = 0, dt = 0;
    void* tables[2] = {nullptr, nullptr};  // [0] f64, [1] f32: 9 arrays of max(Nr, Nt) + 1
    size_t tlen = 0;
    FomCtl* ctl = nullptr;
    cudaStream_t cap = nullptr;
    std::mutex mu;
    std::map<std::vector<long long>, cudaGraphExec_t> graphs;
    int passes = 1;          // 1: fused single pass (default), 2: velocity and stress passes
    void* ws = nullptr;      // second state buffer set of the fused form
    size_t ws_bytes = 0;
    void* pad = nullptr;     // first buffer set of padded runs: ws_bytes, or not there
    bool no_pad = false;     // there was no memory for it beside this ws
};

namespace {

template <typename T>
FomTables<T> tables_of(const rom_fom_s* f) {
    const T* b = static_cast<const T*>(f->tables[sizeof(T) == 8 ? 0 : 1]);
    const size_t L = f->tlen;
    return {b, b + L, b + 2 * L, b + 3 * L, b + 4 * L, b + 5 * L, b + 6 * L, b + 7 * L, b + 8 * L};
}

// Launch shape of a run: 16-byte vectors along m when every row starts on a
// 16-byte boundary; a block is bx realization groups x by polar points.
struct FomShape {
    bool wide;
    int bx, by;
};
template <typename T>
FomShape fom_shape(int M, std::initializer_list<const void*> bufs, bool allow_wide = true) {
    constexpr int VWIDE = 16 / (int)sizeof(T);
    FomShape s{allow_wide && M % VWIDE == 0, 1, 0};
    for (const void* p : bufs) s.wide = s.wide && ((uintptr_t)p % 16 == 0);
    const int vw = s.wide ? VWIDE : 1;
    while (s.bx * vw < M && s.bx < 32) s.bx *= 2;
    s.by = kFomThreads / s.bx;
    return s;
}

int fom_sm_count() {
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    return nsm > 0 ? nsm : 1;
}

unsigned fom_blocks(long long work) {
    const long long b = (work + kFomThreads - 1) / kFomThreads;
    return (unsigned)(b < 1 ? 1 : (b > 1024 ? 1024 : b));
}

// Radial rows per block.  A block's time is its rows (seg plus the NS + 1 it
// recomputes or looks ahead) and about two rows' worth of start-up; the blocks
// run in waves of the resident ones.  Short segments fill the GPU when a grid
// or M is small, long ones waste fewer rows.  Measured, us a step, FP32 on
// 512 x 2048: M = 1 (9 strips) 6.4 / 5.8 / 7.2 / 12.2 at 8 / 16 / 32 / 64
// rows, M = 32 (71 strips) 73 / 67 / 65 / 63 / 61 at 8 / 16 / 32 / 64 / 128;
// the rule takes 16 and 128.
template <int NS>
int fom_seg_rows(int Nr, int nstrip, int nsm) {
    const long long slots = (long long)nsm * fom_occupancy<NS>();
    long long best = 0;
    int seg = 1;
    for (int s = 1; s <= kFomMaxSeg && s <= Nr; ++s) {
        const long long waves = ((long long)nstrip * ((Nr + s - 1) / s) + slots - 1) / slots;
        const long long t = waves * (s + NS + 3);
        if (s == 1 || t < best) { best = t; seg = s; }
    }
    return seg;
}

template <typename T, int NS>
cudaError_t launch_march(FomPass<T> a, const FomShape& s, int nsm, cudaStream_t st) {
    constexpr int VWIDE = 16 / (int)sizeof(T);
    const int TJ = s.by - (2 * NS - 1);
    const int nstrip = (a.Nt - 1 + TJ - 1) / TJ;
    a.seg_rows = fom_seg_rows<NS>(a.Nr, nstrip, nsm);
    a.nmarch = nstrip * ((a.Nr + a.seg_rows - 1) / a.seg_rows);
    const unsigned grid = (unsigned)a.nmarch + (a.traces ? fom_blocks((long long)a.nrecv * a.Mt) : 0u);
    const dim3 blk(s.bx, s.by, 1);
    const size_t smem = ((size_t)(2 * NS + 4 * fom_stages<NS>()) * kFomThreads * (s.wide ? VWIDE : 1) +
                         (size_t)8 * (a.seg_rows + NS + 3)) * sizeof(T);
    const void* fn = s.wide ? (const void*)fom_march_kernel<T, VWIDE, NS> : (const void*)fom_march_kernel<T, 1, NS>;
    if (smem > 48 * 1024) {
        const cudaError_t e = allow_smem(fn, smem);
        if (e != cudaSuccess) return e;
    }
    // An FP32 pass may start before the last one has ended: its launch, and what
    // it does before it needs the state, are then hidden (us a step, M = 1:
    // 512 x 2048 6.0 -> 5.7, 40 x 100 2.45 -> 2.12; M = 2, 128 x 512 3.1 -> 2.5).
    // Blocks that come early take whichever SM has room, which costs more than
    // that where the SMs' load matters and the grid leaves some idle (FP64
    // 40 x 100, M = 16 8.6 -> 14; FP32 with four realizations a thread there,
    // M = 33 4.7 -> 5.0).
    const bool early = sizeof(T) == 4 && (!s.wide || a.nmarch >= nsm * fom_occupancy<NS>());
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = blk;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = early ? 1 : 0;
    void* args[] = {(void*)&a};
    return cudaLaunchKernelExC(&cfg, fn, args);
}

// Passes over `count` steps from step a.off on, two steps a pass in FP32.
// The buffers alternate from pass to pass; with an odd number of passes the
// result ends in the second set (*odd).  Of the FP32 splits of `count` into
// two-step and one-step passes the one with the fewest passes of an even
// number is taken (count = 1 alone has none), so no copy follows.
template <typename T>
cudaError_t march_steps(FomPass<T> a, const FomShape& s, int nsm, int count, cudaStream_t st, bool* odd) {
    int pairs = sizeof(T) == 4 ? count / 2 : 0;
    if ((count - pairs) % 2 != 0 && pairs > 0) --pairs;
    const int passes = count - pairs;
    cudaError_t e = cudaSuccess;
    for (int p = 0; p < passes && e == cudaSuccess; ++p) {
        const bool two = p < pairs;
        if (two) e = launch_march<T, sizeof(T) == 4 ? 2 : 1>(a, s, nsm, st);
        else e = launch_march<T, 1>(a, s, nsm, st);
        a.off += two ? 2 : 1;
        T *v = const_cast<T*>(a.Vo), *s1 = const_cast<T*>(a.S1o), *s2 = const_cast<T*>(a.S2o);
        a.Vo = a.Vn; a.S1o = a.S1n; a.S2o = a.S2n;
        a.Vn = v; a.S1n = s1; a.S2n = s2;
    }
    *odd = passes % 2 != 0;
    return e;
}

cudaError_t end_capture(cudaStream_t cap, cudaError_t e, cudaGraphExec_t* out) {
    cudaGraph_t g = nullptr;
    const cudaError_t e2 = cudaStreamEndCapture(cap, &g);
    if (e == cudaSuccess) e = e2;
    if (e == cudaSuccess) e = cudaGraphInstantiate(out, g, 0);
    if (g) cudaGraphDestroy(g);
    return e;
}

// The fused form's graph: kFomGraphSteps steps from step ctl->step on.
template <typename T>
cudaError_t capture_march(rom_fom_s* f, FomPass<T> a, const FomShape& s, int nsm, cudaGraphExec_t* out) {
    cudaError_t e = cudaStreamBeginCapture(f->cap, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return e;
    bool odd = false;
    a.off = 0;
    e = march_steps<T>(a, s, nsm, kFomGraphSteps, f->cap, &odd);
    if (e == cudaSuccess) {
        fom_advance_kernel<<<1, 1, 0, f->cap>>>(f->ctl, kFomGraphSteps);
        e = cudaGetLastError();
    }
    return end_capture(f->cap, e, out);
}

// The two-pass form's graph: kFomGraphSteps steps, steps past nsteps idle.
template <typename T>
cudaError_t capture_steps(rom_fom_s* f, const FomArgs<T>& a, const FomShape& s, int nsm, cudaGraphExec_t* out) {
    constexpr int VWIDE = 16 / (int)sizeof(T);
    const dim3 blk(s.bx, s.by, 1);
    // persistent grids: the resident blocks of every SM stride over the tiles
    auto grid_for = [&](const void* fn, long long tiles) {
        int per = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, kFomThreads, 0) != cudaSuccess || per < 1)
            per = 1;
        const long long g = (long long)nsm * per;
        return (unsigned)(tiles < g ? (tiles < 1 ? 1 : tiles) : g);
    };
    const long long gx = (a.Nt - 1 + s.by - 1) / s.by;
    const void* fv = s.wide ? (const void*)fom_velocity_kernel<T, VWIDE> : (const void*)fom_velocity_kernel<T, 1>;
    const void* fs = s.wide ? (const void*)fom_stress_kernel<T, VWIDE> : (const void*)fom_stress_kernel<T, 1>;
    const unsigned gv = grid_for(fv, (long long)a.Nr * gx);
    const unsigned gs = grid_for(fs, (long long)(2 * a.Nr - 1) * gx);
    cudaError_t e = cudaStreamBeginCapture(f->cap, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return e;
    for (int k = 0; k < kFomGraphSteps && e == cudaSuccess; ++k) {
        if (s.wide) fom_velocity_kernel<T, VWIDE><<<gv, blk, 0, f->cap>>>(a);
        else fom_velocity_kernel<T, 1><<<gv, blk, 0, f->cap>>>(a);
        if (a.Tper) fom_source_kernel<T><<<fom_blocks(a.M), kFomThreads, 0, f->cap>>>(a);
        if (a.traces) fom_record_kernel<T><<<fom_blocks((long long)a.nrecv * a.M), kFomThreads, 0, f->cap>>>(a);
        if (s.wide) fom_stress_kernel<T, VWIDE><<<gs, blk, 0, f->cap>>>(a);
        else fom_stress_kernel<T, 1><<<gs, blk, 0, f->cap>>>(a);
        fom_tick_kernel<<<1, 1, 0, f->cap>>>(const_cast<FomCtl*>(a.ctl));
        e = cudaGetLastError();
    }
    return end_capture(f->cap, e, out);
}

// The checked arguments of one rom_fom_run call.
struct FomRun {
    void *V, *S1, *S2, *V2, *S12, *S22;
    const void* T;
    const int* recv;
    void* traces;
    int M, nsteps;
    long n0;
    int src, wavelet, nrecv, r;
    bool fused;
    int Mp;             // realizations per row of the fused form's buffers: M, or padded
    void *Vp, *S1p, *S2p;  // padded: the first buffer set (V2, S12, S22 are the second)
};

// Should a thread of the fused FP32 form take 4 realizations with 16-byte
// accesses (n unknowns)?  One realization a thread shortens the chain of a row
// while the grid does not fill the GPU; with more, it is bound by its scalar
// accesses and, above 16 realizations, by the strips that 32 lanes along m
// leave.  us a step, one / four (padded to a multiple of 4): 512 x 2048
// M = 2 9.0 / 11.6, 3 16.1 / 11.7, 9 66 / 33, 17 154 / 59, 33 304 / 119;
// 256 x 1024 M = 3 5.8 / 6.8, 5 9.2 / 8.0; 128 x 512 M = 9 6.3 / 6.5,
// 13 6.3 / 6.3, 17 13.0 / 7.9; 64 x 256 M = 15 3.6 / 4.7, 26 5.1 / 5.6,
// 33 8.9 / 6.6; 40 x 100 M = 5 2.5 / 4.4, 33 5.0 / 4.7.
bool fom_wide(long long n, int M) {
    return M > 32 || (M >= 3 && n * M >= (M > 16 ? 1500000 : 2500000));
}
// A run of that kind whose M is not a multiple of 4 marches on copies padded to
// one, except for a few steps, which the copies would cost as much as, and where
// there is no memory for the copies.
bool fom_padded(long long n, int M, int nsteps) { return M % 4 != 0 && nsteps >= 16 && fom_wide(n, M); }

// The buffers of the fused form for sets of `need` bytes.  They grow to `want`
// (rows of a multiple of 16 bytes, so that a padded run asks for no more than a
// run of its M) where there is room.
cudaError_t fom_grow(rom_fom_s* f, size_t need, size_t want, cudaStream_t st) {
    if (f->ws_bytes >= need) return cudaSuccess;
    cudaStreamSynchronize(st);
    cudaDeviceSynchronize();
    for (auto& kv : f->graphs) cudaGraphExecDestroy(kv.second);
    f->graphs.clear();
    cudaFree(f->ws);
    cudaFree(f->pad);
    f->ws = f->pad = nullptr;
    f->ws_bytes = 0;
    f->no_pad = false;
    cudaError_t e = cudaMalloc(&f->ws, want);
    if (e == cudaErrorMemoryAllocation && want > need) {
        cudaGetLastError();
        want = need;
        e = cudaMalloc(&f->ws, want);
    }
    if (e == cudaSuccess) f->ws_bytes = want;
    return e;
}

// Are there copies for a padded run with sets of `bytes`?  They have the size of
// the second set, whatever this run needs: so they are allocated once for it,
// and no later run frees what a caller's graph may hold.  Not allocated in a
// stream capture; a failure is remembered.
bool fom_pad_buffers(rom_fom_s* f, size_t bytes, cudaStream_t st) {
    if (f->ws_bytes < bytes || f->no_pad) return false;
    if (f->pad) return true;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return false;
    }
    const cudaError_t e = cudaMalloc(&f->pad, f->ws_bytes);
    if (e == cudaSuccess) return true;
    cudaGetLastError();
    f->pad = nullptr;
    f->no_pad = e == cudaErrorMemoryAllocation;
    return false;
}

// The graph of a run's buffers and arguments, captured on its first use.
template <typename F>
cudaError_t cached_graph(rom_fom_s* f, const std::vector<long long>& key, cudaStream_t st, F capture,
                         cudaGraphExec_t* out) {
    auto it = f->graphs.find(key);
    if (it == f->graphs.end()) {
        cudaGraphExec_t ge = nullptr;
        const cudaError_t e = capture(&ge);
        if (e != cudaSuccess) return e;
        if (f->graphs.size() >= 16) {  // keep the cache small
            cudaStreamSynchronize(st);
            for (auto& kv : f->graphs) cudaGraphExecDestroy(kv.second);
            f->graphs.clear();
        }
        it = f->graphs.emplace(key, ge).first;
    }
    *out = it->second;
    return cudaSuccess;
}

template <typename T>
cudaError_t run_fom(rom_fom_s* f, const FomRun& q, cudaStream_t st) {
    const size_t nv = (size_t)f->Nr * (f->Nt - 1), n1 = (size_t)(f->Nr - 1) * (f->Nt - 1),
                 n2 = (size_t)f->Nr * (f->Nt - 2);
    const int nsm = fom_sm_count();
    const bool pad = q.Mp != q.M;
    void *V = pad ? q.Vp : q.V, *S1 = pad ? q.S1p : q.S1, *S2 = pad ? q.S2p : q.S2;
    const FomShape s = fom_shape<T>(q.Mp, {V, S1, S2, q.V2, q.S12, q.S22},
                                    !q.fused || sizeof(T) == 8 || fom_wide((long long)(nv + n1 + n2), q.M));
    const std::vector<long long> key = {(long long)(uintptr_t)V, (long long)(uintptr_t)S1,
                                        (long long)(uintptr_t)S2, q.M, q.Mp, q.src, (long long)(uintptr_t)q.T,
                                        q.wavelet, (long long)(uintptr_t)q.recv, q.nrecv, q.traces ? q.r : 0,
                                        (long long)(uintptr_t)q.traces, (long long)sizeof(T), q.fused,
                                        (long long)(uintptr_t)q.V2};
    cudaGraphExec_t ge = nullptr;
    cudaError_t e = cudaSuccess;
    if (!q.fused) {
        const FomArgs<T> a = {tables_of<T>(f), static_cast<T*>(q.V), static_cast<T*>(q.S1), static_cast<T*>(q.S2),
                              static_cast<const T*>(q.T), q.recv, static_cast<T*>(q.traces), f->ctl, f->Nr, f->Nt,
                              q.M, q.src, q.nrecv, q.r, q.wavelet, f->dt, f->rho};
        e = cached_graph(f, key, st, [&](cudaGraphExec_t* g) { return capture_steps<T>(f, a, s, nsm, g); }, &ge);
        if (e != cudaSuccess) return e;
        fom_set_kernel<<<1, 1, 0, st>>>(f->ctl, q.nsteps, q.n0);
        e = cudaGetLastError();
        for (int k = 0; k < (q.nsteps + kFomGraphSteps - 1) / kFomGraphSteps && e == cudaSuccess; ++k)
            e = cudaGraphLaunch(ge, st);
        return e;
    }
    FomPass<T> a{};
    a.tb = tables_of<T>(f);
    a.Vo = static_cast<T*>(V), a.S1o = static_cast<T*>(S1), a.S2o = static_cast<T*>(S2);
    a.Vn = static_cast<T*>(q.V2), a.S1n = static_cast<T*>(q.S12), a.S2n = static_cast<T*>(q.S22);
    a.Tper = static_cast<const T*>(q.T);
    a.recv = q.recv;
    a.traces = static_cast<T*>(q.traces);
    a.n0 = q.n0;
    a.Nr = f->Nr, a.Nt = f->Nt, a.M = q.Mp, a.Mt = q.M;
    a.nrecv = q.nrecv, a.r = q.r, a.wavelet = q.wavelet;
    a.src_i = q.src >= 0 ? q.src / (f->Nt - 1) : -1;
    a.src_j = q.src >= 0 ? q.src % (f->Nt - 1) + 1 : -1;
    a.dt = f->dt, a.rho = f->rho;
    auto copies = [&](bool in, void* v, void* s1, void* s2) {
        const std::pair<void*, size_t> user[3] = {{q.V, nv}, {q.S1, n1}, {q.S2, n2}};
        void* own[3] = {v, s1, s2};
        for (int i = 0; i < 3; ++i) {
            const long long n = (long long)user[i].second;
            const long long b = (n * q.Mp + kFomThreads - 1) / kFomThreads;
            const unsigned grid = (unsigned)(b < 8LL * nsm ? b : 8LL * nsm);
            float *u = static_cast<float*>(user[i].first), *p = static_cast<float*>(own[i]);
            if (in) fom_pad_kernel<true><<<grid, kFomThreads, 0, st>>>(u, n, q.M, q.Mp, p);
            else fom_pad_kernel<false><<<grid, kFomThreads, 0, st>>>(p, n, q.M, q.Mp, u);
        }
        return cudaGetLastError();
    };
    if (pad) {
        e = copies(true, V, S1, S2);
        if (e != cudaSuccess) return e;
    }
    // whole groups of kFomGraphSteps steps by graph, the rest launched
    const int reps = q.nsteps / kFomGraphSteps;
    if (reps > 0) {
        FomPass<T> g = a;
        g.ctl = f->ctl;
        e = cached_graph(f, key, st, [&](cudaGraphExec_t* x) { return capture_march<T>(f, g, s, nsm, x); }, &ge);
        if (e != cudaSuccess) return e;
        fom_set_kernel<<<1, 1, 0, st>>>(f->ctl, q.nsteps, q.n0);
        e = cudaGetLastError();
        for (int k = 0; k < reps && e == cudaSuccess; ++k) e = cudaGraphLaunch(ge, st);
    }
    bool odd = false;
    a.off = (long long)reps * kFomGraphSteps;
    if (e == cudaSuccess) e = march_steps<T>(a, s, nsm, q.nsteps - reps * kFomGraphSteps, st, &odd);
    const T* Vend = static_cast<const T*>(odd ? q.V2 : V);
    if (e == cudaSuccess && pad) {
        e = copies(false, odd ? q.V2 : V, odd ? q.S12 : S1, odd ? q.S22 : S2);
    } else if (e == cudaSuccess && odd) {
        e = cudaMemcpyAsync(q.V, q.V2, nv * q.M * sizeof(T), cudaMemcpyDeviceToDevice, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(q.S1, q.S12, n1 * q.M * sizeof(T), cudaMemcpyDeviceToDevice, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(q.S2, q.S22, n2 * q.M * sizeof(T), cudaMemcpyDeviceToDevice, st);
    }
    if (e == cudaSuccess && a.traces && q.nsteps % q.r == 0) {
        // a pass records the velocity it finds: the last step's record is left
        fom_last_record_kernel<T><<<fom_blocks((long long)q.nrecv * q.M), kFomThreads, 0, st>>>(
            Vend, q.recv, q.nrecv, q.Mp, q.M,
            a.traces + (size_t)(q.nsteps / q.r - 1) * q.nrecv * q.M);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace

extern "C" {

rom_status rom_fom_create(int Nr, int Ntheta, double r_cmb, double r_earth, double rho, double vs,
                          double dt, rom_fom_t* out) {
    if (!out) return ROM_E_INVAL;
    *out = nullptr;
    if (Nr < 2 || Nr > 65535 || Ntheta < 3 || !(r_cmb > 0.0) || !(r_earth > r_cmb) || !(rho > 0.0) || !(vs > 0.0) ||
        !(dt > 0.0) || !isfinite(r_earth) || !isfinite(rho) || !isfinite(vs) || !isfinite(dt))
        return ROM_E_INVAL;
    const long long nv = (long long)Nr * (Ntheta - 1);
    if (nv * 3 > (1LL << 31)) return ROM_E_INVAL;  // unknown indices stay below 2^31 per field
    rom_fom_s* f = new (std::nothrow) rom_fom_s();
    if (!f) return ROM_E_NOMEM;
    f->Nr = Nr;
    f->Nt = Ntheta;
    f->r_cmb = r_cmb;
    f->r_earth = r_earth;
    f->rho = rho;
    f->vs = vs;
    f->dt = dt;
    const size_t L = (size_t)(Nr > Ntheta ? Nr : Ntheta) + 1;
    f->tlen = L;
    // the stencil factors in FP64 on the host (see the header comment)
    const double dr = (r_earth - r_cmb) / Nr, dth = 3.14159265358979323846 / Ntheta;
    const double mu = rho * vs * vs;
    std::vector<double> t(9 * L, 0.0);
    double *cr_p = &t[0], *cr_m = &t[L], *inv_rh = &t[2 * L], *pt_p = &t[3 * L], *pt_m = &t[4 * L];
    double *q_u = &t[5 * L], *q_d = &t[6 * L], *w_p = &t[7 * L], *w_m = &t[8 * L];
    for (int i = 0; i < Nr; ++i) {
        const double rm = r_cmb + i * dr, rp = r_cmb + (i + 1) * dr, rh = r_cmb + (i + 0.5) * dr;
        const double rh3 = rh * rh * rh;
        cr_p[i] = i + 1 < Nr ? rp * rp * rp / (rho * rh3 * dr) : 0.0;
        cr_m[i] = i >= 1 ? rm * rm * rm / (rho * rh3 * dr) : 0.0;
        inv_rh[i] = 1.0 / rh;
        if (i >= 1) {
            const double rl = r_cmb + (i - 0.5) * dr;
            q_u[i] = mu * rm / (rh * dr);
            q_d[i] = mu * rm / (rl * dr);
        }
    }
    for (int j = 1; j < Ntheta; ++j) {
        const double s = sin(j * dth), sp = sin((j + 0.5) * dth), sm = sin((j - 0.5) * dth);
        pt_p[j] = j <= Ntheta - 2 ? sp * sp / (rho * s * s * dth) : 0.0;
        pt_m[j] = j >= 2 ? sm * sm / (rho * s * s * dth) : 0.0;
        if (j <= Ntheta - 2) {
            w_p[j] = mu * sp / (sin((j + 1) * dth) * dth);
            w_m[j] = mu * sp / (s * dth);
        }
    }
    std::vector<float> tf(t.begin(), t.end());
    cudaError_t e = cudaMalloc(&f->tables[0], t.size() * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&f->tables[1], tf.size() * sizeof(float));
    if (e == cudaSuccess) e = cudaMemcpy(f->tables[0], t.data(), t.size() * sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(f->tables[1], tf.data(), tf.size() * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMalloc(&f->ctl, sizeof(FomCtl));
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&f->cap, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
        cudaFree(f->tables[0]);
        cudaFree(f->tables[1]);
        cudaFree(f->ctl);
        if (f->cap) cudaStreamDestroy(f->cap);
        delete f;
        set_last_error(cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? ROM_E_NOMEM : ROM_E_CUDA;
    }
    *out = f;
    return ROM_OK;
}

rom_status rom_fom_destroy(rom_fom_t f) {
    if (!f) return ROM_E_INVAL;
    cudaDeviceSynchronize();
    for (auto& kv : f->graphs) cudaGraphExecDestroy(kv.second);
    cudaFree(f->tables[0]);
    cudaFree(f->tables[1]);
    cudaFree(f->ctl);
    cudaFree(f->ws);
    cudaFree(f->pad);
    if (f->cap) cudaStreamDestroy(f->cap);
    delete f;
    return ROM_OK;
}

rom_status rom_fom_set_passes(rom_fom_t f, int passes) {
    if (!f || (passes != 1 && passes != 2)) return ROM_E_INVAL;
    std::lock_guard<std::mutex> lk(f->mu);
    f->passes = passes;
    return ROM_OK;
}

rom_status rom_fom_dims(rom_fom_t f, int* nv, int* n1, int* n2) {
    if (!f) return ROM_E_INVAL;
    if (nv) *nv = f->Nr * (f->Nt - 1);
    if (n1) *n1 = (f->Nr - 1) * (f->Nt - 1);
    if (n2) *n2 = f->Nr * (f->Nt - 2);
    return ROM_OK;
}

rom_status rom_fom_run(rom_fom_t f, void* V, void* S1, void* S2, int M, int nsteps, long n0,
                       int src, const void* T, int wavelet, const int* recv, int nrecv, int r,
                       void* traces, int prec, void* stream) {
    if (!f || !V || !S1 || !S2 || M < 1 || nsteps < 0 || n0 < 0) return ROM_E_INVAL;
    if (prec != ROM_FP32 && prec != ROM_FP64) return ROM_E_UNSUPPORTED;
    if (wavelet != ROM_WAVELET_RICKER && wavelet != ROM_WAVELET_GAUSS1) return ROM_E_INVAL;
    const long long nv = (long long)f->Nr * (f->Nt - 1);
    const long long ns = (long long)(f->Nr - 1) * (f->Nt - 1) + (long long)f->Nr * (f->Nt - 2);
    if (src >= nv || (T && src < 0)) return ROM_E_INVAL;
    if (traces && (r < 1 || nrecv < 1 || !recv)) return ROM_E_INVAL;
    if ((long long)M * (nv > ns ? nv : ns) > (1LL << 40)) return ROM_E_INVAL;
    cudaPointerAttributes at;
    for (const void* p : {(const void*)V, (const void*)S1, (const void*)S2, T, (const void*)recv,
                          (const void*)traces}) {
        if (!p) continue;
        if (cudaPointerGetAttributes(&at, p) != cudaSuccess ||
            (at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged)) {
            cudaGetLastError();
            set_last_error("rom_fom_run: device buffers only");
            return ROM_E_INVAL;
        }
    }
    if (nsteps == 0) return ROM_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    std::lock_guard<std::mutex> lk(f->mu);
    // the fused pass writes every other step into a second buffer set
    const bool fused = f->passes == 1;
    const size_t es = prec == ROM_FP64 ? 8 : 4;
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const long long n1 = (long long)(f->Nr - 1) * (f->Nt - 1), n2 = (long long)f->Nr * (f->Nt - 2);
    auto set_bytes = [&](long long m) {
        return al((size_t)(nv * m) * es) + al((size_t)(n1 * m) * es) + al((size_t)(n2 * m) * es);
    };
    const long long per = 16 / (long long)es, Mw = (M + per - 1) / per * per;
    bool pad = false;
    if (fused) {
        const cudaError_t em = fom_grow(f, set_bytes(M), set_bytes(Mw), st);
        if (em != cudaSuccess) {
            set_last_error(cudaGetErrorString(em));
            return em == cudaErrorMemoryAllocation ? ROM_E_NOMEM : ROM_E_CUDA;
        }
        pad = prec == ROM_FP32 && fom_padded(nv + ns, M, nsteps) && fom_pad_buffers(f, set_bytes(Mw), st);
    }
    const int Mp = pad ? (int)Mw : M;
    FomRun q{V, S1, S2, nullptr, nullptr, nullptr, T, recv, traces, M, nsteps, n0, src, wavelet, nrecv,
             traces ? r : 1, fused, Mp, nullptr, nullptr, nullptr};
    if (fused) {
        const size_t bV = al((size_t)(nv * Mp) * es), b1 = al((size_t)(n1 * Mp) * es);
        char* w = static_cast<char*>(f->ws);
        q.V2 = w, q.S12 = w + bV, q.S22 = w + bV + b1;
        w = static_cast<char*>(f->pad);
        if (pad) q.Vp = w, q.S1p = w + bV, q.S2p = w + bV + b1;
    }
    const cudaError_t e = prec == ROM_FP64 ? run_fom<double>(f, q, st) : run_fom<float>(f, q, st);
    if (e != cudaSuccess) {
        set_last_error(cudaGetErrorString(e));
        return ROM_E_CUDA;
    }
    return ROM_OK;
}

}  // extern "C"
