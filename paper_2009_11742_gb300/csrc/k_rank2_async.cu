// Host planning / launch of the one-block kernel with asynchronous exchange
// (FP32, Kp <= 512; FP64, Kp <= 256).
#include <cuda_runtime.h>

#include "rank2_async_launch.cuh"
#include "rank2_launch.cuh"

namespace romk {

template <typename T>
static void* async_kernel(int KI, int cb) { return async_instance<T, false>(KI, cb); }

// Does a run take its traces in tiles of receivers (rpc of them a CTA)?  us a step
// with one dot product a warp at a time / in tiles, records on every step: rank-1
// FP32 K = 512 16 receivers (1 a CTA) 1.35 / 1.39, 100 (7) 1.53 / 1.42, 1000 8.4
// / 2.1; FP64 K = 256, M = 100 1000 receivers 174 / 110.  In FP64 a tile of few
// receivers keeps one warp at it where several shared the dot products.
static bool async_many(const Rank2Args& a, int cb, bool f64) {
    return a.traces && (f64 ? a.rpc >= 32 : cb < 4 && a.rpc >= 6);
}

// The column group for w columns.  FP64 is bound by the FP64 units, so no
// column that is not there is computed unless the wider group's cheaper
// reduction and epilogue make up for it; FP32 takes the widest group in use.
static int async_group(int w, bool f64) {
    if (!f64) return w >= 3 ? 4 : w;
    int best = 1;
    double t = 1e30;
    for (int cb : {4, 2, 1}) {
        const double x = (w + cb - 1) / cb * cb * (cb == 4 ? 1.0 : cb == 2 ? 1.06 : 1.2);
        if (x < t) {
            t = x;
            best = cb;
        }
    }
    return best;
}

template <typename T>
static bool plan_async(int Kp, int M, int R, Rank2Plan* p) {
    if (Kp <= 0 || Kp % 64 != 0 || Kp > (sizeof(T) == 4 ? 512 : 256) || M <= 0) return false;
    p->KI = Kp / 64;
    p->cs = Kp / kRowsPerCta;
    p->nrt = 1;
    p->resident = true;
    p->variant = 1;
    const int rpc = (R + p->cs - 1) / p->cs;
    const size_t smax = (size_t)device_smem_optin();
    auto bytes = [&](int w, int cb, int nC) { return async_smem_layout<T>(w, w / cb, Kp, nC).total; };
    // one CTA per SM
    void* probe_fn = async_kernel<T>(p->KI, 4);
    const size_t probe_smem = smax / 2 + 1024;
    if (prepare_kernel<T>(probe_fn, probe_smem) != cudaSuccess) return false;
    ClusterLaunch probe(p->cs, 1, kThreads, probe_smem);
    p->max_active_clusters = probe.max_active(probe_fn);
    if (p->max_active_clusters <= 0) return false;
    int w = (M + p->max_active_clusters - 1) / p->max_active_clusters;
    p->cb = async_group(w, sizeof(T) == 8);
    w = (w + p->cb - 1) / p->cb * p->cb;
    // receiver rows are staged while they take at most 64 KB, or fit beside the
    // columns
    p->c_global = (size_t)rpc * Kp * sizeof(T) > 64 * 1024 && bytes(w, p->cb, rpc) > smax;
    const int nC = p->c_global ? 0 : rpc;
    while (w > p->cb && bytes(w, p->cb, nC) > smax) w -= p->cb;
    p->Wv = p->Wa = w;
    p->nclusters = (M + w - 1) / w;
    p->smem = bytes(w, p->cb, nC);
    p->async = p->smem <= smax;
    return p->async;
}

template <typename T>
static cudaError_t launch_async(const Rank2Args& a_in, const Rank2Plan& p, cudaStream_t st) {
    Rank2Args a = a_in;
    a.Wv = p.Wv;
    a.Wa = p.Wa;
    a.rpc = (a.R + p.cs - 1) / p.cs;
    a.c_global = p.c_global ? 1 : 0;
    void* fn = async_many(a, p.cb, sizeof(T) == 8) ? async_many_kernel(sizeof(T) == 8, p.KI, p.cb)
                                                   : async_kernel<T>(p.KI, p.cb);
    if (!fn || a.group) return cudaErrorInvalidValue;
    cudaError_t e = prepare_kernel<T>(fn, p.smem);
    if (e != cudaSuccess) return e;
    ClusterLaunch L(p.cs, p.nclusters, kThreads, p.smem, st);
    void* args[] = {(void*)&a};
    return L.launch(fn, args);
}

bool plan_rank2_async(int Kp, int M, int R, bool f64, Rank2Plan* p) {
    return f64 ? plan_async<double>(Kp, M, R, p) : plan_async<float>(Kp, M, R, p);
}

// us a step, this kernel / two-block kernel, at W columns per cluster (the
// two-block kernel with the same M: two blocks of 4):
//     K = 192: W = 4 1.21 / 1.39, 8 1.96 / 1.40
//     K = 256: W = 4 1.43 / 1.59, 8 2.21 / 1.66
//     K = 384: W = 4 1.77 / 2.12, 8 2.96 / 2.13
//     K = 512: W = 2 1.72 / 2.59, 4 2.29 / 2.60, 8 3.71 / 2.61
// Above 4 the two-block kernel's 4 rows a thread (half the operand reads per
// product) win over the shorter chain of a half-step.
bool async_beats_two_block(int W) { return W <= 4; }
cudaError_t launch_rank2_async(const Rank2Args& a, const Rank2Plan& p, bool f64, cudaStream_t st) {
    return f64 ? launch_async<double>(a, p, st) : launch_async<float>(a, p, st);
}

}  // namespace romk
