// Host planning / launch of the split-role FP32 rank-2 kernel.
#include <cuda_runtime.h>

#include "rank2_launch.cuh"
#include "rank2_split.cuh"

namespace romk {

// mode: the instance (0 plain, 1 with the reduced reference state, 2 rank-3 grouped).
static void* two_block_kernel(int KI, int mode = 0) {
#define ROM_TB_CASE(k)                                                          \
    case k:                                                                     \
        return mode == 2   ? (void*)&rank2_split_kernel<k, 2>                   \
               : mode == 1 ? (void*)&rank2_split_kernel<k, 1>                   \
                           : (void*)&rank2_split_kernel<k, 0>;
    switch (KI) {
        ROM_TB_CASE(1) ROM_TB_CASE(2) ROM_TB_CASE(3) ROM_TB_CASE(4)
        ROM_TB_CASE(5) ROM_TB_CASE(6) ROM_TB_CASE(7) ROM_TB_CASE(8)
        default: return nullptr;
    }
#undef ROM_TB_CASE
}

bool plan_rank2_split_f32(int Kp, int M, int R, Rank2Plan* p, int cluster_budget) {
    if (Kp <= 0 || Kp % 64 != 0 || Kp > 512 || M <= 0) return false;
    p->KI = Kp / 64;
    p->cs = Kp / 32;  // H = Kp / 64 CTAs per role
    p->cb = kSplitCB;
    p->resident = true;
    p->variant = 2;
    const int H = p->cs / 2;
    const int rpc = (R + H - 1) / H;
    const int smax = device_smem_optin();
    int wcap = 0;
    for (int w = kSplitBlock; w <= 2048; w += kSplitBlock) {
        if (split_smem_layout(w, Kp, rpc).total > (size_t)smax) break;
        wcap = w;
    }
    if (wcap == 0) return false;
    void* fn = two_block_kernel(p->KI);
    if (!fn) return false;
    const size_t smem_probe = split_smem_layout(wcap, Kp, rpc).total;
    if (prepare_kernel<float>(fn, smem_probe) != cudaSuccess) return false;
    ClusterLaunch probe(p->cs, 1, kThreads, smem_probe);
    const int nact = probe.max_active(fn);
    if (nact <= 0) return false;
    p->max_active_clusters = nact;
    const int budget = cluster_budget > 0 && cluster_budget < nact ? cluster_budget : nact;
    p->nrt = 1;
    int wv = (M + 2 * budget - 1) / (2 * budget);
    wv = ((wv + kSplitBlock - 1) / kSplitBlock) * kSplitBlock;
    if (wv > wcap) {
        // more than one wave: as few as shared memory allows, of equal width
        const int waves = (M + 2 * budget * wcap - 1) / (2 * budget * wcap);
        wv = (M + 2 * budget * waves - 1) / (2 * budget * waves);
        wv = ((wv + kSplitBlock - 1) / kSplitBlock) * kSplitBlock;
    }
    p->Wv = wv;
    p->Wa = wv;
    const int nblocks = (M + wv - 1) / wv;
    p->nclusters = (nblocks + 1) / 2;
    p->smem = split_smem_layout(p->Wa, Kp, rpc).total;
    return true;
}

cudaError_t launch_rank2_split_f32(const Rank2Args& a_in, const Rank2Plan& p, cudaStream_t st, cudaEvent_t started) {
    Rank2Args a = a_in;
    a.Wv = p.Wv;
    a.Wa = p.Wa;
    const int H = p.cs / 2;
    a.rpc = (a.R + H - 1) / H;
    const int mode = a.group ? 2 : (a.Xv != nullptr || a.Xs != nullptr ? 1 : 0);
    if (a.group && (a.Xv || a.Xs)) return cudaErrorInvalidValue;
    void* fn = two_block_kernel(p.KI, mode);
    if (!fn) return cudaErrorInvalidValue;
    cudaError_t e = prepare_kernel<float>(fn, p.smem);
    if (e != cudaSuccess) return e;
    ClusterLaunch L(p.cs, p.nclusters, kThreads, p.smem, st);
    if (started) L.record_started(started);
    void* args[] = {(void*)&a};
    return L.launch(fn, args);
}

}  // namespace romk
