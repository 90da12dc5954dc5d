// Host planning / launch of the one-CTA rank-2 kernel (FP32, Kp <= 128).
#include <cuda_runtime.h>

#include "rank2_cta.cuh"
#include "rank2_launch.cuh"

namespace romk {

template <int KI, bool XR>
static void* cta_kernel_for(int cb) {
    return cb == 1   ? (void*)&rank2_cta_kernel<KI, 1, XR>
           : cb == 2 ? (void*)&rank2_cta_kernel<KI, 2, XR>
                     : (void*)&rank2_cta_kernel<KI, 4, XR>;
}
static void* cta_kernel(int KI, int cb, bool xr) {
    if (KI == 1) return xr ? cta_kernel_for<1, true>(cb) : cta_kernel_for<1, false>(cb);
    return xr ? cta_kernel_for<2, true>(cb) : cta_kernel_for<2, false>(cb);
}

// One block of Wv columns per CTA, as few as spread M over the CTAs that are
// resident at once (one per SM at Kp = 128, two at Kp = 64).  Receiver rows
// are staged while they take less than 64 KB.
bool plan_rank2_cta_f32(int Kp, int M, int R, Rank2Plan* p) {
    if ((Kp != 64 && Kp != 128) || M <= 0) return false;
    p->KI = Kp / 64;
    p->cs = 1;
    p->nrt = 1;
    p->resident = true;
    p->variant = 5;
    p->c_global = (size_t)R * Kp * sizeof(float) > 64 * 1024;
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (nsm <= 0) return false;
    const int slots = nsm * (Kp == 64 ? 2 : 1);
    p->max_active_clusters = slots;
    int w = (M + slots - 1) / slots;
    const int smax = device_smem_optin();
    const int nC = p->c_global ? 0 : R;
    w = w <= 2 ? w : (w + 3) / 4 * 4;
    while (w > 4 && cta_smem_layout(w, Kp, nC).total > (size_t)smax / (Kp == 64 ? 2 : 1)) w -= 4;
    p->cb = w <= 2 ? w : 4;
    p->Wv = p->Wa = w;
    p->nclusters = (M + w - 1) / w;
    p->smem = cta_smem_layout(w, Kp, nC).total;
    return p->smem <= (size_t)smax;
}

cudaError_t launch_rank2_cta_f32(const Rank2Args& a_in, const Rank2Plan& p, cudaStream_t st) {
    Rank2Args a = a_in;
    a.Wv = p.Wv;
    a.Wa = p.Wa;
    a.c_global = p.c_global ? 1 : 0;
    void* fn = cta_kernel(p.KI, p.cb, a.Xv != nullptr || a.Xs != nullptr);
    cudaError_t e = allow_smem(fn, p.smem);
    if (e != cudaSuccess) return e;
    void* args[] = {(void*)&a};
    return cudaLaunchKernel(fn, dim3((unsigned)p.nclusters), dim3(kThreads), args, p.smem, st);
}

}  // namespace romk
