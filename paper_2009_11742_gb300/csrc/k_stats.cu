// Ensemble statistics of receiver traces (mean and quantile bands over the
// realizations, Sec. 4.5.2).  A column is the M values of one (record,
// receiver) pair.  A block stages a tile of columns in shared memory (the
// receivers of a record are contiguous, so its reads are), and one warp (2 or
// 4 above 1024 values) sorts a column in registers and reads the order
// statistics of the Hyndman-Fan type 7 quantiles off it.
//
// Bound: the ALU pipe, by the network's min / max (45 steps of 16 elements a
// lane at M = 512).  1000 records x 64 receivers x 512 realizations: 180 us
// against 774 us for one block per column with a shared-memory bitonic network
// behind 45 block barriers, whose reads took 4 bytes of every sector; the
// traces alone are 20 us of HBM traffic.  FP64 is kept out of the columns'
// loop: a warp's FP64 addition holds an SM's FP64 units for 16 cycles, so
// adding up the means there would by itself take about 90 us.
#include <cuda_runtime.h>
#include <math.h>

#include "../../include/rom.h"
#include "rom_internal.h"

namespace romk {

constexpr int kStatThreads = 256;
constexpr int kStatWarps = kStatThreads / 32;
constexpr int kStatMaxM = 4096;
constexpr int kStatMaxP = 16;

struct StatArgs {
    const float* traces;
    double* mean_out;
    double* q_out;
    double t[kStatMaxP];   // interpolation weight of each quantile
    int lo[kStatMaxP];     // and its lower order statistic
    int nrec, R, M, nprobs;
    int G;                 // columns per tile
    int nj, nr;            // a tile's receivers and records (nj nr <= G)
};

// Float bits in an order-preserving integer form, and back.
__device__ __forceinline__ int stat_key(int b) { return b ^ ((b >> 31) & 0x7fffffff); }

// Compare-exchange with the partner's value: keep the larger if up.
__device__ __forceinline__ int stat_keep(int x, int o, bool up) { return up ? max(x, o) : min(x, o); }

// The merging steps of strides TOP, TOP / 2, .. 1 (element index: lane EPL + e).
template <int EPL, int TOP>
__device__ __forceinline__ void stat_halve(int (&x)[EPL], int lane) {
    if constexpr (TOP >= EPL) {
        const int o = TOP / EPL;
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int e = 0; e < EPL; ++e) x[e] = stat_keep(x[e], __shfl_xor_sync(0xffffffffu, x[e], o), up);
    } else {
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
            if ((e & TOP) == 0) {
                const int a = x[e], b = x[e + TOP];
                x[e] = min(a, b);
                x[e + TOP] = max(a, b);
            }
        }
    }
    if constexpr (TOP > 1) stat_halve<EPL, TOP / 2>(x, lane);
}

// Bitonic sort of the warp's 32 EPL values, ascending in the element index.
// Each merge of SIZE starts with the mirrored partner (index ^ (SIZE - 1)), so
// that every comparison runs the same way.
template <int EPL, int SIZE>
__device__ __forceinline__ void stat_sort(int (&x)[EPL], int lane) {
    if constexpr (SIZE > 2) stat_sort<EPL, SIZE / 2>(x, lane);
    if constexpr (SIZE > EPL) {
        const int mask = SIZE / EPL - 1;
        const bool up = (lane & (SIZE / EPL / 2)) != 0;
#pragma unroll
        for (int e = 0; e < (EPL + 1) / 2; ++e) {
            const int a = __shfl_xor_sync(0xffffffffu, x[EPL - 1 - e], mask);
            if (e != EPL - 1 - e) {
                const int b = __shfl_xor_sync(0xffffffffu, x[e], mask);
                x[EPL - 1 - e] = stat_keep(x[EPL - 1 - e], b, up);
            }
            x[e] = stat_keep(x[e], a, up);
        }
    } else {
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
            const int o = e ^ (SIZE - 1);
            if (e < o) {
                const int a = x[e], b = x[o];
                x[e] = min(a, b);
                x[o] = max(a, b);
            }
        }
    }
    if constexpr (SIZE > 2) stat_halve<EPL, SIZE / 4>(x, lane);
}

// The mean's sum, without FP64 and without rounding: with |v| <= 2^B, the
// integers n1 = rint(v), n2 = rint((v - n1) 2^(B+1)) and n3 = rint of what is
// left of that times 2^(B+1) hold v to 2^-(3 B + 2) of the column's largest
// value: B = 21 up to 512 values a column, 18 (2^-56) up to 4096.  Each is
// read off the low bits of v + 1.5 2^23 and summed exactly in 32 bits.
constexpr unsigned kStatMagicBits = 0x4B400000u;  // 1.5 2^23
template <int B>
__device__ __forceinline__ void stat_split(float v, unsigned (&s)[3]) {
    const float magic = __uint_as_float(kStatMagicBits);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float m = __fadd_rn(v, magic);
        s[k] += __float_as_uint(m);
        v = __fmul_rn(__fsub_rn(v, __fsub_rn(m, magic)), (float)(1 << (B + 1)));
    }
}

struct StatSmem {
    size_t ord, sums, eb, xb, tile, total;
};
__host__ __device__ inline StatSmem stat_smem_layout(int M, int G, int nprobs, int W) {
    StatSmem s{};
    size_t o = 0;
    s.ord = o;  o += (size_t)2 * nprobs * G * 4;               // [2 p + h][column] order statistics
    s.sums = o; o += (size_t)3 * W * G * 4;                    // [part][warp][column]
    s.eb = o;   o += (size_t)W * G * 4;                        // [warp][column] largest |bits|
    s.xb = o;   o += W > 1 ? (size_t)kStatWarps * 1024 * 4 : 0;  // exchange between a column's warps
    s.tile = o; o += (size_t)M * (G + 1) * 4;                  // [m][column], odd stride
    s.total = o;
    return s;
}

// One value stored by another warp of the column, through shared memory.
template <int EPL>
__device__ __forceinline__ void stat_exchange(int (&x)[EPL], int* xb, int wcol, int partner, bool mirror, int lane) {
    __syncthreads();
#pragma unroll
    for (int e = 0; e < EPL; ++e) xb[wcol * 1024 + e * 32 + lane] = x[e];
    __syncthreads();
    const bool up = wcol > partner;
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
        const int o = mirror ? xb[partner * 1024 + (EPL - 1 - e) * 32 + (31 - lane)]
                             : xb[partner * 1024 + e * 32 + lane];
        x[e] = stat_keep(x[e], o, up);
    }
}

// Resident blocks an SM: as many as the tiles leave shared memory for hide the
// chains of the network's steps (1000 x 64 x M = 512 217 us without a bound on
// the registers, 198 with 6 blocks, 209 with 7; 500 x 64 x 1000 265, 208 with 4,
// 218 with 5).
template <int EPL, int W>
__host__ __device__ constexpr int stat_blocks() { return EPL <= 16 ? 6 : (W == 1 ? 4 : 2); }

// log2 of the threads that read a row of nj receivers side by side.
__host__ __device__ inline int stat_row_lanes(int nj) {
    int lg = 0;
    while ((1 << lg) < nj) ++lg;
    return lg;
}

// EPL values a lane, W warps a column (W > 1: EPL = 32).  SHORT: the tile's
// records are short, and their rows are read in one loop (the rows of a record
// follow those of the last), whose bookkeeping costs long ones (1000 x 64 x 512:
// 180 us, 215 with it), as does its mere presence beside the other (182).
template <int EPL, int W, bool SHORT>
__global__ void __launch_bounds__(kStatThreads, stat_blocks<EPL, W>()) trace_stats_kernel(const StatArgs a) {
    static_assert(W == 1 || EPL == 32, "wide columns hold 1024 values a warp");
    constexpr int B = EPL * 32 * W <= 512 ? 21 : 18;
    extern __shared__ __align__(16) unsigned char smem[];
    const StatSmem L = stat_smem_layout(a.M, a.G, a.nprobs, W);
    int* ord = reinterpret_cast<int*>(smem + L.ord);
    int* sums = reinterpret_cast<int*>(smem + L.sums);
    unsigned* top = reinterpret_cast<unsigned*>(smem + L.eb);
    int* xb = reinterpret_cast<int*>(smem + L.xb);
    float* tile = reinterpret_cast<float*>(smem + L.tile);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int M = a.M, G = a.G, TS = G + 1;
    const int ntj = (a.R + a.nj - 1) / a.nj;
    const int k0 = (int)(blockIdx.x / ntj) * a.nr, j0 = (int)(blockIdx.x % ntj) * a.nj;
    const int nr = min(a.nr, a.nrec - k0), nj = min(a.nj, a.R - j0);
    const int nc = nr * nj;                        // column c = rr nj + jj
    // ---- the tile: consecutive threads on consecutive receivers
    {
        const int lg = stat_row_lanes(nj);
        const int jj = tid & ((1 << lg) - 1), step = kStatThreads >> lg;
        if constexpr (SHORT) {
            const float* src = a.traces + (size_t)k0 * M * a.R + j0 + jj;
            int m = tid >> lg, c = jj;             // row of the record, column of the tile
#pragma unroll 4
            for (int p = m; p < (jj < nj ? nr * M : 0); p += step) {
                if (m >= M) {
                    c += m / M * nj;
                    m %= M;
                }
                tile[m * TS + c] = src[(size_t)p * a.R];
                m += step;
            }
        } else {
            for (int rr = 0; rr < nr; ++rr) {
                const float* src = a.traces + (size_t)(k0 + rr) * M * a.R + j0 + jj;
                if (jj < nj) {
#pragma unroll 4
                    for (int m = tid >> lg; m < M; m += step) tile[m * TS + rr * nj + jj] = src[(size_t)m * a.R];
                }
            }
        }
    }
    __syncthreads();
    constexpr int CPI = kStatWarps / W;            // columns in work at a time
    const int w = warp % W;
    for (int cb = 0; cb < nc; cb += CPI) {         // uniform
        const int c = cb + warp / W;
        const bool live = c < nc;
        const float* col = tile + min(c, nc - 1);
        int x[EPL];
        unsigned mx = 0;
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
            const int m = (w * EPL + e) * 32 + lane;
            x[e] = m < M ? __float_as_int(col[m * TS]) : 0;
            mx = max(mx, (unsigned)x[e] & 0x7fffffffu);
        }
        if (a.mean_out) {
            mx = __reduce_max_sync(0xffffffffu, mx);
            if (W > 1) {
                __syncthreads();
                if (lane == 0 && live) top[w * G + c] = mx;
                __syncthreads();
#pragma unroll
                for (int k = 0; k < W; ++k) mx = max(mx, top[k * G + min(c, nc - 1)]);
            } else if (lane == 0 && live) {
                top[c] = mx;
            }
            // |value| < 2^(eb - 126): scaled to 2^B (columns outside the
            // scale's range are summed in FP64 below)
            const int eb = (int)(mx >> 23);
            const float scale = __int_as_float(min(max(B + 253 - eb, 1), 254) << 23);
            unsigned s[3] = {0, 0, 0};  // modulo 2^32
#pragma unroll
            for (int e = 0; e < EPL; ++e) stat_split<B>(__int_as_float(x[e]) * scale, s);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const unsigned t = __reduce_add_sync(0xffffffffu, s[k]);
                if (lane == 0 && live) sums[(k * W + w) * G + c] = (int)(t - EPL * 32u * kStatMagicBits);
            }
        }
        if (a.q_out) {
#pragma unroll
            for (int e = 0; e < EPL; ++e) {
                const int m = (w * EPL + e) * 32 + lane;
                x[e] = m < M ? stat_key(x[e]) : 0x7fffffff;  // absent values sort last
            }
            stat_sort<EPL, 32 * EPL>(x, lane);
            if constexpr (W > 1) {
                int* xc = xb + (warp / W) * W * 1024;
                stat_exchange<EPL>(x, xc, w, w ^ 1, true, lane);
                stat_halve<EPL, 16 * EPL>(x, lane);
                if constexpr (W > 2) {
                    stat_exchange<EPL>(x, xc, w, w ^ 3, true, lane);
                    stat_exchange<EPL>(x, xc, w, w ^ 1, false, lane);
                    stat_halve<EPL, 16 * EPL>(x, lane);
                }
            }
            for (int p = 0; p < a.nprobs; ++p) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int i = min(a.lo[p] + h, M - 1);
                    int v = 0;
#pragma unroll
                    for (int e = 0; e < EPL; ++e) v = e == i % EPL ? x[e] : v;
                    if (live && w * 32 + lane == i / EPL) ord[(2 * p + h) * G + c] = stat_key(v);
                }
            }
        }
    }
    __syncthreads();
    // ---- FP64 only from here on: one value per thread
    if (a.q_out) {
        for (int idx = tid; idx < nc * a.nprobs; idx += kStatThreads) {
            const int p = idx / nc, c = idx - p * nc;
            const double lo = (double)__int_as_float(ord[2 * p * G + c]);
            const double hi = (double)__int_as_float(ord[(2 * p + 1) * G + c]);
            const double t = a.t[p];
            // explicit round-to-nearest operations: no contraction into FMAs
            const double d = __dsub_rn(hi, lo);
            const double q = t >= 0.5 ? __dsub_rn(hi, __dmul_rn(d, __dsub_rn(1.0, t)))
                                      : __dadd_rn(lo, __dmul_rn(d, t));
            a.q_out[((size_t)p * a.nrec + k0 + c / nj) * a.R + j0 + c % nj] = q;
        }
    }
    if (a.mean_out) {
        // the last warps take the means, so that they run beside the quantiles
        for (int c = kStatThreads - 1 - tid; c < nc; c += kStatThreads) {
            unsigned mx = 0;
            int s[3] = {0, 0, 0};
#pragma unroll
            for (int k = 0; k < W; ++k) {
                mx = max(mx, top[k * G + c]);
#pragma unroll
                for (int q = 0; q < 3; ++q) s[q] += sums[(q * W + k) * G + c];
            }
            const int eb = (int)(mx >> 23);
            double sum;
            if (eb == 255 || (mx != 0 && eb < B)) {
                // infinities, NaN, or a scale beyond FP32's range
                sum = 0.0;
                for (int m = 0; m < M; ++m) sum = __dadd_rn(sum, (double)tile[m * TS + c]);
            } else {
                // s0 2^(B+1) + s1 is below 2^53
                const long long hi = (long long)s[0] * (1 << (B + 1)) + s[1];
                sum = scalbn(__fma_rn((double)hi, (double)(1 << (B + 1)), (double)s[2]), eb - 126 - B - 2 * (B + 1));
            }
            a.mean_out[(size_t)(k0 + c / nj) * a.R + j0 + c % nj] = sum / (double)M;
        }
    }
}

// Columns per tile.  16 keep 6 blocks on an SM at M = 512.  With less than two
// tiles an SM, a tile has fewer: first down to one turn of the block's warps,
// then to as few as give every tile an SM of its own (a turn takes as long for
// one column as for a warp each, but two one-column blocks on an SM may share a
// scheduler: 300 columns of M = 1000 in 200 blocks 18.8 us, in 100 below 15).  us
// a call with one receiver, tiles of 8 to 32 columns whatever their number /
// these / one block a column: M = 256, 100 records 20.7 / 12.6 / 14.3, M = 512,
// 100 records 18.5 / 12.6 / 14.5, M = 4000, 10 records 53.5 / 16.8 / 37.2 (about
// 12.5 is the host's part).  Smaller tiles beyond that cost turns and reads:
// 1000 records of 20 receivers, M = 200, tiles of 20 39, of 10 51.
static void stat_tiles(StatArgs& a, int W, long long* nblk) {
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    // the tiles for at most G columns: receivers of one record, or with few of
    // them several records
    auto cut = [&](int G) {
        a.G = G;
        a.nj = a.R < G ? a.R : G;
        a.nr = G / a.nj;
        return *nblk = ((long long)(a.nrec + a.nr - 1) / a.nr) * ((a.R + a.nj - 1) / a.nj);
    };
    int G = a.M <= 256 ? 32 : (a.M <= 512 ? 16 : 8);
    while (cut(G) < 2 * nsm && G > kStatWarps / W) G /= 2;
    if (G <= kStatWarps / W)
        while (G > 1 && cut(G / 2) <= nsm) G /= 2;
    cut(G);
}

template <bool SHORT>
static const void* stat_kernel(int M) {
    if (M <= 32) return (const void*)trace_stats_kernel<1, 1, SHORT>;
    if (M <= 64) return (const void*)trace_stats_kernel<2, 1, SHORT>;
    if (M <= 128) return (const void*)trace_stats_kernel<4, 1, SHORT>;
    if (M <= 256) return (const void*)trace_stats_kernel<8, 1, SHORT>;
    if (M <= 512) return (const void*)trace_stats_kernel<16, 1, SHORT>;
    if (M <= 1024) return (const void*)trace_stats_kernel<32, 1, SHORT>;
    return M <= 2048 ? (const void*)trace_stats_kernel<32, 2, false> : (const void*)trace_stats_kernel<32, 4, false>;
}

static bool device_pointer(const void* p) {
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

}  // namespace romk

extern "C" rom_status rom_trace_stats(const float* traces, int nrec, int R, int M, const double* probs,
                                      int nprobs, double* mean_out, double* q_out, void* stream) {
    using namespace romk;
    if (!traces || nrec < 1 || R < 1 || M < 1 || M > kStatMaxM || nprobs < 0 || nprobs > kStatMaxP)
        return ROM_E_INVAL;
    if (nprobs > 0 && (!probs || !q_out)) return ROM_E_INVAL;
    if (!device_pointer(traces) || (mean_out && !device_pointer(mean_out)) ||
        (q_out && !device_pointer(q_out)))
        return ROM_E_INVAL;
    StatArgs a{};
    for (int i = 0; i < nprobs; ++i) {
        if (!(probs[i] >= 0.0 && probs[i] <= 1.0)) return ROM_E_INVAL;
    }
    if (!mean_out && nprobs == 0) return ROM_OK;
    a.traces = traces;
    a.mean_out = mean_out;
    a.q_out = nprobs > 0 ? q_out : nullptr;
    a.nrec = nrec;
    a.R = R;
    a.M = M;
    a.nprobs = nprobs;
    for (int i = 0; i < nprobs; ++i) {
        const volatile double h = (double)(M - 1) * probs[i];  // rounded before it is used below
        int lo = (int)floor(h);
        if (lo > M - 1) lo = M - 1;
        a.lo[i] = lo;
        a.t[i] = h - (double)lo;
    }
    const int W = M <= 1024 ? 1 : (M <= 2048 ? 2 : 4);
    long long nblk = 0;
    stat_tiles(a, W, &nblk);
    if ((long long)nrec * R > 0x7fffffffLL) return ROM_E_INVAL;
    // several records a tile, too short to keep 3 loads a thread in flight each
    const bool shrt = a.nr > 1 && M < 3 * (kStatThreads >> stat_row_lanes(a.nj));
    const void* fn = shrt ? stat_kernel<true>(M) : stat_kernel<false>(M);
    const size_t smem = stat_smem_layout(M, a.G, nprobs, W).total;
    cudaError_t e = cudaSuccess;
    if (smem > 48 * 1024) e = allow_smem(fn, smem);
    if (e == cudaSuccess) {
        void* args[] = {(void*)&a};
        e = cudaLaunchKernel(fn, dim3((unsigned)nblk), dim3(kStatThreads), args, smem, static_cast<cudaStream_t>(stream));
    }
    return e == cudaSuccess ? ROM_OK : ROM_E_CUDA;
}
