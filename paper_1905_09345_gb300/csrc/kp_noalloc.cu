// kp_noalloc.cu -- one plain-Lloyd iteration that allocates nothing.
//
// For callers that may not allocate device memory at all: a host framework
// that owns every byte of device memory through its own pool, a
// latency-critical loop in which cudaMalloc / cudaFree would synchronise the
// device, or a deployment that must reserve all memory at start-up.  They
// pass X, C and the output arrays; every intermediate (FP64 cluster sums,
// counts, a padded centroid copy, the control block) lives in the
// file-scope array below, which each GPU that loads the library holds until
// the process exits.  The paper has no counterpart to this entry point.
#include <cuda.h>

#include <cmath>
#include <cstring>
#include <mutex>

#include "kp_common.cuh"

namespace kp {
namespace {

constexpr int kNaMaxK = 1024;  // KM_NOALLOC_MAX_K
constexpr int kNaMaxD = 128;   // KM_NOALLOC_MAX_D
constexpr int kNaMaxDp = 132;  // padded centroid row stride for D <= 128

// byte offsets inside the scratch array (each 256-byte aligned)
constexpr size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
constexpr size_t kOffCtrl = 0;
constexpr size_t kOffStats = align256(kOffCtrl + sizeof(Ctrl));
constexpr size_t kOffC = align256(kOffStats + sizeof(kmeans_iter_stats));
constexpr size_t kOffS = align256(kOffC + sizeof(float) * kNaMaxK * kNaMaxDp);
constexpr size_t kOffQ = align256(kOffS + sizeof(double) * kNaMaxK * kNaMaxD);
constexpr size_t kOffCnt = align256(kOffQ + sizeof(double) * kNaMaxK);
constexpr size_t kOffJk = align256(kOffCnt + sizeof(unsigned long long) * kNaMaxK);
constexpr size_t kOffDelta = align256(kOffJk + sizeof(double) * kNaMaxK);
constexpr size_t kOffGrp = align256(kOffDelta + sizeof(float) * kNaMaxK);
constexpr size_t kOffGstart = align256(kOffGrp + sizeof(int32_t) * kNaMaxK);
constexpr size_t kOffDc = align256(kOffGstart + sizeof(int32_t) * 4);
constexpr size_t kOffDg = align256(kOffDc + sizeof(float) * 2 * kNaMaxK);
constexpr size_t kOffDm = align256(kOffDg + sizeof(float) * 2 * 4);
constexpr size_t kScratchBytes = align256(kOffDm + sizeof(float) * 2);  // about 1.6 MB

// The scratch itself.  Host code may not use `g_noalloc_scratch` as an
// address: its device address comes from cudaGetSymbolAddress, per device.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

// Device address of the array, per device ordinal, with the context it was
// looked up in: a context destroyed and made again (cudaDeviceReset) loads the
// module again, so the address is looked up again when the context differs.
struct ScratchSlot {
    CUcontext ctx;
    void *ptr;
};
std::mutex g_mu;
ScratchSlot g_scratch[256] = {};

// the calling thread's current context (driver entry point, fetched once)
CUcontext current_context() {
    using Fn = CUresult (*)(CUcontext *);
    static std::once_flag once;
    static Fn fn = nullptr;
    std::call_once(once, [] {
        cudaDriverEntryPointQueryResult q;
        void *f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<Fn>(f);
    });
    CUcontext c = nullptr;
    if (!fn || fn(&c) != CUDA_SUCCESS) return nullptr;
    return c;
}

// Before the step: the array keeps the previous call's contents, so clear what
// this one accumulates into or reads before writing, and lay the centroids out
// with the padded stride (padding zero).  One group holds every centroid.
__global__ void __launch_bounds__(256) k_noalloc_begin(Params p, const float *C, int4 *ctrl, int nctrl,
                                                       int32_t *grp, int32_t *gstart, float *drift, int ndrift) {
    const int i0 = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
    for (int i = i0; i < nctrl; i += step) ctrl[i] = make_int4(0, 0, 0, 0);
    for (int i = i0; i < ndrift; i += step) drift[i] = 0.f;
    for (int i = i0; i < p.K * p.Dp; i += step) {
        const int k = i / p.Dp, d = i - k * p.Dp;
        p.C[i] = d < p.D ? C[k * p.D + d] : 0.f;
    }
    for (int i = i0; i < p.K * p.D; i += step) p.S[i] = 0.0;
    for (int i = i0; i < p.K; i += step) {
        p.Q[i] = 0.0;
        p.cnt[i] = 0ull;
        grp[i] = 0;
    }
    if (i0 < 2) gstart[i0] = i0 * p.K;
}

// After it: the centroids back to dense rows, and the J_t of the iteration
// (kept in the stats record).
__global__ void __launch_bounds__(256) k_noalloc_end(Params p, float *C_new, double *objective) {
    const int i0 = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
    for (int i = i0; i < p.K * p.D; i += step) {
        const int k = i / p.D, d = i - k * p.D;
        C_new[i] = p.C[(size_t)k * p.Dp + d];
    }
    if (i0 == 0) *objective = p.stats->objective;
}

// Cluster sums of all points, without N-sized scratch: S_k = sum x,
// Q_k = sum ||x - R_k||^2 and the sizes.
//
// One atomic per point and coordinate in FP64 is what a direct sum costs, and
// the L2 does about 60 of them a nanosecond.  So a block first sorts its points
// by label, in shared memory (ids and labels packed in one word), and each
// warp sums a run of the sorted points before it touches the global sums: one
// atomic per cluster and coordinate that the block has met.  The fewer the
// blocks per coordinate, the fewer the atomics: a block takes 32 coordinates,
// and the rows are cut in D / 32 times longer segments instead.
//
// FP64 arithmetic is slow on these SMs (two operations a cycle), so the runs
// are summed in FP32 triples: TwoSum into (h, l), the rounding of l itself
// kept in m, which leaves an error of the order of 2^-70 of the sum of the
// magnitudes; the triple is rounded to FP64 once when it is added to the
// global sum.  What bounds the kernel now is issuing those operations, some 45
// a coordinate.
//
// Measured (every point's sums, K = 256): 262,144 x 64: 292 -> 57 us; 600,000
// x 32: 619 -> 62; 600,000 x 8: 617 -> 62; 600,000 x 128: 752 -> 241 (one FP64
// atomic per point and coordinate before).  A block's code has to stay short:
// with the end of a cluster's run unrolled into the loop over the points it
// waited for instructions most of the time (75 us).
constexpr int kSumThreads = 1024;
constexpr int kSumWarps = kSumThreads / 32;
constexpr int kSumTile = 1 << 13;       // points sorted at a time (13 bits of the word; the label has 10)
constexpr int kSumBatch = 8;            // points whose loads are in flight together

struct Sum3 {
    float h, l, m;
    __device__ __forceinline__ void clear() { h = l = m = 0.f; }
    __device__ __forceinline__ void add(float x) {
        float e, f;
        two_sum(h, x, h, e);
        two_sum(l, e, l, f);
        m = __fadd_rn(m, f);
    }
    // FP32 -> FP64 on the integer units (the conversion instruction shares the
    // slow FP64 pipe); zeros here, what is left (subnormals, infinities, NaN) there
    static __device__ __forceinline__ double widen(float x) {
        const uint32_t u = __float_as_uint(x), a = u & 0x7fffffffu;
        if (a == 0u || (a >= 0x00800000u && a < 0x7f800000u))
            return __hiloint2double((int)(a ? (u & 0x80000000u) | ((a >> 3) + (896u << 20)) : u), (int)(u << 29));
        return (double)x;
    }
    __device__ __forceinline__ double value() const { return widen(h) + (widen(l) + widen(m)); }
};

__global__ void __launch_bounds__(kSumThreads) k_noalloc_sums(Params p, int segs) {
    extern __shared__ uint32_t order[];  // kSumTile sorted points | K counters | parts of Q: triples, clusters
    __shared__ int wsum[kSumWarps];
    __shared__ int nparts;
    int *cur = reinterpret_cast<int *>(order + kSumTile);
    const int most = p.K + kSumWarps;  // a cluster's points lie in one run, or in runs next to each other
    float *part = reinterpret_cast<float *>(cur + p.K);
    int *part_k = reinterpret_cast<int *>(part + 3 * most);
    const int K = p.K, D = p.D;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int seg = blockIdx.x % segs, slice = blockIdx.x / segs;
    const int i = slice * 32 + lane;  // this lane's coordinate
    const bool on = i < D;
    const int64_t n0 = p.N * seg / segs, n1 = p.N * (seg + 1) / segs;
    for (int64_t base = n0; base < n1; base += kSumTile) {
        const int count = (int)min((int64_t)kSumTile, n1 - base);
        // counting sort of the tile by label
        for (int k = threadIdx.x; k < K; k += kSumThreads) cur[k] = 0;
        if (threadIdx.x == 0) nparts = 0;
        __syncthreads();
        for (int e = threadIdx.x; e < count; e += kSumThreads) {
            const int k = checked_label(p, base + e);
            if (k >= 0) atomicAdd(&cur[k], 1);
        }
        __syncthreads();
        const int per = (K + kSumThreads - 1) / kSumThreads;
        const int k0 = min((int)threadIdx.x * per, K), k1 = min(k0 + per, K);
        int run = 0;
        for (int k = k0; k < k1; ++k) {
            const int c = cur[k];
            if (slice == 0 && c) atomicAdd(&p.cnt[k], (unsigned long long)c);
            run += c;
        }
        int incl = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        int off = incl - run, placed = 0;
        for (int w = 0; w < kSumWarps; ++w) {
            if (w < warp) off += wsum[w];
            placed += wsum[w];
        }
        for (int k = k0; k < k1; ++k) {
            const int c = cur[k];
            cur[k] = off;
            off += c;
        }
        __syncthreads();
        for (int e = threadIdx.x; e < count; e += kSumThreads) {
            const int k = checked_label(p, base + e);
            if (k >= 0) order[atomicAdd(&cur[k], 1)] = (uint32_t)k << 13 | (uint32_t)e;
        }
        __syncthreads();
        // the warps' runs; which warp takes which is rotated from block to
        // block, so that blocks do not add to the same clusters at one time
        const int w = (warp + blockIdx.x) % kSumWarps;
        const int r0 = placed * w / kSumWarps, r1 = placed * (w + 1) / kSumWarps;
        Sum3 s, q;
        for (int r = r0; r < r1;) {  // a cluster's points in the run: [r, end)
            const int k = (int)(order[r] >> 13), from = r, end = min(cur[k], r1);
            const float ref = on ? p.R[(size_t)k * p.Dp + i] : 0.f;
            s.clear();
            q.clear();
            for (; r < end; r += kSumBatch) {
                float xv[kSumBatch];
#pragma unroll
                for (int b = 0; b < kSumBatch; ++b)
                    xv[b] = on ? __ldg(p.X + (base + (order[min(r + b, end - 1)] & (kSumTile - 1))) * D + i) : 0.f;
#pragma unroll
                for (int b = 0; b < kSumBatch; ++b) {
                    if (r + b >= end) break;  // warp-uniform
                    s.add(xv[b]);
                    // (x - r)^2 exactly but for 2^-47 of it: x - r = dh + dl, its
                    // square sq + sqe, and 2 dh dl + dl^2
                    float dh, dl, e;
                    two_sum(xv[b], -ref, dh, dl);
                    const float sq = __fmul_rn(dh, dh);
                    const float sqe = __fmaf_rn(dh, dh, -sq);
                    q.add(sq);
                    const float cross = __fmaf_rn(__fmul_rn(2.f, dh), dl, __fmul_rn(dl, dl));
                    two_sum(q.l, __fadd_rn(sqe, cross), q.l, e);
                    q.m = __fadd_rn(q.m, e);
                }
            }
            r = end;
            double v = s.value();
            if (!isfinite(s.h)) {  // a sum beyond FP32, or an infinity among the points: in FP64
                v = 0.0;
                for (int a = from; a < end; ++a)
                    if (on) v += (double)__ldg(p.X + (base + (order[a] & (kSumTile - 1))) * D + i);
            }
            if (on && v != 0.0) atomicAdd(&p.S[(size_t)k * D + i], v);
            // the lanes' parts of Q, still in FP32
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float h = __shfl_xor_sync(0xffffffffu, q.h, o), l = __shfl_xor_sync(0xffffffffu, q.l, o);
                const float m = __shfl_xor_sync(0xffffffffu, q.m, o);
                float e;
                q.m = __fadd_rn(q.m, m);
                two_sum(q.l, l, q.l, e);
                q.m = __fadd_rn(q.m, e);
                q.add(h);
            }
            if (__any_sync(0xffffffffu, !isfinite(q.h))) {  // (as for S; the points' own squares may fit FP32)
                double t = 0.0;
                for (int a = from; a < end; ++a) {
                    const double d = on ? (double)__ldg(p.X + (base + (order[a] & (kSumTile - 1))) * D + i) - (double)ref : 0.0;
                    t += d * d;
                }
                t = warp_sum_d(t);
                if (lane == 0) atomicAdd(&p.Q[k], t);
            } else if (lane == 0) {
                const int at = atomicAdd(&nparts, 1);
                part[at] = q.h;
                part[most + at] = q.l;
                part[2 * most + at] = q.m;
                part_k[at] = k;
            }
        }
        __syncthreads();
        // Q's parts, 32 to an FP64 instruction
        for (int a = threadIdx.x; a < nparts; a += kSumThreads) {
            q.h = part[a];
            q.l = part[most + a];
            q.m = part[2 * most + a];
            atomicAdd(&p.Q[part_k[a]], q.value());
        }
        __syncthreads();
    }
}

float up32(double x) {
    float f = (float)x;
    return (double)f < x ? nextafterf(f, INFINITY) : f;
}
float dn32(double x) {
    float f = (float)x;
    return (double)f > x ? nextafterf(f, -INFINITY) : f;
}

bool on_device(const void *ptr, int dev) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, ptr) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) && a.device == dev;
}

// the message is read back with kmeans_last_error(NULL)
int fail(int code, const char *msg) {
    set_thread_error(msg);
    return code;
}

}  // namespace
}  // namespace kp

using namespace kp;

extern "C" {

KM_API int kmeans_lloyd_step_noalloc(const float *X, int64_t N, int32_t D, const float *C, int32_t K,
                                     int32_t *labels, float *C_new, double *objective, void *stream) {
    if (!X || !C || !labels || !C_new || !objective) return fail(KM_EINVAL, "a pointer argument is NULL");
    if (N < 1 || N >= ((int64_t)1 << 31)) return fail(KM_EINVAL, "N out of range [1, 2^31)");
    if (D < 1 || D > kNaMaxD) return fail(KM_EINVAL, "D out of range [1, 128] for the allocation-free step");
    if (K < 1 || K > kNaMaxK || (int64_t)K > N)
        return fail(KM_EINVAL, "K out of range [1, min(N, 1024)] for the allocation-free step");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return fail(KM_ECUDA, "cudaGetDevice failed");
    if (!on_device(X, dev) || !on_device(C, dev) || !on_device(labels, dev) || !on_device(C_new, dev) ||
        !on_device(objective, dev))
        return fail(KM_EINVAL, "every array must be device memory of the current device");

    // set-up once per device (and again if its context was made anew): the
    // scratch array's device address, looked up with that device current
    void *base = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        const CUcontext cur = current_context();
        if (!cur) return fail(KM_ECUDA, "no current CUDA context");
        if (!g_scratch[dev].ptr || g_scratch[dev].ctx != cur) {
            void *p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess || !p) return fail(KM_ECUDA, "cudaGetSymbolAddress of the scratch array failed");
            g_scratch[dev].ptr = p;
            g_scratch[dev].ctx = cur;
        }
        base = g_scratch[dev].ptr;
    }
    unsigned char *b = static_cast<unsigned char *>(base);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int num_sms = 0;
    if (cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return fail(KM_ECUDA, "cudaDeviceGetAttribute failed");

    Params p;
    memset(&p, 0, sizeof(p));
    p.X = X;
    p.N = N;
    p.D = D;
    p.K = K;
    p.G = 1;
    const int dp = dense_dp(D);
    p.Dp = ((dp / 4) % 2 == 0) ? dp + 4 : dp;
    p.Gp = 4;
    p.tcap = 2;
    p.x_vec4 = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(X) & 15) == 0);
    p.label = labels;
    p.C = reinterpret_cast<float *>(b + kOffC);
    p.S = reinterpret_cast<double *>(b + kOffS);
    p.Q = reinterpret_cast<double *>(b + kOffQ);
    p.R = p.C;  // reference points = the centroids of this step (the update reads each before writing it)
    p.cnt = reinterpret_cast<unsigned long long *>(b + kOffCnt);
    p.Jk = reinterpret_cast<double *>(b + kOffJk);
    p.delta = reinterpret_cast<float *>(b + kOffDelta);
    p.grp = reinterpret_cast<const int32_t *>(b + kOffGrp);
    p.gstart = reinterpret_cast<const int32_t *>(b + kOffGstart);
    p.Dc = reinterpret_cast<float *>(b + kOffDc);
    p.Dg = reinterpret_cast<float *>(b + kOffDg);
    p.Dm = reinterpret_cast<float *>(b + kOffDm);
    p.ctrl = reinterpret_cast<Ctrl *>(b + kOffCtrl);
    p.stats = reinterpret_cast<kmeans_iter_stats *>(b + kOffStats);
    const double eps = (D + 4) * std::ldexp(1.0, -24) * (1.0 + 1.0 / 1024);
    p.eps_hi = up32(1.0 + 2.0 * eps);
    p.eps_lo = dn32(1.0 - eps);
    p.tiny = std::ldexp((float)(D + 4), -149);
    p.algo = KM_ALGO_LLOYD;

#define NA_CUDA(call)                                                           \
    do {                                                                        \
        cudaError_t e_ = (call);                                                \
        if (e_ != cudaSuccess) return fail(KM_ECUDA, cudaGetErrorString(e_));   \
    } while (0)
    const unsigned wide = (unsigned)std::min(num_sms, (K * p.Dp + 255) / 256);
    k_noalloc_begin<<<wide, 256, 0, s>>>(p, C, reinterpret_cast<int4 *>(b), (int)(kOffC / 16),
                                         reinterpret_cast<int32_t *>(b + kOffGrp),
                                         reinterpret_cast<int32_t *>(b + kOffGstart),
                                         reinterpret_cast<float *>(b + kOffDc), (int)((kScratchBytes - kOffDc) / 4));
    NA_CUDA(cudaGetLastError());
    count_launch();
    NA_CUDA(launch_dense_assign(p, s, 1, 0, num_sms, 0));
    {
        // a block per SM; a segment of at least 1024 points
        const int slices = (D + 31) / 32;
        const int segs = (int)std::max<int64_t>(1, std::min<int64_t>(num_sms / slices, N / 1024));
        const size_t smem = sizeof(uint32_t) * (kSumTile + (size_t)K + 4 * (size_t)(K + kSumWarps));
        NA_CUDA(cudaFuncSetAttribute(k_noalloc_sums, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        k_noalloc_sums<<<(unsigned)(segs * slices), kSumThreads, smem, s>>>(p, segs);
        NA_CUDA(cudaGetLastError());
        count_launch();
    }
    NA_CUDA(launch_update(p, s, 0, 0, num_sms));
    k_noalloc_end<<<wide, 256, 0, s>>>(p, C_new, objective);
    NA_CUDA(cudaGetLastError());
    count_launch();
#undef NA_CUDA
    return KM_OK;
}

}  // extern "C"
