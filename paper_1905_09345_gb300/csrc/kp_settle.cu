// kp_settle.cu -- the exact settle behind the tensor-core dense passes.
//
// The tensor-core passes (kp_dense_tc.cu, kp_dense_tcb.cu) estimate every
// distance with a bounded error; a row whose runner-up lies inside the error
// window of its winner is queued (a per-row request and one bit in a bitmap),
// and the kernels here decide it exactly from FP32 direct differences, from
// compensated FP32 sums where their error bound cannot order the two smallest, and
// in FP64 where those cannot either or a third is as near, so that the labels are
// those of the exact argmin (KPynq Sec. I: the distance calculator's result).
#include "kp_common.cuh"

namespace kp {
namespace {

constexpr int kSettleThreads = 256;
constexpr int kSettleWarps = kSettleThreads / 32;
constexpr int kSub = 8;              // lanes per request
constexpr int kPer = 32 / kSub;      // requests a warp works on at a time
constexpr int kGrabMax = 4 * kPer;   // requests a warp claims at a time, at most
constexpr int kSettleStaged = 160 << 10;  // bytes of centroids kept in shared memory, at most

// The bitmap's set bits, compacted into the settle queue: a warp takes 32
// words, scans their populations and reserves its slots with one atomic.
__global__ void k_settle_gather(Params p, int respect_done) {
    Ctrl *ctrl = p.ctrl;
    count_kernel(ctrl);
    if (respect_done && *(volatile int *)&ctrl->done) return;
    if (*(volatile int *)&ctrl->path != KM_PATH_DENSE_TC) return;
    const int lane = threadIdx.x & 31;
    const int64_t nwords = (p.N + 31) / 32;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t w0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; w0 < nwords; w0 += stride) {
        const int64_t w = w0 + lane;
        const uint32_t bits = w < nwords ? p.sbits[w] : 0u;
        const int c = __popc(bits);
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const int tot = __shfl_sync(0xffffffffu, incl, 31);
        int base = 0;
        if (lane == 31 && tot) base = atomicAdd(&ctrl->settle_count, tot);
        base = __shfl_sync(0xffffffffu, base, 31);
        int64_t pos = (int64_t)base + incl - c;
        for (uint32_t b = bits; b; b &= b - 1u) {
            const int64_t n = w * 32 + (__ffs(b) - 1);
            if (pos < p.N && n < p.N) p.squeue[pos] = (int32_t)n;
            ++pos;
        }
    }
}

// FP64 squared distance, i ascending, no fused multiply-add
__device__ __forceinline__ double settle_fp64(const float *x, const float *c, int D) {
    double s = 0.0;
    for (int i = 0; i < D; ++i) {
        const double t = __dsub_rn((double)__ldg(x + i), (double)c[i]);
        s = __dadd_rn(s, __dmul_rn(t, t));
    }
    return s;
}

// FP32 squared distance by one lane (D a multiple of 4)
__device__ __forceinline__ float settle_fp32(const float *x, const float *c, int D) {
    float a0 = 0.f, a1 = 0.f;
#pragma unroll 4
    for (int i = 0; i < D; i += 4) {
        const float4 xv = __ldg(reinterpret_cast<const float4 *>(x + i)), cv = *reinterpret_cast<const float4 *>(c + i);
        const float d0 = xv.x - cv.x, d1 = xv.y - cv.y, d2 = xv.z - cv.z, d3 = xv.w - cv.w;
        a0 = fmaf(d0, d0, a0);
        a1 = fmaf(d1, d1, a1);
        a0 = fmaf(d2, d2, a0);
        a1 = fmaf(d3, d3, a1);
    }
    return a0 + a1;
}

// The three smallest FP32 distances met so far, the first two with their
// centroids.
struct Top3 {
    float s1, s2, s3;
    int i1, i2;
    __device__ __forceinline__ void add(float s, int c) {  // (a NaN is never below anything)
        const bool f = s < s1, g = s < s2;
        s3 = g ? s2 : fminf(s3, s);
        s2 = f ? s1 : (g ? s : s2);
        i2 = f ? i1 : (g ? c : i2);
        s1 = f ? s : s1;
        i1 = f ? c : i1;
    }
    // with the list of the lane `o` away; both lanes get the same result
    __device__ __forceinline__ void merge(int o) {
        const unsigned full = 0xffffffffu;
        const float b1 = __shfl_xor_sync(full, s1, o), b2 = __shfl_xor_sync(full, s2, o);
        const float b3 = __shfl_xor_sync(full, s3, o);
        const int j1 = __shfl_xor_sync(full, i1, o), j2 = __shfl_xor_sync(full, i2, o);
        const bool f = b1 < s1 || (b1 == s1 && j1 < i1);
        const float x1 = f ? s1 : b1, x2 = f ? s2 : b2;                       // the list that lost
        const float y2 = f ? b2 : s2, y3 = f ? b3 : s3;                       // what is left of the other
        const int k1 = f ? i1 : j1, k2 = f ? j2 : i2;
        s1 = f ? b1 : s1;
        i1 = f ? j1 : i1;
        const bool g = x1 < y2 || (x1 == y2 && k1 < k2);
        s2 = g ? x1 : y2;
        i2 = g ? k1 : k2;
        s3 = g ? fminf(x2, y2) : fminf(x1, y3);
    }
};

// ---------------------------------------------------------------------------
// k_settle: the exact decision for the rows the tensor-core epilogue queued
// (runner-up inside the error window).  The candidates are the centroids of
// the groups whose tensor-core minimum lies in the window (a group mask, or --
// for the streamed-centroid pass -- the groups whose written bound is within
// the window's edge).  The smallest FP32 distance decides; where FP32 cannot
// separate it from the runner-up alone the two are ordered by pair_order, and what is left (three
// that FP32 cannot separate, exact ties) by the FP64 distances of every
// candidate, lanes over centroids, ties to the lowest index.  Writes the
// label, corrects u / lb / lbg when the winner is not i1, and appends label
// changes to the moved-point list 32 at a time.
//
// Bound by the latency of the chain count -> request -> row -> candidates and,
// with many requests, by the shared-memory reads of the candidates' rows.
// Eight lanes per request: lane l reads the 16-byte pieces l, l + 8, ... of a
// candidate's row, so that the eight read 128 consecutive bytes and the four
// requests of a warp never conflict, whatever rows they are at.  (A thread
// per request read rows of its own: up to 32 rows a read, twelve times the
// wavefronts, and as many trips as the longest of 32 lists.)  Four candidates
// go together: their partial sums are handed over in a transposing shuffle
// that leaves each pair of lanes one of the four.
//
// Measured, a pass: 31,000 of 300,007 x 64 rows, K = 200: 64 -> 25 us (20 us of it
// FP64 near-ties, a dozen of them); 115,000 of 1,048,576 x 64, K = 256: 85 -> 65;
// 500,000 of 4,194,304 x 128, K = 1024 (centroids in L2): 1270 -> 560.
// ---------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(kSettleThreads, 2) k_settle(Params p, int first, int respect_done, int staged) {
    constexpr int NC = D / 32;  // 16-byte pieces of a row per lane
    extern __shared__ __align__(128) float sm_settle[];  // C (K x D) | group starts
    __shared__ int32_t mv_n[kSettleWarps][32], mv_old[kSettleWarps][32];  // moves not yet appended
    Ctrl *ctrl = p.ctrl;
    count_kernel(ctrl);
    if (respect_done && *(volatile int *)&ctrl->done) return;
    // the requests of this iteration's dense pass, if it ran on the tensor cores
    if (*(volatile int *)&ctrl->path != KM_PATH_DENSE_TC) return;
    int total = *(volatile int *)&ctrl->settle_count;
    if (total < 0 || total > p.N) {  // cannot happen: at most one request per row
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicExch(&ctrl->err, kErrQueue);
        total = 0;
    }
    const unsigned full = 0xffffffffu;
    const int warp_in = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane / kSub, sl = lane % kSub;
    // requests per claim: enough claims for every warp of the grid
    const int64_t nwarps = (int64_t)gridDim.x * kSettleWarps;
    const int grab = (int)min((int64_t)kGrabMax, max((int64_t)kPer, total / (2 * nwarps) / kPer * kPer));
    if ((int64_t)blockIdx.x * grab >= total) return;  // uniform per block
    const int K = p.K, G = p.G;
    // C in shared memory (row stride D) when it fits, else read from L2
    const int cst = staged ? D : p.Dp;
    const float *Cb = staged ? sm_settle : p.C;
    int32_t *gs_s = reinterpret_cast<int32_t *>(sm_settle + (staged ? (size_t)K * D : 0));
    if (staged)
        for (int i = threadIdx.x; i < K * (D / 4); i += kSettleThreads) {
            const int row = i / (D / 4), q4 = i - row * (D / 4);
            reinterpret_cast<float4 *>(sm_settle + (size_t)row * D)[q4] =
                __ldg(reinterpret_cast<const float4 *>(p.C + (size_t)row * p.Dp) + q4);
        }
    for (int i = threadIdx.x; i <= G; i += kSettleThreads) gs_s[i] = p.gstart[i];
    __syncthreads();
    const bool bounds = p.algo == KM_ALGO_FILTERED;
    int c_changed = 0, c_recheck = 0;
    int mcount = 0;  // warp-uniform
    // append the buffered moves (one slot reservation per warp)
    auto flush_moves = [&]() {
        if (mcount) {
            int base = 0;
            if (lane == 0) base = atomicAdd(&ctrl->moved_count, mcount);
            base = __shfl_sync(full, base, 0);
            if (lane < mcount) {
                p.moved[base + lane] = mv_n[warp_in][lane];
                p.moved_old[base + lane] = mv_old[warp_in][lane];
            }
            __syncwarp();
            mcount = 0;
        }
    };
    // the candidates of a request: the centroids of the masked groups; all K
    // when the mask holds every group
    auto all_of = [&](unsigned long long gmask) { return gmask == ~0ull || (gmask == 0ull && !p.lb); };
    // dynamic schedule: a warp claims `grab` requests (they differ in work),
    // its lanes read them, and its sub-warps take them kPer at a time
    for (;;) {
        int r0 = 0;
        if (lane == 0) r0 = atomicAdd(&ctrl->settle_next, grab);
        r0 = __shfl_sync(full, r0, 0);
        if (r0 >= total || r0 < 0) break;
        const int cnt = min(grab, total - r0);
        SettleReq mine;
        mine.n = -1;
        mine.old = -1;
        mine.i1 = 0;
        mine.lb_alt = 0.f;
        mine.gmask[0] = mine.gmask[1] = 0ull;
        if (lane < cnt) {
            const int n = p.squeue[r0 + lane];
            if (n >= 0 && n < p.N) mine = p.sreq[n];
            if (n < 0 || n >= p.N || mine.n != n || (unsigned)mine.i1 >= (unsigned)K) {
                atomicExch(&ctrl->err, kErrQueue);
                mine.n = -1;
            }
        }
        float mine_lim = 0.f;
        unsigned long long mine_mask = mine.gmask[0] | mine.gmask[1];
        if (K > 256) {  // requests of the streamed-centroid pass
            mine_lim = __uint_as_float((uint32_t)mine.gmask[1]);
            mine_mask = 0ull;
        }
        for (int j = 0; j < cnt; j += kPer) {  // warp-uniform
            const int from = j + sub;  // < 32
            const int n = __shfl_sync(full, mine.n, from), old = __shfl_sync(full, mine.old, from);
            const int w1 = __shfl_sync(full, mine.i1, from);
            const float lim = __shfl_sync(full, mine_lim, from), lb_alt = __shfl_sync(full, mine.lb_alt, from);
            const unsigned long long gmask = __shfl_sync(full, mine_mask, from);
            const bool act = n >= 0;
            const int64_t row = act ? n : 0;
            ulonglong2 xv[NC];
#pragma unroll
            for (int k = 0; k < NC; ++k)
                xv[k] = __ldg(reinterpret_cast<const ulonglong2 *>(p.X + row * D) + sl + kSub * k);
            Top3 t;
            t.s1 = t.s2 = t.s3 = INFINITY;
            t.i1 = t.i2 = w1;
            // the walk: centroids [col, cend) of the current group, then the next
            // group of the mask m (group ids base + bit).  For the bounds' window
            // m is refilled with 32 groups at a time, four per lane.
            const bool window = gmask == 0ull && p.lb;
            int col = 0, cend = act && all_of(gmask) ? K : 0;
            unsigned long long m = act && !all_of(gmask) && !window ? gmask : 0ull;
            int seg = act && window ? 0 : G;  // next group of the row's bounds to test
            const float *lbr = p.lb + row * p.Gp;
            const float4 none = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
            auto bounds4 = [&](int g) {
                return g < p.Gp ? *reinterpret_cast<const float4 *>(lbr + g) : none;
            };
            float4 ahead = seg < G ? bounds4(4 * sl) : none;
            int base = 0;
            for (;;) {  // warp-uniform trips
                if (col >= cend && m) {
                    const int b = __ffsll((long long)m) - 1;
                    m &= m - 1;
                    // (a window's mask has bit 8 t + l for group base + 4 l + t)
                    const int g = window ? base + 4 * (b & 7) + (b >> 3) : b;
                    if (g < G) {
                        col = gs_s[g];
                        cend = gs_s[g + 1];
                    }
                }
                const bool dry = col >= cend && !m;
                if (__any_sync(full, dry && seg < G)) {
                    const bool take = dry && seg < G;
                    const float4 v = ahead;
                    unsigned mk = 0;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float b = k == 0 ? v.x : (k == 1 ? v.y : (k == 2 ? v.z : v.w));
                        const unsigned in = __ballot_sync(full, b <= lim && seg + 4 * sl + k < G);
                        mk |= ((in >> (sub * kSub)) & 0xffu) << (8 * k);
                    }
                    if (take) {
                        m = mk;
                        base = seg;
                        seg += 32;
                        if (seg < G) ahead = bounds4(seg + 4 * sl);
                    }
                    continue;
                }
                if (!__any_sync(full, col < cend || m)) break;
                if (!__any_sync(full, col < cend)) continue;  // (an empty group)
                const int last = max(cend - 1, 0);
                float s[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const ulonglong2 *c = reinterpret_cast<const ulonglong2 *>(Cb + (size_t)min(col + k, last) * cst) + sl;
                    f32x2 a0 = 0ull, a1 = 0ull;
#pragma unroll
                    for (int q = 0; q < NC; ++q) {
                        const ulonglong2 c2 = c[kSub * q];
                        const f32x2 d0 = sub2(xv[q].x, c2.x), d1 = sub2(xv[q].y, c2.y);
                        a0 = fma2(d0, d0, a0);
                        a1 = fma2(d1, d1, a1);
                    }
                    s[k] = sum2(a0) + sum2(a1);
                }
                // lanes 4 apart: two candidates each; 2 apart: one each; then the pair's sum
                const bool u4 = sl & 4, u2 = sl & 2;
                const float r0v = (u4 ? s[2] : s[0]) + __shfl_xor_sync(full, u4 ? s[0] : s[2], 4);
                const float r1v = (u4 ? s[3] : s[1]) + __shfl_xor_sync(full, u4 ? s[1] : s[3], 4);
                float sx = (u2 ? r1v : r0v) + __shfl_xor_sync(full, u2 ? r0v : r1v, 2);
                sx += __shfl_xor_sync(full, sx, 1);
                const int cc = col + (u4 ? 2 : 0) + (u2 ? 1 : 0);
                if (cc < cend) t.add(sx, cc);
                col += 4;
            }
            t.merge(2);
            t.merge(4);
            // near-ties, one request after another, by the whole warp
            int bi = t.i1;
            float bs = t.s1;
            unsigned rm = __ballot_sync(full, sl == 0 && act && t.s2 != INFINITY && unresolved(t.s1, t.s2, p));
            while (rm) {
                const int src = __ffs(rm) - 1;
                rm &= rm - 1;
                const int64_t nr = __shfl_sync(full, n, src);
                const int a1 = __shfl_sync(full, t.i1, src), a2 = __shfl_sync(full, t.i2, src);
                const float v1 = __shfl_sync(full, t.s1, src), v2 = __shfl_sync(full, t.s2, src);
                const float v3 = __shfl_sync(full, t.s3, src);
                const float *xg = p.X + nr * D;
                int bj = a1;
                float bsr = v1;
                int o = -1;
                if (v3 == INFINITY || !unresolved(v1, v3, p)) {
                    const float *c1 = Cb + (size_t)a1 * cst, *c2 = Cb + (size_t)a2 * cst;
                    o = pair_order(xg, c1, c2, D);
                    // (narrower rows: the scan below is as fast, and the call costs every launch 0.4 us)
                    if (D > 64 && o < 0) o = pair_order_f64(xg, c1, c2, D, tie_key(p, a2) < tie_key(p, a1));
                }
                if (o == 1) {
                    bj = a2;
                    bsr = v2;
                } else if (o < 0) {
                    const unsigned long long gm = __shfl_sync(full, gmask, src);
                    const float lm = __shfl_sync(full, lim, src);
                    const float *lbn = p.lb + nr * p.Gp;
                    double bd = INFINITY;
                    bj = 0x7fffffff;
                    for (int c = lane; c < K; c += 32) {
                        bool cand = all_of(gm);
                        if (!cand) {
                            const int g = p.grp[c];
                            cand = gm == 0ull ? lbn[g] <= lm : (g < 64 && ((gm >> g) & 1ull));
                        }
                        if (!cand || !unresolved(v1, settle_fp32(xg, Cb + (size_t)c * cst, D), p)) continue;
                        const double d64 = settle_fp64(xg, Cb + (size_t)c * cst, D);
                        if (d64 < bd || (d64 == bd && tie_key(p, c) < tie_key(p, bj))) {
                            bd = d64;
                            bj = c;
                        }
                    }
#pragma unroll
                    for (int w = 16; w > 0; w >>= 1) {
                        const double ov = __shfl_xor_sync(full, bd, w);
                        const int oi = __shfl_xor_sync(full, bj, w);
                        if (ov < bd || (ov == bd && tie_key(p, oi) < tie_key(p, bj))) {
                            bd = ov;
                            bj = oi;
                        }
                    }
                    if (bj == 0x7fffffff) bj = a1;
                    // for u: its FP32 distance, or the smallest (it is no farther than a1)
                    bsr = bj == a2 ? v2 : v1;
                }
                if (lane / kSub == src / kSub) {
                    bi = bj;
                    bs = bsr;
                }
                c_recheck += lane == 0;
            }
            bool moved = false;
            if (act && sl == 0) {
                p.label[n] = bi;
                if (bounds) {
                    p.u[n] = dist_up(bs, p);
                    if (bi != w1) {
                        p.lb[row * p.Gp + p.grp[w1]] = lb_alt;
                        p.lb[row * p.Gp + p.grp[bi]] = lb_alt;
                        p.lbg[n] = lb_alt;
                    }
                }
                moved = bi != old;
                c_changed += moved;
            }
            // label changes: the sub-warp leaders' moves, appended 32 at a time
            if (!first) {
                const unsigned mm = __ballot_sync(full, moved);
                if (mm) {
                    const int k = mcount + __popc(mm & ((1u << lane) - 1u));
                    if (moved) {
                        mv_n[warp_in][k] = n;
                        mv_old[warp_in][k] = old;
                    }
                    mcount += __popc(mm);
                    __syncwarp();
                    if (mcount > 32 - kPer) flush_moves();
                }
            }
        }
    }
    if (!first) flush_moves();
    c_changed = __reduce_add_sync(full, c_changed);
    c_recheck = __reduce_add_sync(full, c_recheck);
    if (lane == 0) {
        if (c_changed) atomicAdd(&ctrl->n_changed, (unsigned long long)c_changed);
        if (c_recheck) atomicAdd(&ctrl->n_recheck, (unsigned long long)c_recheck);
    }
}

}  // namespace

cudaError_t launch_settle(const Params &p, cudaStream_t s, int first, int respect_done, int num_sms) {
    if (p.D != 32 && p.D != 64 && p.D != 128) return cudaErrorInvalidValue;
    // compact the request bitmap (one warp per 32 words), then the requests
    const int64_t words = (p.N + 31) / 32;
    const int64_t gblocks = std::max<int64_t>(1, std::min<int64_t>((words + 255) / 256, (int64_t)num_sms * 8));
    count_launch();
    k_settle_gather<<<(unsigned)gblocks, 256, 0, s>>>(p, respect_done);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // C in shared memory when it fits (up to 160 KB), else read from L2
    const int staged = (size_t)p.K * p.D * 4 <= (size_t)kSettleStaged;
    const size_t smem = (staged ? (size_t)p.K * p.D * 4 : 0) + (size_t)(p.G + 1) * 4;
    auto kern = p.D == 32 ? k_settle<32> : (p.D == 64 ? k_settle<64> : k_settle<128>);
    // (one value for every context: it is the process's, and another thread's
    // context may be launching; K of a tensor-core pass is at most 4096)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSettleStaged + 4 * (4096 + 1));
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kSettleThreads, smem);
    if (e != cudaSuccess) return e;
    count_launch();
    kern<<<(unsigned)(num_sms * std::max(per_sm, 1)), kSettleThreads, smem, s>>>(p, first, respect_done, staged);
    return cudaGetLastError();
}

}  // namespace kp
