// kp_stats.cu -- cluster statistics (S_k = sum x in FP64, Q_k = sum
// ||x - R_k||^2 about a reference point R_k, n_k) for the centroid update.
//
// Two ways, chosen on the device after each assignment, both on the same
// three kernels: a counting sort of entries by cluster (k_stats_hist counts
// and lays out the segments, k_stats_scatter places the entries), then each
// warp sums a run of sorted entries (64; 16 when few points moved)
// coordinate-parallel and adds one partial per cluster it met to the global
// FP64 sums.  Global atomics then
// touch each cluster a few times instead of once per point.
//   * full recompute (iteration 0, or more than N/2 labels changed): one
//     entry per point, under its label; S, Q and the counts start from zero;
//   * incremental (few labels changed): two entries per relabelled point,
//     +x under its new label and -x under its old one (the sign in bit 31 of
//     the entry's id), added to the sums as they stand; the counts change by
//     the entries' signs.
// When only a handful of labels changed, k_stats_hist moves those points
// itself, one atomic per coordinate, and the other two have nothing to do.
#include <type_traits>

#include "kp_common.cuh"

namespace kp {

constexpr int kStatsThreads = 256;
constexpr int kStatsTile = kStatsThreads * 4;  // points per block step of the scatter
constexpr int kSumRun = 64;                    // sorted entries per warp in k_stats_sum (full mode)
constexpr int kSumRunMoved = 16;               // the same for at most N/8 moved points' entries
                                               // (few, so shorter runs put more warps on them)
constexpr int kSumMaxPer = 8;                  // coordinates per lane (D <= 256)

// full when the moved points' entries (two each) would outnumber the points
__device__ __forceinline__ bool stats_full_rule(const Params &p, int all_points) {
    return all_points || (int64_t)p.ctrl->moved_count * 2 > p.N;
}

// Few moved points: at most so many, per cluster and in coordinates.  An FP64
// atomic per coordinate costs less than the sort's three chains of dependent
// loads as long as the L2 takes them (60 a nanosecond in all, one address about
// every 40 ns) in the time of one such chain; the bounds keep the worst case,
// every move between the same two clusters, near 40 us.  Measured, the three
// kernels of an iteration: 16,384 x 16, K = 16, 25 moved points: 14.6 us sorted,
// 9.6 moved one by one, but 3,300 moved points 15 sorted and 64 one by one;
// 200,003 x 17, K = 100, 500 to 800 moved points: 20 sorted, 9 one by one.  Whole
// fits with 2, 4, 8, 16, 32 points per cluster (48 problems): 15.3, 15.1, 15.0,
// 15.0, 15.0 ms, sorted always 15.7.
constexpr int64_t kDirectCoords = 1 << 17;
constexpr int64_t kDirectPer = 8;
constexpr int64_t kDirectMax = 1024;
constexpr int kStatsSorted = 0, kStatsFull = 1, kStatsDirect = 2;  // Ctrl::stats_full

constexpr uint32_t kNegEntry = 0x80000000u;  // entry id bit: subtract the point

// Entries of the sort: full mode, point e under its label; incremental mode,
// moved point e under its new label (e < m) or, subtracted, under its old
// label (m <= e < 2m).  Returns the cluster (-1: none) and the entry's id.
__device__ __forceinline__ int stats_entry(const Params &p, bool full, int64_t m, int64_t e, uint32_t &id) {
    if (full) {
        id = (uint32_t)e;
        return checked_label(p, e);
    }
    if (e < m) {
        const int64_t n = p.moved[e];
        id = (uint32_t)n;
        return checked_label(p, n);
    }
    const int64_t n = p.moved[e - m];
    const int old = p.moved_old[e - m];
    id = (uint32_t)n | kNegEntry;
    if (old < 0) return -1;  // the point had no cluster
    if (old >= p.K) {
        atomicExch(&p.ctrl->err, kErrLabel);
        return -1;
    }
    return old;
}
__device__ __forceinline__ int64_t stats_entries(const Params &p, bool full) {
    return full ? p.N : 2 * (int64_t)p.ctrl->moved_count;
}

// Decide the mode; move the points if they are few; in full mode zero S and Q;
// count the entries per cluster (shared-memory histogram when K fits), and let
// the last block turn the counts into segment offsets (hcur) and, in full mode,
// the new cluster sizes (cnt).
__global__ void __launch_bounds__(kStatsThreads) k_stats_hist(Params p, int all_points, int respect_done) {
    extern __shared__ int hist[];
    __shared__ int last;
    __shared__ int wsum[kStatsThreads / 32];
    Ctrl *ctrl = p.ctrl;
    count_kernel(ctrl);
    if (respect_done && *(volatile int *)&ctrl->done) return;
    const bool full = stats_full_rule(p, all_points);
    const int K = p.K, D = p.D;
    const bool local = K <= p.hist_smem_k;
    const int64_t m = full ? 0 : (int64_t)ctrl->moved_count;
    const bool direct = !full && m <= kDirectMax && m <= kDirectPer * K && m * D <= kDirectCoords;
    if (blockIdx.x == 0 && threadIdx.x == 0)
        ctrl->stats_full = full ? kStatsFull : (direct ? kStatsDirect : kStatsSorted);
    if (direct) {
        for (int64_t it = ((int64_t)blockIdx.x * kStatsThreads + threadIdx.x) >> 5; it < m;
             it += ((int64_t)gridDim.x * kStatsThreads) >> 5)
            move_point(p, p.moved[it], p.moved_old[it]);
        return;
    }
    const int64_t ne = stats_entries(p, full);
    // blocks taking part: one per tile of entries (the others leave at once;
    // few moved points need few blocks)
    const unsigned used = (unsigned)max((int64_t)1, min((int64_t)gridDim.x, (ne + kStatsTile - 1) / kStatsTile));
    if (blockIdx.x >= used) return;
    const int64_t tid = (int64_t)blockIdx.x * kStatsThreads + threadIdx.x;
    const int64_t nthr = (int64_t)used * kStatsThreads;
    if (full) {
        for (int64_t i = tid; i < (int64_t)K * D; i += nthr) p.S[i] = 0.0;
        for (int64_t i = tid; i < K; i += nthr) p.Q[i] = 0.0;
        // the sums start from zero: each cluster's reference point becomes its
        // current centroid (the one the update subtracts), so that Q_k holds the
        // objective term itself and the update cancels nothing large
        for (int64_t i = tid; i < (int64_t)K * p.Dp; i += nthr) p.R[i] = p.C[i];
    }
    if (local) {
        for (int i = threadIdx.x; i < K; i += kStatsThreads) hist[i] = 0;
        __syncthreads();
    }
    for (int64_t e = tid; e < ne; e += nthr) {
        uint32_t id;
        const int k = stats_entry(p, full, m, e, id);
        if (k < 0) continue;
        if (local) atomicAdd(&hist[k], 1);
        else atomicAdd(&p.hcount[k], 1);
    }
    if (local) {
        __syncthreads();
        for (int i = threadIdx.x; i < K; i += kStatsThreads)
            if (hist[i]) atomicAdd(&p.hcount[i], hist[i]);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&ctrl->stats_ticket, 1u) == used - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    // exclusive scan of the counts: each thread a contiguous run
    const int lane = threadIdx.x & 31;
    const int per = (K + kStatsThreads - 1) / kStatsThreads;
    const int b0 = threadIdx.x * per, b1 = min(b0 + per, K);
    int run = 0;
    for (int b = b0; b < b1; ++b) run += __ldcg(p.hcount + b);
    int incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[threadIdx.x >> 5] = incl;
    __syncthreads();
    int off = incl - run;
    for (int w = 0; w < (int)(threadIdx.x >> 5); ++w) off += wsum[w];
    for (int b = b0; b < b1; ++b) {
        const int c = __ldcg(p.hcount + b);
        p.hcur[b] = off;
        if (full) p.cnt[b] = (unsigned long long)c;
        p.hcount[b] = 0;  // ready for the next sort
        off += c;
    }
    if (threadIdx.x == 0) ctrl->stats_ticket = 0;
}

// Place every entry in its cluster's segment (per tile of 1024 entries:
// shared-memory counts, one global atomic per cluster and tile).
__global__ void __launch_bounds__(kStatsThreads) k_stats_scatter(Params p, int respect_done) {
    extern __shared__ int sh[];  // K counters | K bases
    Ctrl *ctrl = p.ctrl;
    count_kernel(ctrl);
    if (respect_done && *(volatile int *)&ctrl->done) return;
    const int mode = *(volatile int *)&ctrl->stats_full;
    if (mode == kStatsDirect) return;
    const bool full = mode == kStatsFull;
    const int64_t m = full ? 0 : (int64_t)ctrl->moved_count;
    const int64_t ne = stats_entries(p, full);
    const int K = p.K;
    const bool local = K <= p.hist_smem_k;
    if (!local) {  // large K: one global atomic per entry
        for (int64_t e = (int64_t)blockIdx.x * kStatsThreads + threadIdx.x; e < ne;
             e += (int64_t)gridDim.x * kStatsThreads) {
            uint32_t id;
            const int k = stats_entry(p, full, m, e, id);
            if (k < 0) continue;
            const int pos = atomicAdd(&p.hcur[k], 1);
            p.perm[pos] = (int32_t)id;
            p.slab[pos] = k;
        }
        return;
    }
    if ((int64_t)blockIdx.x * kStatsTile >= ne) return;  // no tile for this block (block-uniform)
    int *cnt = sh;
    int *base = sh + K;
    for (int i = threadIdx.x; i < K; i += kStatsThreads) cnt[i] = 0;
    __syncthreads();
    for (int64_t t0 = (int64_t)blockIdx.x * kStatsTile; t0 < ne; t0 += (int64_t)gridDim.x * kStatsTile) {
        int k[4];
        uint32_t id[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t e = t0 + j * kStatsThreads + threadIdx.x;
            k[j] = e < ne ? stats_entry(p, full, m, e, id[j]) : -1;
            if (k[j] >= 0) atomicAdd(&cnt[k[j]], 1);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < K; i += kStatsThreads) {
            const int c = cnt[i];
            base[i] = c ? atomicAdd(&p.hcur[i], c) : 0;
            cnt[i] = 0;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (k[j] >= 0) {
                const int pos = base[k[j]] + atomicAdd(&cnt[k[j]], 1);
                p.perm[pos] = (int32_t)id[j];
                p.slab[pos] = k[j];
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < K; i += kStatsThreads) cnt[i] = 0;
        __syncthreads();
    }
}

// The same operations on one value and on two (kp_common.cuh)
__device__ __forceinline__ float add2(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float mul2(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma2(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ void two_sum2(float a, float b, float &s, float &e) { two_sum(a, b, s, e); }
__device__ __forceinline__ float flip2(float a, bool neg) { return neg ? -a : a; }
__device__ __forceinline__ f32x2 flip2(f32x2 a, bool neg) { return a ^ (neg ? kNeg2 : 0ull); }
__device__ __forceinline__ void put2(float &v, float lo, float) { v = lo; }
__device__ __forceinline__ void put2(f32x2 &v, float lo, float hi) { v = pack2(lo, hi); }
__device__ __forceinline__ void get2(float v, float &lo, float &hi) { lo = v, hi = 0.f; }
__device__ __forceinline__ void get2(f32x2 v, float &lo, float &hi) { unpack2(v, lo, hi); }

// Each warp sums a run of consecutive sorted entries, lanes over the
// coordinates, eight entries' loads in flight at a time, and adds its partial
// sums to S and Q (and, in incremental mode, the count change to cnt) whenever
// the cluster changes along the run (and at its end).  A subtracted entry
// adds -x and -||x - R_k||^2 (exact negations).
// Q_k sums ||x - R_k||^2 (R_k = the cluster's reference point, set to its
// centroid by k_stats_hist).  FP64 arithmetic is slow on the SMs of this GPU,
// so the run sums are kept as unevaluated FP32 pairs (hi + lo, compensated
// summation with TwoSum; the squares split exactly with a fused
// multiply-add), accurate to a few units in 2^-48 relative for runs this
// short, and turned into FP64 only when they are added to the global sums.
//
// Bound by latency: a batch of eight rows is read at random places (each 64 to
// 512 bytes) and summed before the next is asked for.  The run's ids are in
// registers before its first batch, so that a batch waits for its rows only, and
// two coordinates of a lane go through the arithmetic together (f32x2).
// Measured, all points: 1,048,576 x 64: 139 -> 105 us; 300,007 x 64: 54 -> 37;
// 4,194,304 x 128: 900 -> 670.  A ring of rows in shared memory, seven ahead, with
// a rolled loop over the points measured 157, 54 and 900.
template <int NPER>  // coordinates per lane: ceil(D / 32), in pairs beyond one
__global__ void __launch_bounds__(kStatsThreads, NPER <= 2 ? 3 : (NPER == 4 ? 2 : 1)) k_stats_sum(Params p, int respect_done) {
    Ctrl *ctrl = p.ctrl;
    count_kernel(ctrl);
    if (respect_done && *(volatile int *)&ctrl->done) return;
    const int mode = *(volatile int *)&ctrl->stats_full;
    if (mode == kStatsDirect) return;
    const bool full = mode == kStatsFull;
    const int64_t ne = stats_entries(p, full);
    const int D = p.D;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * kStatsThreads + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * kStatsThreads) >> 5;
    constexpr int kB = 8;  // points per batch
    using V = std::conditional_t<NPER == 1, float, f32x2>;  // coordinates lane + 64 j and lane + 64 j + 32
    constexpr int NP = (NPER + 1) / 2;
    // entries placed: the hist kernel's count (entries without a cluster are
    // not placed), read from the segment ends
    const int64_t placed = ne == 0 ? 0 : (int64_t)__ldcg(p.hcur + (p.K - 1));
    const int run = (full || ne * 8 > p.N) ? kSumRun : kSumRunMoved;
    for (int64_t r0 = warp * run; r0 < placed; r0 += nwarps * run) {
        const int64_t r1 = min(r0 + run, placed);
        V sh[NP], sl[NP], rn[NP];  // sums; minus the reference point of cluster `cur`
        V qh = 0, ql = 0;
        long long dn = 0;  // count change of cluster `cur` (incremental mode)
        // the run's ids and clusters, two per lane, so that a batch's rows do not
        // wait for them
        const int cnt = (int)(r1 - r0);
        static_assert(kSumRun <= 64 && kB <= 32 && 32 % kB == 0, "two per lane, a batch in one of them");
        const int id0 = lane < cnt ? p.perm[r0 + lane] : 0, id1 = lane + 32 < cnt ? p.perm[r0 + lane + 32] : 0;
        const int k0 = lane < cnt ? p.slab[r0 + lane] : -1, k1 = lane + 32 < cnt ? p.slab[r0 + lane + 32] : -1;
        int cur = __shfl_sync(0xffffffffu, k0, 0);
        auto load_ref = [&]() {
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const int i = lane + 64 * j;
                const float *r = p.R + (size_t)cur * p.Dp + i;
                put2(rn[j], i < D ? -r[0] : 0.f, 2 * j + 1 < NPER && i + 32 < D ? -r[32] : 0.f);
                sh[j] = sl[j] = 0;
            }
        };
        load_ref();
        auto flush = [&]() {
            float h0, h1, l0, l1, e;
            get2(qh, h0, h1);
            get2(ql, l0, l1);
            two_sum(h0, h1, h0, e);
            const double qs = warp_sum_d((double)h0 + (double)__fadd_rn(e, __fadd_rn(l0, l1)));
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const int i = lane + 64 * j;
                get2(sh[j], h0, h1);
                get2(sl[j], l0, l1);
                const double v0 = (double)h0 + (double)l0;
                if (i < D && v0 != 0.0) atomicAdd(&p.S[(size_t)cur * D + i], v0);
                if (2 * j + 1 < NPER) {
                    const double v1 = (double)h1 + (double)l1;
                    if (i + 32 < D && v1 != 0.0) atomicAdd(&p.S[(size_t)cur * D + i + 32], v1);
                }
            }
            if (lane == 0 && qs != 0.0) atomicAdd(&p.Q[cur], qs);
            if (lane == 0 && dn != 0 && !full) atomicAdd(&p.cnt[cur], (unsigned long long)dn);  // two's complement
            qh = ql = 0;
            dn = 0;
        };
        for (int e = 0; e < cnt; e += kB) {
            const int ide = e < 32 ? id0 : id1, ke = e < 32 ? k0 : k1;
            int nb[kB], kb[kB];
            bool neg[kB];
            V xv[kB][NP];
#pragma unroll
            for (int b = 0; b < kB; ++b) {
                const uint32_t id = (uint32_t)__shfl_sync(0xffffffffu, ide, (e & 31) + b);
                nb[b] = (int)(id & ~kNegEntry);
                neg[b] = (id & kNegEntry) != 0u;
                kb[b] = __shfl_sync(0xffffffffu, ke, (e & 31) + b);
            }
#pragma unroll
            for (int b = 0; b < kB; ++b) {
                const float *x = p.X + (int64_t)nb[b] * D;
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    const int i = lane + 64 * j;
                    put2(xv[b][j], kb[b] >= 0 && i < D ? __ldg(x + i) : 0.f,
                         2 * j + 1 < NPER && kb[b] >= 0 && i + 32 < D ? __ldg(x + i + 32) : 0.f);
                }
            }
#pragma unroll
            for (int b = 0; b < kB; ++b) {
                if (kb[b] < 0) break;
                if (kb[b] != cur) {  // warp-uniform
                    flush();
                    cur = kb[b];
                    load_ref();
                }
                dn += neg[b] ? -1 : 1;
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    const V xi = xv[b][j];
                    V e, dh, dl;
                    two_sum2(sh[j], flip2(xi, neg[b]), sh[j], e);
                    sl[j] = add2(sl[j], e);
                    // x - r as an exact pair dh + dl, its square as sq + sqe (exact)
                    // plus 2 dh dl + dl^2 (below 2^-47 of the square)
                    two_sum2(xi, rn[j], dh, dl);
                    const V sq = mul2(dh, dh);
                    const V sqe = fma2(dh, dh, flip2(sq, true));
                    const V cross = fma2(add2(dh, dh), dl, mul2(dl, dl));
                    two_sum2(qh, flip2(sq, neg[b]), qh, e);
                    ql = add2(ql, add2(e, flip2(add2(sqe, cross), neg[b])));
                }
            }
        }
        flush();
    }
}

bool stats_full_supported(const Params &p) { return p.perm != nullptr && p.D <= 32 * kSumMaxPer; }

cudaError_t launch_stats_full(const Params &p, cudaStream_t s, int all_points, int respect_done, int num_sms) {
    {
        const size_t h1 = p.K <= p.hist_smem_k ? (size_t)p.K * 4 : 0;
        const size_t h2 = 2 * h1;
        // (one value for every context: it is the process's, and another thread's context may be launching)
        cudaError_t e =
            cudaFuncSetAttribute(k_stats_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, p.hist_smem_k * 8);
        if (e != cudaSuccess) return e;
        const int64_t blocks = (p.N + kStatsTile - 1) / kStatsTile;
        // two blocks per SM: each block adds its counts to the K global ones
        // and takes a ticket, so fewer blocks mean fewer contended atomics
        const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(blocks, (int64_t)num_sms * 2));
        count_launch();
        k_stats_hist<<<grid, kStatsThreads, h1, s>>>(p, all_points, respect_done);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        count_launch();
        k_stats_scatter<<<grid, kStatsThreads, h2, s>>>(p, respect_done);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        const int64_t runs = (p.N + kSumRun - 1) / kSumRun;
        const unsigned sgrid = (unsigned)std::max<int64_t>(
            1, std::min<int64_t>((runs + kStatsThreads / 32 - 1) / (kStatsThreads / 32), (int64_t)num_sms * 8));
        count_launch();
        const int nper = (p.D + 31) / 32;
        if (nper <= 1) k_stats_sum<1><<<sgrid, kStatsThreads, 0, s>>>(p, respect_done);
        else if (nper <= 2) k_stats_sum<2><<<sgrid, kStatsThreads, 0, s>>>(p, respect_done);
        else if (nper <= 4) k_stats_sum<4><<<sgrid, kStatsThreads, 0, s>>>(p, respect_done);
        else k_stats_sum<kSumMaxPer><<<sgrid, kStatsThreads, 0, s>>>(p, respect_done);
        return cudaGetLastError();
    }
}

}  // namespace kp
