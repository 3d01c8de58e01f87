// kp_kmeanspp.cu -- k-means++ seeding on the GPU.
//
// The paper takes its initial centroids as given; the library also offers the
// D^2 seeding of k-means++ (Arthur and Vassilvitskii, SODA 2007): the first
// centre is a point drawn uniformly, each further one a point drawn with
// probability proportional to D(x)^2, its squared distance to the nearest
// centre chosen so far.  The random numbers are inputs (one uniform in [0, 1)
// per centre) and every decision is exact, so that any implementation given
// the same uniforms picks the same points:
//   D(x)^2   FP64, sum_i (x_i - c_i)^2 with i ascending and no fused
//            multiply-add, minimised over the centres chosen so far;
//   weights  q(x) = floor(D(x)^2 * 2^s) (64-bit integers), 2^s the power of two
//            that puts max_x D(x)^2 in [2^31, 2^32) -- an exact scaling, and
//            integer sums are exact in any order;
//   draw     T = floor(u_j * W), W = sum q (T = W - 1 if the product rounds up
//            to W); the centre is the first point (in index order) whose
//            running sum of q exceeds T; W = 0: floor(u_j * N); first: floor(u_0 * N).
//
// FP64 runs at 1/64 of the FP32 rate, so D(x)^2 is kept in FP64 but evaluated
// only where it can change: per centre an FP32 distance with a rigorous error
// bound settles, for all but about N / j of the points after j centres, that
// the new centre is not nearer.  The others are collected per block (FP64
// costs a warp the same for one lane as for 32) and get their FP64 distance;
// the conversions of x to FP64, which share that pipe, are made on the integer
// one.
//
// Nor does every point need its FP32 distance: with the nearest centre a(x)
// kept beside D(x)^2, ||c - a(x)||^2 >= 4 D(x)^2 shows by the triangle
// inequality that the new centre c is not nearer, from eight bytes of the point
// and a table of the distances between c and the other centres, which every
// block makes for itself.  What is left of X to read per centre are the rows
// near c and those that no centre is near to yet.  (For few points a block there
// is no table: making it would cost more than reading them.)
//
// The weights need no FP64 either: for max D^2 in [2^(e-1), 2^e), q(x) is a
// shift of the significand of D(x)^2.  e = e0 - k, with 2^e0 > max D^2 when e0
// was set and k the first occupied bin of a histogram of the points by the
// binary orders that D(x)^2 lies below 2^e0.  The histogram and the chunk sums
// of q change only with the points that change; a second set of sums is kept
// for k + 1, so that the usual step of k costs a re-summation during the next
// sweep only.  When the maximum falls further (the first centres do that, and
// outliers) the sums are made anew by all blocks: the next launch does that
// instead of a sweep, and the host makes up for the launches spent so (one to
// spare is always launched).
// (16,777,216 x 2, K = 4, one such fall: 35 ms with the last block making the
// sums, 1.4 now, 1.9 with FP64 distances to every point.)
//
// Scratch: D(x)^2, and beside it what the bound's filter reads (a(x) and D(x)^2
// in FP32).  Where memory for the second half is short the sweeps do without
// that filter.
//
// One launch per centre as a rule (k_pp_step): the distances to the centre drawn
// last, the sums, and -- in the last block to finish -- the next draw: the chunk
// holding T, then the point in it, copied to the output centroids.  Every
// block owns a run of chunks.
// Measured on GB300 (1,048,576 x 32, K = 128): 337 us per centre and 43.9 ms in
// all with FP64 distances to every point; 50 us and 6.9 ms with the FP32 filter
// alone (21 the read of X, 8 the FP64 distances, 8 the draw, 5 the launch);
// 38 us and 5.4 ms with the bound's filter before it; 4.9 ms without a copy of the
// arguments in local memory.  3,878 x 100: 45 -> 22 us per centre with the FP32
// filter.
#include <cmath>

#include "kp_common.cuh"

namespace kp {
namespace {

constexpr int kPPThreads = 256;
constexpr int kPPWarps = kPPThreads / 32;
// blocks per SM of the sweep and row groups a warp has in flight: 96 KB of rows
// per SM either way; 4 blocks with 4 or 6 groups measured 7.3 ms for the job
// above, 3 with 8 groups 7.0 ms (fewer spills)
constexpr int kPPBlocks = 3, kPPU = 8;
constexpr int kPPSegment = 2048;   // points filtered between two looks at the list
constexpr int kPPList = 2 * kPPSegment;
constexpr int kPPTable = 1024;     // centres whose distances to the new one the first filter uses
constexpr int kPPMaxD = 4096;      // coordinates of a point (the centre is in shared memory)
constexpr int kPPMaxChunks = 4096; // chunk size: the power of two >= 32 that gives at most so many
constexpr int kPPBins = 65;        // binary orders of D^2 below 2^e0 (64: more, or zero)

// what the next launch does
enum PPTodo : int {
    kPPSweep,  // the distances to the last centre
    kPPSums,   // the chunk sums anew
    kPPMax,    // the largest distance
    kPPHist    // the histogram and the chunk sums anew
};

struct PPState {
    int chosen;               // centres chosen so far
    int err;                  // nonzero: an index out of range was produced
    long long pick;           // the centre chosen last
    unsigned long long wmax;  // bit pattern of max D^2 (doubles >= 0 order as their bits)
    int todo;                 // PPTodo
    int e0;                   // scale of the histogram
    int k;                    // its first occupied bin when the last draw was made
    int cur;                  // the set of sums of the weights at k; the other: at k + 1
    int resum;                // the other set must be made anew
    unsigned ticket;          // blocks done
    unsigned long long hist[kPPBins];  // points by the binary order of D^2 (NaN: in none)
};

__device__ __forceinline__ long long uniform_index(double u, long long N) {
    long long i = (long long)floor(__dmul_rn(u, (double)N));
    return i < 0 ? 0 : (i >= N ? N - 1 : i);
}

// e with d = m 2^e, m in [0.5, 1) (d normal: a nonzero squared distance between
// FP32 points is at least 2^-298)
__device__ __forceinline__ int exponent_of(unsigned long long bits) { return (int)((bits >> 52) & 0x7ff) - 1022; }

// the weights floor(d 2^(32 - e)) for 0 <= d < 2^e, from the bits of d (NaN: 0;
// infinity: the largest integer), at e and at e - 1
struct Weights {
    unsigned long long at, next;
};
__device__ __forceinline__ Weights weights(double d, int e) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(d);
    const int ex = (int)(bits >> 52);  // d = m 2^(ex - 1075)
    const unsigned long long m = ex == 0 || d != d ? 0ull : (bits & 0xfffffffffffffull) | 0x10000000000000ull;
    const unsigned long long next = m >> (min(max(1043 + e - ex, 1), 64) - 1);
    if (ex == 0x7ff && m != 0ull) return {~0ull, ~0ull};
    return {next >> 1, next};
}

// the bin of d (not NaN)
__device__ __forceinline__ int bin_of(double d, int e0) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(d);
    return (bits >> 52) ? min(max(e0 - exponent_of(bits), 0), 64) : 64;
}

// float to double on the integer pipe, exact for zero and normal numbers;
// others set `odd` (no branch, so that several conversions and products are in
// flight at once)
__device__ __forceinline__ double widen(float x, bool &odd) {
    const unsigned u = __float_as_uint(x), m = u & 0x7fffffffu;
    odd |= m != 0u && m - 0x00800000u >= 0x7f000000u;
    const unsigned h = m == 0u ? 0u : (m >> 3) + 0x38000000u;
    return __hiloint2double((int)((u & 0x80000000u) | h), (int)(u << 29));
}

// FP64 squared distance, i ascending, no fused multiply-add (VEC: D a multiple
// of 4, rows 16-byte aligned); c in FP64
template <bool VEC>
__device__ __forceinline__ double dist2(const float *x, const double *c, int D) {
    constexpr int B = 8;  // coordinates whose squares are formed before they are summed
    double s = 0.0;
    bool odd = false;
    int i = 0;
    for (; i + B <= D; i += B) {
        float xv[B];
        if constexpr (VEC) {
#pragma unroll
            for (int k = 0; k < B; k += 4) {
                const float4 v = __ldg(reinterpret_cast<const float4 *>(x + i + k));
                xv[k] = v.x;
                xv[k + 1] = v.y;
                xv[k + 2] = v.z;
                xv[k + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < B; ++k) xv[k] = __ldg(x + i + k);
        }
        double t[B];
#pragma unroll
        for (int k = 0; k < B; ++k) t[k] = __dsub_rn(widen(xv[k], odd), c[i + k]);
#pragma unroll
        for (int k = 0; k < B; ++k) t[k] = __dmul_rn(t[k], t[k]);
#pragma unroll
        for (int k = 0; k < B; ++k) s = __dadd_rn(s, t[k]);
    }
    for (; i < D; ++i) {
        const double t = __dsub_rn(widen(__ldg(x + i), odd), c[i]);
        s = __dadd_rn(s, __dmul_rn(t, t));
    }
    if (odd) {  // a subnormal, infinite or NaN coordinate
        s = 0.0;
        for (i = 0; i < D; ++i) {
            const double t = __dsub_rn((double)__ldg(x + i), c[i]);
            s = __dadd_rn(s, __dmul_rn(t, t));
        }
    }
    return s;
}

// inclusive scan of one value per thread across the block
__device__ __forceinline__ unsigned long long block_scan_incl(unsigned long long v, unsigned long long *sh,
                                                              unsigned long long *total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    if (lane == 31) sh[w] = v;
    __syncthreads();
    unsigned long long before = 0, all = 0;
#pragma unroll
    for (int i = 0; i < kPPWarps; ++i) {
        if (i < w) before += sh[i];
        all += sh[i];
    }
    if (total) *total = all;
    __syncthreads();
    return v + before;
}
__device__ __forceinline__ unsigned long long warp_sum_u(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ unsigned long long warp_max_u(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

struct PPArgs {
    const float *X;
    long long N;
    int D, K;
    double *dmin;                 // N: D(x)^2
    float2 *ub;                   // N: D(x)^2 rounded up to FP32 (the filters' bound); the nearest
                                  // centre so far (an int in the second half); may be missing
    unsigned long long *sums0, *sums1;  // chunk sums of the weights (two sets)
    int csh;                      // log2 of the chunk size
    long long nb;                 // chunks
    const double *u;
    PPState *st;
    float *C;
    long long *idx;
};

// (an index into the kernel's arguments would copy them to local memory)
__device__ __forceinline__ unsigned long long *sums_of(const PPArgs &a, int set) { return set ? a.sums1 : a.sums0; }

// a load that stays where it is written
__device__ __forceinline__ int ld_now(const int *p) {
    int v;
    asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ long long ld_now(const long long *p) {
    long long v;
    asm volatile("ld.global.s64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}

// the chunks of this block: [first, last)
__device__ __forceinline__ long long chunk0(const PPArgs &a, unsigned blk) {
    return (long long)blk * a.nb / gridDim.x;
}

// centre j is point `pick`: its row to C, its index to idx
__device__ __forceinline__ void take_centre(const PPArgs &a, int j, long long pick) {
    for (int i = threadIdx.x; i < a.D; i += kPPThreads) a.C[(long long)j * a.D + i] = a.X[pick * a.D + i];
    if (threadIdx.x == 0) {
        a.idx[j] = pick;
        a.st->pick = pick;
    }
}

// d = D(x_n)^2 of the points n of chunk b, lanes over the points, four loads in
// flight
template <class F>
__device__ __forceinline__ void each_distance(const PPArgs &a, long long b, F f) {
    const long long n1 = min(a.N, (b + 1) << a.csh);
    for (long long n0 = (b << a.csh) + (threadIdx.x & 31); n0 < n1; n0 += 128) {
        double d[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) d[v] = n0 + 32 * v < n1 ? __ldcg(a.dmin + n0 + 32 * v) : 0.0;
#pragma unroll
        for (int v = 0; v < 4; ++v)
            if (n0 + 32 * v < n1) f(n0 + 32 * v, d[v]);
    }
}

// A block's part of what a fall of the maximum asks for (PPTodo); with `ub` also
// the filter's bound of every point, nearest centre 0.
__device__ __forceinline__ void remake(const PPArgs &a, int todo, float2 *ub) {
    __shared__ int hist[kPPBins];
    if (threadIdx.x < kPPBins) hist[threadIdx.x] = 0;
    __syncthreads();
    const PPState *st = a.st;
    const int e0 = st->e0, e = e0 - st->k, cur = st->cur, lane = threadIdx.x & 31;
    const long long c1 = chunk0(a, blockIdx.x + 1);
    unsigned long long m = 0;
    for (long long b = chunk0(a, blockIdx.x) + (threadIdx.x >> 5); b < c1; b += kPPWarps) {
        if (todo == kPPMax) {
            each_distance(a, b, [&](long long, double d) {
                if (d == d) m = max(m, (unsigned long long)__double_as_longlong(d));
            });
            continue;
        }
        unsigned long long s0 = 0, s1 = 0;
        each_distance(a, b, [&](long long n, double d) {
            if (ub) ub[n] = make_float2(d == d ? __double2float_ru(d) : INFINITY, __int_as_float(0));
            const Weights w = weights(d, e);
            s0 += w.at;
            s1 += w.next;
            if (todo == kPPHist && d == d) atomicAdd(&hist[bin_of(d, e0)], 1);
        });
        s0 = warp_sum_u(s0);
        s1 = warp_sum_u(s1);
        if (lane == 0) {
            sums_of(a, cur)[b] = s0;
            sums_of(a, cur ^ 1)[b] = s1;
        }
    }
    m = warp_max_u(m);
    if (lane == 0 && m) atomicMax(&a.st->wmax, m);
    __syncthreads();
    if (threadIdx.x < kPPBins && hist[threadIdx.x])  // (a block's points fit 31 bits, all together need not)
        atomicAdd(&a.st->hist[threadIdx.x], (unsigned long long)hist[threadIdx.x]);
}

// The last block to finish (whole block): the draw of the next centre from the
// chunk sums, or the order to remake them first.  Every other block's results are
// visible (fence and ticket).
__device__ __forceinline__ void draw(const PPArgs &a) {
    __shared__ unsigned long long sh[kPPWarps];
    __shared__ unsigned long long s_before;
    __shared__ long long s_block, s_pick;
    __shared__ int s_k;
    __shared__ unsigned long long s_sum[kPPMaxChunks + kPPMaxChunks / 16];
    constexpr int kPer = kPPMaxChunks / kPPThreads;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    PPState *st = a.st;
    int cur = ld_now(&st->cur);
    const int kg = ld_now(&st->k), j = ld_now(&st->chosen), e0 = ld_now(&st->e0), todo = ld_now(&st->todo);
    // the sums at k, read before k is known to stand
    unsigned long long v[kPer];
    auto load_sums = [&](const unsigned long long *bs) {
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const long long b = i * kPPThreads + tid;
            v[i] = b < a.nb ? __ldcg(bs + b) : 0ull;
        }
    };
    load_sums(sums_of(a, cur));
    const double u = *const_cast<const volatile double *>(a.u + min(j, a.K - 1));  // (now: nothing else depends on it yet)
    if (warp == 0) {  // the first occupied bin
        const unsigned long long h0 = __ldcg(&st->hist[lane]), h1 = __ldcg(&st->hist[32 + lane]);
        const unsigned b0 = __ballot_sync(0xffffffffu, h0 != 0), b1 = __ballot_sync(0xffffffffu, h1 != 0);
        if (lane == 0) s_k = b0 ? __ffs(b0) - 1 : (b1 ? 31 + __ffs(b1) : 64);
    }
    if (tid == 0) {
        s_block = -1;
        s_pick = a.N;
    }
    __syncthreads();
    if (todo == kPPMax) {  // the scale; then the histogram
        if (tid < kPPBins) st->hist[tid] = 0ull;
        if (tid == 0) {
            const unsigned long long w = __ldcg(&st->wmax);
            if (w) st->e0 = exponent_of(w);
            st->k = w ? 0 : 64;  // all zero: it stays so
            st->todo = kPPHist;
            st->ticket = 0u;
        }
        return;
    }
    const int kt = s_k, resum = kt == kg + 1 && kt < 64;
    if (resum) {
        cur ^= 1;
    } else if (kt != kg) {  // (not after kPPSums and kPPHist)
        // the maximum fell by more than a factor of two, or (64) there was or is
        // none in the histogram's reach
        if (tid == 0) {
            if (kt == 64 || kg == 64) {
                st->todo = kPPMax;
                st->wmax = 0ull;
            } else {
                st->todo = kPPSums;
                st->k = kt;
            }
            st->ticket = 0u;
        }
        return;
    }
    const int e = e0 - kt;
    if (resum) load_sums(sums_of(a, cur));
    // per-thread run of consecutive chunk sums, scanned across the block
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int b = i * kPPThreads + tid;
        s_sum[b + (b >> 4)] = v[i];
    }
    __syncthreads();
    const int per = (int)((a.nb + kPPThreads - 1) / kPPThreads);  // at most kPer
    const int b0 = tid * per;
    unsigned long long run = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int b = b0 + i;
        v[i] = i < per && b < a.nb ? s_sum[b + (b >> 4)] : 0ull;
        run += v[i];
    }
    unsigned long long W = 0;
    const unsigned long long incl = block_scan_incl(run, sh, &W);
    if (W == 0) {  // every weight is zero: a uniform draw
        if (tid == 0) s_pick = uniform_index(u, a.N);
    } else {
        unsigned long long T = (unsigned long long)floor(__dmul_rn(u, (double)W));
        if (T >= W) T = W - 1;
        unsigned long long acc = incl - run;
        if (acc <= T && T < incl) {  // exactly one thread: its run holds T
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                if (acc <= T && acc + v[i] > T) {
                    s_block = b0 + i;
                    s_before = acc;
                }
                acc += v[i];
            }
        }
        __syncthreads();
        const long long b = s_block;
        if (b >= 0) {
            // the chunk, 256 points at a time, until the running sum exceeds T
            unsigned long long before = s_before;
            const long long n1 = min(a.N, (b + 1) << a.csh);
            for (long long n0 = b << a.csh; n0 < n1; n0 += kPPThreads) {
                const long long n = n0 + tid;
                const unsigned long long q = n < n1 ? weights(__ldcg(a.dmin + n), e).at : 0ull;
                unsigned long long tot;
                const unsigned long long in = before + block_scan_incl(q, sh, &tot);
                if (in > T && in - q <= T) s_pick = n;  // the first run above T
                before += tot;
                if (before > T) break;  // block-uniform
            }
        }
    }
    __syncthreads();
    long long pick = s_pick;
    if (pick < 0 || pick >= a.N) {  // cannot happen: the chunk sums and the scan agree
        if (tid == 0) st->err = 1;
        pick = 0;
    }
    take_centre(a, j, pick);
    if (tid == 0) {
        st->k = kt;
        st->cur = cur;
        st->resum = resum;
        st->chosen = j + 1;
        st->todo = kPPSweep;
        st->ticket = 0u;
    }
}

// true in every thread of the last block to get here
__device__ __forceinline__ bool last_block(PPState *st) {
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&st->ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Centre 0, drawn uniformly: every point's FP64 distance, and the scale of the
// weights.
template <bool VEC>
__global__ void __launch_bounds__(kPPThreads) k_pp_first(PPArgs a) {
    extern __shared__ double sd[];  // the centre (D)
    const long long pick = uniform_index(a.u[0], a.N);
    for (int i = threadIdx.x; i < a.D; i += kPPThreads) sd[i] = (double)a.X[pick * a.D + i];
    __syncthreads();
    unsigned long long m = 0;
    for (long long n = (long long)blockIdx.x * kPPThreads + threadIdx.x; n < a.N; n += (long long)gridDim.x * kPPThreads) {
        const double d = dist2<VEC>(a.X + n * a.D, sd, a.D);
        a.dmin[n] = d;
        if (d == d) m = max(m, (unsigned long long)__double_as_longlong(d));
    }
    m = warp_max_u(m);
    if ((threadIdx.x & 31) == 0 && m) atomicMax(&a.st->wmax, m);
    if (blockIdx.x == 0) take_centre(a, 0, pick);
    if (!last_block(a.st)) return;
    if (threadIdx.x == 0) {
        const unsigned long long w = __ldcg(&a.st->wmax);
        a.st->e0 = w ? exponent_of(w) : 0;
        a.st->k = w ? 0 : 64;
        a.st->chosen = 1;
        a.st->ticket = 0u;
    }
}

// The filter's bound of every point, the chunk sums and the histogram, the draw
// of centre 1
__global__ void __launch_bounds__(kPPThreads) k_pp_weigh(PPArgs a) {
    remake(a, kPPHist, a.ub);
    if (last_block(a.st)) draw(a);
}

// The centre drawn last: the distances it shortens, and the sums.  A row is read
// by LPR = 2^lprl lanes, 16 bytes each (VEC: D a multiple of 4 and 16-byte
// aligned rows) or one coordinate each, so that a warp's loads are contiguous;
// successive centres sweep a block's points in opposite directions (`odd`), so
// that the end of one sweep is found in L2 by the next.  BOUND: the bound's
// filter comes first.
template <bool VEC, bool BOUND>
__device__ __forceinline__ void sweep(const PPArgs &a, int chosen, long long pick, int e0, int k, int cur, int resum,
                                      int odd, int table, int lprl, float eps_lo, float tiny) {
    // the centre: FP64 (D), then FP32 padded to a multiple of LPR vectors with
    // zeros; the first filter's table (kPPTable) and list (kPPSegment)
    extern __shared__ double sd[];
    __shared__ unsigned list[kPPList];
    __shared__ int hist[kPPBins];
    __shared__ int nlist, nkept;
    __shared__ int newest, s_e0, s_k, s_cur;  // the centre drawn last; of the state (registers are short)
    const int D = a.D, LPR = 1 << lprl, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *sc = reinterpret_cast<float *>(sd + ((D + 1) & ~1));
    constexpr int W = VEC ? 4 : 1;
    const int nv = D / W;                      // vectors of a row
    const int steps = (nv + LPR - 1) >> lprl;  // vectors per lane
    float *far = sc + steps * LPR * W;         // what D(x)^2 has to exceed for the new centre to matter
    unsigned short *kept = reinterpret_cast<unsigned short *>(far + kPPTable);
    {
        const float *c = a.X + pick * D;
        for (int i = threadIdx.x; i < steps * LPR * W; i += kPPThreads) {
            const float v = i < D ? c[i] : 0.f;
            sc[i] = v;
            if (i < D) sd[i] = (double)v;
        }
    }
    if (threadIdx.x < kPPBins) hist[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        nlist = nkept = 0;
        newest = chosen - 1;
        s_e0 = e0;
        s_k = k;
        s_cur = cur;
    }
    const long long c0 = chunk0(a, blockIdx.x), c1 = chunk0(a, blockIdx.x + 1);
    const long long p0 = c0 << a.csh, p1 = min(a.N, c1 << a.csh);  // this block's points
    if (resum)
        for (long long b = c0 + warp; b < c1; b += kPPWarps) {
            unsigned long long s = 0;
            const long long n1 = min(a.N, (b + 1) << a.csh);
            for (long long n = (b << a.csh) + lane; n < n1; n += 32) s += weights(a.dmin[n], e0 - k).next;
            s = warp_sum_u(s);
            if (lane == 0) sums_of(a, cur ^ 1)[b] = s;
        }
    __syncthreads();

    const int sub = lane >> lprl, l = lane & (LPR - 1), rows = 32 >> lprl;
    // a quarter of the squared distances between the new centre and the others,
    // rounded down with room for the FP64 sums' own error: a point whose D^2 is
    // no larger is, by the triangle inequality, no nearer to the new centre
    const int ntab = BOUND ? min(chosen - 1, table) : 0;
    for (int g0 = warp * rows; g0 < ntab; g0 += kPPWarps * rows) {  // warp-uniform
        const int g = g0 + sub;
        float s = 0.f;
        for (int t = 0; t < steps; ++t) {
            const int q = l + (t << lprl);
            if (g < ntab && q < nv) {
                if constexpr (VEC) {
                    const float4 x = *(reinterpret_cast<const float4 *>(a.C + (long long)g * D) + q);
                    const float4 cc = *reinterpret_cast<const float4 *>(sc + 4 * q);
                    const float d0 = x.x - cc.x, d1 = x.y - cc.y, d2 = x.z - cc.z, d3 = x.w - cc.w;
                    s = fmaf(d3, d3, fmaf(d2, d2, fmaf(d1, d1, fmaf(d0, d0, s))));
                } else {
                    const float d = a.C[(long long)g * D + q] - sc[q];
                    s = fmaf(d, d, s);
                }
            }
        }
        for (int o = LPR >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (l == 0 && g < ntab)
            far[g] = s < INFINITY ? __fmul_rd(__fsub_rd(__fmul_rd(s, eps_lo), tiny), 0.249997f) : -1.f;
    }
    __syncthreads();
    auto bound = [&](long long n) {
        if constexpr (BOUND) return a.ub[n].x;
        const double d = a.dmin[n];
        return d == d ? __double2float_ru(d) : INFINITY;
    };
    constexpr int U = kPPU;  // row groups in flight
    for (long long q0 = p0; q0 < p1; q0 += kPPSegment) {
        // the filter, on a segment of this block's points
        const int cnt = (int)min((long long)kPPSegment, p1 - q0);
        // (odd: the segments and their rows from the end)
        const long long s0 = odd ? p1 - (q0 - p0) - cnt : q0;
        // first by the bound alone, a thread per point
        {
            constexpr int kPer = kPPSegment / kPPThreads;
            float2 b[kPer];
#pragma unroll
            for (int v = 0; v < kPer; ++v) {
                const int i = v * kPPThreads + threadIdx.x;
                b[v] = BOUND && i < cnt ? a.ub[s0 + i] : make_float2(-1.f, 0.f);
            }
#pragma unroll
            for (int v = 0; v < kPer; ++v) {
                const int i = v * kPPThreads + threadIdx.x, c = __float_as_int(b[v].y);
                const bool keep = i < cnt && !(BOUND && c < ntab && b[v].x <= far[c]);
                const unsigned m = __ballot_sync(0xffffffffu, keep);
                if (m) {
                    int at = 0;
                    if (lane == 0) at = atomicAdd(&nkept, __popc(m));
                    at = __shfl_sync(0xffffffffu, at, 0);
                    if (keep) kept[at + __popc(m & ((1u << lane) - 1u))] = (unsigned short)i;
                }
            }
        }
        __syncthreads();
        const int nk = nkept;
        // then by the FP32 distance
        for (int g0 = warp * U * rows; g0 < nk; g0 += kPPWarps * U * rows) {
            float s[U], ub[U];
            int r[U];
#pragma unroll
            for (int v = 0; v < U; ++v) {
                s[v] = 0.f;
                r[v] = g0 + v * rows + sub;
                if (odd) r[v] = nk - 1 - r[v];  // below zero past the end
                r[v] = r[v] >= 0 && r[v] < nk ? kept[r[v]] : -1;
                ub[v] = l == 0 && r[v] >= 0 ? bound(s0 + r[v]) : 0.f;
            }
            for (int t = 0; t < steps; ++t) {
                const int q = l + (t << lprl);
                if constexpr (VEC) {
                    float4 x[U];
#pragma unroll
                    for (int v = 0; v < U; ++v)
                        x[v] = r[v] >= 0 && q < nv ? __ldg(reinterpret_cast<const float4 *>(a.X + (s0 + r[v]) * D) + q)
                                                   : make_float4(0.f, 0.f, 0.f, 0.f);
                    const float4 cc = *reinterpret_cast<const float4 *>(sc + 4 * q);
#pragma unroll
                    for (int v = 0; v < U; ++v) {
                        const float d0 = x[v].x - cc.x, d1 = x[v].y - cc.y, d2 = x[v].z - cc.z, d3 = x[v].w - cc.w;
                        s[v] = fmaf(d3, d3, fmaf(d2, d2, fmaf(d1, d1, fmaf(d0, d0, s[v]))));
                    }
                } else {
                    float x[U];
#pragma unroll
                    for (int v = 0; v < U; ++v) x[v] = r[v] >= 0 && q < nv ? __ldg(a.X + (s0 + r[v]) * D + q) : 0.f;
                    const float cc = sc[q];
#pragma unroll
                    for (int v = 0; v < U; ++v) {
                        const float d = x[v] - cc;
                        s[v] = fmaf(d, d, s[v]);
                    }
                }
            }
#pragma unroll
            for (int v = 0; v < U; ++v)
                for (int o = LPR >> 1; o > 0; o >>= 1) s[v] += __shfl_xor_sync(0xffffffffu, s[v], o);
#pragma unroll
            for (int v = 0; v < U; ++v) {
                bool pass = false;
                if (l == 0 && r[v] >= 0) {
                    // not nearer when the distance is certainly at least D^2 (an
                    // overflowed one settles nothing)
                    const float lo = __fsub_rd(__fmul_rd(s[v], eps_lo), tiny);
                    pass = !(lo >= ub[v] && s[v] < INFINITY);
                }
                const unsigned m = __ballot_sync(0xffffffffu, pass);
                if (m) {
                    int base = 0;
                    if (lane == 0) base = atomicAdd(&nlist, __popc(m));
                    base = __shfl_sync(0xffffffffu, base, 0);
                    if (pass) list[base + __popc(m & ((1u << lane) - 1u))] = (unsigned)(s0 + r[v] - p0);
                }
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) nkept = 0;
        // the FP64 distances of the points it kept, when they fill the block or
        // the points end
        const int n = nlist;
        __syncthreads();
        if (n < kPPSegment / 2 && q0 + kPPSegment < p1) continue;  // (room for a whole segment is left)
        for (int i = threadIdx.x; i < n; i += kPPThreads) {
            const long long pt = p0 + list[i];
            const double s = dist2<VEC>(a.X + pt * D, sd, D);
            const double d = a.dmin[pt], m = fmin(d, s);
            if (m < d || (d != d && m == m)) {
                a.dmin[pt] = m;
                if constexpr (BOUND) a.ub[pt] = make_float2(__double2float_ru(m), __int_as_float(newest));
                const long long b = pt >> a.csh;
                const int e = s_e0 - s_k;
                const Weights wm = weights(m, e), wd = weights(d, e);
                atomicAdd(&sums_of(a, s_cur)[b], wm.at - wd.at);  // modulo 2^64
                atomicAdd(&sums_of(a, s_cur ^ 1)[b], wm.next - wd.next);
                if (d == d) atomicAdd(&hist[bin_of(d, s_e0)], -1);
                atomicAdd(&hist[bin_of(m, s_e0)], 1);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) nlist = 0;
        __syncthreads();
    }
    if (threadIdx.x < kPPBins && hist[threadIdx.x])  // (a block's points fit 31 bits, all together need not)
        atomicAdd(&a.st->hist[threadIdx.x], (unsigned long long)(long long)hist[threadIdx.x]);
}

// A sweep and the draw of the next centre, or what has to be done before that
// draw.
template <bool VEC, bool BOUND>
__global__ void __launch_bounds__(kPPThreads, kPPBlocks) k_pp_step(PPArgs a, int odd, int table, int lprl,
                                                                       float eps_lo, float tiny) {
    // the state's fields in one go, before the first of them is looked at
    const int chosen = ld_now(&a.st->chosen), todo = ld_now(&a.st->todo);
    const int e0 = ld_now(&a.st->e0), k = ld_now(&a.st->k), cur = ld_now(&a.st->cur), resum = ld_now(&a.st->resum);
    const long long pick = ld_now(&a.st->pick);
    if (chosen >= a.K) return;
    if (todo == kPPSweep) sweep<VEC, BOUND>(a, chosen, pick, e0, k, cur, resum, odd, table, lprl, eps_lo, tiny);
    else remake(a, todo, nullptr);
    if (last_block(a.st)) draw(a);
}

int kmeanspp_chunk_log2(int64_t N) {
    int c = 5;
    while (((N - 1) >> c) >= kPPMaxChunks) ++c;
    return c;
}

// device memory of a call
struct PPScratch {
    double *dmin;              // N
    float2 *ub;                // N, or NULL: the sweeps do without the bound's filter
    unsigned long long *sums;  // 2 per chunk
    PPState *st;
    double *u;                 // K
    float *C;                  // K x D
    long long *idx;            // K
};

// The launches that choose centres `chosen` .. K - 1, if the maximum falls
// slowly; a launch spent on remaking the sums leaves one centre more to the
// next call.
cudaError_t launch_kmeanspp(const PPScratch &w, const float *X, int64_t N, int D, int K, int chosen, cudaStream_t s,
                            int num_sms) {
    PPArgs a;
    a.X = X;
    a.N = N;
    a.D = D;
    a.K = K;
    a.dmin = w.dmin;
    a.ub = w.ub;
    a.csh = kmeanspp_chunk_log2(N);
    a.nb = (N + ((int64_t)1 << a.csh) - 1) >> a.csh;
    a.sums0 = w.sums;
    a.sums1 = w.sums + a.nb;
    a.u = w.u;
    a.st = w.st;
    a.C = w.C;
    a.idx = w.idx;
    cudaError_t e;
    // 16-byte loads where the rows allow; lanes per row: its vectors rounded up
    // to a power of two, at most a warp
    const bool vec = D % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    const int nv = vec ? D / 4 : D;
    int lprl = 0;
    while ((1 << lprl) < nv && lprl < 5) ++lprl;
    const int steps = (nv + (1 << lprl) - 1) >> lprl;
    const size_t smem = (size_t)((D + 1) & ~1) * 8 + (size_t)steps * (4u << lprl) * (vec ? 4 : 1) + kPPTable * 4 +
                        kPPSegment * 2;
    auto step = a.ub ? (vec ? k_pp_step<true, true> : k_pp_step<false, true>)
                     : (vec ? k_pp_step<true, false> : k_pp_step<false, false>);
    // (one value for every call: it is the process's, and another thread may be launching)
    constexpr int most = kPPMaxD * 12 + kPPTable * 4 + kPPSegment * 2;
    if ((e = cudaFuncSetAttribute(step, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) != cudaSuccess) return e;
    // FP32 error of a D-term sum of squared differences (any order), with room
    // for the FP64 sum's own (2^-53 relative): true >= computed (1 - eps) - tiny
    const double eps = (D + 8) * std::ldexp(1.0, -24) * (1.0 + 1.0 / 1024);
    float eps_lo = (float)(1.0 - eps);
    if ((double)eps_lo > 1.0 - eps) eps_lo = std::nextafter(eps_lo, 0.0f);
    const float tiny = std::ldexp((float)(D + 8), -149);
    // one wave of blocks that own whole chunks
    const unsigned grid = (unsigned)std::min<int64_t>(a.nb, (int64_t)num_sms * kPPBlocks);
    // Every block makes the table for itself: as many distances as half of its
    // points, and none for few points.  K = 300, all centres in the table / half the
    // points / none: 2,000 x 100: 9.8 / 7.4 / 7.1 ms (32 points a block), 40,000 x 32:
    // 5.8 / 5.4 / 5.0 (88), 60,000 x 784: 44 / 44 / 51 (132), 335,544 x 100: 13.2 / 13.2
    // / 21.5 (736), points in clusters; without clusters the table gains nothing and
    // costs 26 / 26 / 21.5 in the last case, 9.9 / 9.0 / 7.4 at 100,000 x 17 (219).
    const int64_t points = N / grid;
    const int table = points < 128 ? 0 : (int)std::min<int64_t>(kPPTable, points / 2);
    const unsigned fg = (unsigned)std::min<int64_t>((N + kPPThreads - 1) / kPPThreads, (int64_t)num_sms * 8);
    if (chosen == 0) {
        if ((e = cudaMemsetAsync(w.st, 0, sizeof(PPState), s)) != cudaSuccess) return e;
        count_launch();
        if (vec) k_pp_first<true><<<fg, kPPThreads, (size_t)D * 8, s>>>(a);
        else k_pp_first<false><<<fg, kPPThreads, (size_t)D * 8, s>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (K > 1) {
            count_launch();
            k_pp_weigh<<<grid, kPPThreads, 0, s>>>(a);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        chosen = 2;
    }
    // (one launch to spare, K - chosen + 1 in all: 2 us against the 25 us of another look)
    for (int j = chosen; j < K + (K > 2); ++j) {
        count_launch();
        step<<<grid, kPPThreads, smem, s>>>(a, j & 1, table, lprl, eps_lo, tiny);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace
}  // namespace kp

using namespace kp;

extern "C" {

KM_API int kmeans_init_kmeanspp(const float *X, int64_t N, int32_t D, int32_t K, const double *u, float *centroids,
                                int64_t *indices, void *stream) {
    auto fail = [](int code, const char *msg) {
        set_thread_error(msg);
        return code;
    };
    if (!X || !u || !centroids) return fail(KM_EINVAL, "a pointer argument is NULL");
    if (N < 1 || N >= ((int64_t)1 << 40) || D < 1 || D > kPPMaxD || K < 1 || (int64_t)K > N)
        return fail(KM_EINVAL, "need 1 <= K <= N < 2^40 and 1 <= D <= 4096");
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, X) != cudaSuccess ||
        (a.type != cudaMemoryTypeDevice && a.type != cudaMemoryTypeManaged)) {
        cudaGetLastError();
        return fail(KM_EINVAL, "X must be device memory");
    }
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                  cudaSuccess)
        return fail(KM_ECUDA, "device query failed");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int64_t nb = ((N - 1) >> kmeanspp_chunk_log2(N)) + 1;
    // one piece of memory, 256-byte aligned parts
    size_t bytes = 0;
    auto part = [&](size_t n) {
        const size_t at = bytes;
        bytes = (bytes + n + 255) & ~(size_t)255;
        return at;
    };
    const size_t o_dmin = part((size_t)N * 8), o_sums = part((size_t)nb * 16), o_st = part(sizeof(PPState)),
                 o_u = part((size_t)K * 8), o_C = part((size_t)K * D * 4), o_idx = part((size_t)K * 8);
    char *base = nullptr;
    PPScratch w = {};
    cudaError_t e = pool_alloc(dev, reinterpret_cast<void **>(&base), bytes, s);
    if (e == cudaSuccess) {
        w.dmin = reinterpret_cast<double *>(base + o_dmin);
        w.sums = reinterpret_cast<unsigned long long *>(base + o_sums);
        w.st = reinterpret_cast<PPState *>(base + o_st);
        w.u = reinterpret_cast<double *>(base + o_u);
        w.C = reinterpret_cast<float *>(base + o_C);
        w.idx = reinterpret_cast<long long *>(base + o_idx);
        e = cudaMemcpyAsync(w.u, u, (size_t)K * 8, cudaMemcpyDefault, s);
    }
    if (e == cudaSuccess && K > 2) {  // (the sweeps' only; they can do without)
        e = pool_alloc(dev, reinterpret_cast<void **>(&w.ub), (size_t)N * 8, s);
        if (e == cudaErrorMemoryAllocation) {
            cudaGetLastError();
            w.ub = nullptr;
            e = cudaSuccess;
        }
    }
    struct {
        int chosen, err;  // as in PPState
    } h = {0, 0};
    // every launch chooses a centre or gets nearer to it, at most three to a centre
    for (int64_t round = 0; e == cudaSuccess && h.chosen < K && !h.err && round <= 3 * (int64_t)K; ++round) {
        e = launch_kmeanspp(w, X, N, D, K, h.chosen, s, sms);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&h, w.st, sizeof(h), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaMemcpyAsync(centroids, w.C, (size_t)K * D * 4, cudaMemcpyDefault, s);
        if (e == cudaSuccess && indices) e = cudaMemcpyAsync(indices, w.idx, (size_t)K * 8, cudaMemcpyDefault, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    }
    for (void *p : {(void *)base, (void *)w.ub})
        if (p) cudaFreeAsync(p, s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(e == cudaErrorMemoryAllocation ? KM_ENOMEM : KM_ECUDA, cudaGetErrorString(e));
    }
    if (h.err || h.chosen < K) return fail(KM_ECUDA, "the draw produced an index out of range");
    return KM_OK;
}

}  // extern "C"
