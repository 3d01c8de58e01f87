// kp_dense.cu -- dense assignment (every point against every centroid) and
// the cluster-statistics update for the points it moved.
//
// Used for iteration 0 of the filtered method, where every bound is created
// (KPynq Sec. I: the distance calculator evaluates whatever the filters have
// not removed, and at t = 0 nothing is removed yet), and for every iteration
// of plain Lloyd, the comparison baseline.
//
// The distance is the direct difference sum (x_i - c_i)^2 in FP32; its rounding
// error is bounded (Params::eps_hi/eps_lo), and when the two nearest FP32
// values cannot be ordered by that bound the two are ordered by compensated FP32
// sums (pair_order), or, where those decide nothing or a third is as near, in FP64
// with the summation order of the FP64 definition, so labels are exact.
#include "kp_common.cuh"

namespace kp {

constexpr int kDenseThreads = 128;
constexpr int kDenseWarps = kDenseThreads / 32;
constexpr int kDenseTileBytes = 64 * 1024;
constexpr int kDenseLbBytes = 48 * 1024;

// acc += d d (in place: fma2 in its stead takes up to 8 registers more here)
__device__ __forceinline__ void fma2_sq(f32x2 &acc, f32x2 d) {
    asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(acc) : "l"(d));
}
// any D: x and c in global memory (c with stride Dp)
__device__ __forceinline__ float sqdist_gen(const float *__restrict__ x, const float *__restrict__ c, int D) {
    float a0 = 0.f, a1 = 0.f;
    int i = 0;
    for (; i + 1 < D; i += 2) {
        float t0 = x[i] - c[i], t1 = x[i + 1] - c[i + 1];
        a0 = fmaf(t0, t0, a0);
        a1 = fmaf(t1, t1, a1);
    }
    if (i < D) {
        float t0 = x[i] - c[i];
        a0 = fmaf(t0, t0, a0);
    }
    return a0 + a1;
}

// the same for a centroid's row in global memory, 16 bytes at a time (it is
// aligned, and zero from D up to a multiple of 4)
__device__ __forceinline__ float sqdist_row(const float *__restrict__ x, const float *__restrict__ c, int D) {
    float a0 = 0.f, a1 = 0.f;
    for (int i = 0; i < D; i += 4) {
        const float4 cv = *reinterpret_cast<const float4 *>(c + i);
        const float t0 = x[i] - cv.x, t1 = (i + 1 < D ? x[i + 1] : 0.f) - cv.y;
        const float t2 = (i + 2 < D ? x[i + 2] : 0.f) - cv.z, t3 = (i + 3 < D ? x[i + 3] : 0.f) - cv.w;
        a0 = fmaf(t0, t0, a0);
        a1 = fmaf(t1, t1, a1);
        a0 = fmaf(t2, t2, a0);
        a1 = fmaf(t3, t3, a1);
    }
    return a0 + a1;
}

// What the scan over the centroids leaves of a point.
struct Nearest {
    float s1, s2;    // smallest and second smallest value
    int best;        // centroid of s1
    float bg_m2;     // smallest value in the best's group without the best
    float gm1, gm2;  // the same two of the group being scanned
    int ga;          // its best centroid

    __device__ __forceinline__ void init() {
        s1 = s2 = bg_m2 = gm1 = gm2 = INFINITY;
        best = ga = 0;
    }
    // (a NaN is never below anything and leaves both minima alone)
    __device__ __forceinline__ void visit(int c, float s) {
        const bool q = s < gm1;
        gm2 = fminf(gm2, q ? gm1 : s);
        gm1 = fminf(gm1, s);
        ga = q ? c : ga;
    }
    // end of a group: its smallest value, for the caller's bound
    __device__ __forceinline__ float close() {
        const float m = gm1;
        if (gm1 < s1) {
            s2 = fminf(s1, gm2);
            s1 = gm1;
            best = ga;
            bg_m2 = gm2;
        } else {
            s2 = fminf(s2, gm1);
        }
        gm1 = gm2 = INFINITY;
        return m;
    }
};

__device__ __forceinline__ float bound_dn(float s, const Params &p) { return s == INFINITY ? INFINITY : dist_dn(s, p); }

// Finish a warp's points (lane: point n if active, its scan's result; row: its
// group bounds, in shared or global memory).  Near-ties are settled by the
// whole warp, one point at a time: the lanes share the centroids out; a single
// one that the FP32 bound cannot separate from the best is ordered by
// pair_order, several (or what that leaves open) by their FP64 distances.
// Returns the lane's number of settled points; `changed` counts its moves.
__device__ __forceinline__ int finish_points(const Params &p, Ctrl *ctrl, bool active, int64_t n, Nearest &t,
                                             float *row, bool bounds, int first, int v, int &changed) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool near = active && t.s2 != INFINITY && unresolved(t.s1, t.s2, p);
    unsigned todo = __ballot_sync(full, near);
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const int64_t m = __shfl_sync(full, n, src);
        const float ref = __shfl_sync(full, t.s1, src);
        const int was = __shfl_sync(full, t.best, src);
        const float *xr = p.X + m * p.D;
        // the centroids that FP32 cannot separate from the best
        int many = 0, other = was;
        float so = ref;
        for (int c0 = 0; c0 < p.K; c0 += 32) {
            const int c = c0 + lane;
            const float s = c < p.K ? sqdist_row(xr, p.C + (size_t)c * p.Dp, p.D) : INFINITY;
            const unsigned in = __ballot_sync(full, c < p.K && c != was && unresolved(ref, s, p));
            many += __popc(in);
            if (in) {
                other = c0 + __ffs(in) - 1;
                so = __shfl_sync(full, s, __ffs(in) - 1);
            }
        }
        int bi = was;
        float bs = ref;
        const int o =
            many == 1 ? pair_order(xr, p.C + (size_t)was * p.Dp, p.C + (size_t)other * p.Dp, p.D) : (many ? -1 : 0);
        if (o == 1) {
            bi = other;
            bs = so;
        } else if (o < 0) {
            // two: a lane each, at the same time; several: the lanes share them out
            double bd = INFINITY;
            const int step = many == 1 ? p.K : 32;
            for (int c = many > 1 ? lane : (lane == 0 ? was : (lane == 1 ? other : p.K)); c < p.K; c += step) {
                const float s = sqdist_row(xr, p.C + (size_t)c * p.Dp, p.D);
                if (c != was && !unresolved(ref, s, p)) continue;
                const double d = dist2_f64(xr, p.C + (size_t)c * p.Dp, p.D);
                if (d < bd || (d == bd && tie_key(p, c) < tie_key(p, bi))) { bd = d; bi = c; bs = s; }
            }
#pragma unroll
            for (int w = 16; w > 0; w >>= 1) {
                const double od = __shfl_xor_sync(full, bd, w);
                const int oi = __shfl_xor_sync(full, bi, w);
                const float os = __shfl_xor_sync(full, bs, w);
                if (od < bd || (od == bd && tie_key(p, oi) < tie_key(p, bi))) { bd = od; bi = oi; bs = os; }
            }
        }
        if (bi != was) {
            if (bounds) {  // group bounds must now exclude the new best
                float *r = reinterpret_cast<float *>(__shfl_sync(full, reinterpret_cast<unsigned long long>(row), src));
                for (int g = lane; g < p.G; g += 32) {
                    float mn = INFINITY;
                    for (int c = p.gstart[g]; c < p.gstart[g + 1]; ++c)
                        if (c != bi) mn = fminf(mn, sqdist_row(xr, p.C + (size_t)c * p.Dp, p.D));
                    r[g] = bound_dn(mn, p);
                }
                __syncwarp();
            }
            if (lane == src) {
                t.best = bi;
                t.s1 = bs;
                t.bg_m2 = -1.f;  // already written
            }
        }
    }
    int old = t.best;
    if (active) {
        if (bounds) {
            if (t.bg_m2 >= 0.f) row[p.grp[t.best]] = bound_dn(t.bg_m2, p);
            p.u[n] = dist_up(t.s1, p);
            p.stamp[n] = make_stamp(v, v);
        }
        old = first ? -1 : p.label[n];
        p.label[n] = t.best;
    }
    const bool moved = old != t.best;
    changed += moved;
    if (!first) {
        const unsigned mv = __ballot_sync(full, moved);
        if (mv) {
            int slot = 0;
            if (lane == __ffs(mv) - 1) slot = atomicAdd(&ctrl->moved_count, __popc(mv));
            slot = __shfl_sync(full, slot, __ffs(mv) - 1) + __popc(mv & ((1u << lane) - 1u));
            if (moved) {
                p.moved[slot] = (int)n;
                p.moved_old[slot] = old;
            }
        }
    }
    return near;
}

// counters: one atomic per warp
__device__ __forceinline__ void add_counters(Ctrl *ctrl, int changed, int settled, int64_t dist) {
    changed = __reduce_add_sync(0xffffffffu, changed);
    settled = __reduce_add_sync(0xffffffffu, settled);
    if ((threadIdx.x & 31) == 0) {
        if (changed) atomicAdd(&ctrl->n_changed, (unsigned long long)changed);
        if (settled) atomicAdd(&ctrl->n_recheck, (unsigned long long)settled);
        if (dist) atomicAdd(&ctrl->n_dist, (unsigned long long)dist);
    }
}

// Dense assignment, D <= 128.  first: iteration 0 of this context (all points
// count as moved and are added to the sums by the caller).  Writes labels; for
// the filtered method also u, lbg, lb and stamps (exact at the current
// version).
//
// Bound by the FP32 pipe: a subtraction and a multiply-add per point, centroid
// and coordinate.  Both go through the packed instructions (f32x2), which halve
// the issue slots, and every value read from shared memory serves P points per
// lane, held in registers, of Q centroids at a time, so that 4 P packed
// instructions follow a 16-byte broadcast read and 2 P Q sums are in flight.
// Rows of more than 64 coordinates are cut over L lanes (32 / L lanes apart),
// whose partial sums meet in a transposing shuffle that leaves each lane the
// P / L points it owns.
//
// Measured, K = 256 (before: one point per lane, scalar, two centroids): 262,144
// x 64: 599 -> 310 us, the FP32 pipe busy in 75% of the cycles; 600,000 x 8:
// 286 -> 124; x 16: 377 -> 212; x 32: 673 -> 399; x 50: 1177 -> 667; x 128: 3358
// -> 1699.
template <int DPL, int L, int P, int Q, int MB>
__global__ void __launch_bounds__(kDenseThreads, MB) k_dense_assign(Params p, int first, int respect_done,
                                                                   int if_dense) {
    extern __shared__ __align__(128) float smem[];
    constexpr int OWN = P / L;                   // points a lane owns
    constexpr int PW = 32 * OWN;                 // points of a warp
    constexpr int PB = PW * kDenseWarps;         // points of a block
    constexpr int SEG = L > 1 ? DPL + 4 : DPL;   // a lane's part of a staged row (skewed: no bank conflicts)
    constexpr int RS = L * SEG;                  // staged row stride
    static_assert(DPL % 4 == 0 && P % L == 0 && (L == 1 || L == 2), "shape");
    Ctrl *ctrl = p.ctrl;
    count_kernel(ctrl);
    if (respect_done && *(volatile int *)&ctrl->done) return;
    if (if_dense && !*(volatile int *)&ctrl->dense_mode) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) ctrl->path = KM_PATH_DENSE_FP32;
    const int v = ctrl->v;
    const int K = p.K, D = p.D;
    const bool bounds = p.algo == KM_ALGO_FILTERED;
    const int KT = min(K, kDenseTileBytes / (RS * 4));
    const bool resident = KT == K;
    float *cs = smem;
    const int ls = p.Gp + 1;
    const bool stage_lb = bounds && (size_t)ls * PB * 4 <= kDenseLbBytes;
    float *lbs = smem + (size_t)KT * RS;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int part = lane / (32 / L);      // which coordinates
    const int lidx = lane % (32 / L);      // which points

    auto stage = [&](int c0, int kt) {
        for (int i = threadIdx.x; i < kt * (L * DPL / 4); i += kDenseThreads) {
            const int r = i / (L * DPL / 4), q = (i % (L * DPL / 4)) * 4;
            const float *c = p.C + (size_t)(c0 + r) * p.Dp;
            float4 w;
            if (q + 4 <= p.Dp) {  // the padding up to Dp is zero
                w = *reinterpret_cast<const float4 *>(c + q);
            } else {
                w.x = w.y = w.z = w.w = 0.f;
            }
            *reinterpret_cast<float4 *>(cs + r * RS + (q / DPL) * SEG + q % DPL) = w;
        }
    };
    if (resident) {
        stage(0, K);
        __syncthreads();
    }

    int changed = 0, settled = 0;
    int64_t dist = 0;
    for (int64_t base = (int64_t)blockIdx.x * PB; base < p.N; base += (int64_t)gridDim.x * PB) {
        const int64_t w0 = base + warp * PW;  // the warp's points, 32 / L apart per lane
        f32x2 x[P][DPL / 2];
#pragma unroll
        for (int j = 0; j < P; ++j) {
            const int64_t n = w0 + j * (32 / L) + lidx;
            const float *row = p.X + min(n, p.N - 1) * D;
            if (p.x_vec4) {
#pragma unroll
                for (int i = 0; i < DPL; i += 4) {
                    ulonglong2 w = make_ulonglong2(0ull, 0ull);
                    if (part * DPL + i < D) w = __ldg(reinterpret_cast<const ulonglong2 *>(row + part * DPL + i));
                    x[j][i / 2] = w.x;
                    x[j][i / 2 + 1] = w.y;
                }
            } else {
#pragma unroll
                for (int i = 0; i < DPL; i += 2) {
                    const int q = part * DPL + i;
                    const float a = q < D ? __ldg(row + q) : 0.f, b = q + 1 < D ? __ldg(row + q + 1) : 0.f;
                    asm("mov.b64 %0, {%1, %2};" : "=l"(x[j][i / 2]) : "f"(a), "f"(b));
                }
            }
        }
        // the point in slot o of this lane
        auto own = [&](int o) { return w0 + (part * OWN + o) * (32 / L) + lidx; };
        auto lb_row = [&](int o) {
            const int64_t n = min(own(o), p.N - 1);
            return stage_lb ? lbs + (int)(own(o) - base) * ls : p.lb + n * p.Gp;
        };
        Nearest t[OWN];
#pragma unroll
        for (int o = 0; o < OWN; ++o) t[o].init();
        int g = 0, gend = bounds ? p.gstart[1] : K;
        auto close_group = [&]() {
#pragma unroll
            for (int o = 0; o < OWN; ++o) {
                const float m = t[o].close();
                if (bounds && (stage_lb || own(o) < p.N)) lb_row(o)[g] = bound_dn(m, p);
            }
        };
        // centroid c's sums of this lane's part of its P points, to the owners
        auto visit = [&](int c, const f32x2 *acc) {
            while (c == gend) {  // same for all threads
                close_group();
                gend = p.gstart[++g + 1];
            }
            float s[P];
#pragma unroll
            for (int j = 0; j < P; ++j) s[j] = sum2(acc[j]);
#pragma unroll
            for (int h = L / 2; h > 0; h >>= 1) {  // h: the bit of `part` that this step settles
                const bool up = part & h;
                const int half = OWN * h;
#pragma unroll
                for (int j = 0; j < half; ++j) {
                    const float mine = up ? s[j + half] : s[j], give = up ? s[j] : s[j + half];
                    s[j] = mine + __shfl_xor_sync(0xffffffffu, give, h * (32 / L));
                }
            }
#pragma unroll
            for (int o = 0; o < OWN; ++o) t[o].visit(c, s[o]);
        };
        for (int c0 = 0; c0 < K; c0 += KT) {
            const int kt = min(KT, K - c0);
            if (!resident) {
                __syncthreads();
                stage(c0, kt);
                __syncthreads();
            }
            const float *cp = cs + part * SEG;
            for (int k = 0; k < kt; k += Q) {
                f32x2 acc[Q][P];
                const float *c[Q];
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    c[q] = cp + min(k + q, kt - 1) * RS;
#pragma unroll
                    for (int j = 0; j < P; ++j) acc[q][j] = 0ull;
                }
#pragma unroll
                for (int i = 0; i < DPL / 2; i += 2) {
#pragma unroll
                    for (int q = 0; q < Q; ++q) {
                        const ulonglong2 u = *reinterpret_cast<const ulonglong2 *>(c[q] + 2 * i);
#pragma unroll
                        for (int j = 0; j < P; ++j) {
                            fma2_sq(acc[q][j], sub2(x[j][i], u.x));
                            fma2_sq(acc[q][j], sub2(x[j][i + 1], u.y));
                        }
                    }
                }
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    if (k + q < kt) visit(c0 + k + q, acc[q]);
            }
        }
        while (true) {  // the last group, and empty ones behind it
            close_group();
            if (!bounds || ++g >= p.G) break;
        }
        __syncwarp();
#pragma unroll
        for (int o = 0; o < OWN; ++o) {
            const int64_t n = own(o);
            settled += finish_points(p, ctrl, n < p.N, n, t[o], lb_row(o), bounds, first, v, changed);
        }
        dist += max((int64_t)0, min((int64_t)PW, p.N - w0)) * K;
        if (bounds) {
            __syncwarp();
            // lbg = min over the row, then a coalesced copy of the warp's rows
#pragma unroll
            for (int o = 0; o < OWN; ++o) {
                if (own(o) < p.N) {
                    const float *r = lb_row(o);
                    float m = INFINITY;
                    for (int q = 0; q < p.G; ++q) m = fminf(m, r[q]);
                    p.lbg[own(o)] = m;
                }
            }
            if (stage_lb && w0 < p.N) {
                const int count = (int)min((int64_t)PW, p.N - w0) * p.Gp;
                const float *src = lbs + warp * PW * ls;
                float *dst = p.lb + w0 * p.Gp;
                for (int i = lane; i < count; i += 32) {
                    const int r = i / p.Gp, q = i - r * p.Gp;
                    dst[i] = q < p.G ? src[r * ls + q] : 0.f;
                }
            }
            __syncwarp();
        }
    }
    add_counters(ctrl, changed, settled, lane == 0 ? dist : 0);
}

// Dense assignment, any D: one point per lane, operands in global memory.
__global__ void __launch_bounds__(kDenseThreads) k_dense_assign_any(Params p, int first, int respect_done,
                                                                    int if_dense) {
    Ctrl *ctrl = p.ctrl;
    count_kernel(ctrl);
    if (respect_done && *(volatile int *)&ctrl->done) return;
    if (if_dense && !*(volatile int *)&ctrl->dense_mode) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) ctrl->path = KM_PATH_DENSE_FP32;
    const int v = ctrl->v;
    const bool bounds = p.algo == KM_ALGO_FILTERED;
    int changed = 0, settled = 0;
    int64_t dist = 0;
    for (int64_t base = (int64_t)blockIdx.x * kDenseThreads; base < p.N; base += (int64_t)gridDim.x * kDenseThreads) {
        const int64_t n = base + threadIdx.x;
        const bool active = n < p.N;
        const int64_t row = min(n, p.N - 1);
        float *lb = p.lb + row * p.Gp;
        Nearest t;
        t.init();
        if (active) {
            const float *x = p.X + row * p.D;
            int g = 0, gend = bounds ? p.gstart[1] : p.K;
            for (int c = 0; c <= p.K; ++c) {
                while (c == gend) {
                    const float m = t.close();
                    if (!bounds) break;
                    lb[g] = bound_dn(m, p);
                    if (++g == p.G) break;
                    gend = p.gstart[g + 1];
                }
                if (c < p.K) t.visit(c, sqdist_gen(x, p.C + (size_t)c * p.Dp, p.D));
            }
        }
        settled += finish_points(p, ctrl, active, n, t, lb, bounds, first, v, changed);
        dist += active ? p.K : 0;
        if (bounds) {
            __syncwarp();
            if (active) {
                float m = INFINITY;
                for (int g = 0; g < p.G; ++g) m = fminf(m, lb[g]);
                p.lbg[n] = m;
                for (int g = p.G; g < p.Gp; ++g) lb[g] = 0.f;
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dist += __shfl_xor_sync(0xffffffffu, dist, o);
    add_counters(ctrl, changed, settled, (threadIdx.x & 31) == 0 ? dist : 0);
}

// Cluster statistics for moved points: S[new] += x, S[old] -= x (FP64),
// Q (sum of ||x||^2) and counts likewise.  One warp per point, lanes over the
// coordinates, so each point's atomics are coalesced.
__global__ void __launch_bounds__(256) k_apply_moves(Params p, int all_points, int respect_done, int if_dense) {
    Ctrl *ctrl = p.ctrl;
    count_kernel(ctrl);
    if (respect_done && *(volatile int *)&ctrl->done) return;
    if (if_dense && !*(volatile int *)&ctrl->dense_mode) return;
    if (*(volatile int *)&ctrl->stats_full) return;  // recomputed in full instead
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t count = all_points ? p.N : (int64_t)ctrl->moved_count;
    for (int64_t it = warp; it < count; it += nwarps) {
        int64_t n;
        int old;
        if (all_points) { n = it; old = -1; }
        else { n = p.moved[it]; old = p.moved_old[it]; }
        move_point(p, n, old);
    }
}

int dense_dp(int D) {
    if (D <= 4) return 4;
    if (D <= 8) return 8;
    if (D <= 16) return 16;
    if (D <= 32) return 32;
    if (D <= 64) return 64;
    if (D <= 128) return 128;
    return 0;
}

template <int DPL, int L, int P, int Q, int MB>
static cudaError_t launch_dense_t(const Params &p, cudaStream_t s, int first, int respect_done, int num_sms,
                                  int if_dense) {
    constexpr int PB = P / L * kDenseThreads;
    constexpr int RS = L * (L > 1 ? DPL + 4 : DPL);
    size_t smem = (size_t)std::min(p.K, kDenseTileBytes / (RS * 4)) * RS * 4;
    const size_t lb = (size_t)(p.Gp + 1) * PB * 4;
    if (p.algo == KM_ALGO_FILTERED && lb <= (size_t)kDenseLbBytes) smem += lb;
    auto kernel = k_dense_assign<DPL, L, P, Q, MB>;
    // (one value for every context: it is the process's, and another thread's context may be launching)
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kDenseTileBytes + kDenseLbBytes);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kDenseThreads, smem);
    if (e != cudaSuccess) return e;
    const int64_t tiles = (p.N + PB - 1) / PB;
    const int64_t grid = std::min<int64_t>(tiles, (int64_t)num_sms * std::max(per_sm, 1));
    count_launch();
    kernel<<<(unsigned)grid, kDenseThreads, smem, s>>>(p, first, respect_done, if_dense);
    return cudaGetLastError();
}

cudaError_t launch_dense_assign(const Params &p, cudaStream_t s, int first, int respect_done, int num_sms,
                                int if_dense) {
    // few points: one per lane, so that they spread over more warps
    // (200 centroids in 17 dimensions: 60,000 points 33 us against 35, 120,000
    // the same, 250,000 101 against 92)
    // Otherwise P and Q by width, as measured (600,000 points, K = 256): up to 8
    // coordinates 4 points and 2 centroids (123 us against 136 with 2 and 4),
    // beyond 2 and 4 (D = 16: 212 against 224; 32: 400 against 387, but 65 against
    // 71 for K = 32); D = 128: a row on two lanes 1699, on one 1689, on four 1805
    const bool few = p.N < (int64_t)num_sms * kDenseThreads * 4;
#define DENSE(DPL, L, P, Q, MB) return launch_dense_t<DPL, L, P, Q, MB>(p, s, first, respect_done, num_sms, if_dense)
#define DENSE_F(DPL, P, Q, MB)            \
    do {                                  \
        if (few) DENSE(DPL, 1, 1, 4, MB); \
        else DENSE(DPL, 1, P, Q, MB);     \
    } while (0)
    if (p.D <= 32) switch ((p.D + 3) / 4) {
        case 1: DENSE_F(4, 4, 2, 4);
        case 2: DENSE_F(8, 4, 2, 4);
        case 3: DENSE_F(12, 2, 4, 4);
        case 4: DENSE_F(16, 2, 4, 4);
        case 5: DENSE_F(20, 2, 4, 4);
        case 6: DENSE_F(24, 2, 4, 4);
        case 7: DENSE_F(28, 2, 4, 4);
        default: DENSE_F(32, 2, 4, 3);
        }
    if (p.D <= 64) switch ((p.D + 7) / 8) {
        case 5: DENSE_F(40, 2, 4, 2);
        case 6: DENSE_F(48, 2, 4, 2);
        case 7: DENSE_F(56, 2, 4, 2);
        default: DENSE_F(64, 2, 4, 2);
        }
    if (p.D <= 128) switch ((p.D + 15) / 16) {
        case 5: DENSE(40, 2, 2, 4, 2);
        case 6: DENSE(48, 2, 2, 4, 2);
        case 7: DENSE(56, 2, 2, 4, 2);
        default: DENSE(64, 2, 2, 4, 2);
        }
#undef DENSE_F
#undef DENSE
    const int64_t grid = std::min<int64_t>((p.N + kDenseThreads - 1) / kDenseThreads, (int64_t)num_sms * 8);
    count_launch();
    k_dense_assign_any<<<(unsigned)grid, kDenseThreads, 0, s>>>(p, first, respect_done, if_dense);
    return cudaGetLastError();
}

cudaError_t launch_apply_moves(const Params &p, cudaStream_t s, int all_points, int respect_done, int num_sms,
                               int if_dense) {
    int64_t items = all_points ? p.N : p.N;  // moved count is only known on the device
    int64_t grid = std::min<int64_t>((items + 7) / 8, (int64_t)num_sms * 8);
    grid = std::max<int64_t>(grid, 1);
    count_launch();
    k_apply_moves<<<(unsigned)grid, 256, 0, s>>>(p, all_points, respect_done, if_dense);
    return cudaGetLastError();
}

}  // namespace kp
