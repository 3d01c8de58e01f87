// kp_dense_tc.cu -- dense assignment on the 5th-generation tensor cores.
//
// The distance calculator of KPynq (Sec. I) evaluates every pair the filters
// leave; when that is (nearly) every pair -- iteration 0, plain Lloyd, or a
// filtered iteration in which most points survive -- the evaluation is a
// dense contraction, ||x||^2 - 2 x.c + ||c||^2, and belongs on the tensor
// cores.
//
// Mixed precision with a bounded error ("BF16x3"): every FP32 value v is
// split into two bfloat16 numbers, v_h = bf16(v) and v_l = bf16(v - v_h), and
//     x.c ~ x_h.c_h + x_h.c_l + x_l.c_h
// is accumulated in FP32 by tcgen05.mma (kind::f16, M=128 points x N<=256
// centroids, K=16 per instruction, three instructions per K step).  X is
// split once per context into two bfloat16 copies that TMA loads with
// 128-byte swizzle; the centroid block is split into shared memory by the
// CTA itself.  Accumulators live in TMEM, double-buffered across two
// epilogue warp groups.
//
// Persistent CTA per SM: warp 0 issues TMA, one thread of warp 1 issues the
// MMAs, warps 2..17 (two groups of eight, two warps per TMEM lane quadrant,
// each scanning half of the columns) read the accumulators back with
// tcgen05.ld, one TMEM lane (= point) per thread, and turn
// t_k = ||c_k||^2 - 2 x.c_k into the winner, the runner-up and the per-group
// minima, four columns at a time (Scan4 in kp_tc.cuh).  Lower bounds are
// t-based with the error E(x) subtracted, the upper
// bound adds it; when the runner-up lies within 2E of the winner the point is
// settled exactly by kp_settle.cu (FP32 direct differences, then compensated FP32
// sums, then FP64, each where the one before cannot decide), so labels are exact.
//
// Bound by the scan: of 200 us for 1,048,576 x 64, K = 256, G = 26, loads,
// products and TMEM reads alone take 76, the scan 80 (the minima and maxima of
// four columns are 13 instructions on the half-rate pipe), the rows' bounds and
// labels 45.  Measured: that pass 226 -> 200 us, 300,007 x 64, K = 200, plain
// Lloyd, 55 -> 47 (column-by-column scan, rows finished by one of the two
// halves, a lane per centroid's norm before).
//
// Error model of t_k (per point; c_max = max ||c_k||, c2_max = max ||c_k||^2):
//   the split leaves |v - v_h - v_l| <= 2^-16 |v| (bfloat16 unit roundoff
//   2^-8, twice), so the three products miss at most 3.05 2^-16 |x_i c_i|;
//   products are exact in FP32 and the accumulation of 3D of them adds at
//   most 3D 2^-23 (Cauchy-Schwarz bounds sum |x_i c_i| by ||x|| ||c||);
//   ||c||^2 is an FP32 sum of squares and the final fma rounds once:
//     |t~ - t| <= (6.1 2^-16 + (6D+1) 2^-23) ||x|| ||c|| + (D+3) 2^-24 ||c||^2,
//   used with a 1.25x margin as E(x).
#include "kp_tc.cuh"

namespace kp {

namespace {

constexpr int kEpiWarps = 8;      // warps per epilogue group: two per TMEM lane quadrant
constexpr int kGroups = 2;        // epilogue groups = TMEM buffers
constexpr int kTcThreads = 64 + kGroups * kEpiWarps * 32;

// the two warps of a quadrant (named barrier `id`, 64 threads): every thread
// contributes v, every thread gets the AND
__device__ __forceinline__ bool pair_and(bool v, int id) {
    int out;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbar.red.and.pred q, %2, 64, p;\n\t"
        "selp.s32 %0, 1, 0, q;\n\t}"
        : "=r"(out)
        : "r"((int)v), "r"(id)
        : "memory");
    return out != 0;
}
__device__ __forceinline__ void pair_sync(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }

struct TcCfg {
    int Kp;        // centroid rows in shared memory (multiple of 32, <= 256)
    int stages;    // A pipeline depth
    int tmem_cols; // allocated TMEM columns (2 buffers)
    int buf_cols;  // columns per buffer (>= Kp, power of two)
    uint32_t off_A, off_cn, off_gs, off_stage, off_bar;
    int num_tiles;
    float e_lin;   // 1.25 (6.1 2^-16 + (6D+1) 2^-23), rounded up
    float e_c2;    // 1.25 (D+3) 2^-24, rounded up
    float xn_lo, xn_hi;  // relative error of the precomputed ||x - mu||^2
};

template <int D>
__global__ void __launch_bounds__(kTcThreads, 1)
    k_dense_tc(const __grid_constant__ CUtensorMap tmh, const __grid_constant__ CUtensorMap tml, Params p, TcCfg cfg,
               int first, int respect_done, int if_dense) {
    extern __shared__ uint8_t raw[];
    Ctrl *ctrl = p.ctrl;
    count_kernel(ctrl);
    if (respect_done && *(volatile int *)&ctrl->done) return;
    if (if_dense && !*(volatile int *)&ctrl->dense_mode) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) ctrl->path = KM_PATH_DENSE_TC;
    constexpr int NA = D / 64;  // 64-element atoms per row
    uint8_t *sm = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~(uintptr_t)1023);
    const int Kp = cfg.Kp;
    const int b_atom = Kp * 128;
    uint8_t *sBh = sm;
    uint8_t *sBl = sm + NA * b_atom;
    uint8_t *sA = sm + cfg.off_A;  // stage s: [NA atoms of x_h][NA atoms of x_l]
    float *cn = reinterpret_cast<float *>(sm + cfg.off_cn);  // [Kp] ||c||^2 (+inf: padding)
    int32_t *gtab = reinterpret_cast<int32_t *>(cn + Kp);  // [Kp] group of each column (padding: the last)
    uint32_t *bm = reinterpret_cast<uint32_t *>(sm + cfg.off_gs);  // [Kp / 32] group-start masks
    float *stage = reinterpret_cast<float *>(sm + cfg.off_stage);  // [2 groups x 128 rows][Gp + 1]
    float4 *t4 = reinterpret_cast<float4 *>(stage + (size_t)kGroups * kTM * (p.Gp + 1));  // one per scanning lane
    uint64_t *bars = reinterpret_cast<uint64_t *>(sm + cfg.off_bar);
    const int S = cfg.stages;
    uint64_t *full_a = bars;
    uint64_t *empty_a = bars + S;
    uint64_t *acc_full = bars + 2 * S;  // [kGroups]
    uint64_t *acc_empty = bars + 2 * S + kGroups;
    uint64_t *mma_done = bars + 2 * S + 2 * kGroups;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * S + 2 * kGroups + 1);
    float *c2max_s = reinterpret_cast<float *>(tmem_slot + 1);

    // (the broadcast tells the compiler that the warp index is warp-uniform)
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int v = ctrl->v;
    const int K = p.K, G = p.G;

    // a tile of points to stage s
    auto load_tile = [&](int tile, int s) {
        uint8_t *st = sA + (size_t)s * 2 * NA * kAtomBytes;
        mbar_arrive_expect_tx(&full_a[s], (uint32_t)(2 * NA * kAtomBytes));
        for (int a = 0; a < NA; ++a) {
            tma_2d(st + a * kAtomBytes, &tmh, 64 * a, tile * kTM, &full_a[s]);
            tma_2d(st + (NA + a) * kAtomBytes, &tml, 64 * a, tile * kTM, &full_a[s]);
        }
    };
    if (threadIdx.x == 0) {
        for (int i = 0; i < S; ++i) {
            bar_init(&full_a[i], 1);
            bar_init(&empty_a[i], 1);  // the commit of the MMAs that read the stage
        }
        for (int g = 0; g < kGroups; ++g) {
            bar_init(&acc_full[g], 1);
            bar_init(&acc_empty[g], kEpiWarps);
        }
        bar_init(mma_done, 1);
        *c2max_s = 0.f;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // the first tiles of points, on their way while the centroids are split
        int s = 0;
        for (int tile = blockIdx.x; tile < cfg.num_tiles && s < S; tile += gridDim.x, ++s) load_tile(tile, s);
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(cfg.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int c = threadIdx.x; c < Kp / 32; c += blockDim.x) bm[c] = 0u;
    // The centroid block, split into x_h / x_l bfloat16 tiles (128-byte swizzle),
    // and the FP32 norms of the values split (padding rows: zero tiles, norm
    // +inf).  Eight coordinates per thread, a row on D / 8 neighbouring lanes;
    // the loads of four rounds go out together, so that every launch pays their
    // latency once or twice.
    float cm = 0.f;
    constexpr int kRounds = 4;
    for (int i0 = threadIdx.x; i0 < Kp * (D / 8); i0 += kRounds * kTcThreads) {  // (whole warps: Kp D / 8 is a multiple of 32)
        const int q = i0 % (D / 8);  // the same in every round: kTcThreads is a multiple of D / 8
        float4 w[kRounds][2], m[2];
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        const bool in = q * 8 < p.D;  // coordinates beyond D: zero padding
#pragma unroll
        for (int s = 0; s < kRounds; ++s) {
            const int row = (i0 + s * kTcThreads) / (D / 8);
            const float4 *c = reinterpret_cast<const float4 *>(p.C + (size_t)min(row, K - 1) * p.Dp + q * 8);
            w[s][0] = in ? c[0] : zero;
            w[s][1] = in ? c[1] : zero;
        }
        const float4 *mu = reinterpret_cast<const float4 *>(p.mu + q * 8);  // (mu's padding columns are zero)
        m[0] = in && p.mu ? mu[0] : zero;
        m[1] = in && p.mu ? mu[1] : zero;
#pragma unroll
        for (int s = 0; s < kRounds; ++s) {
            const int row = (i0 + s * kTcThreads) / (D / 8);
            if (row >= Kp) break;  // warp-uniform
            const bool real = row < K;
            float vals[8] = {__fsub_rn(w[s][0].x, m[0].x), __fsub_rn(w[s][0].y, m[0].y), __fsub_rn(w[s][0].z, m[0].z),
                             __fsub_rn(w[s][0].w, m[0].w), __fsub_rn(w[s][1].x, m[1].x), __fsub_rn(w[s][1].y, m[1].y),
                             __fsub_rn(w[s][1].z, m[1].z), __fsub_rn(w[s][1].w, m[1].w)};
            float ss = 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                vals[k] = real ? vals[k] : 0.f;
                ss = fmaf(vals[k], vals[k], ss);
            }
            uint4 h, l;
            split8(vals, h, l);
            *reinterpret_cast<uint4 *>(sBh + swz_chunk(row, q, b_atom)) = h;
            *reinterpret_cast<uint4 *>(sBl + swz_chunk(row, q, b_atom)) = l;
#pragma unroll
            for (int o = D / 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
            if (q == 0) {
                cn[row] = real ? ss : INFINITY;
                gtab[row] = real ? p.grp[row] : G - 1;
            }
            if (real) cm = fmaxf(cm, ss);
        }
    }
    cm = warp_max(cm);
    __syncthreads();  // c2max_s and the masks initialised
    if (lane == 0 && cm > 0.f) atomicMax(reinterpret_cast<int *>(c2max_s), __float_as_int(cm));
    // group g >= 1 starts at column gstart[g] (< K <= Kp)
    for (int g = 1 + threadIdx.x; g < G; g += blockDim.x) {
        const int col = p.gstart[g];
        if ((unsigned)col < (unsigned)Kp) atomicOr(&bm[col >> 5], 1u << (col & 31));
    }
    // generic-proxy writes of the B tiles must be visible to the tensor cores
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA
        if (lane == 0) {
            int i = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < cfg.num_tiles && ok; tile += gridDim.x, ++i) {
                const int s = i % S, f = i / S;
                if (f == 0) continue;  // (issued above)
                ok = bar_wait(&empty_a[s], (f - 1) & 1, ctrl);
                if (!ok) break;
                load_tile(tile, s);
            }
            // drain: every issued copy has landed before the block can exit
            const int issued = i;
            for (int j = issued - S < 0 ? 0 : issued - S; j < issued; ++j)
                bar_wait(&full_a[j % S], (j / S) & 1, ctrl);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA
        if (lane == 0) {
            // kind::f16: F32 accumulate, BF16 A and B, K-major, N = Kp, M = 128
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(Kp >> 3) << 17) |
                                   ((uint32_t)(kTM >> 4) << 24);
            bool ok = true;
            int i = 0;
            for (int tile = blockIdx.x; tile < cfg.num_tiles && ok; tile += gridDim.x, ++i) {
                const int s = i % S, f = i / S;
                const int buf = i % kGroups, u = i / kGroups;
                if (u > 0 && !(ok = bar_wait(&acc_empty[buf], (u - 1) & 1, ctrl))) break;
                if (!(ok = bar_wait(&full_a[s], f & 1, ctrl))) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem + (uint32_t)(buf * cfg.buf_cols);
                const uint8_t *st = sA + (size_t)s * 2 * NA * kAtomBytes;
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks) {
                    if (D == 64 && 16 * ks >= p.D) break;  // 32 coordinates: the padding to 64 adds nothing
                    const int a = ks >> 2, j = ks & 3;
                    const uint64_t dah = desc_sw128(smem_u32(st + a * kAtomBytes + j * 32));
                    const uint64_t dal = desc_sw128(smem_u32(st + (NA + a) * kAtomBytes + j * 32));
                    const uint64_t dbh = desc_sw128(smem_u32(sBh + a * b_atom + j * 32));
                    const uint64_t dbl = desc_sw128(smem_u32(sBl + a * b_atom + j * 32));
                    const uint32_t acc = ks > 0;
                    asm volatile(
                        "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 q, %4, %4;\n\t"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %5, %3, q;\n\t"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %6, %2, %3, q;\n\t}" ::"r"(d_tmem),
                        "l"(dah), "l"(dbh), "r"(idesc), "r"(acc), "l"(dbl), "l"(dal)
                        : "memory");
                }
                // the A stage is free once these MMAs have read it
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 smem_u32(&empty_a[s]))
                             : "memory");
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 smem_u32(&acc_full[buf]))
                             : "memory");
            }
            // every MMA of this thread is complete before TMEM is freed
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(mma_done))
                         : "memory");
            bar_wait(mma_done, 0, ctrl);
        }
    } else {
        // ------------------------------------------------------- epilogue
        // Two warps per TMEM lane quadrant and group, one lane per row in both:
        // half 0 scans the first half of the accumulator columns, half 1 the
        // second.  They meet three times a tile (64-thread named barriers 1..8):
        // at its start, when half 1's result is in shared memory, and when half
        // 0's merged result is.  Everything else is each half's own: the group
        // minima it has scanned (half 0's slots are the group numbers, half 1's
        // the group numbers plus one), their bounds, and its share of the row.
        const int e = warp - 2;
        const int grp_id = e / kEpiWarps;
        const int half = (e % kEpiWarps) / 4;
        const int pid = 1 + grp_id * 4 + (e & 3);
        const int q = warp & 3;  // TMEM lane quadrant of this warp
        const int r = q * 32 + lane;
        const bool bounds = p.algo == KM_ALGO_FILTERED;
        const float c2max = __fmul_ru(*c2max_s, 1.0f + 1.0f / 1024);
        const float cmax = sqrt_hi(c2max);
        const float ec2 = __fmul_ru(cfg.e_c2, c2max);
        const uint32_t row = smem_u32(stage + (size_t)(grp_id * kTM + r) * (p.Gp + 1));  // shared by the pair
        // halves in steps of 16 columns; the group open across their border has
        // a part in both
        const int csplit = ((Kp >> 4) + 1) / 2 * 16;
        const int c0 = half ? csplit : 0, c1 = half ? Kp : csplit;
        const int gsplit = __shfl_sync(0xffffffffu, gtab[csplit - 1], 0);
        // the groups whose bounds this half writes, and the slot of group 0
        const int glo = half ? gsplit + 1 : 0, ghi = half || gsplit == G - 1 ? G : gsplit + 1;
        const uint32_t slot0 = row + 4u * half;
        const uint32_t mine = smem_u32(t4 + e * 32 + lane), other = smem_u32(t4 + (e ^ 4) * 32 + lane);
        Scan4 sc;
        sc.row = row;
        sc.t4 = mine;
        int c_changed = 0;
        int64_t c_dist = 0;
        auto put4 = [](uint32_t at, float x, float y, int z, float w) {
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at), "f"(x), "f"(y), "f"(__int_as_float(z)), "f"(w)
                         : "memory");
        };
        auto get4 = [](uint32_t at) {
            float4 v;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(at) : "memory");
            return v;
        };
        int i = grp_id;
        for (int tile = blockIdx.x + grp_id * gridDim.x; tile < cfg.num_tiles;
             tile += kGroups * gridDim.x, i += kGroups) {
            const int u = i / kGroups;
            const int64_t n = (int64_t)tile * kTM + r;
            const bool valid = n < p.N;
            // read now, so that their latency hides behind the wait and the scan
            const int old = half == 0 && valid && !first ? p.label[n] : -1;
            const float xn = valid ? p.xnorm[n] : 0.f;
            // waits are warp-uniform (the TMEM loads below are warp-collective)
            // and pair-uniform (the named barriers need both warps)
            const bool ok = __all_sync(0xffffffffu, bar_wait(&acc_full[grp_id], u & 1, ctrl));
            if (!pair_and(ok, pid)) break;
            tc_fence_after();
            const uint32_t tb = tmem + (uint32_t)(grp_id * cfg.buf_cols) + ((uint32_t)(q * 32) << 16);

            // group minima, winner (lowest index on ties) and runner-up over this
            // half's columns, 16 at a time, the next 16 in flight
            sc.b1 = sc.b2 = sc.gm = INFINITY;
            sc.c4 = c0;
            sc.pend = half ? gsplit + 1 : 0;
            auto sixteen = [&](const uint32_t(&acc)[16], int c) {
                // (a broadcast, so that the compiler knows the mask to be warp-uniform)
                const uint32_t m16 = __shfl_sync(0xffffffffu, bm[c >> 5], 0) >> (c & 31);
                const float4 *cn4 = reinterpret_cast<const float4 *>(cn + c);
#pragma unroll
                for (int j = 0; j < 16; j += 4) sc.four(&acc[j], cn4[j >> 2], (m16 >> j) & 15u, c + j);
            };
            {
                uint32_t ra[16], rb[16];
                tmem_ld16_async(tb + c0, ra);
#pragma unroll 1
                for (int c = c0; c < c1; c += 32) {
                    tmem_wait16(ra);
                    if (c + 16 < c1) tmem_ld16_async(tb + c + 16, rb);
                    sixteen(ra, c);
                    if (c + 16 < c1) {
                        tmem_wait16(rb);
                        if (c + 32 < c1) tmem_ld16_async(tb + c + 32, ra);
                        sixteen(rb, c + 16);
                    }
                }
            }
            // accumulators no longer needed
            tc_fence_before();
            __syncwarp();
            if (lane == 0) bar_arrive(&acc_empty[grp_id]);
            // the open group's minimum, and this half's result
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(row + 4u * (uint32_t)sc.pend), "f"(sc.gm) : "memory");
            float b1 = sc.b1, b2 = sc.b2;
            int i1 = sc.winner();
            if (half) put4(mine, b1, b2, i1, lds_f(slot0 + 4u * (uint32_t)gsplit));
            pair_sync(pid);
            if (half == 0) {
                const float4 m = get4(other);
                const bool bw = m.x < b1;  // half 0 holds the lower indices: it wins ties
                b2 = fminf(fminf(b2, m.y), fmaxf(b1, m.x));
                i1 = bw ? __float_as_int(m.z) : i1;
                b1 = fminf(b1, m.x);
                put4(mine, b1, b2, i1, 0.f);
                const uint32_t at = row + 4u * (uint32_t)gsplit;
                const float gm = fminf(lds_f(at), m.w);
                asm volatile("st.shared.f32 [%0], %1;" ::"r"(at), "f"(gm) : "memory");
            }
            pair_sync(pid);
            if (half) {
                const float4 m = get4(other);
                b1 = m.x;
                b2 = m.y;
                i1 = __float_as_int(m.z);
            }
            const float xlo = __fmul_rd(xn, cfg.xn_lo), xup = __fmul_ru(xn, cfg.xn_hi);
            const float R = __fadd_ru(sqrt_hi(xup), cmax);  // bounds ||x - mu|| + ||c - mu||
            const float E = __fmaf_ru(p.e_cen, __fmul_ru(R, R), __fmaf_ru(cfg.e_lin, __fmul_ru(sqrt_hi(xup), cmax), ec2));
            const float thr = __fadd_ru(b1, __fmul_ru(2.f, E));
            auto bound_of = [&](float t) { return t == INFINITY ? INFINITY : sqrt_lo(__fsub_rd(__fadd_rd(xlo, t), E)); };

            // Rows whose runner-up is inside the error window go to the settle
            // queue: k_settle decides them exactly afterwards from FP32 (and
            // FP64) distances to the centroids of the groups whose minimum lies
            // in the window (every other centroid is strictly farther than the
            // tensor-core winner i1, which is among them).  The epilogue writes
            // such a row's bounds as if i1 won; k_settle corrects them when it
            // does not.
            const bool need = valid && b2 <= thr;
            const unsigned nm = __ballot_sync(0xffffffffu, need);
            const bool moved = half == 0 && valid && !need && old != i1;
            int mbase = 0;
            const unsigned mm = __ballot_sync(0xffffffffu, moved);
            if (half == 0) {
                // label changes: one slot reservation per warp, used at the end
                if (mm && !first && lane == 0) mbase = atomicAdd(&ctrl->moved_count, __popc(mm));
                c_changed += moved;
                c_dist += valid ? K : 0;
                // the warp's 32 rows in the request bitmap (every word is written
                // by every dense pass, so the bitmap needs no clearing)
                if (lane == 0) p.sbits[(int64_t)tile * (kTM / 32) + q] = nm;
                if (valid && !need) p.label[n] = i1;
            }
            // this half's groups that can hold a window column (at most 64
            // groups; more: all of them), before the winner's own is replaced
            unsigned long long gmask = G <= 64 ? 0ull : ~0ull;
            if (nm && G <= 64)
                for (int g = glo; g < ghi; ++g)
                    gmask |= lds_f(slot0 + 4u * (uint32_t)g) <= thr ? 1ull << g : 0ull;
            if (bounds) {
                // the winner's group must exclude the winner: every other column
                // is at least the runner-up b2.  The bound is monotone in t, so the
                // smallest group bound is the bound of the runner-up.
                const int gb = gtab[i1];
                if (gb >= glo && gb < ghi)
                    asm volatile("st.shared.f32 [%0], %1;" ::"r"(slot0 + 4u * (uint32_t)gb), "f"(b2) : "memory");
                if (half && valid) {
                    p.lbg[n] = bound_of(b2);
                    p.u[n] = sqrt_hi(__fadd_ru(__fadd_ru(xup, b1), E));
                    p.stamp[n] = make_stamp(v, v);
                }
                // s_c >= xn_lo + t_c - E for every column c: the bounds of the
                // groups, four at a time to the row (the four that both halves
                // have a part of one by one; the padding with the last group)
                float *lbrow = p.lb + n * p.Gp;
                for (int g = glo & ~3; g < ghi; g += 4) {
                    float o[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int gk = min(max(g + k, glo), ghi - 1);
                        o[k] = g + k < G ? bound_of(lds_f(slot0 + 4u * (uint32_t)gk)) : 0.f;
                    }
                    if (valid) {
                        if (g >= glo && (g + 4 <= ghi || ghi == G)) {  // warp-uniform
                            *reinterpret_cast<float4 *>(lbrow + g) = make_float4(o[0], o[1], o[2], o[3]);
                        } else {
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                if (g + k >= glo && (g + k < ghi || ghi == G)) lbrow[g + k] = o[k];
                        }
                    }
                }
            }
            if (need) {
                SettleReq *rq = p.sreq + n;
                rq->gmask[half] = gmask;
                if (half == 0) {
                    rq->n = (int32_t)n;
                    rq->old = old;
                    rq->i1 = i1;
                    // every column is at least b1: when i1 loses, this bounds both i1's
                    // group (which now keeps i1) and the winner's group
                    rq->lb_alt = bound_of(b1);
                }
            }
            if (mm && !first) {
                mbase = __shfl_sync(0xffffffffu, mbase, 0);
                if (moved) {
                    const int slot = mbase + __popc(mm & ((1u << lane) - 1u));
                    p.moved[slot] = (int)n;
                    p.moved_old[slot] = old;
                }
            }
        }
        c_changed = __reduce_add_sync(0xffffffffu, c_changed);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c_dist += __shfl_xor_sync(0xffffffffu, c_dist, o);
        if (lane == 0) {
            if (c_changed) atomicAdd(&ctrl->n_changed, (unsigned long long)c_changed);
            if (c_dist) atomicAdd(&ctrl->n_dist, (unsigned long long)c_dist);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cfg.tmem_cols)
                     : "memory");
    }
}

// X -> (x_h, x_l) bfloat16 copies with rows of Dt >= D coordinates (zero
// padding), four elements per thread, and each row's ||x - mu||^2 (FP32 sum of
// the squares of the values split, reduced over the Dt / 4 lanes of the row).
// Dt / 4 is 16 or 32 and the loop steps by whole warps, so a row's lanes are
// one aligned half-warp or warp and all of them run every iteration.
__global__ void k_split_x(const float *X, int64_t N, int D, int Dt, uint2 *Xh, uint2 *Xl, float4 *Xcopy,
                          const float *mu, float *xnorm) {
    const int q4n = Dt / 4;
    const int64_t n4 = N * q4n;
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n4; base += stride) {
        const int64_t i = base + lane;
        const bool act = i < n4;
        const int64_t row = i / q4n;
        const int q4 = (int)(i - row * q4n);
        float ss = 0.f;
        if (act) {
            const float4 a =
                q4 * 4 < D ? *reinterpret_cast<const float4 *>(X + row * D + q4 * 4) : make_float4(0, 0, 0, 0);
            if (Xcopy && q4 * 4 < D) Xcopy[(row * D + q4 * 4) / 4] = a;  // the device copy, in the same pass
            // x - mu, rounded once to FP32 (the padding stays exactly zero)
            const float4 m =
                (mu && q4 * 4 < D) ? *reinterpret_cast<const float4 *>(mu + q4 * 4) : make_float4(0, 0, 0, 0);
            const float vv[4] = {__fsub_rn(a.x, m.x), __fsub_rn(a.y, m.y), __fsub_rn(a.z, m.z), __fsub_rn(a.w, m.w)};
            uint32_t hw[2], lw[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                __nv_bfloat16 h0 = __float2bfloat16_rn(vv[2 * k]), h1 = __float2bfloat16_rn(vv[2 * k + 1]);
                __nv_bfloat16 l0 = __float2bfloat16_rn(vv[2 * k] - __bfloat162float(h0));
                __nv_bfloat16 l1 = __float2bfloat16_rn(vv[2 * k + 1] - __bfloat162float(h1));
                hw[k] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                lw[k] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
            }
            Xh[i] = make_uint2(hw[0], hw[1]);
            Xl[i] = make_uint2(lw[0], lw[1]);
#pragma unroll
            for (int k = 0; k < 4; ++k) ss = fmaf(vv[k], vv[k], ss);
        }
        for (int o = q4n >> 1; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        if (act && q4 == 0 && xnorm) xnorm[row] = ss;
    }
}

int pow2_at_least(int x) {
    int p2 = 32;
    while (p2 < x) p2 <<= 1;
    return p2;
}

bool plan(const Params &p, size_t smem_limit, TcCfg &cfg, size_t &smem) {
    const int Dt = tc_dim(p.D);
    if (!Dt || p.K > 256) return false;
    cfg.Kp = ((p.K + 31) / 32) * 32;
    cfg.buf_cols = pow2_at_least(cfg.Kp);
    cfg.tmem_cols = kGroups * cfg.buf_cols;
    if (cfg.tmem_cols > 512) return false;
    const size_t NA = Dt / 64;
    const size_t b_bytes = 2 * NA * (size_t)cfg.Kp * 128;
    const size_t a_stage = 2 * NA * (size_t)kAtomBytes;
    const size_t cn_bytes = (size_t)cfg.Kp * 8;  // norms and groups of the columns
    const size_t gs_bytes = (((size_t)cfg.Kp / 32) * 4 + 15) & ~size_t(15);  // group-start masks
    // the rows' minima, and 16 bytes per scanning lane.  A shape is taken when two
    // stages of points fit beside half of those; at the border one stage is left.
    const size_t rows_bytes = (size_t)kGroups * kTM * (p.Gp + 1) * 4, lane_bytes = (size_t)kGroups * kEpiWarps * 32 * 16;
    const size_t stage_bytes = rows_bytes + lane_bytes;
    const size_t fixed = 1024 + b_bytes + cn_bytes + gs_bytes + stage_bytes + 64 * 8 + 64;
    if (fixed - lane_bytes / 2 + 2 * a_stage > smem_limit) return false;
    cfg.stages = (int)std::min<size_t>(6, (smem_limit - fixed) / a_stage);
    size_t off = b_bytes;
    cfg.off_A = (uint32_t)off;
    off += cfg.stages * a_stage;
    cfg.off_cn = (uint32_t)off;
    off += cn_bytes;
    cfg.off_gs = (uint32_t)off;
    off += gs_bytes;
    cfg.off_stage = (uint32_t)off;
    off += stage_bytes;
    off = (off + 7) & ~size_t(7);
    cfg.off_bar = (uint32_t)off;
    off += (2 * cfg.stages + 2 * kGroups + 1) * 8 + 16;
    smem = 1024 + off;
    if (smem > smem_limit) return false;
    cfg.num_tiles = (int)((p.N + kTM - 1) / kTM);
    const double D = Dt;  // the padded width: its zero products add nothing, the bound stays valid
    cfg.e_lin = (float)(1.25 * (6.1 * std::ldexp(1.0, -16) + (6 * D + 1) * std::ldexp(1.0, -23)) * (1 + 1e-6));
    cfg.e_c2 = (float)(1.25 * (D + 3) * std::ldexp(1.0, -24) * (1 + 1e-6));
    // ||x - mu||^2 from k_split_x: an FP32 sum of non-negative terms in which
    // each term meets at most 4 + log2(Dt / 4) <= 9 roundings, so the relative
    // error is below 9.01 2^-24 < 2^-20
    const double rel = std::ldexp(1.0, -20);
    cfg.xn_lo = (float)(1.0 - rel);
    cfg.xn_hi = (float)(1.0 + rel);
    return true;
}

template <int D>
cudaError_t launch_t(const Params &p, cudaStream_t s, int first, int respect_done, int num_sms, size_t smem_limit,
                     int if_dense) {
    TcCfg cfg;
    size_t smem;
    if (!plan(p, smem_limit, cfg, smem) || !p.Xh || !p.Xl || !p.xnorm) return cudaErrorNotSupported;
    auto enc = encoder();
    if (!enc) return cudaErrorNotSupported;
    CUtensorMap tmh, tml;
    const int Dt = tc_dim(p.D);
    cuuint64_t gx[2] = {(cuuint64_t)Dt, (cuuint64_t)p.N}, sx[1] = {(cuuint64_t)Dt * 2};
    cuuint32_t bx[2] = {64, (cuuint32_t)kTM}, es[2] = {1, 1};
    if (enc(&tmh, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t *>(p.Xh), gx, sx, bx, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    if (enc(&tml, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t *>(p.Xl), gx, sx, bx, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    // (one value for every context: it is the process's, and another thread's context may be launching)
    cudaError_t e = cudaFuncSetAttribute(k_dense_tc<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_limit);
    if (e != cudaSuccess) return e;
    const int grid = std::min(cfg.num_tiles, num_sms);
    count_launch();
    k_dense_tc<D><<<grid, kTcThreads, smem, s>>>(tmh, tml, p, cfg, first, respect_done, if_dense);
    return cudaGetLastError();
}

}  // namespace

bool dense_tc_eligible(const Params &p, size_t smem_limit) {
    TcCfg cfg;
    size_t smem;
    return encoder() != nullptr && plan(p, smem_limit, cfg, smem);
}

cudaError_t launch_split_x(const float *X, int64_t N, int D, int Dt, uint16_t *Xh, uint16_t *Xl, cudaStream_t s,
                           int num_sms, float *Xcopy, const float *mu, float *xnorm) {
    if (Dt != 64 && Dt != 128) return cudaErrorInvalidValue;  // a row's lanes: one half-warp or warp
    const int64_t n4 = N * Dt / 4;  // D and Dt are multiples of 4
    const int64_t grid = std::min<int64_t>((n4 + 255) / 256, (int64_t)num_sms * 16);
    count_launch();
    k_split_x<<<(unsigned)std::max<int64_t>(grid, 1), 256, 0, s>>>(X, N, D, Dt, reinterpret_cast<uint2 *>(Xh),
                                                                    reinterpret_cast<uint2 *>(Xl),
                                                                    reinterpret_cast<float4 *>(Xcopy), mu, xnorm);
    return cudaGetLastError();
}

cudaError_t launch_dense_tc(const Params &p, cudaStream_t s, int first, int respect_done, int num_sms,
                            size_t smem_limit, int if_dense) {
    if (p.K > 256) return launch_dense_tcb(p, s, first, respect_done, num_sms, smem_limit, if_dense);
    switch (tc_dim(p.D)) {
    case 64: return launch_t<64>(p, s, first, respect_done, num_sms, smem_limit, if_dense);
    case 128: return launch_t<128>(p, s, first, respect_done, num_sms, smem_limit, if_dense);
    default: return cudaErrorNotSupported;
    }
}

}  // namespace kp
