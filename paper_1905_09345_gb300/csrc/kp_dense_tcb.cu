// kp_dense_tcb.cu -- dense assignment on the tensor cores when the centroids
// do not fit one accumulator (K > 256).
//
// The same contraction as kp_dense_tc.cu (Sec. I: the distance calculator on
// the pairs the filters leave, here all of them): t_k = ||c_k||^2 - 2 x.c_k
// from BF16x3 tcgen05.mma, exact decisions through the settle queue.  The
// centroids stream through shared memory in blocks of 128 (both bfloat16
// halves, loaded by TMA from a split copy made at the start of each pass),
// and each row's scan -- group minima, winner, runner-up -- carries across
// the blocks.
//
// Persistent CTA per SM, 576 threads: warp 0 issues TMA, one thread of warp 1
// the MMAs, warps 2..17 read the accumulators.  Tiles of 128 points go in
// pairs; both tiles of a pair use each centroid block while it is in shared
// memory.  The scan bounds the kernel (about 12 instructions per row and
// column at half of the issue rate; the tensor pipe is active 25-40% of the
// time), so every tile has eight warps:
// two per TMEM lane quadrant, one for the blocks of the first half of the
// centroids, one for those of the second half (each warp's columns stay one
// ascending run, so its group minima close in order).  The blocks are issued
// alternately from the two halves, and each (tile, half) owns one of the four
// TMEM buffers of 128 columns, so three buffers are scanned or waiting while
// the fourth is multiplied.
// The bfloat16 halves of a block have shared-memory slots of their own and
// the products with the high half come first (x_h c_h, x_l c_h of both
// tiles, then x_h c_l), so that one half loads while the other is multiplied.
//
// Measured on GB300 (one pass): 4,194,304 x 128, K = 1024, G = 103: 5.2 ms with
// four scanning warps per tile and a column-by-column scan, 3.5 ms now;
// 1,048,576 x 32, K = 4096, G = 410: 4.9 -> 2.7 ms.  Blocks of 64 columns with
// two buffers per (tile, half) measured 5.9 and 4.2 ms, a sixteen-column
// tournament 5.5 and 3.7 (spills, and the code outgrows the instruction cache).
#include "kp_tc.cuh"

namespace kp {
namespace {

constexpr int kNB = 128;                       // centroids per block (MMA N)
constexpr int kBAtom = kNB * 128;              // one 64-element column block of a centroid block
constexpr int kQuadWarps = 4;                  // warps of a (tile, half): the TMEM lane quadrants
constexpr int kEpi = 4 * kQuadWarps;           // two tiles x two halves
constexpr int kThreads = 64 + kEpi * 32;
constexpr int kMaxKp = 4096;
constexpr int kSlots = 7;                      // staged group minima per row: 3 left over + those that
                                               // four columns can close, whatever the groups' sizes
constexpr int kCnSlots = 4;                    // blocks of norms per half

struct TcbCfg {
    int Kp;          // K padded to a multiple of kNB
    int nb, hb;      // centroid blocks; blocks of the first half
    int hs;          // slots of half a centroid block (even, 2 or 4)
    uint32_t off_B, off_cn, off_bm, off_stage, off_t4, off_mrg, off_bar;
    int num_tiles;
    float e_lin, e_c2, xn_lo, xn_hi;
};

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
    k_dense_tcb(const __grid_constant__ CUtensorMap tmh, const __grid_constant__ CUtensorMap tml,
                const __grid_constant__ CUtensorMap tmch, const __grid_constant__ CUtensorMap tmcl, Params p,
                TcbCfg cfg, int first, int respect_done, int if_dense) {
    extern __shared__ uint8_t raw[];
    Ctrl *ctrl = p.ctrl;
    count_kernel(ctrl);
    if (respect_done && *(volatile int *)&ctrl->done) return;
    if (if_dense && !*(volatile int *)&ctrl->dense_mode) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) ctrl->path = KM_PATH_DENSE_TC;
    constexpr int NA = D / 64;
    uint8_t *sm = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~(uintptr_t)1023);
    const int nb = cfg.nb, hb = cfg.hb, HS = cfg.hs;
    uint8_t *sA = sm;               // 2 tiles: [NA atoms x_h][NA atoms x_l]
    uint8_t *sB = sm + cfg.off_B;   // HS slots of NA atoms: c_h, c_l of successive blocks
    float *cnr = reinterpret_cast<float *>(sm + cfg.off_cn);  // [2 halves][kCnSlots][kNB] ||c||^2 (+inf: padding)
    uint32_t *bm = reinterpret_cast<uint32_t *>(sm + cfg.off_bm);  // [Kp / 32] group-start masks
    float4 *mrg = reinterpret_cast<float4 *>(sm + cfg.off_mrg);    // [2 tiles][128 rows] the second half's result
    uint64_t *bars = reinterpret_cast<uint64_t *>(sm + cfg.off_bar);
    uint64_t *full_a = bars;               // [2]
    uint64_t *empty_a = bars + 2;          // [2]
    uint64_t *acc_full = bars + 4;         // [2 tiles][2 halves]
    uint64_t *acc_empty = bars + 8;        // [2][2]
    uint64_t *mfull = bars + 12;           // [2 tiles][4 quadrants]
    uint64_t *mempty = bars + 20;          // [2][4]
    uint64_t *cn_full = bars + 28;         // [2 halves][kCnSlots]
    uint64_t *mma_done = bars + 36;
    uint64_t *full_b = bars + 37;          // [HS]
    uint64_t *empty_b = full_b + HS;       // [HS]
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(empty_b + HS);
    float *c2max_s = reinterpret_cast<float *>(tmem_slot + 1);

    // (the broadcast tells the compiler that the warp index is warp-uniform)
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int v = ctrl->v;
    const int K = p.K, G = p.G;
    // this CTA's tiles: blockIdx.x + i * gridDim.x; pairs (2pr, 2pr + 1)
    const int ntile = cfg.num_tiles > (int)blockIdx.x
                          ? (cfg.num_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x
                          : 0;
    const int npair = (ntile + 1) >> 1;

    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            bar_init(&full_a[i], 1);
            bar_init(&empty_a[i], 1);
        }
        for (int i = 0; i < 4; ++i) {
            bar_init(&acc_full[i], 1);
            bar_init(&acc_empty[i], kQuadWarps);
        }
        for (int i = 0; i < 8; ++i) {
            bar_init(&mfull[i], 1);
            bar_init(&mempty[i], 1);
            bar_init(&cn_full[i], 1);
        }
        for (int i = 0; i < HS; ++i) {
            bar_init(&full_b[i], 1);
            bar_init(&empty_b[i], 1);
        }
        bar_init(mma_done, 1);
        *c2max_s = 0.f;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // largest norm, group-start masks
    for (int c = threadIdx.x; c < cfg.Kp / 32; c += blockDim.x) bm[c] = 0u;
    {
        float cm = 0.f;
        for (int k = threadIdx.x; k < K; k += blockDim.x) cm = fmaxf(cm, p.cnorm[k]);
        cm = warp_max(cm);
        __syncthreads();  // c2max_s and the masks initialised
        if (lane == 0 && cm > 0.f) atomicMax(reinterpret_cast<int *>(c2max_s), __float_as_int(cm));
        for (int g = 1 + threadIdx.x; g < G; g += blockDim.x) {
            const int col = p.gstart[g];
            if ((unsigned)col < (unsigned)cfg.Kp) atomicOr(&bm[col >> 5], 1u << (col & 31));
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // step k of a tile pair takes block blk(k): alternately from the two halves
    // (the first half has the odd block)
    auto blk = [&](int k) { return (k & 1) ? hb + (k >> 1) : (k >> 1); };

    if (warp == 0) {
        // ------------------------------------------------------------ TMA
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmh) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tml) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmch) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmcl) : "memory");
            bool ok = true;
            int nl = 0;            // half blocks issued
            int ia[2] = {0, 0};    // tiles issued into each A stage
            int uh[2] = {0, 0};    // blocks of norms issued per half
            for (int pr = 0; pr < npair && ok; ++pr) {
                for (int g = 0; g < 2 && ok; ++g) {
                    const int i = 2 * pr + g;
                    if (i >= ntile) break;
                    if (pr > 0 && !(ok = bar_wait(&empty_a[g], (pr - 1) & 1, ctrl))) break;
                    ++ia[g];
                    const int tile = (int)blockIdx.x + i * (int)gridDim.x;
                    uint8_t *st = sA + (size_t)g * 2 * NA * kAtomBytes;
                    mbar_arrive_expect_tx(&full_a[g], (uint32_t)(2 * NA * kAtomBytes));
                    for (int a = 0; a < NA; ++a) {
                        tma_2d(st + a * kAtomBytes, &tmh, 64 * a, tile * kTM, &full_a[g]);
                        tma_2d(st + (NA + a) * kAtomBytes, &tml, 64 * a, tile * kTM, &full_a[g]);
                    }
                }
                for (int k = 0; k < nb && ok; ++k) {
                    const int j = blk(k), h = k & 1;
                    for (int part = 0; part < 2; ++part) {
                        const int bs = nl % HS, fb = nl / HS;
                        if (fb > 0 && !(ok = bar_wait(&empty_b[bs], (fb - 1) & 1, ctrl))) break;
                        ++nl;
                        uint8_t *sb = sB + (size_t)bs * NA * kBAtom;
                        mbar_arrive_expect_tx(&full_b[bs], (uint32_t)(NA * kBAtom));
                        for (int a = 0; a < NA; ++a)
                            tma_2d(sb + a * kBAtom, part ? &tmcl : &tmch, 64 * a, j * kNB, &full_b[bs]);
                        if (part == 0) {
                            // the block's norms.  Their slot was last read for this half's
                            // block four uses ago; the slot of c_h just waited for (at most
                            // two blocks back) was multiplied after the scan of this half's
                            // block three uses ago had released its accumulators, and a warp
                            // that releases one block has read the one before (a second
                            // tile without a successor: see `late` below).
                            uint64_t *cb = &cn_full[h * kCnSlots + (uh[h] & (kCnSlots - 1))];
                            mbar_arrive_expect_tx(cb, kNB * 4);
                            tma_bulk_g2s(cnr + (h * kCnSlots + (uh[h] & (kCnSlots - 1))) * kNB, p.cnorm + j * kNB,
                                         kNB * 4, cb);
                            ++uh[h];
                        }
                    }
                }
            }
            // drain: the last loads of each barrier have landed before the block exits
            for (int g = 0; g < 2; ++g)
                if (ia[g] > 0) bar_wait(&full_a[g], (ia[g] - 1) & 1, ctrl);
            for (int b = 0; b < HS; ++b) {
                const int uses = nl > b ? (nl - b + HS - 1) / HS : 0;
                if (uses > 0) bar_wait(&full_b[b], (uses - 1) & 1, ctrl);
            }
            for (int h = 0; h < 2; ++h)
                for (int b = 0; b < kCnSlots; ++b) {
                    const int uses = uh[h] > b ? (uh[h] - b + kCnSlots - 1) / kCnSlots : 0;
                    if (uses > 0) bar_wait(&cn_full[h * kCnSlots + b], (uses - 1) & 1, ctrl);
                }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA
        if (lane == 0) {
            // kind::f16: F32 accumulate, BF16 A and B, K-major, N = 128, M = 128
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kNB >> 3) << 17) |
                                   ((uint32_t)(kTM >> 4) << 24);
            bool ok = true;
            int nl = 0;
            // [d_tmem] (+)= A atom rows at sa . B atom rows at sb, over the D coordinates
            auto product = [&](uint32_t d_tmem, const uint8_t *sa, const uint8_t *sb, bool fresh) {
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks) {
                    if (D == 64 && 16 * ks >= p.D) break;  // 32 coordinates: the padding to 64 adds nothing
                    const int a = ks >> 2, jj = ks & 3;
                    const uint64_t da = desc_sw128(smem_u32(sa + a * kAtomBytes + jj * 32));
                    const uint64_t db = desc_sw128(smem_u32(sb + a * kBAtom + jj * 32));
                    const uint32_t acc = !(fresh && ks == 0);
                    asm volatile(
                        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
                        "l"(da), "l"(db), "r"(idesc), "r"(acc)
                        : "memory");
                }
            };
            auto commit = [&](uint64_t *b) {
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 smem_u32(b))
                             : "memory");
            };
            for (int pr = 0; pr < npair && ok; ++pr) {
                const int ng = 2 * pr + 1 < ntile ? 2 : 1;
                for (int g = 0; g < ng && ok; ++g) ok = bar_wait(&full_a[g], pr & 1, ctrl);
                if (!ok) break;
                tc_fence_after();
                for (int k = 0; k < nb && ok; ++k) {
                    const int h = k & 1;
                    const uint32_t uses = (uint32_t)(pr * (h ? nb - hb : hb) + (k >> 1));
                    for (int part = 0; part < 2 && ok; ++part, ++nl) {
                        const int bs = nl % HS, fb = nl / HS;
                        if (!(ok = bar_wait(&full_b[bs], fb & 1, ctrl))) break;
                        tc_fence_after();
                        const uint8_t *sb = sB + (size_t)bs * NA * kBAtom;
                        if (part == 0 && uses > 0) {
                            // the (tile, half) buffers are read; at a pair's start also a
                            // missing second tile's, whose last release follows its last
                            // read of the norms
                            for (int g = 0; g < (k < 2 ? 2 : ng) && ok; ++g)
                                ok = bar_wait(&acc_empty[g * 2 + h], (uses - 1) & 1, ctrl);
                            if (!ok) break;
                            tc_fence_after();
                        }
                        for (int g = 0; g < ng; ++g) {
                            const uint32_t d_tmem = tmem + (uint32_t)((g * 2 + h) * kNB);
                            const uint8_t *st = sA + (size_t)g * 2 * NA * kAtomBytes;
                            if (part == 0) {
                                product(d_tmem, st, sb, true);                      // x_h c_h
                                product(d_tmem, st + NA * kAtomBytes, sb, false);   // x_l c_h
                            } else {
                                product(d_tmem, st, sb, false);                     // x_h c_l
                                commit(&acc_full[g * 2 + h]);
                            }
                        }
                        commit(&empty_b[bs]);  // the slot is free once these MMAs have read it
                    }
                }
                if (!ok) break;
                for (int g = 0; g < ng; ++g) commit(&empty_a[g]);
            }
            // every MMA of this thread is complete before TMEM is freed
            commit(mma_done);
            bar_wait(mma_done, 0, ctrl);
        }
    } else {
        // ------------------------------------------------------- epilogue
        const int e = warp - 2;
        const int h = e >> 3;          // half of the centroids
        const int g = (e >> 2) & 1;    // tile of the pair
        const int q = warp & 3;        // TMEM lane quadrant of this warp
        const int r = q * 32 + lane;
        const int pair = g * 4 + q;    // the two warps of a quadrant meet at mfull / mempty
        const float c2max = __fmul_ru(*c2max_s, 1.0f + 1.0f / 1024);
        const float cmax = sqrt_hi(c2max);
        const float ec2 = __fmul_ru(cfg.e_c2, c2max);
        // the filtered method keeps every bound; plain Lloyd keeps only the
        // group bounds, for the exact settle's candidate groups
        const bool bounds = p.algo == KM_ALGO_FILTERED;
        const bool has_lb = p.lb != nullptr;
        const int j0 = h ? hb : 0, nblk = h ? nb - hb : hb;
        // the group open across the two halves' border: both halves hold a part
        // of it, and the second half starts in its slot
        const int gsplit = __shfl_sync(0xffffffffu, p.grp[kNB * hb - 1], 0);
        Scan4 sc;
        sc.row = smem_u32(sm + cfg.off_stage) + (uint32_t)((e * 32 + lane) * kSlots) * 4u;
        sc.t4 = smem_u32(sm + cfg.off_t4) + (uint32_t)(e * 32 + lane) * 16u;
        const float4 *cnh = reinterpret_cast<const float4 *>(cnr + h * kCnSlots * kNB);
        unsigned long long c_changed = 0, c_dist = 0;
        for (int pr = 0; pr < npair; ++pr) {
            const int i = 2 * pr + g;
            if (i >= ntile) break;
            const int tile = (int)blockIdx.x + i * (int)gridDim.x;
            const int64_t n = (int64_t)tile * kTM + r;
            const bool valid = n < p.N;
            const float xn = valid ? p.xnorm[n] : 0.f;
            const float xlo = __fmul_rd(xn, cfg.xn_lo), xup = __fmul_ru(xn, cfg.xn_hi);
            const float R = __fadd_ru(sqrt_hi(xup), cmax);  // bounds ||x - mu|| + ||c - mu||
            const float E = __fmaf_ru(p.e_cen, __fmul_ru(R, R), __fmaf_ru(cfg.e_lin, __fmul_ru(sqrt_hi(xup), cmax), ec2));
            float *lbrow = p.lb + n * p.Gp;
            const bool store = has_lb && valid;
            auto bound_of = [&](float t) { return t == INFINITY ? INFINITY : sqrt_lo(__fsub_rd(__fadd_rd(xlo, t), E)); };

            sc.b1 = sc.b2 = sc.gm = INFINITY;
            sc.c4 = kNB * j0;
            sc.pend = h ? (gsplit & 3) : 0;
            int gq = h ? (gsplit & ~3) : 0;  // group of slot 0 (a multiple of four)
            float gsp = INFINITY;            // second half: its part of group gsplit
            bool head = h != 0;              // its slots still start with that group's four
            // slots [0, cnt) of the four that group gsplit lies in (second half)
            auto head_slots = [&](int cnt) {
                const int s0 = gsplit & 3;
                gsp = lds_f(sc.row + 4u * (uint32_t)s0);
                for (int s = s0 + 1; s < cnt; ++s) {
                    const float b = bound_of(lds_f(sc.row + 4u * (uint32_t)s));
                    if (store) lbrow[gq + s] = b;
                }
                head = false;
            };
            bool ok = true;
            for (int b = 0; b < nblk; ++b) {
                const uint32_t u = (uint32_t)(pr * nblk + b);
                ok = __all_sync(0xffffffffu, bar_wait(&acc_full[g * 2 + h], u & 1, ctrl) &&
                                                 bar_wait(&cn_full[h * kCnSlots + (u & (kCnSlots - 1))],
                                                          (u / kCnSlots) & 1, ctrl));
                if (!ok) break;
                tc_fence_after();
                const uint32_t tb = tmem + (uint32_t)((g * 2 + h) * kNB) + ((uint32_t)(q * 32) << 16);
                const float4 *cn4 = cnh + (u & (kCnSlots - 1)) * (kNB / 4);
                const int cb = kNB * (j0 + b);
                // four columns, then -- when four groups have closed -- their bounds to lb
                auto sixteen = [&](const uint32_t(&acc)[16], int c0) {
                    // (a broadcast, so that the compiler knows the mask to be warp-uniform)
                    const uint32_t m16 = __shfl_sync(0xffffffffu, bm[(cb + c0) >> 5], 0) >> ((cb + c0) & 31);
#pragma unroll
                    for (int j = 0; j < 16; j += 4) {
                        const uint32_t nib = (m16 >> j) & 15u;
                        sc.four(&acc[j], cn4[(c0 + j) >> 2], nib, cb + c0 + j);
                        if (nib && sc.pend >= 4) {  // warp-uniform
                            if (head) {
                                head_slots(4);
                            } else {  // whole groups, never empty: a finite minimum
                                float4 o;
                                o.x = sqrt_lo(__fsub_rd(__fadd_rd(xlo, lds_f(sc.row)), E));
                                o.y = sqrt_lo(__fsub_rd(__fadd_rd(xlo, lds_f(sc.row + 4)), E));
                                o.z = sqrt_lo(__fsub_rd(__fadd_rd(xlo, lds_f(sc.row + 8)), E));
                                o.w = sqrt_lo(__fsub_rd(__fadd_rd(xlo, lds_f(sc.row + 12)), E));
                                if (store) *reinterpret_cast<float4 *>(lbrow + gq) = o;
                            }
                            gq += 4;
                            sc.pend -= 4;
                            for (int s = 0; s < sc.pend; ++s) {
                                const float t = lds_f(sc.row + 16u + 4u * (uint32_t)s);
                                asm volatile("st.shared.f32 [%0], %1;" ::"r"(sc.row + 4u * (uint32_t)s), "f"(t));
                            }
                        }
                    }
                };
                // A second tile's warps are not waited for again when the CTA's last pair
                // lacks it: their last release before that pair says that the block's
                // norms are read too, so that their slot may be filled again.
                const bool late = g == 1 && b == nblk - 1 && i + 2 >= ntile;
                auto release = [&]() {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) bar_arrive(&acc_empty[g * 2 + h]);
                };
                uint32_t ra[16], rb[16];
                tmem_ld16_async(tb, ra);
#pragma unroll 1
                for (int c0 = 0; c0 < kNB; c0 += 32) {
                    tmem_wait16(ra);
                    tmem_ld16_async(tb + c0 + 16, rb);
                    sixteen(ra, c0);
                    tmem_wait16(rb);
                    if (c0 + 32 < kNB) {
                        tmem_ld16_async(tb + c0 + 32, ra);
                    } else if (!late) {  // the accumulators are read: release them
                        release();
                    }
                    sixteen(rb, c0 + 16);
                }
                if (late) release();
            }
            if (!ok) break;  // a wait timed out (error recorded)
            // the open group's minimum
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(sc.row + 4u * (uint32_t)sc.pend), "f"(sc.gm) : "memory");
            ++sc.pend;
            if (h) {
                if (head) {
                    head_slots(sc.pend);
                } else {
                    for (int s = 0; s < sc.pend; ++s) {
                        const float b = bound_of(lds_f(sc.row + 4u * (uint32_t)s));
                        if (store) lbrow[gq + s] = b;
                    }
                }
                const int ci = sc.winner();
                if (pr > 0 && !__all_sync(0xffffffffu, bar_wait(&mempty[pair], (pr - 1) & 1, ctrl))) break;
                mrg[g * kTM + r] = make_float4(sc.b1, sc.b2, __int_as_float(ci), gsp);
                __syncwarp();
                if (lane == 0) bar_arrive(&mfull[pair]);  // with the bounds stored above
                continue;
            }
            const int old = valid ? (first ? -1 : p.label[n]) : -1;
            const int ai = sc.winner();
            if (!__all_sync(0xffffffffu, bar_wait(&mfull[pair], pr & 1, ctrl))) break;
            const float4 mg = mrg[g * kTM + r];
            __syncwarp();
            if (lane == 0) bar_arrive(&mempty[pair]);
            for (int s = 0; s < sc.pend; ++s) {  // the last of them is gsplit
                float t = lds_f(sc.row + 4u * (uint32_t)s);
                if (s == sc.pend - 1) t = fminf(t, mg.w);
                const float b = bound_of(t);
                if (store) lbrow[gq + s] = b;
            }
            // the first half holds the lower indices: it wins ties
            const bool bw = mg.x < sc.b1;
            const float b1 = bw ? mg.x : sc.b1;
            const int i1 = bw ? __float_as_int(mg.z) : ai;
            const float b2 = fminf(fminf(sc.b2, mg.y), fmaxf(sc.b1, mg.x));
            const float thr = __fadd_ru(b1, __fmul_ru(2.f, E));
            const bool need = valid && b2 <= thr;
            const unsigned nm = __ballot_sync(0xffffffffu, need);
            if (need) {
                // candidates of the exact settle: the groups whose bound does not
                // exceed the bound of the window's edge (lb is written by now)
                SettleReq rq;
                rq.n = (int32_t)n;
                rq.old = old;
                rq.i1 = i1;
                rq.lb_alt = sqrt_lo(__fsub_rd(__fadd_rd(xlo, b1), E));
                rq.gmask[0] = 0ull;
                rq.gmask[1] = __float_as_uint(sqrt_hi(__fsub_ru(__fadd_ru(xup, thr), E)));
                p.sreq[n] = rq;
            }
            if (lane == 0) p.sbits[(int64_t)tile * (kTM / 32) + q] = nm;
            const int best = i1;
            if (valid) {
                c_dist += (unsigned long long)K;
                if (!need) p.label[n] = best;
                // the winner's group excludes the winner: every other column is
                // at least the runner-up; the smallest group bound is that bound
                const float lw = bound_of(b2);
                if (has_lb) lbrow[p.grp[best]] = lw;
                if (bounds) {
                    p.lbg[n] = lw;
                    p.u[n] = sqrt_hi(__fadd_ru(__fadd_ru(xup, b1), E));
                    p.stamp[n] = make_stamp(v, v);
                }
            }
            {
                const bool moved = valid && !need && old != best;
                const unsigned mm = __ballot_sync(0xffffffffu, moved);
                c_changed += moved ? 1 : 0;
                if (mm && !first) {
                    int base = 0;
                    if (lane == 0) base = atomicAdd(&ctrl->moved_count, __popc(mm));
                    base = __shfl_sync(0xffffffffu, base, 0);
                    if (moved) {
                        const int slot = base + __popc(mm & ((1u << lane) - 1u));
                        p.moved[slot] = (int)n;
                        p.moved_old[slot] = old;
                    }
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            c_changed += __shfl_xor_sync(0xffffffffu, c_changed, o);
            c_dist += __shfl_xor_sync(0xffffffffu, c_dist, o);
        }
        if (lane == 0) {
            if (c_changed) atomicAdd(&ctrl->n_changed, c_changed);
            if (c_dist) atomicAdd(&ctrl->n_dist, c_dist);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// C -> (c_h, c_l) bfloat16 copies (K padded to Kp with zero rows) and the
// FP32 norms (padding: +inf), as the kernel above reads them; gated like the
// dense pass.  A warp per centroid.
__global__ void k_split_c(Params p, int Kp, int respect_done, int if_dense) {
    Ctrl *ctrl = p.ctrl;
    count_kernel(ctrl);
    if (respect_done && *(volatile int *)&ctrl->done) return;
    if (if_dense && !*(volatile int *)&ctrl->dense_mode) return;
    const int D = p.D, Dt = tc_dim(p.D);
    const int lane = threadIdx.x & 31;
    const int wid = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int nw = (int)((gridDim.x * blockDim.x) >> 5);
    for (int k = wid; k < Kp; k += nw) {
        float s2 = 0.f;
        for (int d = lane; d < Dt; d += 32) {
            float x = (k < p.K && d < D) ? p.C[(size_t)k * p.Dp + d] : 0.f;  // zero padding
            if (p.mu && k < p.K && d < D) x = __fsub_rn(x, p.mu[d]);  // c - mu
            const __nv_bfloat16 h = __float2bfloat16_rn(x);
            const __nv_bfloat16 l = __float2bfloat16_rn(x - __bfloat162float(h));
            p.Ch[(size_t)k * Dt + d] = __bfloat16_as_ushort(h);
            p.Cl[(size_t)k * Dt + d] = __bfloat16_as_ushort(l);
            s2 = fmaf(x, x, s2);  // ||c - mu||^2 of the values split
        }
        s2 = warp_sum(s2);
        if (lane == 0) p.cnorm[k] = k < p.K ? s2 : INFINITY;
    }
}

bool plan_b(const Params &p, size_t smem_limit, TcbCfg &cfg, size_t &smem) {
    const int Dt = tc_dim(p.D);
    if (!Dt || p.K <= 256) return false;
    cfg.Kp = ((p.K + kNB - 1) / kNB) * kNB;
    if (cfg.Kp > kMaxKp) return false;
    cfg.nb = cfg.Kp / kNB;
    cfg.hb = (cfg.nb + 1) / 2;
    // The shapes that this engine takes are those of an earlier layout, which kept
    // every norm and the minima of 64 columns' groups (under the contiguous grouping
    // j -> j G / K, whatever the context's) in shared memory.  The present layout
    // needs less, and at most 229,208 bytes: 128 coordinates with K = 4096, with K =
    // 1024 and more than 368 groups, or with K = 257 and more than 106 would fit too
    // and still go to the FP32 engine.
    int most = 0;
    for (int j = 0; j < cfg.Kp / 64; ++j) {
        const int64_t c0 = (int64_t)j * 64, c1 = std::min<int64_t>((int64_t)(j + 1) * 64, p.K) - 1;
        if (c0 >= p.K) break;
        const int g0 = (int)(c0 * p.G / p.K), g1 = (int)(c1 * p.G / p.K);
        most = std::max(most, g1 - g0 + 1);
    }
    const int srow = (most + 2) | 1;
    const size_t NA = Dt / 64;
    const size_t a_bytes = 2 * 2 * NA * (size_t)kAtomBytes;
    const size_t half = NA * (size_t)kBAtom;
    if (1024 + a_bytes + 2 * half + (size_t)cfg.Kp * 8 + (size_t)cfg.Kp / 32 * 4 + 256 * (size_t)srow * 4 + 184 >
        smem_limit)
        return false;
    size_t off = a_bytes;
    cfg.off_B = (uint32_t)off;
    cfg.hs = 4;
    const size_t fixed = 2 * kCnSlots * kNB * 4 + ((size_t)cfg.Kp / 32 * 4 + 15) / 16 * 16 +
                         (size_t)kEpi * 32 * (kSlots * 4 + 16) + 2 * kTM * 16 + (37 + 2 * 4) * 8 + 16;
    if (1024 + off + 4 * half + fixed > smem_limit) cfg.hs = 2;
    off += cfg.hs * half;
    cfg.off_cn = (uint32_t)off;
    off += 2 * kCnSlots * kNB * 4;
    cfg.off_bm = (uint32_t)off;
    off += ((size_t)cfg.Kp / 32 * 4 + 15) / 16 * 16;
    cfg.off_t4 = (uint32_t)off;
    off += (size_t)kEpi * 32 * 16;
    cfg.off_mrg = (uint32_t)off;
    off += 2 * kTM * 16;
    cfg.off_stage = (uint32_t)off;
    off += (size_t)kEpi * 32 * kSlots * 4;
    cfg.off_bar = (uint32_t)off;  // a multiple of 8: every part above is a multiple of 16
    off += (37 + 2 * cfg.hs) * 8 + 16;
    smem = 1024 + off;
    if (smem > smem_limit) return false;
    cfg.num_tiles = (int)((p.N + kTM - 1) / kTM);
    const double D = Dt;  // the padded width (zero products add nothing)
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
cudaError_t launch_b(const Params &p, cudaStream_t s, int first, int respect_done, int num_sms, size_t smem_limit,
                     int if_dense) {
    TcbCfg cfg;
    size_t smem;
    if (!plan_b(p, smem_limit, cfg, smem) || !p.Xh || !p.Xl || !p.xnorm || !p.Ch || !p.Cl || !p.cnorm)
        return cudaErrorNotSupported;
    auto enc = encoder();
    if (!enc) return cudaErrorNotSupported;
    CUtensorMap tmh, tml, tmch, tmcl;
    const int Dt = tc_dim(p.D);
    cuuint64_t gx[2] = {(cuuint64_t)Dt, (cuuint64_t)p.N}, sx[1] = {(cuuint64_t)Dt * 2};
    cuuint64_t gc[2] = {(cuuint64_t)Dt, (cuuint64_t)cfg.Kp};
    cuuint32_t bx[2] = {64, (cuuint32_t)kTM}, bc[2] = {64, (cuuint32_t)kNB}, es[2] = {1, 1};
    struct M {
        CUtensorMap *m;
        const uint16_t *src;
        cuuint64_t *g;
        cuuint32_t *b;
    } maps[4] = {{&tmh, p.Xh, gx, bx}, {&tml, p.Xl, gx, bx}, {&tmch, p.Ch, gc, bc}, {&tmcl, p.Cl, gc, bc}};
    for (auto &m : maps)
        if (enc(m.m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t *>(m.src), m.g, sx, m.b, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    {
        const int64_t grid = std::max<int64_t>(1, std::min<int64_t>((cfg.Kp + 7) / 8, (int64_t)num_sms * 4));
        count_launch();
        k_split_c<<<(unsigned)grid, 256, 0, s>>>(p, cfg.Kp, respect_done, if_dense);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    // (one value for every context: it is the process's, and another thread's context may be launching)
    cudaError_t e = cudaFuncSetAttribute(k_dense_tcb<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_limit);
    if (e != cudaSuccess) return e;
    const int grid = std::min(cfg.num_tiles, num_sms);
    count_launch();
    k_dense_tcb<D><<<grid, kThreads, smem, s>>>(tmh, tml, tmch, tmcl, p, cfg, first, respect_done, if_dense);
    return cudaGetLastError();
}

}  // namespace

bool dense_tcb_eligible(const Params &p, size_t smem_limit) {
    TcbCfg cfg;
    size_t smem;
    return encoder() != nullptr && plan_b(p, smem_limit, cfg, smem);
}

int dense_tcb_kp(const Params &p) { return ((p.K + kNB - 1) / kNB) * kNB; }

cudaError_t launch_dense_tcb(const Params &p, cudaStream_t s, int first, int respect_done, int num_sms,
                             size_t smem_limit, int if_dense) {
    switch (tc_dim(p.D)) {
    case 64: return launch_b<64>(p, s, first, respect_done, num_sms, smem_limit, if_dense);
    case 128: return launch_b<128>(p, s, first, respect_done, num_sms, smem_limit, if_dense);
    default: return cudaErrorNotSupported;
    }
}

}  // namespace kp
