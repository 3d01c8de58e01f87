// kp_mlp.cu -- the learned group proposal's network on the 5th-generation
// tensor cores: inference, and training (forward, backward, Adam).
//
// The paper's filters (Sec. I) start from bounds that iteration 0 makes; the
// proposal is the library's layered form that predicts each point's centroid
// group so that those bounds can be seeded without a dense pass.  The network
// is a multilayer perceptron  D -> H -> H -> G  with GELU activations (the
// exact erf form), trained with softmax cross-entropy (mean over the batch)
// and Adam, FP32 master weights and bfloat16 compute weights.
//
// Inference is one kernel for the three layers, k_mlp_infer (below).  In
// training every matrix product is one kernel, k_mlp_gemm:
//     C[M x N] = A[M x K] . B[N x K]^T
// with both operands bfloat16 and K-major in global memory, staged into shared
// memory by TMA (128-byte swizzle, one 64-element K slice per stage, a ring of
// stages), multiplied by tcgen05.mma (kind::f16, M = 128 rows per CTA, up to
// two N chunks of <= 256 columns) into FP32 accumulators in TMEM, and read back
// by sixteen epilogue warps (four per TMEM lane quadrant, each a quarter of the
// columns, one row per thread) that apply the layer's fused epilogue:
//     GELU     bias + GELU -> bfloat16 activations (row-major and/or
//              transposed) and the FP32 derivative GELU'(z) for the backward
//              pass;
//     SOFTMAX  bias + softmax cross-entropy: the loss, and the logit gradient
//              (p - onehot(y)) / B as bfloat16 (row-major and transposed), with
//              its per-warp column sums (the bias gradient);
//     MUL      the backpropagated gradient times GELU'(z) (row-major and/or
//              transposed bfloat16, per-warp column sums);
//     F32      the FP32 tile itself (split-K partial products of a weight
//              gradient, summed by the update kernel).
// The weight-gradient products contract over the batch, so the forward and
// backward epilogues also write the transposed copies those products read
// K-major; every operand stays in the layout the tensor cores take directly.
// A step's products are small (B = 8192 gives 64 to 128 CTAs of a few K
// slices), so latency bounds them: sixteen epilogue warps share a tile, the
// three weight gradients are one launch, the launches (tensor maps included)
// are planned once per batch size and each may start its set-up while the one
// ahead ends.  Measured on GB300, B = 8192, 32 -> 256 -> 256 -> 410: a
// gradient 249 us with four epilogue warps and eight separate launches, 119
// now; a training step 201 -> 107 us.
//
// Shapes are padded once: D to Dk (a multiple of 64, the K slice), the hidden
// width H to Hp (a multiple of 64) with zero weights and biases (a padded unit
// computes GELU(0) = 0 and has zero outgoing weights, so it changes nothing
// and its gradients stay zero), G to Gk (a multiple of 64) for the products
// that contract over the classes.
#include <cmath>
#include <cstdarg>
#include <cstddef>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "kp_tc.cuh"

namespace kp {
namespace {

constexpr int kMM = 128;       // rows per tile (TMEM lanes)
constexpr int kMK = 64;        // K per stage: one 128-byte row of bfloat16
constexpr int kMParts = 4;     // epilogue warps per TMEM lane quadrant
constexpr int kMThreads = 64 + kMParts * 128; // warp 0 TMA, warp 1 MMA (and TMEM allocation), warps 2..17 epilogue
constexpr uint32_t kMPolls = 1u << 22;

enum Epi : int { E_GELU = 0, E_SOFTMAX = 1, E_MUL = 3, E_F32 = 4 };

struct GemmCfg {
    int M, N;          // valid output rows / columns
    int mt, nt;        // CTAs along M and N (the rest of a product's CTAs split K)
    int k_steps;       // K slices of 64 per CTA (split-K: the CTA's split selects the slice range)
    int nch, bn;       // N chunks per CTA and columns per chunk (multiple of 16, <= 256)
    int mode;          // Epi
    const float *bias; // N (GELU, SOFTMAX)
    uint16_t *out;     // row-major bfloat16 M x ldo (nullable)
    int ldo;
    uint16_t *outT;    // transposed bfloat16 N x ldt (nullable)
    int ldt;
    float *aux;        // FP32 M x lda: GELU'(z) (written by GELU, read by MUL; nullable in GELU)
    int lda;
    float *part;       // F32: split z at part + z * part_split, row stride ldp
    int ldp;
    int64_t part_split;
    float *colsum;     // per-warp column sums: [M / 32] x ldc (nullable)
    int ldc;
    const int32_t *y;  // SOFTMAX: class of each row
    float scale;       // SOFTMAX: 1 / batch
    double *loss;      // SOFTMAX: [0] += cross-entropy, [1] += correct predictions, [2] += rows
    int *err;          // KM_ETIMEOUT when a bounded wait gave up
};

__device__ __forceinline__ bool mwait(uint64_t *b, uint32_t parity, int *err) {
    for (uint32_t i = 0; i < kMPolls; ++i)
        if (mbar_try_wait(b, parity)) return true;
    atomicExch(err, (int)KM_ETIMEOUT);
    return false;
}

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
// d/dz [z Phi(z)] = Phi(z) + z phi(z)
__device__ __forceinline__ float gelu_d(float z) {
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.3989422804014327f * expf(-0.5f * z * z);
}
__device__ __forceinline__ uint16_t bf16_bits(float v) { return __bfloat16_as_ushort(__float2bfloat16_rn(v)); }

// 16 bfloat16 values to 32 contiguous bytes (16-byte aligned)
__device__ __forceinline__ void store_bf16x16(uint16_t *dst, const float (&v)[16]) {
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = (uint32_t)bf16_bits(v[2 * i]) | ((uint32_t)bf16_bits(v[2 * i + 1]) << 16);
    uint4 *d = reinterpret_cast<uint4 *>(dst);
    d[0] = make_uint4(w[0], w[1], w[2], w[3]);
    d[1] = make_uint4(w[4], w[5], w[6], w[7]);
}

// sum over the 32 lanes (rows) of a warp
__device__ __forceinline__ float lane_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sums over the lanes of sixteen columns, each by lane_sum's tree, in 16
// shuffles instead of 80: at every step a lane passes on the half of its
// columns that the partner keeps.  Even lanes return their column's sum (*col).
__device__ __forceinline__ float lane_sums16(const float (&v)[16], int lane, int &col) {
    float a[8];
    const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4, h2 = lane & 2;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const float got = __shfl_xor_sync(0xffffffffu, h16 ? v[k] : v[k + 8], 16);
        a[k] = (h16 ? v[k + 8] : v[k]) + got;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float got = __shfl_xor_sync(0xffffffffu, h8 ? a[k] : a[k + 4], 8);
        a[k] = (h8 ? a[k + 4] : a[k]) + got;
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float got = __shfl_xor_sync(0xffffffffu, h4 ? a[k] : a[k + 2], 4);
        a[k] = (h4 ? a[k + 2] : a[k]) + got;
    }
    const float got = __shfl_xor_sync(0xffffffffu, h2 ? a[0] : a[1], 2);
    a[0] = (h2 ? a[1] : a[0]) + got;
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
    col = (h16 ? 8 : 0) + (h8 ? 4 : 0) + (h4 ? 2 : 0) + (h2 ? 1 : 0);
    return a[0];
}

// Up to three products in one launch: CTAs [first[p], first[p + 1]) are product p's.
struct GemmBatch {
    CUtensorMap ta[3], tb[3];
    GemmCfg g[3];
    int first[4];
    int stages;         // of the largest product
    uint32_t st_bytes;  // stage size of the largest
    int tmem_cols;
};

// The epilogue warps' named barrier (1): every thread contributes v, gets the AND.
__device__ __forceinline__ bool epi_all(bool v) {
    int out;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbar.red.and.pred q, 1, %2, p;\n\t"
        "selp.s32 %0, 1, 0, q;\n\t}"
        : "=r"(out)
        : "r"((int)v), "n"(kMParts * 128)
        : "memory");
    return out != 0;
}

// Programmatic dependent launch: the next kernel of the chain may start its
// set-up on idle SMs once a thread of every CTA has said so (trigger); it
// touches nothing that earlier kernels write or read before they have finished
// (wait).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__global__ void __launch_bounds__(kMThreads, 1) k_mlp_gemm(const __grid_constant__ GemmBatch gb) {
    extern __shared__ uint8_t raw[];
    uint8_t *sm = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~(uintptr_t)1023);
    const int pb = (int)blockIdx.x >= gb.first[2] ? 2 : ((int)blockIdx.x >= gb.first[1] ? 1 : 0);
    const GemmCfg &g = gb.g[pb];
    const int S = gb.stages;
    constexpr uint32_t a_bytes = kMM * 128;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sm + (size_t)S * gb.st_bytes);
    uint64_t *full = bars, *empty = bars + S, *accb = bars + 2 * S;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 2 * S + 1);
    float4 *red = reinterpret_cast<float4 *>(bars + 2 * S + 2);  // [kMParts][128] (softmax)
    float *sbias = reinterpret_cast<float *>(red + kMParts * kMM);  // [512]
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int cta = (int)blockIdx.x - gb.first[pb];
    const int bx = cta % g.mt, by = cta / g.mt % g.nt, bz = cta / (g.mt * g.nt);
    const int m0 = bx * kMM;
    const int nb = by * g.nch * g.bn;  // first output column of this CTA
    const int ks0 = bz * g.k_steps;

    if (threadIdx.x == 0) {
        for (int i = 0; i < S; ++i) {
            bar_init(&full[i], 1);
            bar_init(&empty[i], 1);
        }
        bar_init(accb, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(gb.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        // Only now may the next product's CTAs come: they take TMEM columns and hold
        // them until this kernel has ended, which it could not if it still needed them.
        pdl_trigger();
    }
    pdl_wait();
    if (g.bias)  // this CTA's columns, zero past the output
        for (int i = threadIdx.x; i < g.nch * g.bn; i += kMThreads) sbias[i] = nb + i < g.N ? g.bias[nb + i] : 0.f;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA
        if (lane == 0) {
            const CUtensorMap *ta = &gb.ta[pb], *tb = &gb.tb[pb];
            asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)ta) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)tb) : "memory");
            const uint32_t bytes = a_bytes + (uint32_t)(g.nch * g.bn) * 128u;
            int i = 0;
            for (; i < g.k_steps; ++i) {
                const int s = i % S, f = i / S;
                if (f > 0 && !mwait(&empty[s], (f - 1) & 1, g.err)) break;
                uint8_t *st = sm + (size_t)s * gb.st_bytes;
                mbar_arrive_expect_tx(&full[s], bytes);
                const int kc = (ks0 + i) * kMK;
                tma_2d(st, ta, kc, m0, &full[s]);
                for (int c = 0; c < g.nch; ++c) tma_2d(st + a_bytes + c * g.bn * 128, tb, kc, nb + c * g.bn, &full[s]);
            }
            // every issued copy has landed before the block can exit
            for (int j = i - S < 0 ? 0 : i - S; j < i; ++j) mwait(&full[j % S], (j / S) & 1, g.err);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA
        if (lane == 0) {
            // kind::f16: F32 accumulate, BF16 A and B, both K-major, N = bn, M = 128
            const uint32_t idesc =
                (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(g.bn >> 3) << 17) | ((uint32_t)(kMM >> 4) << 24);
            for (int i = 0; i < g.k_steps; ++i) {
                const int s = i % S;
                if (!mwait(&full[s], (i / S) & 1, g.err)) break;
                tc_fence_after();
                const uint8_t *st = sm + (size_t)s * gb.st_bytes;
#pragma unroll
                for (int j = 0; j < 4; ++j) {  // four K = 16 steps inside the 128-byte row
                    const uint64_t da = desc_sw128(smem_u32(st + j * 32));
                    for (int c = 0; c < g.nch; ++c) {
                        const uint64_t db = desc_sw128(smem_u32(st + a_bytes + c * g.bn * 128 + j * 32));
                        const uint32_t acc = (i > 0 || j > 0) ? 1u : 0u;
                        asm volatile(
                            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(
                                tmem + (uint32_t)(c * g.bn)),
                            "l"(da), "l"(db), "r"(idesc), "r"(acc)
                            : "memory");
                    }
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 smem_u32(&empty[s]))
                             : "memory");
            }
            // the accumulators are complete (and no MMA of this thread is in
            // flight) once accb completes
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(accb))
                         : "memory");
            mwait(accb, 0, g.err);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------- epilogue
        const int part = (warp - 2) >> 2;  // quarter of the columns
        const int q = warp & 3;            // TMEM lane quadrant of this warp
        const int r = q * 32 + lane;
        const int row = m0 + r;
        const bool valid = row < g.M;
        const bool ok = epi_all(mwait(accb, 0, g.err));
        tc_fence_after();
        const uint32_t tb_ = tmem + ((uint32_t)(q * 32) << 16);
        const int units = g.nch * g.bn >> 4;  // of 16 columns
        const int u0 = part * units / kMParts, u1 = (part + 1) * units / kMParts;
        const int rw = (m0 + q * 32) >> 5;  // row warp (for the per-warp column sums)
        if (ok && g.mode != E_SOFTMAX) {
            for (int u = u0; u < u1; ++u) {
                const int c0 = u * 16, n0 = nb + c0;
                if (n0 >= g.N) break;  // warp-uniform; N is a multiple of 16
                uint32_t v[16];
                tmem_ld16_async(tb_ + c0, v);
                tmem_wait16(v);
                float a[16];
                if (g.mode == E_GELU) {
                    float d[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float z = __uint_as_float(v[j]) + sbias[c0 + j];
                        a[j] = gelu(z);
                        d[j] = gelu_d(z);
                    }
                    if (valid) {
                        store_bf16x16(g.out + (size_t)row * g.ldo + n0, a);
                        float4 *ap = reinterpret_cast<float4 *>(g.aux + (size_t)row * g.lda + n0);
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            ap[j] = make_float4(d[4 * j], d[4 * j + 1], d[4 * j + 2], d[4 * j + 3]);
                    }
                } else if (g.mode == E_MUL) {
                    if (valid) {
                        const float4 *ap = reinterpret_cast<const float4 *>(g.aux + (size_t)row * g.lda + n0);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float4 dd = ap[j];
                            a[4 * j] = __uint_as_float(v[4 * j]) * dd.x;
                            a[4 * j + 1] = __uint_as_float(v[4 * j + 1]) * dd.y;
                            a[4 * j + 2] = __uint_as_float(v[4 * j + 2]) * dd.z;
                            a[4 * j + 3] = __uint_as_float(v[4 * j + 3]) * dd.w;
                        }
                        if (g.out) store_bf16x16(g.out + (size_t)row * g.ldo + n0, a);
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; ++j) a[j] = 0.f;
                    }
                    int col;
                    const float cs = lane_sums16(a, lane, col);
                    if (!(lane & 1)) g.colsum[(size_t)rw * g.ldc + n0 + col] = cs;
                } else {  // E_F32
                    if (valid) {
                        float4 *pp = reinterpret_cast<float4 *>(g.part + (size_t)bz * g.part_split +
                                                                (size_t)row * g.ldp + n0);
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            pp[j] = make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                                                __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3]));
                    }
                    continue;
                }
                if (g.outT && valid) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) g.outT[(size_t)(n0 + j) * g.ldt + row] = bf16_bits(a[j]);
                }
            }
        } else if (ok) {  // E_SOFTMAX (one N tile: nb == 0); a row's four warps meet in shared memory
            float mx = -INFINITY;
            int bi = 0;
            for (int u = u0; u < u1; ++u) {
                uint32_t v[16];
                tmem_ld16_async(tb_ + u * 16, v);
                tmem_wait16(v);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const int n = u * 16 + j;
                    if (n < g.N) {
                        const float l = __uint_as_float(v[j]) + sbias[n];
                        if (l > mx) {
                            mx = l;
                            bi = n;
                        }
                    }
                }
            }
            red[part * kMM + r] = make_float4(mx, __int_as_float(bi), 0.f, 0.f);
            epi_all(true);
            mx = -INFINITY;
            bi = 0;
#pragma unroll
            for (int k = 0; k < kMParts; ++k) {  // ascending columns: the first largest
                const float4 o = red[k * kMM + r];
                if (o.x > mx) {
                    mx = o.x;
                    bi = __float_as_int(o.y);
                }
            }
            epi_all(true);  // read before it is written again
            const int y = valid ? g.y[row] : -1;
            // exp(l - max) takes the logits' place in TMEM
            float ly = 0.f;
            for (int u = u0; u < u1; ++u) {
                uint32_t v[16];
                tmem_ld16_async(tb_ + u * 16, v);
                tmem_wait16(v);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const int n = u * 16 + j;
                    const float l = __uint_as_float(v[j]) + sbias[n];
                    if (n == y) ly = l;
                    v[j] = __float_as_uint(n < g.N ? expf(l - mx) : 0.f);
                }
                tmem_st16(tb_ + u * 16, v);
            }
            // their sum in ascending columns (one running sum per row, handed from
            // quarter to quarter: the rounding of a plain loop over the classes)
            float s = 0.f;
#pragma unroll 1
            for (int k = 0; k < kMParts; ++k) {
                if (part == k) {
                    if (k > 0) s = red[(k - 1) * kMM + r].x;
                    for (int u = u0; u < u1; ++u) {
                        uint32_t v[16];
                        tmem_ld16_async(tb_ + u * 16, v);
                        tmem_wait16(v);
#pragma unroll
                        for (int j = 0; j < 16; ++j) s += __uint_as_float(v[j]);  // zero past the classes
                    }
                    red[k * kMM + r] = make_float4(s, ly, 0.f, 0.f);
                }
                asm volatile("bar.sync %0, %1;" ::"r"(2 + q), "n"(kMParts * 32) : "memory");
            }
            s = red[(kMParts - 1) * kMM + r].x;
            ly = 0.f;
#pragma unroll
            for (int k = 0; k < kMParts; ++k) ly += red[k * kMM + r].y;  // the other quarters hold zero
            const float inv_s = 1.0f / s;
            for (int u = u0; u < u1; ++u) {
                const int c0 = u * 16;
                uint32_t v[16];
                tmem_ld16_async(tb_ + c0, v);
                tmem_wait16(v);
                float d[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const int n = c0 + j;
                    d[j] = (valid && n < g.N) ? (__uint_as_float(v[j]) * inv_s - (n == y ? 1.f : 0.f)) * g.scale : 0.f;
                }
                if (valid) {
                    store_bf16x16(g.out + (size_t)row * g.ldo + c0, d);
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (c0 + j < g.N) g.outT[(size_t)(c0 + j) * g.ldt + row] = bf16_bits(d[j]);
                }
                int col;
                const float cs = lane_sums16(d, lane, col);
                if (!(lane & 1) && c0 + col < g.N) g.colsum[(size_t)rw * g.ldc + c0 + col] = cs;
            }
            if (part == 0) {
                const float ce = valid ? (logf(s) + mx - ly) : 0.f;
                const float hit = (valid && bi == y) ? 1.f : 0.f;
                const float ces = lane_sum(ce), hits = lane_sum(hit), rows = lane_sum(valid ? 1.f : 0.f);
                if (lane == 0) {
                    atomicAdd(&g.loss[0], (double)ces);
                    atomicAdd(&g.loss[1], (double)hits);
                    atomicAdd(&g.loss[2], (double)rows);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(gb.tmem_cols)
                     : "memory");
    }
}

// ---------------------------------------------------------------------------
// inference: the three layers and the largest logit in one kernel
// ---------------------------------------------------------------------------
// Persistent CTA per SM; tiles of 128 rows go alternately to two groups of
// eight epilogue warps (two per TMEM lane quadrant, one per half of the
// columns).  A tile's activations never leave the SM: its group stages the
// rows as bfloat16 into its A buffer, the tensor cores multiply it by W1, the
// group turns the accumulators into GELU(z + b) in the same A buffer, and so
// on for W2; the logits (in chunks of at most 256 columns) only pass through
// registers for the running maximum.  The weights stream from L2 through a
// ring of 64-element K slices; while one group works on its accumulators (256
// TMEM columns each), the other's product runs.
// The GELU (an erff per activation) bounds it.  Measured on GB300, 1,048,576 x
// 32 -> 256 -> 256 -> 410: 2.69 ms as a cast and three products per 131,072
// rows with the activations through memory, 0.86 ms now (436 TFLOP/s); 2,090 x
// 64 -> 256 -> 256 -> 33: 66 -> 42 us.
constexpr int kInGroupWarps = 8;
constexpr int kInThreads = 64 + 2 * kInGroupWarps * 32;

struct InferCfg {
    const float *X;
    int64_t N;
    int D, Dk, Hp, C;   // row width, padded; padded hidden width; classes
    int nch, bn;        // logit chunks and columns per chunk
    int x_vec;          // rows allow 16-byte loads
    int stages;         // weight ring
    int64_t tiles;
    uint32_t a_bytes, w_bytes;  // an A buffer; a ring stage
    const float *b1, *b2, *b3;
    int32_t *pred;
    int *err;
};

// the two warps of a quadrant (named barrier `id`, 64 threads): every thread
// contributes v, every thread gets the AND
__device__ __forceinline__ bool pair_all(bool v, int id) {
    int out;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbar.red.and.pred q, %2, 64, p;\n\t"
        "selp.s32 %0, 1, 0, q;\n\t}"
        : "=r"(out)
        : "r"((int)v), "r"(id)
        : "memory");
    return out != 0;
}

__global__ void __launch_bounds__(kInThreads, 1)
    k_mlp_infer(const __grid_constant__ CUtensorMap t1, const __grid_constant__ CUtensorMap t2,
                const __grid_constant__ CUtensorMap t3, InferCfg c) {
    extern __shared__ uint8_t raw[];
    uint8_t *sm = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~(uintptr_t)1023);
    const int S = c.stages;
    uint8_t *ring = sm + 2 * (size_t)c.a_bytes;
    float *sb1 = reinterpret_cast<float *>(ring + (size_t)S * c.w_bytes);
    float *sb2 = sb1 + c.Hp;
    float *sb3 = sb2 + c.Hp;  // nch * bn; -inf past the classes, so that they are never the largest
    float2 *mrg = reinterpret_cast<float2 *>(sb3 + c.nch * c.bn);  // [2][128]
    uint64_t *bars = reinterpret_cast<uint64_t *>(mrg + 2 * kMM);
    uint64_t *a_ready = bars, *acc_full = bars + 2, *done = bars + 4, *full = bars + 5, *empty = full + S;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(empty + S);
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int phases = 2 + c.nch;
    // this CTA's tiles: blockIdx.x + i * gridDim.x; group g takes i = g, g + 2, ...
    const int64_t mine = c.tiles > (int64_t)blockIdx.x
                             ? (c.tiles - (int64_t)blockIdx.x + (int64_t)gridDim.x - 1) / (int64_t)gridDim.x
                             : 0;

    if (threadIdx.x == 0) {
        for (int g = 0; g < 2; ++g) {
            bar_init(&a_ready[g], kInGroupWarps);
            bar_init(&acc_full[g], 1);
        }
        bar_init(done, 1);
        for (int i = 0; i < S; ++i) {
            bar_init(&full[i], 1);
            bar_init(&empty[i], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int i = threadIdx.x; i < c.Hp; i += blockDim.x) {
        sb1[i] = c.b1[i];
        sb2[i] = c.b2[i];
    }
    for (int i = threadIdx.x; i < c.nch * c.bn; i += blockDim.x) sb3[i] = i < c.C ? c.b3[i] : -INFINITY;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&t1) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&t2) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&t3) : "memory");
            uint32_t nl = 0;  // slices issued
            bool ok = true;
            for (int64_t i0 = 0; i0 < mine && ok; i0 += 2)
                for (int ph = 0; ph < phases && ok; ++ph)
                    for (int g = 0; g < 2 && i0 + g < mine && ok; ++g) {
                        const CUtensorMap *t = ph == 0 ? &t1 : (ph == 1 ? &t2 : &t3);
                        const int ks = (ph == 0 ? c.Dk : c.Hp) / kMK;
                        const uint32_t rows = (uint32_t)(ph < 2 ? c.Hp : c.bn);
                        const int r0 = ph < 2 ? 0 : (ph - 2) * c.bn;
                        for (int k = 0; k < ks; ++k, ++nl) {
                            const uint32_t st = nl % S, f = nl / S;
                            if (f > 0 && !(ok = mwait(&empty[st], (f - 1) & 1, c.err))) break;
                            mbar_arrive_expect_tx(&full[st], rows * 128u);
                            tma_2d(ring + (size_t)st * c.w_bytes, t, k * kMK, r0, &full[st]);
                        }
                    }
            // every issued copy has landed before the block can exit
            for (uint32_t j = nl > (uint32_t)S ? nl - S : 0; j < nl; ++j) mwait(&full[j % S], (j / S) & 1, c.err);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA
        if (lane == 0) {
            uint32_t nl = 0;
            uint32_t na[2] = {0, 0};  // phases issued per group
            bool ok = true;
            for (int64_t i0 = 0; i0 < mine && ok; i0 += 2)
                for (int ph = 0; ph < phases && ok; ++ph)
                    for (int g = 0; g < 2 && i0 + g < mine && ok; ++g) {
                        const int ks = (ph == 0 ? c.Dk : c.Hp) / kMK;
                        const int nn = ph < 2 ? c.Hp : c.bn;
                        // kind::f16: F32 accumulate, BF16 A and B, both K-major, M = 128
                        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(nn >> 3) << 17) |
                                               ((uint32_t)(kMM >> 4) << 24);
                        // the group's A operand is in place and its accumulators are read
                        if (!(ok = mwait(&a_ready[g], na[g] & 1, c.err))) break;
                        ++na[g];
                        tc_fence_after();
                        const uint8_t *A = sm + (size_t)g * c.a_bytes;
                        for (int k = 0; k < ks; ++k, ++nl) {
                            const uint32_t st = nl % S;
                            if (!(ok = mwait(&full[st], (nl / S) & 1, c.err))) break;
                            tc_fence_after();
                            const uint8_t *B = ring + (size_t)st * c.w_bytes;
#pragma unroll
                            for (int j = 0; j < 4; ++j) {  // four K = 16 steps inside the 128-byte row
                                const uint64_t da = desc_sw128(smem_u32(A + k * (kMM * 128) + j * 32));
                                const uint64_t db = desc_sw128(smem_u32(B + j * 32));
                                const uint32_t acc = (k > 0 || j > 0) ? 1u : 0u;
                                asm volatile(
                                    "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(
                                        tmem + (uint32_t)(g * 256)),
                                    "l"(da), "l"(db), "r"(idesc), "r"(acc)
                                    : "memory");
                            }
                            asm volatile(
                                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                    smem_u32(&empty[st]))
                                : "memory");
                        }
                        if (!ok) break;
                        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                         smem_u32(&acc_full[g]))
                                     : "memory");
                    }
            // every MMA of this thread is complete before TMEM is freed
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(done))
                         : "memory");
            mwait(done, 0, c.err);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------- epilogue
        const int e = warp - 2;
        const int g = e >> 3, half = (e >> 2) & 1;
        const int q = warp & 3;  // TMEM lane quadrant of this warp
        const int r = q * 32 + lane;
        const int pid = 1 + g * 4 + q;
        const int gt = (e & 7) * 32 + lane;  // thread of the group
        uint8_t *A = sm + (size_t)g * c.a_bytes;
        const uint32_t tb = tmem + (uint32_t)(g * 256) + ((uint32_t)(q * 32) << 16);
        uint32_t na = 0;  // accumulators awaited
        auto release = [&]() {  // A written (generic proxy) and TMEM read: the next product may run
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0) bar_arrive(&a_ready[g]);
        };
        auto await = [&]() {  // pair-uniform: a named barrier needs both warps
            const bool ok = __all_sync(0xffffffffu, mwait(&acc_full[g], na & 1, c.err));
            ++na;
            const bool both = pair_all(ok, pid);
            tc_fence_after();
            return both;
        };
        for (int64_t i = g; i < mine; i += 2) {
            const int64_t m0 = ((int64_t)blockIdx.x + i * (int64_t)gridDim.x) * kMM;
            // the rows as bfloat16, zero-padded to Dk, in 16-byte chunks
            const int cq = c.Dk >> 3;
            for (int idx = gt; idx < kMM * cq; idx += kInGroupWarps * 32) {
                const int rr = idx / cq, ch = idx - rr * cq, d0 = ch * 8;
                const int64_t n = m0 + rr;
                float v[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = 0.f;
                if (n < c.N) {
                    const float *x = c.X + n * c.D;
                    if (c.x_vec) {
#pragma unroll
                        for (int k = 0; k < 8; k += 4)
                            if (d0 + k < c.D) {
                                const float4 t = __ldg(reinterpret_cast<const float4 *>(x + d0 + k));
                                v[k] = t.x;
                                v[k + 1] = t.y;
                                v[k + 2] = t.z;
                                v[k + 3] = t.w;
                            }
                    } else {
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            if (d0 + k < c.D) v[k] = __ldg(x + d0 + k);
                    }
                }
                uint32_t w[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    w[k] = (uint32_t)bf16_bits(v[2 * k]) | ((uint32_t)bf16_bits(v[2 * k + 1]) << 16);
                *reinterpret_cast<uint4 *>(A + swz_chunk(rr, ch, kMM * 128)) = make_uint4(w[0], w[1], w[2], w[3]);
            }
            release();
            bool ok = true;
            // the hidden layers: this warp's half of the columns, 16 at a time
            for (int layer = 0; layer < 2; ++layer) {
                if (!(ok = await())) break;
                const float *bias = layer ? sb2 : sb1;
                const int c1 = (half + 1) * (c.Hp >> 1);
#pragma unroll 1
                for (int c0 = half * (c.Hp >> 1); c0 < c1; c0 += 16) {
                    uint32_t v[16];
                    tmem_ld16_async(tb + c0, v);
                    float b[16];
#pragma unroll
                    for (int k = 0; k < 16; k += 4) {
                        const float4 t = *reinterpret_cast<const float4 *>(bias + c0 + k);
                        b[k] = t.x;
                        b[k + 1] = t.y;
                        b[k + 2] = t.z;
                        b[k + 3] = t.w;
                    }
                    tmem_wait16(v);
                    uint32_t w[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float a0 = gelu(__uint_as_float(v[2 * k]) + b[2 * k]);
                        const float a1 = gelu(__uint_as_float(v[2 * k + 1]) + b[2 * k + 1]);
                        w[k] = (uint32_t)bf16_bits(a0) | ((uint32_t)bf16_bits(a1) << 16);
                    }
                    *reinterpret_cast<uint4 *>(A + swz_chunk(r, c0 >> 3, kMM * 128)) =
                        make_uint4(w[0], w[1], w[2], w[3]);
                    *reinterpret_cast<uint4 *>(A + swz_chunk(r, (c0 >> 3) + 1, kMM * 128)) =
                        make_uint4(w[4], w[5], w[6], w[7]);
                }
                release();
            }
            if (!ok) break;  // a wait timed out (error recorded)
            // the logits: the first largest over this warp's half of every chunk
            float best = -INFINITY;
            int bi = 0;
            for (int h = 0; h < c.nch; ++h) {
                if (!(ok = await())) break;
                const int nu = c.bn >> 4, hu = (nu + 1) >> 1;
                const int u1 = half ? nu : hu;
#pragma unroll 1
                for (int u = half ? hu : 0; u < u1; ++u) {
                    uint32_t v[16];
                    tmem_ld16_async(tb + u * 16, v);
                    tmem_wait16(v);
                    const int n0 = h * c.bn + u * 16;
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        const float l = __uint_as_float(v[k]) + sb3[n0 + k];
                        if (l > best) {
                            best = l;
                            bi = n0 + k;
                        }
                    }
                }
                if (h + 1 < c.nch) release();
            }
            if (!ok) break;
            if (half) mrg[g * kMM + r] = make_float2(best, __int_as_float(bi));
            pair_all(true, pid);
            if (!half) {
                // (the next write of the slot follows this warp's next a_ready arrival)
                const float2 o = mrg[g * kMM + r];
                const int oi = __float_as_int(o.y);
                if (o.x > best || (o.x == best && oi < bi)) bi = oi;
                if (m0 + r < c.N) c.pred[m0 + r] = bi;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// ---------------------------------------------------------------------------
// data movement and the update
// ---------------------------------------------------------------------------
// SplitMix64 (Steele, Lea and Flood, OOPSLA 2014): a counter-based generator
__device__ __host__ __forceinline__ uint64_t splitmix64(uint64_t z) {
    z += 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

struct MlpState {
    int32_t t;      // Adam steps taken
    int32_t err;    // KM_ETIMEOUT when a bounded wait gave up
    double loss[3]; // cross-entropy sum, correct predictions, rows (since the last read)
};

// Batch of B rows: random rows of the training set (with replacement, a
// counter-based draw per (seed, step, row)), or rows 0..B-1 when seed is
// ~0ull.  Writes Xb (B x Dk bfloat16, zero padding), XbT (Dn x B, rows >= D
// zero) and the classes yb (labels mapped to contiguous groups when K > 0).
// A block per 32 rows: the rows pass through shared memory, so that both copies
// are written in runs of consecutive elements.
constexpr int kGatherRows = 32, kGatherThreads = 256;
__global__ void __launch_bounds__(kGatherThreads)
    k_mlp_gather(const float *X, int64_t N, int D, const int32_t *labels, int K, int G, int B, int Dk, int Dn,
                 uint64_t seed, const MlpState *st, uint16_t *Xb, uint16_t *XbT, int32_t *yb) {
    __shared__ uint16_t tile[kGatherRows][256 + 2];  // Dk <= 256
    pdl_trigger();
    const int i0 = blockIdx.x * kGatherRows;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = warp; k < kGatherRows && i0 + k < B; k += kGatherThreads / 32) {
        const int i = i0 + k;
        int64_t src = i;
        if (seed != ~0ull) src = (int64_t)(splitmix64(seed ^ splitmix64(((uint64_t)st->t << 32) | (uint32_t)i)) % (uint64_t)N);
        for (int d = lane; d < Dk; d += 32) {
            const uint16_t b = bf16_bits(d < D ? X[src * D + d] : 0.f);
            Xb[(size_t)i * Dk + d] = b;
            tile[k][d] = b;
        }
        if (lane == 0) {
            int y = labels[src];
            if (K > 0) y = (int)(((int64_t)y * G) / K);
            yb[i] = (y >= 0 && y < G) ? y : 0;
        }
    }
    __syncthreads();
    if (i0 + lane < B)
        for (int d = warp; d < Dn; d += kGatherThreads / 32) XbT[(size_t)d * B + i0 + lane] = tile[lane][d];
}

struct MlpDims {
    int D, H, G;        // logical sizes
    int Dk, Dn, Hp, Gk; // padded
    int64_t oW1, ob1, oW2, ob2, oW3, ob3, P;  // offsets of W1 b1 W2 b2 W3 b3 in the parameter vector
};

struct ApplyArgs {
    int mode;           // 0: gradient out, 1: Adam step, 2: copy the masters to the compute weights
    int wblocks;        // blocks for the weights (the others take the biases)
    float *master, *m1, *m2;
    const float *pW1, *pW2, *pW3;  // split-K partials
    int s1, s2, s3;
    int64_t ps1, ps2, ps3;         // floats between splits
    const float *cs1, *cs2, *cs3;  // per-warp column sums
    int nrw;                       // row warps (B / 32)
    float *grad;                   // mode 0
    float lr, b1, b2, eps;
    MlpState *st;
    uint16_t *W1b, *W2b, *W2T, *W3b, *W3T;
    float *b1p, *b2p, *b3p;
};

// One thread per parameter: its gradient (sum of the split-K partials or of
// the per-warp column sums), then the requested action; the compute copies
// (bfloat16 weights, padded FP32 biases) are rewritten from the masters.  The
// last blocks take the biases, 32 a block: eight warps sum an eighth of the
// row warps each (one thread over all of them took 20 us).
constexpr int kApplyThreads = 256;
__device__ __forceinline__ void apply_one(const MlpDims &d, const ApplyArgs &a, int64_t i, float gsum, float bc1,
                                          float bc2) {
    // Adam (Kingma and Ba): bias-corrected first and second moments
    const float m = a.b1 * a.m1[i] + (1.0f - a.b1) * gsum;
    const float v = a.b2 * a.m2[i] + (1.0f - a.b2) * gsum * gsum;
    a.m1[i] = m;
    a.m2[i] = v;
    a.master[i] -= a.lr * (m / bc1) / (sqrtf(v / bc2) + a.eps);
}
__global__ void __launch_bounds__(kApplyThreads) k_mlp_apply(MlpDims d, ApplyArgs a) {
    __shared__ float part[kApplyThreads];
    pdl_trigger();
    pdl_wait();
    const int t1 = a.mode == 1 ? a.st->t + 1 : 0;
    const float bc1 = a.mode == 1 ? 1.0f - powf(a.b1, (float)t1) : 1.f;
    const float bc2 = a.mode == 1 ? 1.0f - powf(a.b2, (float)t1) : 1.f;
    if ((int)blockIdx.x >= a.wblocks) {
        // biases: b1, b2 (H each), b3 (G) as one run
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const int o = ((int)blockIdx.x - a.wblocks) * 32 + lane;
        const bool in = o < 2 * d.H + d.G;
        const int seg = o < d.H ? 0 : (o < 2 * d.H ? 1 : 2);
        const int c = seg == 0 ? o : (seg == 1 ? o - d.H : o - 2 * d.H);
        const int64_t i = (seg == 0 ? d.ob1 : (seg == 1 ? d.ob2 : d.ob3)) + c;
        float gsum = 0.f;
        if (a.mode != 2) {
            const float *cs = seg == 0 ? a.cs1 : (seg == 1 ? a.cs2 : a.cs3);
            const int ld = seg == 2 ? d.G : d.Hp;
            float sum = 0.f;
            if (in) {
#pragma unroll 8
                for (int w = warp; w < a.nrw; w += kApplyThreads / 32) sum += cs[(int64_t)w * ld + c];
            }
            part[threadIdx.x] = sum;
            __syncthreads();
            if (warp == 0)
                for (int w = 0; w < kApplyThreads / 32; ++w) gsum += part[w * 32 + lane];
        }
        if (warp != 0 || !in) return;
        if (a.mode == 0) {
            a.grad[i] = gsum;
            return;
        }
        if (a.mode == 1) apply_one(d, a, i, gsum, bc1, bc2);
        (seg == 0 ? a.b1p : (seg == 1 ? a.b2p : a.b3p))[c] = a.master[i];
        return;
    }
    // weights: W1, W2, W3 as one run
    const int64_t n1 = (int64_t)d.H * d.D, n2 = (int64_t)d.H * d.H, nw = n1 + n2 + (int64_t)d.G * d.H;
    for (int64_t o = (int64_t)blockIdx.x * kApplyThreads + threadIdx.x; o < nw; o += (int64_t)a.wblocks * kApplyThreads) {
        const int seg = o < n1 ? 0 : (o < n1 + n2 ? 1 : 2);
        const int64_t w = seg == 0 ? o : (seg == 1 ? o - n1 : o - n1 - n2);
        const int64_t i = (seg == 0 ? d.oW1 : (seg == 1 ? d.oW2 : d.oW3)) + w;
        const int ld = seg == 0 ? d.D : d.H;
        const int r = (int)(w / ld), c = (int)(w - (int64_t)r * ld);  // (row, column) of the weight
        if (a.mode != 2) {
            const float *pw = seg == 0 ? a.pW1 : (seg == 1 ? a.pW2 : a.pW3);
            const int sn = seg == 0 ? a.s1 : (seg == 1 ? a.s2 : a.s3);
            const int64_t ps = seg == 0 ? a.ps1 : (seg == 1 ? a.ps2 : a.ps3);
            pw += (int64_t)r * (seg == 0 ? d.Dn : d.Hp) + c;
            float gsum = 0.f;
#pragma unroll 8
            for (int z = 0; z < sn; ++z) gsum += pw[z * ps];
            if (a.mode == 0) {
                a.grad[i] = gsum;
                continue;
            }
            apply_one(d, a, i, gsum, bc1, bc2);
        }
        const uint16_t wb = bf16_bits(a.master[i]);
        if (seg == 0) {
            a.W1b[(size_t)r * d.Dk + c] = wb;
        } else if (seg == 1) {
            a.W2b[(size_t)r * d.Hp + c] = wb;
            a.W2T[(size_t)c * d.Hp + r] = wb;
        } else {
            a.W3b[(size_t)r * d.Hp + c] = wb;
            a.W3T[(size_t)c * d.Gk + r] = wb;
        }
    }
}

__global__ void k_mlp_step_end(MlpState *st) { st->t += 1; }

// Xavier-uniform weights U(-a, a), a = sqrt(6 / (fan_in + fan_out)), zero
// biases, from the counter-based generator (seed, parameter index)
__global__ void k_mlp_init(MlpDims d, float *master, uint64_t seed) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < d.P; i += (int64_t)gridDim.x * blockDim.x) {
        float a = 0.f;
        if (i < d.ob1) a = sqrtf(6.0f / (float)(d.D + d.H));
        else if (i >= d.oW2 && i < d.ob2) a = sqrtf(6.0f / (float)(2 * d.H));
        else if (i >= d.oW3 && i < d.ob3) a = sqrtf(6.0f / (float)(d.H + d.G));
        const float u = (float)(splitmix64(seed ^ splitmix64((uint64_t)i)) >> 40) * (1.0f / 16777216.0f);
        master[i] = a * (2.0f * u - 1.0f);
    }
}

int round_up(int x, int m) { return (x + m - 1) / m * m; }
int pow2_at_least(int x) {
    int p = 32;
    while (p < x) p <<= 1;
    return p;
}

}  // namespace
}  // namespace kp

using namespace kp;

// ---------------------------------------------------------------------------
// the network object
// ---------------------------------------------------------------------------
struct kmeans_mlp {
    int dev = 0, num_sms = 0;
    size_t smem_optin = 0;
    cudaStream_t stream = nullptr;
    MlpDims d{};
    int nch3 = 1, bn3 = 16;  // layer-3 N chunks
    int bnH = 64;            // columns per CTA of the hidden-layer products
    float *master = nullptr, *m1 = nullptr, *m2 = nullptr;
    uint16_t *W1b = nullptr, *W2b = nullptr, *W2T = nullptr, *W3b = nullptr, *W3T = nullptr;
    float *b1p = nullptr, *b2p = nullptr, *b3p = nullptr;
    MlpState *st = nullptr;
    int *err = nullptr;  // &st->err
    // training buffers (batch B)
    int B = 0;
    uint16_t *Xb = nullptr, *XbT = nullptr, *A1 = nullptr, *A1T = nullptr, *A2 = nullptr, *A2T = nullptr,
             *dZ3 = nullptr, *dZ3T = nullptr, *dZ2 = nullptr, *dZ2T = nullptr, *dZ1T = nullptr;
    float *G1 = nullptr, *G2 = nullptr, *pW1 = nullptr, *pW2 = nullptr, *pW3 = nullptr, *cs1 = nullptr,
          *cs2 = nullptr, *cs3 = nullptr;
    int32_t *yb = nullptr;
    int s1 = 1, s2 = 1, s3 = 1;
    // the training products of a batch of B rows, as launched: layers 1, 2, 3, dZ2,
    // dZ1, and the three weight gradients together
    static constexpr int kPlans = 6;
    GemmBatch plan[kPlans];
    int grid[kPlans] = {};
    size_t smem[kPlans] = {};
    std::vector<void *> batch_allocs;
    std::vector<void *> allocs;
    char errmsg[512] = "";
};

namespace kp {
namespace {

thread_local char g_mlp_err[512] = "";

int mlp_fail(kmeans_mlp *m, int code, const char *fmt, ...) {
    char *buf = m ? m->errmsg : g_mlp_err;
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, 512, fmt, ap);
    va_end(ap);
    if (!m) set_thread_error(buf);
    return code;
}

#define MLP_CUDA(m, call)                                                                                   \
    do {                                                                                                    \
        cudaError_t e_ = (call);                                                                            \
        if (e_ != cudaSuccess)                                                                              \
            return mlp_fail((m), e_ == cudaErrorMemoryAllocation ? KM_ENOMEM : KM_ECUDA, "%s: %s (%s:%d)", #call, \
                            cudaGetErrorString(e_), __FILE__, __LINE__);                                    \
    } while (0)

template <class T>
cudaError_t mlp_alloc(kmeans_mlp *m, T **p, size_t n, std::vector<void *> &list) {
    void *v = nullptr;
    cudaError_t e = pool_alloc(m->dev, &v, std::max<size_t>(n, 1) * sizeof(T), m->stream);
    if (e != cudaSuccess) return e;
    list.push_back(v);
    *p = static_cast<T *>(v);
    return cudaMemsetAsync(v, 0, std::max<size_t>(n, 1) * sizeof(T), m->stream);
}

// 2D bfloat16 tensor map: `rows` rows of `cols` elements (row stride `ld`
// elements), boxes of 64 x box_rows with 128-byte swizzle
int make_map(kmeans_mlp *m, CUtensorMap *map, const uint16_t *base, int64_t rows, int64_t cols, int64_t ld,
             int box_rows) {
    auto enc = encoder();
    if (!enc) return mlp_fail(m, KM_ECUDA, "cuTensorMapEncodeTiled is not available");
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)(ld * 2)};
    cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1u, 1u};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t *>(base), dims, strides, box, es,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return mlp_fail(m, KM_ECUDA, "tensor map encoding failed (%d)", (int)r);
    return KM_OK;
}

// One product C = A . B^T.  A: rows x K (row stride lda_el), B: N rows x K.
// K must be a multiple of 64 (splits * 64 * k_steps).
struct GemmSpec {
    const uint16_t *A;
    int64_t a_rows, a_ld;
    const uint16_t *Bm;
    int64_t b_rows, b_ld;
    int64_t K;       // contraction length (multiple of 64 * splits)
    int M, N;        // valid output extent
    int nch, bn;     // columns per CTA: nch * bn
    int ntiles;      // CTAs along N
    int splits;
};

// adds a product to launch `k` of the network's plan
int plan_add(kmeans_mlp *m, int k, int idx, const GemmSpec &sp, GemmCfg g) {
    GemmBatch &b = m->plan[k];
    if (idx == 0) {
        memset(&b, 0, sizeof(b));
        m->grid[k] = 0;
    }
    int rc;
    if ((rc = make_map(m, &b.ta[idx], sp.A, sp.a_rows, sp.K, sp.a_ld, kMM))) return rc;
    if ((rc = make_map(m, &b.tb[idx], sp.Bm, sp.b_rows, sp.K, sp.b_ld, sp.bn))) return rc;
    g.M = sp.M;
    g.N = sp.N;
    g.mt = (sp.M + kMM - 1) / kMM;
    g.nt = sp.ntiles;
    g.nch = sp.nch;
    g.bn = sp.bn;
    g.k_steps = (int)(sp.K / kMK / sp.splits);
    g.err = m->err;
    b.g[idx] = g;
    b.first[idx] = m->grid[k];
    m->grid[k] += g.mt * g.nt * sp.splits;
    for (int i = idx + 1; i < 4; ++i) b.first[i] = m->grid[k];
    b.st_bytes = std::max<uint32_t>(b.st_bytes, (uint32_t)kMM * 128u + (uint32_t)(sp.nch * sp.bn) * 128u);
    b.tmem_cols = std::max(b.tmem_cols, pow2_at_least(sp.nch * sp.bn));
    const size_t fixed = 1024 + 256 + (size_t)kMParts * kMM * 16 + 512 * 4;  // alignment, barriers, row reductions, bias
    int stages = 4;
    while (stages > 2 && fixed + stages * (size_t)b.st_bytes > m->smem_optin) --stages;
    b.stages = stages;
    m->smem[k] = fixed + stages * (size_t)b.st_bytes;
    if (m->smem[k] > m->smem_optin) return mlp_fail(m, KM_EINVAL, "product tile does not fit in shared memory");
    return KM_OK;
}

// a launch that may begin before the kernel ahead of it on the stream ends
// (the kernel waits for it itself: pdl_wait)
template <class... P, class... A>
cudaError_t launch_pdl(void (*kernel)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t s,
                       const A &...args) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    count_launch();
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

int launch_plan(kmeans_mlp *m, int k, cudaStream_t s) {
    const cudaError_t e = launch_pdl(k_mlp_gemm, (unsigned)m->grid[k], kMThreads, m->smem[k], s, m->plan[k]);
    if (e != cudaSuccess) return mlp_fail(m, KM_ECUDA, "k_mlp_gemm launch: %s", cudaGetErrorString(e));
    return KM_OK;
}

GemmCfg cfg0(int mode) {
    GemmCfg g;
    memset(&g, 0, sizeof(g));
    g.mode = mode;
    return g;
}

// columns per CTA for a hidden-width output: all of them when M is large
// (one pass over A), else split in two for more CTAs
void hidden_tiles(const kmeans_mlp *m, int M, int &bn, int &ntiles) {
    const int Hp = m->d.Hp;
    if (Hp > 128 && (M + kMM - 1) / kMM < m->num_sms) {
        bn = Hp / 2;
        ntiles = 2;
    } else {
        bn = Hp;
        ntiles = 1;
    }
}

// the launches of one batch's forward and backward pass
int plan_batch(kmeans_mlp *m, int B) {
    const MlpDims &d = m->d;
    int rc, bnh, nth;
    hidden_tiles(m, B, bnh, nth);
    // layer 1: A1 = GELU(Xb W1^T + b1), with A1^T and GELU'(z1)
    GemmCfg g = cfg0(E_GELU);
    g.bias = m->b1p; g.out = m->A1; g.ldo = d.Hp; g.outT = m->A1T; g.ldt = B; g.aux = m->G1; g.lda = d.Hp;
    if ((rc = plan_add(m, 0, 0, {m->Xb, B, d.Dk, m->W1b, d.Hp, d.Dk, d.Dk, B, d.Hp, 1, bnh, nth, 1}, g))) return rc;
    // layer 2
    g = cfg0(E_GELU);
    g.bias = m->b2p; g.out = m->A2; g.ldo = d.Hp; g.outT = m->A2T; g.ldt = B; g.aux = m->G2; g.lda = d.Hp;
    if ((rc = plan_add(m, 1, 0, {m->A1, B, d.Hp, m->W2b, d.Hp, d.Hp, d.Hp, B, d.Hp, 1, bnh, nth, 1}, g))) return rc;
    // layer 3 + softmax cross-entropy: dZ3 = (softmax - onehot) / B
    g = cfg0(E_SOFTMAX);
    g.bias = m->b3p; g.out = m->dZ3; g.ldo = d.Gk; g.outT = m->dZ3T; g.ldt = B; g.colsum = m->cs3; g.ldc = d.G;
    g.y = m->yb; g.scale = 1.0f / (float)B; g.loss = m->st->loss;
    if ((rc = plan_add(m, 2, 0, {m->A2, B, d.Hp, m->W3b, d.G, d.Hp, d.Hp, B, d.G, m->nch3, m->bn3, 1, 1}, g)))
        return rc;
    // dZ2 = (dZ3 W3) * GELU'(z2)
    g = cfg0(E_MUL);
    g.aux = m->G2; g.lda = d.Hp; g.out = m->dZ2; g.ldo = d.Hp; g.outT = m->dZ2T; g.ldt = B; g.colsum = m->cs2;
    g.ldc = d.Hp;
    if ((rc = plan_add(m, 3, 0, {m->dZ3, B, d.Gk, m->W3T, d.Hp, d.Gk, d.Gk, B, d.Hp, 1, bnh, nth, 1}, g))) return rc;
    // dZ1 = (dZ2 W2) * GELU'(z1)
    g = cfg0(E_MUL);
    g.aux = m->G1; g.lda = d.Hp; g.outT = m->dZ1T; g.ldt = B; g.colsum = m->cs1; g.ldc = d.Hp;
    if ((rc = plan_add(m, 4, 0, {m->dZ2, B, d.Hp, m->W2T, d.Hp, d.Hp, d.Hp, B, d.Hp, 1, bnh, nth, 1}, g))) return rc;
    // weight gradients, contracted over the batch: dW3 = dZ3^T A2, dW2 = dZ2^T A1, dW1 = dZ1^T X
    g = cfg0(E_F32);
    g.part = m->pW3; g.ldp = d.Hp; g.part_split = (int64_t)d.G * d.Hp;
    if ((rc = plan_add(m, 5, 0, {m->dZ3T, d.G, B, m->A2T, d.Hp, B, B, d.G, d.Hp, 1, d.Hp, 1, m->s3}, g))) return rc;
    g = cfg0(E_F32);
    g.part = m->pW2; g.ldp = d.Hp; g.part_split = (int64_t)d.Hp * d.Hp;
    if ((rc = plan_add(m, 5, 1, {m->dZ2T, d.Hp, B, m->A1T, d.Hp, B, B, d.Hp, d.Hp, 1, d.Hp, 1, m->s2}, g))) return rc;
    g = cfg0(E_F32);
    g.part = m->pW1; g.ldp = d.Dn; g.part_split = (int64_t)d.Hp * d.Dn;
    return plan_add(m, 5, 2, {m->dZ1T, d.Hp, B, m->XbT, d.Dn, B, B, d.Hp, d.Dn, 1, d.Dn, 1, m->s1}, g);
}

int alloc_batch(kmeans_mlp *m, int B) {
    if (m->B == B) return KM_OK;
    for (void *p : m->batch_allocs) cudaFreeAsync(p, m->stream);
    m->batch_allocs.clear();
    m->B = 0;
    const MlpDims &d = m->d;
    auto &L = m->batch_allocs;
    // split-K of the weight gradients: at least 4 slices of 64 per CTA, at most
    // one wave of CTAs for the three products together (fewer partial sums to
    // write and read back than with a wave for each)
    const int tiles = 2 * ((d.Hp + kMM - 1) / kMM) + (d.G + kMM - 1) / kMM;
    int sk = 1;
    while (sk * 2 * tiles <= m->num_sms && (B / 64) % (sk * 2) == 0 && B / 64 / (sk * 2) >= 4) sk *= 2;
    m->s1 = m->s2 = m->s3 = sk;
    MLP_CUDA(m, mlp_alloc(m, &m->Xb, (size_t)B * d.Dk, L));
    MLP_CUDA(m, mlp_alloc(m, &m->XbT, (size_t)d.Dn * B, L));
    MLP_CUDA(m, mlp_alloc(m, &m->A1, (size_t)B * d.Hp, L));
    MLP_CUDA(m, mlp_alloc(m, &m->A1T, (size_t)d.Hp * B, L));
    MLP_CUDA(m, mlp_alloc(m, &m->A2, (size_t)B * d.Hp, L));
    MLP_CUDA(m, mlp_alloc(m, &m->A2T, (size_t)d.Hp * B, L));
    MLP_CUDA(m, mlp_alloc(m, &m->dZ3, (size_t)B * d.Gk, L));
    MLP_CUDA(m, mlp_alloc(m, &m->dZ3T, (size_t)d.G * B, L));
    MLP_CUDA(m, mlp_alloc(m, &m->dZ2, (size_t)B * d.Hp, L));
    MLP_CUDA(m, mlp_alloc(m, &m->dZ2T, (size_t)d.Hp * B, L));
    MLP_CUDA(m, mlp_alloc(m, &m->dZ1T, (size_t)d.Hp * B, L));
    MLP_CUDA(m, mlp_alloc(m, &m->G1, (size_t)B * d.Hp, L));
    MLP_CUDA(m, mlp_alloc(m, &m->G2, (size_t)B * d.Hp, L));
    MLP_CUDA(m, mlp_alloc(m, &m->pW1, (size_t)m->s1 * d.Hp * d.Dn, L));
    MLP_CUDA(m, mlp_alloc(m, &m->pW2, (size_t)m->s2 * d.Hp * d.Hp, L));
    MLP_CUDA(m, mlp_alloc(m, &m->pW3, (size_t)m->s3 * d.G * d.Hp, L));
    MLP_CUDA(m, mlp_alloc(m, &m->cs1, (size_t)(B / 32) * d.Hp, L));
    MLP_CUDA(m, mlp_alloc(m, &m->cs2, (size_t)(B / 32) * d.Hp, L));
    MLP_CUDA(m, mlp_alloc(m, &m->cs3, (size_t)(B / 32) * d.G, L));
    MLP_CUDA(m, mlp_alloc(m, &m->yb, (size_t)B, L));
    const int rc = plan_batch(m, B);
    if (rc) return rc;
    m->B = B;
    return KM_OK;
}

// forward + backward of one batch already gathered into Xb / XbT / yb;
// leaves the split-K partials and the column sums for k_mlp_apply
int enqueue_fwd_bwd(kmeans_mlp *m, cudaStream_t s) {
    for (int k = 0; k < kmeans_mlp::kPlans; ++k)
        if (int rc = launch_plan(m, k, s)) return rc;
    return KM_OK;
}

ApplyArgs apply_args(kmeans_mlp *m, int mode) {
    ApplyArgs a;
    memset(&a, 0, sizeof(a));
    const MlpDims &d = m->d;
    a.mode = mode;
    a.master = m->master; a.m1 = m->m1; a.m2 = m->m2;
    a.pW1 = m->pW1; a.pW2 = m->pW2; a.pW3 = m->pW3;
    a.s1 = m->s1; a.s2 = m->s2; a.s3 = m->s3;
    a.ps1 = (int64_t)d.Hp * d.Dn; a.ps2 = (int64_t)d.Hp * d.Hp; a.ps3 = (int64_t)d.G * d.Hp;
    a.cs1 = m->cs1; a.cs2 = m->cs2; a.cs3 = m->cs3;
    a.nrw = m->B / 32;
    a.st = m->st;
    a.W1b = m->W1b; a.W2b = m->W2b; a.W2T = m->W2T; a.W3b = m->W3b; a.W3T = m->W3T;
    a.b1p = m->b1p; a.b2p = m->b2p; a.b3p = m->b3p;
    a.b1 = 0.9f; a.b2 = 0.999f; a.eps = 1e-8f;
    return a;
}

int launch_apply(kmeans_mlp *m, ApplyArgs a, cudaStream_t s) {
    const MlpDims &d = m->d;
    const int64_t nw = (int64_t)d.H * d.D + (int64_t)d.H * d.H + (int64_t)d.G * d.H;
    a.wblocks = (int)std::min<int64_t>((nw + kApplyThreads - 1) / kApplyThreads, (int64_t)m->num_sms * 8);
    const int bblocks = (2 * d.H + d.G + 31) / 32;
    const cudaError_t e = launch_pdl(k_mlp_apply, (unsigned)(a.wblocks + bblocks), kApplyThreads, 0, s, d, a);
    if (e != cudaSuccess) return mlp_fail(m, KM_ECUDA, "k_mlp_apply launch: %s", cudaGetErrorString(e));
    return KM_OK;
}

// the batch's rows (of N) and classes into Xb / XbT / yb
int launch_gather(kmeans_mlp *m, const float *X, int64_t N, const int32_t *labels, int K, uint64_t seed,
                  cudaStream_t s) {
    const MlpDims &d = m->d;
    count_launch();
    k_mlp_gather<<<(unsigned)((m->B + kGatherRows - 1) / kGatherRows), kGatherThreads, 0, s>>>(
        X, N, d.D, labels, K, d.G, m->B, d.Dk, d.Dn, seed, m->st, m->Xb, m->XbT, m->yb);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return mlp_fail(m, KM_ECUDA, "k_mlp_gather launch: %s", cudaGetErrorString(e));
    return KM_OK;
}

// waits for the stream and reads the state (error flag, loss) back
int read_state(kmeans_mlp *m, MlpState &h) {
    MLP_CUDA(m, cudaMemcpyAsync(&h, m->st, sizeof(h), cudaMemcpyDeviceToHost, m->stream));
    MLP_CUDA(m, cudaStreamSynchronize(m->stream));
    if (h.err) return mlp_fail(m, KM_ETIMEOUT, "a bounded wait in a tensor-core product gave up");
    return KM_OK;
}
int check_err(kmeans_mlp *m) {
    MlpState h;
    return read_state(m, h);
}
// the error flag and the loss sums to zero (not the step counter)
cudaError_t clear_state(kmeans_mlp *m) {
    return cudaMemsetAsync(&m->st->err, 0, sizeof(MlpState) - offsetof(MlpState, err), m->stream);
}

struct DevGuard {
    int prev = -1;
    explicit DevGuard(int dev) {
        if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) cudaSetDevice(dev);
        else prev = -1;
    }
    ~DevGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

bool dev_ptr(const void *p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

// pred[n] = the class with the largest logit (first maximum), on stream s
// (used by the context's seeded iteration 0 and by kmeans_mlp_predict_net)
int mlp_predict_enqueue(kmeans_mlp *m, const float *X, int64_t N, int32_t *pred, cudaStream_t s) {
    const MlpDims &d = m->d;
    InferCfg c;
    c.X = X;
    c.N = N;
    c.D = d.D;
    c.Dk = d.Dk;
    c.Hp = d.Hp;
    c.C = d.G;
    c.nch = m->nch3;
    c.bn = m->bn3;
    c.x_vec = d.D % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    c.tiles = (N + kMM - 1) / kMM;
    c.a_bytes = (uint32_t)(std::max(d.Dk, d.Hp) / 64) * (kMM * 128);
    c.w_bytes = (uint32_t)std::max(d.Hp, m->bn3) * 128u;
    c.b1 = m->b1p;
    c.b2 = m->b2p;
    c.b3 = m->b3p;
    c.pred = pred;
    c.err = m->err;
    const size_t fixed = 1024 + 2 * (size_t)c.a_bytes + (size_t)(2 * d.Hp + c.nch * c.bn) * 4 + 2 * kMM * 8 + 256;
    c.stages = (int)std::min<size_t>(6, (m->smem_optin - fixed) / c.w_bytes);
    if (fixed > m->smem_optin || c.stages < 2)
        return mlp_fail(m, KM_EINVAL, "the network's tiles do not fit in shared memory");
    const size_t smem = fixed + (size_t)c.stages * c.w_bytes;
    CUtensorMap t1, t2, t3;
    int rc;
    if ((rc = make_map(m, &t1, m->W1b, d.Hp, d.Dk, d.Dk, d.Hp))) return rc;
    if ((rc = make_map(m, &t2, m->W2b, d.Hp, d.Hp, d.Hp, d.Hp))) return rc;
    if ((rc = make_map(m, &t3, m->W3b, d.G, d.Hp, d.Hp, m->bn3))) return rc;
    count_launch();
    k_mlp_infer<<<(unsigned)std::min<int64_t>(c.tiles, m->num_sms), kInThreads, smem, s>>>(t1, t2, t3, c);
    MLP_CUDA(m, cudaGetLastError());
    return KM_OK;
}

int mlp_error_flag(kmeans_mlp *m) { return check_err(m); }
const char *mlp_message(const kmeans_mlp *m) { return m->errmsg; }

}  // namespace kp

extern "C" {

KM_API int kmeans_mlp_create(kmeans_mlp **out, int32_t D, int32_t hidden, int32_t classes, uint64_t seed,
                             void *stream) {
    if (!out) return mlp_fail(nullptr, KM_EINVAL, "out is NULL");
    *out = nullptr;
    if (D < 1 || D > 256) return mlp_fail(nullptr, KM_EINVAL, "D out of range [1, 256]");
    if (hidden < 1 || hidden > 256) return mlp_fail(nullptr, KM_EINVAL, "hidden out of range [1, 256]");
    if (classes < 1 || classes > 512) return mlp_fail(nullptr, KM_EINVAL, "classes out of range [1, 512]");
    kmeans_mlp *m = new (std::nothrow) kmeans_mlp();
    if (!m) return mlp_fail(nullptr, KM_ENOMEM, "host allocation failed");
    struct Guard {
        kmeans_mlp *&m;
        bool keep = false;
        ~Guard() {
            if (!keep && m) kmeans_mlp_destroy(m);
        }
    } guard{m};
    if (cudaGetDevice(&m->dev) != cudaSuccess) return mlp_fail(nullptr, KM_ECUDA, "cudaGetDevice failed");
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, m->dev) != cudaSuccess)
        return mlp_fail(nullptr, KM_ECUDA, "cudaDeviceGetAttribute failed");
    m->num_sms = v;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, m->dev) != cudaSuccess)
        return mlp_fail(nullptr, KM_ECUDA, "cudaDeviceGetAttribute failed");
    m->smem_optin = (size_t)v;
    m->stream = static_cast<cudaStream_t>(stream);
    MlpDims &d = m->d;
    d.D = D;
    d.H = hidden;
    d.G = classes;
    d.Dk = round_up(D, 64);
    d.Dn = round_up(D, 16);
    d.Hp = round_up(hidden, 64);
    d.Gk = round_up(classes, 64);
    d.oW1 = 0;
    d.ob1 = d.oW1 + (int64_t)hidden * D;
    d.oW2 = d.ob1 + hidden;
    d.ob2 = d.oW2 + (int64_t)hidden * hidden;
    d.oW3 = d.ob2 + hidden;
    d.ob3 = d.oW3 + (int64_t)classes * hidden;
    d.P = d.ob3 + classes;
    m->nch3 = (classes + 255) / 256;
    m->bn3 = round_up((classes + m->nch3 - 1) / m->nch3, 16);
    int rc;
    auto fail_cuda = [&](cudaError_t e) {
        return mlp_fail(nullptr, e == cudaErrorMemoryAllocation ? KM_ENOMEM : KM_ECUDA, "%s", cudaGetErrorString(e));
    };
    cudaError_t e;
#define MC(call) \
    if ((e = (call)) != cudaSuccess) return fail_cuda(e)
    MC(mlp_alloc(m, &m->master, (size_t)d.P, m->allocs));
    MC(mlp_alloc(m, &m->m1, (size_t)d.P, m->allocs));
    MC(mlp_alloc(m, &m->m2, (size_t)d.P, m->allocs));
    MC(mlp_alloc(m, &m->W1b, (size_t)d.Hp * d.Dk, m->allocs));
    MC(mlp_alloc(m, &m->W2b, (size_t)d.Hp * d.Hp, m->allocs));
    MC(mlp_alloc(m, &m->W2T, (size_t)d.Hp * d.Hp, m->allocs));
    MC(mlp_alloc(m, &m->W3b, (size_t)classes * d.Hp, m->allocs));
    MC(mlp_alloc(m, &m->W3T, (size_t)d.Hp * d.Gk, m->allocs));
    MC(mlp_alloc(m, &m->b1p, (size_t)d.Hp, m->allocs));
    MC(mlp_alloc(m, &m->b2p, (size_t)d.Hp, m->allocs));
    MC(mlp_alloc(m, &m->b3p, (size_t)classes, m->allocs));
    MC(mlp_alloc(m, &m->st, 1, m->allocs));
    m->err = &m->st->err;
    // (one value for every network: it is the process's, and another thread's network may be launching)
    MC(cudaFuncSetAttribute(k_mlp_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)m->smem_optin));
    MC(cudaFuncSetAttribute(k_mlp_infer, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)m->smem_optin));
    count_launch();
    k_mlp_init<<<(unsigned)std::min<int64_t>((d.P + 255) / 256, (int64_t)m->num_sms * 8), 256, 0, m->stream>>>(
        d, m->master, seed);
    MC(cudaGetLastError());
#undef MC
    ApplyArgs a = apply_args(m, 2);
    if ((rc = launch_apply(m, a, m->stream))) return mlp_fail(nullptr, rc, "%s", m->errmsg);
    if (cudaStreamSynchronize(m->stream) != cudaSuccess) return mlp_fail(nullptr, KM_ECUDA, "initialisation failed");
    guard.keep = true;
    *out = m;
    return KM_OK;
}

KM_API int kmeans_mlp_set_params(kmeans_mlp *m, const float *W1, const float *b1, const float *W2, const float *b2,
                                 const float *W3, const float *b3) {
    if (!m) return mlp_fail(nullptr, KM_EINVAL, "network is NULL");
    if (!W1 || !b1 || !W2 || !b2 || !W3 || !b3) return mlp_fail(m, KM_EINVAL, "a parameter pointer is NULL");
    DevGuard dg(m->dev);
    const MlpDims &d = m->d;
    const float *src[6] = {W1, b1, W2, b2, W3, b3};
    const int64_t off[7] = {d.oW1, d.ob1, d.oW2, d.ob2, d.oW3, d.ob3, d.P};
    for (int i = 0; i < 6; ++i)
        MLP_CUDA(m, cudaMemcpyAsync(m->master + off[i], src[i], (size_t)(off[i + 1] - off[i]) * 4, cudaMemcpyDefault,
                                    m->stream));
    MLP_CUDA(m, cudaMemsetAsync(m->m1, 0, (size_t)d.P * 4, m->stream));
    MLP_CUDA(m, cudaMemsetAsync(m->m2, 0, (size_t)d.P * 4, m->stream));
    MLP_CUDA(m, cudaMemsetAsync(m->st, 0, sizeof(MlpState), m->stream));
    int rc;
    if ((rc = launch_apply(m, apply_args(m, 2), m->stream))) return rc;
    MLP_CUDA(m, cudaStreamSynchronize(m->stream));
    return KM_OK;
}

KM_API int kmeans_mlp_get_params(kmeans_mlp *m, float *W1, float *b1, float *W2, float *b2, float *W3, float *b3) {
    if (!m) return mlp_fail(nullptr, KM_EINVAL, "network is NULL");
    DevGuard dg(m->dev);
    const MlpDims &d = m->d;
    float *dst[6] = {W1, b1, W2, b2, W3, b3};
    const int64_t off[7] = {d.oW1, d.ob1, d.oW2, d.ob2, d.oW3, d.ob3, d.P};
    for (int i = 0; i < 6; ++i)
        if (dst[i])
            MLP_CUDA(m, cudaMemcpyAsync(dst[i], m->master + off[i], (size_t)(off[i + 1] - off[i]) * 4,
                                        cudaMemcpyDefault, m->stream));
    MLP_CUDA(m, cudaStreamSynchronize(m->stream));
    return KM_OK;
}

KM_API int kmeans_mlp_gradient(kmeans_mlp *m, const float *X, const int32_t *y, int32_t B, double *loss,
                               float *grad) {
    if (!m) return mlp_fail(nullptr, KM_EINVAL, "network is NULL");
    if (!X || !y || !grad) return mlp_fail(m, KM_EINVAL, "a pointer argument is NULL");
    if (B < 128 || B % 128 != 0 || B > (1 << 20)) return mlp_fail(m, KM_EINVAL, "B must be a multiple of 128 in [128, 2^20]");
    if (!dev_ptr(X) || !dev_ptr(y) || !dev_ptr(grad)) return mlp_fail(m, KM_EINVAL, "X, y and grad must be device memory");
    DevGuard dg(m->dev);
    int rc;
    if ((rc = alloc_batch(m, B))) return rc;
    cudaStream_t s = m->stream;
    MLP_CUDA(m, clear_state(m));
    if ((rc = launch_gather(m, X, B, y, 0, ~0ull, s))) return rc;
    if ((rc = enqueue_fwd_bwd(m, s))) return rc;
    ApplyArgs a = apply_args(m, 0);
    a.grad = grad;
    if ((rc = launch_apply(m, a, s))) return rc;
    MlpState h;
    if ((rc = read_state(m, h))) return rc;
    if (loss) *loss = h.loss[2] > 0 ? h.loss[0] / h.loss[2] : 0.0;
    return KM_OK;
}

KM_API int kmeans_mlp_train(kmeans_mlp *m, const float *X, int64_t N, const int32_t *labels, int32_t K,
                            int64_t steps, int32_t batch, float lr, uint64_t seed, double *mean_loss,
                            double *accuracy) {
    if (!m) return mlp_fail(nullptr, KM_EINVAL, "network is NULL");
    if (!X || !labels) return mlp_fail(m, KM_EINVAL, "a pointer argument is NULL");
    if (N < 1 || steps < 0 || K < 0 || !(lr > 0.f)) return mlp_fail(m, KM_EINVAL, "bad N, steps, K or lr");
    if (batch < 128 || batch % 128 != 0 || batch > (1 << 20))
        return mlp_fail(m, KM_EINVAL, "batch must be a multiple of 128 in [128, 2^20]");
    if (seed == ~0ull && N < batch) return mlp_fail(m, KM_EINVAL, "a fixed batch (seed ~0) needs N >= batch");
    if (!dev_ptr(X) || !dev_ptr(labels)) return mlp_fail(m, KM_EINVAL, "X and labels must be device memory");
    DevGuard dg(m->dev);
    int rc;
    if ((rc = alloc_batch(m, batch))) return rc;
    cudaStream_t s = m->stream;
    MLP_CUDA(m, clear_state(m));
    // one step recorded once as a CUDA graph, replayed `steps` times (the
    // step counter on the device drives the row draw and Adam's bias correction)
    cudaStream_t cap = nullptr;
    MLP_CUDA(m, cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
    struct CapGuard {
        cudaStream_t s;
        ~CapGuard() { cudaStreamDestroy(s); }
    } cg{cap};
    MLP_CUDA(m, cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal));
    rc = launch_gather(m, X, N, labels, K, seed, cap);
    if (!rc) rc = enqueue_fwd_bwd(m, cap);
    if (!rc) {
        ApplyArgs a = apply_args(m, 1);
        a.lr = lr;
        rc = launch_apply(m, a, cap);
    }
    if (!rc) {
        count_launch();
        k_mlp_step_end<<<1, 1, 0, cap>>>(m->st);
    }
    cudaGraph_t graph = nullptr;
    cudaError_t e2 = cudaStreamEndCapture(cap, &graph);
    if (rc) {
        if (graph) cudaGraphDestroy(graph);
        return rc;
    }
    MLP_CUDA(m, e2);
    cudaGraphExec_t ex = nullptr;
    cudaError_t e3 = cudaGraphInstantiate(&ex, graph, 0);
    cudaGraphDestroy(graph);
    MLP_CUDA(m, e3);
    struct ExecGuard {
        cudaGraphExec_t x;
        ~ExecGuard() { cudaGraphExecDestroy(x); }
    } eg{ex};
    for (int64_t i = 0; i < steps; ++i) MLP_CUDA(m, cudaGraphLaunch(ex, s));
    MlpState h;
    if ((rc = read_state(m, h))) return rc;
    if (mean_loss) *mean_loss = h.loss[2] > 0 ? h.loss[0] / h.loss[2] : 0.0;
    if (accuracy) *accuracy = h.loss[2] > 0 ? h.loss[1] / h.loss[2] : 0.0;
    return KM_OK;
}

KM_API int kmeans_mlp_predict_net(kmeans_mlp *m, const float *X, int64_t N, int32_t *pred) {
    if (!m) return mlp_fail(nullptr, KM_EINVAL, "network is NULL");
    if (!X || !pred || N < 1) return mlp_fail(m, KM_EINVAL, "bad X, pred or N");
    if (!dev_ptr(X) || !dev_ptr(pred)) return mlp_fail(m, KM_EINVAL, "X and pred must be device memory");
    DevGuard dg(m->dev);
    MLP_CUDA(m, cudaMemsetAsync(m->err, 0, 4, m->stream));
    int rc;
    if ((rc = mlp_predict_enqueue(m, X, N, pred, m->stream))) return rc;
    return check_err(m);
}

KM_API void kmeans_mlp_destroy(kmeans_mlp *m) {
    if (!m) return;
    DevGuard dg(m->dev);
    for (void *p : m->batch_allocs) cudaFreeAsync(p, m->stream);
    for (void *p : m->allocs) cudaFreeAsync(p, m->stream);
    cudaStreamSynchronize(m->stream);
    delete m;
}

KM_API const char *kmeans_mlp_last_error(const kmeans_mlp *m) { return m ? m->errmsg : kp::g_mlp_err; }

}  // extern "C"
