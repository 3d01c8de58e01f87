// kp_tc.cuh -- pieces shared by the tensor-core dense kernels: mbarrier and
// TMA helpers, tcgen05 descriptors and TMEM loads, the bfloat16 split, the
// 128-byte-swizzled tile layout, and the row scan of the epilogue (group
// minima, winner, runner-up).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <mutex>

#include "kp_common.cuh"

namespace kp {
namespace {

constexpr int kTM = 128;          // points per tile
constexpr uint32_t kPolls = 1u << 22;
constexpr int kAtomBytes = kTM * 128;  // one 64-element bfloat16 column block of a tile

__device__ __forceinline__ uint64_t desc_sw128(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);
    d |= (uint64_t)1 << 16;            // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;  // stride byte offset: 8 rows x 128 B
    d |= (uint64_t)1 << 46;            // descriptor version
    d |= (uint64_t)2 << 61;            // 128-byte swizzle
    return d;
}
__device__ __forceinline__ void bar_init(uint64_t *b, uint32_t n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t *b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
// bounded wait; on time-out records KM_ETIMEOUT and returns false
__device__ __forceinline__ bool bar_wait(uint64_t *b, uint32_t parity, Ctrl *ctrl) {
    for (uint32_t i = 0; i < kPolls; ++i)
        if (mbar_try_wait(b, parity)) return true;
    atomicExch(&ctrl->err, (int)KM_ETIMEOUT);
    return false;
}
__device__ __forceinline__ void tma_2d(void *dst, const CUtensorMap *m, int c0, int c1, uint64_t *b) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_u32(dst)),
        "l"((uint64_t)m), "r"(c0), "r"(c1), "r"(smem_u32(b))
        : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Asynchronous TMEM read of 16 columns; the registers may be used only after
// tmem_wait16 on the same array (which names them, so that the compiler cannot
// move their uses above the wait).
__device__ __forceinline__ void tmem_ld16_async(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait16(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15])
                 :
                 : "memory");
}

// 16 columns back to TMEM, complete on return
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n\t"
        "tcgen05.wait::st.sync.aligned;" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}

// byte offset of the 16-byte chunk holding bfloat16 elements [8q, 8q+8) of
// `row` in a 128-byte-swizzled K-major tile (64 elements per 128-byte row)
__device__ __forceinline__ uint32_t swz_chunk(int row, int q, int atom_bytes) {
    return (uint32_t)((q >> 3) * atom_bytes + row * 128 + (((q & 7) ^ (row & 7)) << 4));
}

__device__ __forceinline__ void split8(const float *v, uint4 &h, uint4 &l) {
    uint32_t hw[4], lw[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        __nv_bfloat16 h0 = __float2bfloat16_rn(v[2 * i]), h1 = __float2bfloat16_rn(v[2 * i + 1]);
        __nv_bfloat16 l0 = __float2bfloat16_rn(v[2 * i] - __bfloat162float(h0));
        __nv_bfloat16 l1 = __float2bfloat16_rn(v[2 * i + 1] - __bfloat162float(h1));
        hw[i] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
        lw[i] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
    }
    h = make_uint4(hw[0], hw[1], hw[2], hw[3]);
    l = make_uint4(lw[0], lw[1], lw[2], lw[3]);
}
__device__ __forceinline__ float min3(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Running scan of one row over an ascending run of accumulator columns, four
// at a time: the smallest value and the runner-up from the sorted pairs of the
// four, the winner as the index of its group of four (whose values the lane
// keeps in shared memory, from which the column is read off at the end), and
// the open group's minimum.  A group boundary among the four columns (the
// same for every row) closes the minimum into the row's next slot.
// The stores carry no memory clobber, so that the scan's loads may move
// across them; what they wrote is read back by volatile accesses only.
struct Scan4 {
    float b1, b2, gm;
    int c4;        // first column of the four that hold b1
    uint32_t row;  // slots of the row's group minima
    uint32_t t4;   // the lane's four values
    int pend;      // the open group's slot (warp-uniform)

    __device__ __forceinline__ void four(const uint32_t *acc, const float4 &cn, uint32_t nib, int c) {
        const f32x2 m2 = 0xc0000000c0000000ull;  // (-2, -2)
        float t[4];
        unpack2(fma2(pack2(__uint_as_float(acc[0]), __uint_as_float(acc[1])), m2, pack2(cn.x, cn.y)), t[0], t[1]);
        unpack2(fma2(pack2(__uint_as_float(acc[2]), __uint_as_float(acc[3])), m2, pack2(cn.z, cn.w)), t[2], t[3]);
        const float l0 = fminf(t[0], t[1]), h0 = fmaxf(t[0], t[1]);
        const float l1 = fminf(t[2], t[3]), h1 = fmaxf(t[2], t[3]);
        const float m = fminf(l0, l1);
        const float s = min3(fmaxf(l0, l1), h0, h1);  // the second smallest of the four
        b2 = min3(b2, s, fmaxf(b1, m));
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.lt.f32 p, %6, %7;\n\t@p st.shared.v4.f32 [%1], {%2, %3, %4, %5};\n\t"
            "selp.s32 %0, %8, %0, p;\n\t}"
            : "+r"(c4)
            : "r"(t4), "f"(t[0]), "f"(t[1]), "f"(t[2]), "f"(t[3]), "f"(m), "f"(b1), "r"(c));
        b1 = fminf(b1, m);
        if (nib == 0) {
            gm = fminf(gm, m);
        } else {  // (branches on nib are warp-uniform)
            auto close = [&](float v) {
                asm volatile("st.shared.f32 [%0], %1;" ::"r"(row + 4u * (uint32_t)pend), "f"(v));
                ++pend;
            };
            if (nib & 1u) {
                close(gm);
                gm = INFINITY;
            }
            if (nib & 2u) {
                close(fminf(gm, t[0]));
                gm = t[1];
            } else {
                gm = fminf(gm, l0);
            }
            if (nib & 4u) {
                close(gm);
                gm = INFINITY;
            }
            if (nib & 8u) {
                close(fminf(gm, t[2]));
                gm = t[3];
            } else {
                gm = fminf(gm, l1);
            }
        }
    }
    // the winner's column (lowest among equal values)
    __device__ __forceinline__ int winner() const {
        float t0, t1, t2, t3;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(t0), "=f"(t1), "=f"(t2), "=f"(t3) : "r"(t4));
        if (b1 == INFINITY) return c4;
        return c4 + (t0 == b1 ? 0 : (t1 == b1 ? 1 : (t2 == b1 ? 2 : 3)));
    }
};

__device__ __forceinline__ float lds_f(uint32_t a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        cudaDriverEntryPointQueryResult q;
        void *f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    });
    return fn;
}

}  // namespace
}  // namespace kp
