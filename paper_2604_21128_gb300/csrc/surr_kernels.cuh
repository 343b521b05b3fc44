// Kernels of the learned surrogate (a convolutional operator that advances
// the QLA state K steps at once).  Every contraction accumulates in FP32 on
// the tensor cores (tcgen05.mma with a TMEM accumulator for the convolutions,
// mma.sync m16n8k16 for the weight gradient).  3x3 convolutions wrap
// periodically, like the lattice.
//
// Layouts.  BF16 activations and pre-activation gradients are blocked by
// eight channels with a one-pixel periodic halo: [image][channel / 8]
// [H + 2][W + 2][8], the halo holding copies of the opposite edge, written
// with the interior.  A convolution tile's input -- any rectangle with its
// 3x3 neighbours -- is then one box of a tensor map: no wrapping in the
// loader, and a pixel's eight channels are the 16 bytes of one row of a
// tensor-core operand.  FP32 gradients are blocked the same way without the
// halo: [image][channel / 8][H][W][8].
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace surr {

using bf16 = __nv_bfloat16;

constexpr float LEAK = 0.1f;   // leaky-ReLU slope

// ---------------------------------------------------------------------------
// Warp-level tensor-core helpers.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_u32(const void *p) {
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void ldsm_x4_t(unsigned (&r)[4], const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_u32(p)));
}

// D += A (16x16, row) * B (16x8, col), BF16 in, FP32 accumulate.
__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4], unsigned b0,
                                         unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void cp16(void *smem, const void *gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem)), "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Start of channel group g (of G) of image b of a blocked BF16 tensor, in
// 16-byte pixels.
__device__ __forceinline__ size_t plane8(int b, int g, int G, int H, int W) {
    return (size_t(b) * G + g) * size_t(H + 2) * size_t(W + 2);
}
__device__ __forceinline__ size_t pixel8(int y, int x, int W) {
    return size_t(y + 1) * (W + 2) + (x + 1);
}

// Eight channels of pixel (y, x) into a blocked plane, halo copies included.
__device__ __forceinline__ void put8(uint4 *plane, int y, int x, int H, int W, uint4 v) {
    uint4 *r = plane + pixel8(y, x, W);
    const bool left = x == 0, right = x == W - 1;
    *r = v;
    if (left) r[W] = v;
    if (right) r[-W] = v;
    const long long col = (long long)H * (W + 2);
    if (y == 0) {
        uint4 *q = r + col;
        *q = v;
        if (left) q[W] = v;
        if (right) q[-W] = v;
    }
    if (y == H - 1) {
        uint4 *q = r - col;
        *q = v;
        if (left) q[W] = v;
        if (right) q[-W] = v;
    }
}

__device__ __forceinline__ void unpack8(uint4 u, float (&v)[8]) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        __nv_bfloat162 b;
        *reinterpret_cast<uint32_t *>(&b) = w[j];
        v[2 * j] = __bfloat162float(b.x);
        v[2 * j + 1] = __bfloat162float(b.y);
    }
}

__device__ __forceinline__ uint4 pack8(const float (&v)[8]) {
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
        w[j] = *reinterpret_cast<const uint32_t *>(&b);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// ---------------------------------------------------------------------------
// mbarriers and TMA.
// ---------------------------------------------------------------------------
constexpr unsigned long long WAIT_NS = 2000000000ull;   // a wait gives up after 2 s
// How long one try may suspend the thread: waiting warps that poll instead
// slow down the warps they wait for.
constexpr unsigned TRY_NS = 1000000;

__device__ __forceinline__ void mbar_init(uint64_t *b, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t a, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(a), "r"(parity), "r"(TRY_NS)
        : "memory");
    return done != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Wait for the phase of the given parity; false once WAIT_NS of wall time
// have passed (try_wait may suspend the thread for a while on each call, so
// the bound is on time, not on the number of calls) or *abort is raised.
__device__ __forceinline__ bool mbar_wait(uint64_t *b, uint32_t parity,
                                          const volatile int *abort = nullptr) {
    const uint32_t a = smem_u32(b);
    if (mbar_try(a, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (;;) {
        if (mbar_try(a, parity)) return true;
        if (abort && *abort) return false;
        if (global_ns() - t0 > WAIT_NS) return false;
    }
}
// 4-D tiled TMA load into shared memory, completing on the mbarrier's
// transaction count.
__device__ __forceinline__ void tma_load_4d(void *dst, const void *map, int c0, int c1, int c2,
                                            int c3, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
        "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void tma_load_2d(void *dst, const void *map, int c0, int c1,
                                            uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(smem_u32(bar))
        : "memory");
}
// `bytes` contiguous bytes (a multiple of 16, 16-byte aligned).
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes,
                                          uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

}  // namespace surr
