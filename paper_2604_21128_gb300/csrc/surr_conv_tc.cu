// 3x3 periodic convolution of the learned surrogate on the fifth-generation
// tensor cores: an implicit GEMM
//   out[p, co] = sum_{tap, ci} w[co][tap][ci] * in[p shifted by tap, ci]
// with M = 128 pixels (an 8 x 16 pixel tile, one TMEM lane each) and N = NT
// output channels per tile.
//
// A tile's input is the 10 x 18 pixel patch around it, 32 channels (or the 16
// of the first layer) per slot, brought by one TMA box (the blocked layout's
// halo makes it a plain rectangle): [channel group][18 rows][10 pixels][16
// bytes].  Rows of eight pixels are 128 contiguous bytes, i.e. the 8-row core
// matrices of the no-swizzle K-major operand layout, image rows 160 bytes
// apart (SBO) and channel groups 2880 bytes apart (LBO), so each of the nine
// taps is the same patch at a different descriptor start.  A patch is 1.4
// times the tile's own pixels (a 128 x 1 row tile needs 3.05 times).
// Weights come as [tap][channel group][output channel][16 bytes] by bulk
// copies, one unit per tap and slot; where all units fit in shared memory
// they are loaded once per CTA, else they stream through a ring.
//
// CTAs are persistent over tiles and warp-specialised: one thread loads, one
// issues tcgen05.mma (K = 16 each), four warps run the epilogue from TMEM.
// Two accumulators alternate, so a tile's epilogue overlaps the next tile's
// MMAs.  The epilogue applies bias, skip and activation and writes the output
// with its halo, and in the same pass the 2x2 average pooling or the nearest
// upsampling that the next layer reads.
//
// Accumulation order: (32-channel slot, tap, K = 16 step) on widths that are
// multiples of 128, (tap, slot, step) on others.  With few channels the
// second order needs every slot of a tile resident; nothing else depends on
// it, but results are reproducible per width, whatever the tiling.
//
// What bounds it: for N = 16 or 32 the operand reads from shared memory (an
// MMA reads 4 KB of pixels for 16 K multiply-adds per output channel), for
// wider N the tensor pipe (conv_cost), and the epilogues.  Batch 8 at 256^2, us per
// layer: 30 18 18 17 21 26 42 39 34 24; with row patches and per-tap gathers, and
// separate pooling and upsampling, 53 32 41 47 47 90 131 113 93 71.
//
// Every wait on an mbarrier gives up after WAIT_NS of %globaltimer time; a CTA
// that gives up raises the caller's flag, lets its copies in flight land, frees
// its TMEM and returns.  After such a timeout the launch's outputs are
// undefined, and so is the TMEM it freed if the wait that ran out was on MMAs
// still in flight (a genuine hang of the tensor pipe rather than a phase that
// never comes): the caller should rebuild the network before trusting another
// result.
#include <cuda.h>

#include "surr_internal.h"

namespace surr {
namespace {

constexpr int PROWS = TY + 2, PCOLS = TX + 2;       // patch rows, pixels per row
constexpr int PROW_BYTES = PCOLS * 16;              // 160
constexpr int PGROUP_BYTES = PROWS * PROW_BYTES;    // 2880
constexpr int MAX_A = 16, MAX_B = 96;               // slots of the two rings
constexpr int EPI_WARPS = 8;                        // two per quarter of the TMEM lanes
constexpr int LOAD_WARP = EPI_WARPS, MMA_WARP = EPI_WARPS + 1;
constexpr int CONV_THREADS = 32 * (EPI_WARPS + 2);

// Test hook (surr_test_stall_conv): CTA 0 of each launch, or (2) of each
// EP_F32 launch, waits for a phase that never completes, so its bounded wait
// runs out; launches that find their flag raised do not.
__device__ int g_conv_tc_stall;

// Shared-memory matrix descriptor (tcgen05 format): start address, leading
// byte offset (K direction), stride byte offset (8-row direction), all in
// 16-byte units; descriptor version 1 at bit 46; no swizzle (bits 61-63 = 0).
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return uint64_t((addr >> 4) & 0x3FFFu) | (uint64_t((lbo >> 4) & 0x3FFFu) << 16) |
           (uint64_t((sbo >> 4) & 0x3FFFu) << 32) | (uint64_t(1) << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), BF16
// A and B (bits 7-9, 10-12 = 1), both K-major (bits 15, 16 = 0), N / 8 at
// bit 17, M / 16 at bit 24.
__device__ __forceinline__ uint32_t umma_idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(n >> 3) << 17) |
           (uint32_t(TM >> 4) << 24);
}

__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// D[tmem] (+)= A[smem] * B[smem]^T, one 128 x N x 16 step.
__device__ __forceinline__ void umma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                     uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(p));
    return p != 0;
}

// Arrive on the mbarrier once every MMA this thread issued so far is done.
__device__ __forceinline__ void umma_commit(uint64_t *b) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            smem_u32(b))
        : "memory");
}

// 16 consecutive FP32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// How a launch is laid out: NT output channels per tile (cout / NT slices),
// patches of kg channel groups, weight units of one tap and bc patches, na
// and nb ring slots (nb = every unit of a tile when resident), tiles per image
// row / column / launch, chunk_major order.
struct ConvPlan {
    int nt, slices, kg, chunks, bc, na, nb, resident, chunk_major, wbox;
    int ntx, nty, tiles, tcols;
};

// Store at *r, part of a pixel of a blocked plane (u parts per pixel), with
// the halo copies that `edge` names: bits 0-3: first column, last column,
// first row, last row of the image.
template <typename V>
__device__ __forceinline__ void put_edge(V *r, int u, unsigned edge, int H, int W, V v) {
    *r = v;
    if (edge == 0) return;
    const long long col = (long long)H * (W + 2) * u, row = (long long)W * u;
    if (edge & 1) r[row] = v;
    if (edge & 2) r[-row] = v;
    if (edge & 4) {
        V *q = r + col;
        *q = v;
        if (edge & 1) q[row] = v;
        if (edge & 2) q[-row] = v;
    }
    if (edge & 8) {
        V *q = r - col;
        *q = v;
        if (edge & 1) q[row] = v;
        if (edge & 2) q[-row] = v;
    }
}
__device__ __forceinline__ float2 unpack2(uint32_t w) {
    __nv_bfloat162 b;
    *reinterpret_cast<uint32_t *>(&b) = w;
    return make_float2(__bfloat162float(b.x), __bfloat162float(b.y));
}
__device__ __forceinline__ unsigned edge_of(int y, int x, int H, int W) {
    return (x == 0 ? 1u : 0u) | (x == W - 1 ? 2u : 0u) | (y == 0 ? 4u : 0u) |
           (y == H - 1 ? 8u : 0u);
}

// Output channels [c_lo, c_hi) of co0's tile for this thread's accumulator
// row (TMEM lane, pixel (y, x) of image b), by mode; `wait` returns once the
// accumulator is complete (false: give up).  bias points to the tile's biases
// in shared memory.  Every thread of the warp takes part in the loads and
// shuffles; only pixels of the image store.  What does not depend on the
// accumulator (addresses, edges, the first skip values) comes before the wait.
template <ConvMode MODE, typename Wait>
__device__ __forceinline__ bool epilogue(const ConvArgs &a, uint32_t tmem_row, int c_lo, int c_hi,
                                         int co0, const float *bias, int b, int y, int x,
                                         Wait wait) {
    const bool valid = y < a.H && x < a.W;
    const int G = a.cout / 8, g0 = (co0 + c_lo) / 8;
    if constexpr (MODE == EP_F32) {
        float4 *o = reinterpret_cast<float4 *>(a.out_f) +
                    2 * (((size_t(b) * G + g0) * a.H + y) * a.W + x);
        const size_t step = 2 * size_t(a.H) * a.W;
        if (!wait()) return false;
#pragma unroll 1
        for (int c0 = c_lo; c0 < c_hi; c0 += 16) {
            float v[16];
            tmem_ld16(tmem_row + uint32_t(c0), v);
#pragma unroll
            for (int h = 0; h < 2; ++h, o += step) {
                if (!valid) continue;
                o[0] = make_float4(v[8 * h], v[8 * h + 1], v[8 * h + 2], v[8 * h + 3]);
                o[1] = make_float4(v[8 * h + 4], v[8 * h + 5], v[8 * h + 6], v[8 * h + 7]);
            }
        }
    } else if constexpr (MODE == EP_OUT) {
        float *o = a.out_f + ((size_t(b) * a.H + y) * a.W + x) * a.n_out;
        if (!wait()) return false;
#pragma unroll 1
        for (int c0 = c_lo; c0 < c_hi; c0 += 16) {
            float v[16];
            tmem_ld16(tmem_row + uint32_t(c0), v);
            if (!valid) continue;
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (co0 + c0 + j < a.n_out) o[co0 + c0 + j] = v[j] + bias[c0 + j];
        }
    } else {
        const size_t step = plane8(0, 1, 1, a.H, a.W);
        const size_t at = plane8(b, g0, G, a.H, a.W) + pixel8(y, x, a.W);
        const uint4 *sk = reinterpret_cast<const uint4 *>(a.skip) + at;
        uint4 *o = reinterpret_cast<uint4 *>(a.out) + at;
        const unsigned edge = edge_of(y, x, a.H, a.W);
        const int h2 = a.H / 2, w2 = a.W / 2, H2 = 2 * a.H, W2 = 2 * a.W;
        const size_t pstep = plane8(0, 1, 1, h2, w2), ustep = plane8(0, 1, 1, H2, W2);
        uint4 *po = reinterpret_cast<uint4 *>(a.pool) + plane8(b, g0, G, h2, w2) +
                    pixel8(y / 2, x / 2, w2);
        const unsigned pedge = edge_of(y / 2, x / 2, h2, w2);
        uint4 *uo = reinterpret_cast<uint4 *>(a.up) + plane8(b, g0, G, H2, W2) +
                    pixel8(2 * y, 2 * x, W2);
        const bool skip = a.skip && valid;
        uint4 s0 = make_uint4(0, 0, 0, 0), s1 = s0, s2 = s0, s3 = s0;
        if (skip) {
            s0 = sk[0];
            s1 = sk[step];
            if (c_lo + 16 < c_hi) {
                s2 = sk[2 * step];
                s3 = sk[3 * step];
            }
        }
        if (!wait()) return false;
#pragma unroll 1
        for (int c0 = c_lo; c0 < c_hi; c0 += 16) {
            float v[16];
            tmem_ld16(tmem_row + uint32_t(c0), v);
            const uint4 sv[2] = {s0, s1};
            s0 = s2;
            s1 = s3;
            if (skip && c0 + 32 < c_hi) {   // skip values two rounds ahead
                s2 = sk[4 * step];
                s3 = sk[5 * step];
                sk += 2 * step;
            }
            const float4 *bb = reinterpret_cast<const float4 *>(bias + c0);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 t = bb[j];
                v[4 * j] += t.x;
                v[4 * j + 1] += t.y;
                v[4 * j + 2] += t.z;
                v[4 * j + 3] += t.w;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float q[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) q[j] = v[8 * h + j];
                if (a.skip) {
                    float s[8];
                    unpack8(sv[h], s);
#pragma unroll
                    for (int j = 0; j < 8; ++j) q[j] += s[j];
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) q[j] = q[j] > 0.f ? q[j] : LEAK * q[j];
                const uint4 r = pack8(q);
                if (valid) put_edge(o, 1, edge, a.H, a.W, r);
                o += step;
                if (a.up) {
                    if (valid) {
                        // the four copies touch the halo where this pixel does
                        put_edge(uo, 1, edge & 5, H2, W2, r);
                        put_edge(uo + 1, 1, edge & 6, H2, W2, r);
                        put_edge(uo + W2 + 2, 1, edge & 9, H2, W2, r);
                        put_edge(uo + W2 + 3, 1, edge & 10, H2, W2, r);
                    }
                    uo += ustep;
                }
                if (a.pool) {
                    // The tile's columns are one lane apart, its rows eight,
                    // and tiles start on even pixels: the four lanes of a
                    // pooled pixel swap words until each holds two channels
                    // of all four pixels.
                    const bool xo = x & 1, yo = y & 1;
                    const uint32_t k0 = xo ? r.z : r.x, k1 = xo ? r.w : r.y;
                    const uint32_t m0 = __shfl_xor_sync(0xffffffffu, xo ? r.x : r.z, 1);
                    const uint32_t m1 = __shfl_xor_sync(0xffffffffu, xo ? r.y : r.w, 1);
                    // (l, r): the row's left and right pixel, words 0 and 1
                    const uint32_t l0 = xo ? m0 : k0, l1 = xo ? m1 : k1;
                    const uint32_t r0 = xo ? k0 : m0, r1 = xo ? k1 : m1;
                    const uint32_t nl = __shfl_xor_sync(0xffffffffu, yo ? l0 : l1, 8);
                    const uint32_t nr = __shfl_xor_sync(0xffffffffu, yo ? r0 : r1, 8);
                    const uint32_t ml = yo ? l1 : l0, mr = yo ? r1 : r0;
                    const float2 p0 = unpack2(yo ? nl : ml), p1 = unpack2(yo ? nr : mr);
                    const float2 p2 = unpack2(yo ? ml : nl), p3 = unpack2(yo ? mr : nr);
                    const __nv_bfloat162 m =
                        __floats2bfloat162_rn(0.25f * (p0.x + p1.x + p2.x + p3.x),
                                              0.25f * (p0.y + p1.y + p2.y + p3.y));
                    if (valid)
                        put_edge(reinterpret_cast<uint32_t *>(po) + (xo ? 2 : 0) + (yo ? 1 : 0), 4,
                                 pedge, h2, w2, *reinterpret_cast<const uint32_t *>(&m));
                    po += pstep;
                }
            }
        }
    }
    return true;
}

template <ConvMode MODE>
__global__ void __launch_bounds__(CONV_THREADS)
k_conv3x3(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ CUtensorMap wmap,
          const ConvArgs a, const ConvPlan pl) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full_a[MAX_A], empty_a[MAX_A], full_b[MAX_B], empty_b[MAX_B];
    __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ __align__(16) float bias_s[256];

    // the warp index through a shuffle: its branches are then uniform
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int slice = int(blockIdx.x) % pl.slices, first = int(blockIdx.x) / pl.slices;
    const int stride = int(gridDim.x) / pl.slices;
    const int co0 = slice * pl.nt;
    const int items = first < pl.tiles ? (pl.tiles - 1 - first) / stride + 1 : 0;
    const int a_bytes = pl.kg * PGROUP_BYTES, b_bytes = pl.bc * pl.kg * pl.nt * 16;
    // TMA destinations must be 128-byte aligned (the launch adds the slack)
    unsigned char *smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    unsigned char *sa = smem, *sb = smem + pl.na * a_bytes;
    const volatile int *abort = &abort_flag;

    if (warp == LOAD_WARP) {
        for (int k = lane; k < pl.na; k += 32) {
            mbar_init(&full_a[k], 1);
            mbar_init(&empty_a[k], 1);
        }
        for (int k = lane; k < pl.nb; k += 32) {
            mbar_init(&full_b[k], 1);
            mbar_init(&empty_b[k], 1);
        }
        if (lane < 2) {
            mbar_init(&acc_full[lane], 1);
            mbar_init(&acc_empty[lane], EPI_WARPS);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid == 0) abort_flag = 0;
    if constexpr (MODE != EP_F32)
        if (tid < pl.nt) bias_s[tid] = a.bias[co0 + tid];
    if (warp == MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_slot)),
                     "r"(pl.tcols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == LOAD_WARP && lane == 0) {
        // loader: patches and weight units in the order the MMAs take them
        // (ring positions step; divisions would cost as much as a unit's MMAs)
        int as = 0, bs = 0, na_used = 0, nb_used = 0;   // slots, and how many ever filled
        uint32_t ap = 1, bp = 1;                        // parity of the slot's last release
        bool ok = true;
        const uint32_t w_bytes = uint32_t(pl.nt) * 16;
        const size_t w_group = size_t(a.cout) * 8, w_tap = w_group * (a.cin / 8);
        auto load_a = [&](int c, int tx, int ty, int b) {
            if (na_used == pl.na) ok = mbar_wait(&empty_a[as], ap, abort);
            else ++na_used;
            if (!ok) return;
            mbar_expect_tx(&full_a[as], uint32_t(a_bytes));
            // patch corner (-1, -1) of the tile is (0, 0) with the halo
            tma_load_4d(sa + as * a_bytes, &tmap, tx * TX * 2, ty * TY, c * pl.kg, b, &full_a[as]);
            if (++as == pl.na) { as = 0; ap ^= 1; }
        };
        auto load_b = [&](int tap, int c) {
            if (nb_used == pl.nb) ok = mbar_wait(&empty_b[bs], bp, abort);
            else ++nb_used;
            if (!ok) return;
            mbar_expect_tx(&full_b[bs], uint32_t(b_bytes));
            const bf16 *src = a.w + tap * w_tap + c * pl.kg * w_group + co0 * 8;
            unsigned char *dst = sb + bs * b_bytes;
            // one copy per unit: contiguous if it has every output channel,
            // else a box of channels x channel groups
            if (pl.slices == 1) bulk_load(dst, src, uint32_t(b_bytes), &full_b[bs]);
            else if (pl.wbox) tma_load_2d(dst, &wmap, co0 * 2, tap * (a.cin / 8) + c * pl.kg, &full_b[bs]);
            else
                for (int g = 0; g < pl.bc * pl.kg; ++g)
                    bulk_load(dst + g * w_bytes, src + g * w_group, w_bytes, &full_b[bs]);
            if (++bs == pl.nb) { bs = 0; bp ^= 1; }
        };
        for (int k = 0; k < items && ok; ++k) {
            int t = first + k * stride;
            const int tx = t % pl.ntx;
            t /= pl.ntx;
            const int ty = t % pl.nty, b = t / pl.nty;
            const bool weights = !pl.resident || k == 0;
            if (pl.chunk_major) {
                for (int c = 0; c < pl.chunks && ok; ++c) {
                    load_a(c, tx, ty, b);
                    for (int tap = 0; weights && tap < 9 && ok; ++tap) load_b(tap, c);
                }
            } else {
                for (int tap = 0; tap < 9 && ok; ++tap)
                    for (int c = 0; c < pl.chunks && ok; ++c) {
                        if (tap == 0) load_a(c, tx, ty, b);
                        if (weights && ok && c % pl.bc == 0) load_b(tap, c);
                    }
            }
        }
        if (!ok) abort_flag = 1;
        // every copy lands (bounded) before the CTA's shared memory is
        // released, also on the way out after a timeout: the slots filled
        // last, newest first (a slot's fill has the parity its release will)
        for (int i = 0; i < na_used; ++i) {
            if (as == 0) { as = pl.na; ap ^= 1; }
            mbar_wait(&full_a[--as], ap ^ 1);
        }
        for (int i = 0; i < nb_used; ++i) {
            if (bs == 0) { bs = pl.nb; bp ^= 1; }
            mbar_wait(&full_b[--bs], bp ^ 1);
        }
    } else if (warp == MMA_WARP) {
        // The whole warp runs the loop, one elected lane issues: branches and
        // descriptors are then uniform.  Descriptors step by precomputed
        // offsets: a unit's two MMAs take 80 (N = 32) to 256 cycles, which a
        // few dozen dependent integer instructions of a single warp exceed
        // (with divisions in the loop a unit took 1000 to 1500).
        const bool leader = elect_one();
        const uint32_t idesc = umma_idesc(pl.nt);
        const uint64_t a0 = umma_desc(smem_u32(sa), PGROUP_BYTES, PROW_BYTES);
        const uint64_t b0 = umma_desc(smem_u32(sb), uint32_t(pl.nt) * 16, 128);
        const uint32_t a_step = uint32_t(a_bytes) / 16, b_step = uint32_t(b_bytes) / 16;
        const uint32_t bk = uint32_t(pl.nt) * 2;   // two channel groups on
        const bool two = pl.kg == 4, stream = !pl.resident;
        int as = 0, bs = 0;
        uint32_t ap = 0, bp = 0;
        bool ok = true;
        auto wait = [&](uint64_t *bar, uint32_t parity) {
            ok = __all_sync(0xffffffffu, mbar_wait(bar, parity, abort));
            tc_fence_after();
        };
        for (int k = 0; k < items && ok; ++k) {
            const int buf = k & 1;
            if (k >= 2) wait(&acc_empty[buf], uint32_t(k / 2 - 1) & 1);
            if (!ok) break;
            const uint32_t d = tmem + uint32_t(buf * pl.nt);
            const bool weights = stream || k == 0;   // weight units to wait for
            uint32_t acc = 0;
            if (!stream) bs = 0;
            constexpr uint32_t ROW = PROW_BYTES / 16;
            if (pl.chunk_major) {
                for (int c = 0; c < pl.chunks && ok; ++c) {
                    wait(&full_a[as], ap);
                    if (!ok) break;
                    const uint64_t da = a0 + uint64_t(as * a_step);
                    if (!weights) {
                        // resident weights: nothing to wait for within a patch
                        if (leader) {
                            uint64_t db = b0 + uint64_t(c * 9 * b_step);
#pragma unroll
                            for (int tap = 0; tap < 9; ++tap, db += b_step) {
                                const uint32_t off = (tap / 3) * ROW + tap % 3;
                                umma(d, da + off, db, idesc, tap > 0 ? 1 : acc);
                                if (two)
                                    umma(d, da + (off + 2 * PGROUP_BYTES / 16), db + bk, idesc, 1);
                            }
                        }
                        acc = 1;
                    } else {
#pragma unroll
                        for (int tap = 0; tap < 9; ++tap) {
                            const uint32_t off = (tap / 3) * ROW + tap % 3;
                            if (ok) wait(&full_b[bs], stream ? bp : 0);
                            if (ok && leader) {
                                const uint64_t db = b0 + uint64_t(bs * b_step);
                                umma(d, da + off, db, idesc, acc);
                                if (two)
                                    umma(d, da + (off + 2 * PGROUP_BYTES / 16), db + bk, idesc, 1);
                                if (stream) umma_commit(&empty_b[bs]);
                            }
                            acc = 1;
                            if (++bs == pl.nb) { bs = 0; bp ^= 1; }
                        }
                    }
                    if (ok && leader) umma_commit(&empty_a[as]);
                    if (++as == pl.na) { as = 0; ap ^= 1; }
                }
            } else {
                // the tile's patches are slots as .. as + chunks - 1 (na is a
                // multiple of chunks)
#pragma unroll 1
                for (int tap = 0; tap < 9 && ok; ++tap) {
                    uint64_t da = a0 + uint64_t(as * a_step + (tap / 3) * ROW + tap % 3);
                    for (int c = 0; c < pl.chunks; c += pl.bc) {
                        if (tap == 0)
                            for (int e = 0; e < pl.bc && ok; ++e) wait(&full_a[as + c + e], ap);
                        if (ok && weights) wait(&full_b[bs], stream ? bp : 0);
                        if (!ok) break;
                        if (leader) {
                            uint64_t db = b0 + uint64_t(bs * b_step);
                            // bc is 1, 2 or 4 patches
                            for (int e = 0; e < pl.bc; ++e) {
                                umma(d, da, db, idesc, acc);
                                if (two) umma(d, da + 2 * PGROUP_BYTES / 16, db + bk, idesc, 1);
                                acc = 1;
                                da += a_step;
                                db += 2 * bk;
                            }
                            if (stream) umma_commit(&empty_b[bs]);
                        }
                        if (++bs == pl.nb) { bs = 0; bp ^= 1; }
                    }
                }
                if (ok && leader)
                    for (int c = 0; c < pl.chunks; ++c) umma_commit(&empty_a[as + c]);
                as += pl.chunks;
                if (as == pl.na) { as = 0; ap ^= 1; }
            }
            if (ok && leader) umma_commit(&acc_full[buf]);
        }
        if (!ok) abort_flag = 1;
    } else if (warp < EPI_WARPS) {
        // warps w and w + 4 share TMEM lanes and split the channels
        const int part = warp >> 2, row = (warp & 3) * 32 + lane;
        const int c_lo = pl.nt >= 32 ? part * (pl.nt / 2) : 0;
        const int c_hi = pl.nt >= 32 ? c_lo + pl.nt / 2 : part == 0 ? pl.nt : 0;
        bool ok = true;
        for (int k = 0; k < items && ok; ++k) {
            const int buf = k & 1;
            int t = first + k * stride;
            const int tx = t % pl.ntx;
            t /= pl.ntx;
            const int ty = t % pl.nty, b = t / pl.nty;
            ok = epilogue<MODE>(
                a, tmem + uint32_t(buf * pl.nt) + (uint32_t((warp & 3) * 32) << 16), c_lo, c_hi,
                co0, bias_s, b, ty * TY + (row >> 3), tx * TX + (row & 7), [&] {
                    // tcgen05.ld is warp-collective: decide for the whole warp
                    const bool f = __all_sync(0xffffffffu,
                                              mbar_wait(&acc_full[buf], (k / 2) & 1, abort));
                    tc_fence_after();
                    return f;
                });
            if (!ok) break;
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[buf]);
        }
        if (ok && items > 0 && blockIdx.x == 0 && g_conv_tc_stall != 0 &&
            (MODE == EP_F32 || g_conv_tc_stall == 1) &&
            *static_cast<const volatile int *>(a.err) == 0)
            // the phase after the last one never completes
            ok = mbar_wait(&acc_full[(items - 1) & 1], (((items - 1) / 2) + 1) & 1, abort);
        if (!ok) abort_flag = 1;
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && abort_flag) atomicExch(a.err, 1);
    if (warp == MMA_WARP)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(pl.tcols)
                     : "memory");
}

using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                 const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                 const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                 CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's tensor-map encoder, looked up once through the runtime.
EncodeTiled encode_tiled() {
    static EncodeTiled fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return EncodeTiled(nullptr);
        return reinterpret_cast<EncodeTiled>(p);
    }();
    return fn;
}

// Weights [tap][cin / 8][cout][8] as rows of output channels: boxes of nt
// channels x kg groups.
bool weight_map(CUtensorMap *map, const bf16 *w, int cout, int cin, int nt, int kg) {
    const EncodeTiled enc = encode_tiled();
    if (!enc || (reinterpret_cast<uintptr_t>(w) & 15)) return false;
    const cuuint64_t dims[2] = {cuuint64_t(cout) * 2, cuuint64_t(9 * (cin / 8))};
    const cuuint64_t strides[1] = {cuuint64_t(cout) * 16};
    const cuuint32_t box[2] = {cuuint32_t(nt * 2), cuuint32_t(kg)};
    const cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, const_cast<bf16 *>(w), dims, strides, box,
               estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Streaming multiprocessors of the current device, read once.
int sm_count() {
    static const int n = [] {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1)
            return 1;
        return v;
    }();
    return n;
}

// Rounds of tiles per SM times a tile's MMAs times what one takes: 32 cycles
// to read 128 pixels x 16 channels from shared memory at 128 bytes a cycle,
// NT / 4 for the weights, against NT / 2 in the tensor pipe.
long long conv_cost(int tiles, int slices, int nt, int sms) {
    const long long rounds = ((long long)tiles * slices + sms - 1) / sms;
    return rounds * std::max(32 + nt / 4, nt / 2);
}

// The layout of slices of pl->nt output channels: false where not even three
// weight units fit beside the patches that have to be resident together (cin
// = 512 with NT = 256 and the taps outermost, the one such pair).
bool lay_out(const ConvArgs &a, ConvPlan *pl, int *smem, int *per_sm) {
    pl->slices = a.cout / pl->nt;
    pl->tcols = std::max(32, 2 * pl->nt);
    // slots of a tile that must be resident together: all of them when the
    // taps are outermost; a weight unit then covers four patches (eight MMAs
    // per wait: with two, the waits and ring steps of a single warp, 400 to
    // 500 cycles per unit, took longer than the MMAs)
    pl->chunk_major = a.W % 128 == 0 || pl->chunks > MAX_A;
    const int need = pl->chunk_major ? 1 : pl->chunks;
    pl->bc = 1;
    const int a_bytes = pl->kg * PGROUP_BYTES;
    // (four ring slots of it have to fit beside a tile's patches)
    if (!pl->chunk_major)
        while (pl->bc < 4 && pl->chunks % (2 * pl->bc) == 0 &&
               4 * (2 * pl->bc * pl->kg * pl->nt * 16) + need * a_bytes <= 222 * 1024)
            pl->bc *= 2;
    const int units = 9 * pl->chunks / pl->bc;
    const int b_bytes = pl->bc * pl->kg * pl->nt * 16;
    // two CTAs per SM where weights and a few patches fit twice, else one;
    // weights resident where they fit, else a ring of what is left
    for (int c = 2; c >= 1; --c) {
        const int budget = (c == 2 ? 110 : 222) * 1024;
        if (pl->tcols * c > 512) continue;
        // patches in whole tiles where the taps are outermost
        const int most = pl->chunk_major ? 4 : 2 * need;
        if (units <= MAX_B && units * b_bytes + (need + (pl->chunk_major ? 1 : 0)) * a_bytes <=
                                  budget) {
            pl->resident = 1;
            pl->nb = units;
            pl->na = std::min(std::min(MAX_A, most), (budget - units * b_bytes) / a_bytes);
        } else if (c == 1) {
            pl->resident = 0;
            pl->na = std::min(std::min(MAX_A, most), (budget - 3 * b_bytes) / a_bytes);
            if (pl->na < need) return false;
            if (!pl->chunk_major) pl->na = pl->na / need * need;
            pl->nb = std::min(std::min(units, MAX_B), (budget - pl->na * a_bytes) / b_bytes);
        } else {
            continue;
        }
        if (!pl->chunk_major) pl->na = pl->na / need * need;
        *smem = 128 + pl->na * a_bytes + pl->nb * b_bytes;
        *per_sm = c;
        return true;
    }
    return false;
}

// The cheapest NT (conv_cost; the wider one of equals) that has a layout.
bool plan_conv(const ConvArgs &a, ConvPlan *pl, int *smem, int *per_sm) {
    const int sms = sm_count();
    pl->ntx = (a.W + TX - 1) / TX;
    pl->nty = (a.H + TY - 1) / TY;
    pl->tiles = a.B * pl->ntx * pl->nty;
    pl->kg = a.cin % 32 == 0 ? 4 : 2;
    pl->chunks = a.cin / (8 * pl->kg);
    ConvPlan t = *pl;
    long long best = -1;
    for (t.nt = 256; t.nt >= 16; t.nt /= 2) {
        if (a.cout % t.nt || (t.nt < 32 && a.cout >= 32)) continue;
        const long long cost = conv_cost(t.tiles, a.cout / t.nt, t.nt, sms);
        int bytes, ctas;
        if ((best >= 0 && cost >= best) || !lay_out(a, &t, &bytes, &ctas)) continue;
        best = cost;
        *pl = t;
        *smem = bytes;
        *per_sm = ctas;
    }
    return best >= 0;
}

template <ConvMode MODE>
cudaError_t launch_conv(const ConvArgs &a, cudaStream_t st) {
    auto k = k_conv3x3<MODE>;
    static const cudaError_t attr = [&] {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             224 * 1024);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     int(cudaSharedmemCarveoutMaxShared));
        return e;
    }();
    if (attr != cudaSuccess) return attr;
    ConvPlan pl;
    int smem = 0, per_sm = 0;
    CUtensorMap map;
    if (!plan_conv(a, &pl, &smem, &per_sm)) return cudaErrorInvalidConfiguration;
    if (!blocked_map(&map, a.in, a.B, a.cin, a.H, a.W, true, PCOLS, PROWS, pl.kg))
        return cudaErrorNotSupported;
    pl.wbox = pl.slices > 1 && pl.nt <= 128;
    CUtensorMap wmap = map;
    if (pl.wbox && !weight_map(&wmap, a.w, a.cout, a.cin, pl.nt, pl.bc * pl.kg))
        return cudaErrorNotSupported;
    // whole slices: every slice gets the same number of CTAs
    int per_slice = std::max(1, sm_count() * per_sm / pl.slices);
    if (per_slice > pl.tiles) per_slice = pl.tiles;
    k<<<unsigned(per_slice) * unsigned(pl.slices), CONV_THREADS, smem, st>>>(map, wmap, a, pl);
    return cudaGetLastError();
}

}  // namespace

bool blocked_map(CUtensorMap *map, const bf16 *t, int B, int C, int H, int W, bool halo, int bx,
                 int by, int bg) {
    const EncodeTiled enc = encode_tiled();
    if (!enc || (reinterpret_cast<uintptr_t>(t) & 15)) return false;
    const cuuint64_t row = cuuint64_t(W + 2) * 16, plane = cuuint64_t(H + 2) * row;
    const int G = C / 8;
    // (a pixel is two 8-byte elements: boxes of up to 128 pixels)
    const cuuint64_t dims[4] = {cuuint64_t(halo ? W + 2 : W) * 2, cuuint64_t(halo ? H + 2 : H),
                                cuuint64_t(G), cuuint64_t(B)};
    const cuuint64_t strides[3] = {row, plane, plane * cuuint64_t(G)};
    const cuuint32_t box[4] = {cuuint32_t(bx * 2), cuuint32_t(by), cuuint32_t(bg), 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const bf16 *base = halo ? t : t + (size_t(W + 2) + 1) * 8;
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 4, const_cast<bf16 *>(base), dims, strides,
               box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t conv3x3(const ConvArgs &a, ConvMode mode, cudaStream_t st) {
    if (a.cin % 16 || (a.cin > 16 && a.cin % 32) || a.cout % 16) return cudaErrorInvalidValue;
    switch (mode) {
    case EP_ACT: return launch_conv<EP_ACT>(a, st);
    case EP_F32: return launch_conv<EP_F32>(a, st);
    default: return launch_conv<EP_OUT>(a, st);
    }
}

cudaError_t conv_tc_stall(int on) {
    return cudaMemcpyToSymbol(g_conv_tc_stall, &on, sizeof(int));
}

}  // namespace surr
