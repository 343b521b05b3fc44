// Kernels of the learned surrogate around the tcgen05 convolution
// (surr_conv_tc.cu): the weight gradient as a split-K GEMM over the pixels
// (warp-level mma.sync), the activation backward with the gradients of
// pooling and upsampling folded in, loss, Adam and the layout conversions.
#include "surr_internal.h"

namespace surr {
namespace {

// ---------------------------------------------------------------------------
// Weight gradient: part[split][co][tap][ci] = sum over this split's pixels p
// of dz[p][co] * in[p shifted by tap][ci].  Splits are contiguous ranges of
// the linear pixel index, summed in order in K = 16 steps of 16 consecutive
// pixels, whichever kernel runs.
//
// Where rows are multiples of 16 pixels: a CTA takes 16 MT CW output channels
// x 8 IW input channels and all nine taps.  Per stage (up to 64 pixels of one
// row, or the 64 / w whole rows of narrow images) TMA brings the pixels of dz
// and the patch of the input around them once; a pixel's eight channels are
// 16 bytes, so eight consecutive pixels are what a transposing ldmatrix takes
// without bank conflicts, and the taps are the same patch at shifted
// addresses.  Warp (cw, iw) owns channels 16 MT cw.. x 8 iw.. of all taps:
// MT + 4.5 ldmatrix.x4 for 9 MT MMAs per K step.  (A CTA per tap that loads
// both operands again each time took 1395 us per training step at batch 8,
// 256^2; it remains below for other widths.)
// ---------------------------------------------------------------------------
constexpr int DW_STAGES = 4, DW_PIX = 64;

// Stage geometry of a level w pixels wide: segments of sw pixels, sr rows.
struct DwGeom {
    int w, h, sw, sr;
    __host__ __device__ int z_group() const { return sw * sr * 16; }          // bytes
    __host__ __device__ int i_row() const { return (sw + 2) * 16; }
    __host__ __device__ int i_group() const { return (sr + 2) * i_row(); }
};

// Walks a split's pixels stage by stage.
struct DwWalk {
    long long p, end;
    int x, y, b;
    __device__ DwWalk(const DwGeom &g, long long q0, long long q1) : p(q0), end(q1) {
        const long long row = q0 / g.w;
        x = int(q0 - row * g.w);
        b = int(row / g.h);
        y = int(row - (long long)b * g.h);
    }
    __device__ bool done() const { return p >= end; }
    // pixels of the stage at the current position
    __device__ int len(const DwGeom &g) const {
        if (g.sr > 1) return DW_PIX;
        int n = min(g.sw, g.w - x);
        if (end - p < n) n = int(end - p);
        return n;
    }
    __device__ void next(const DwGeom &g) {
        const int n = len(g);
        p += n;
        if (g.sr > 1) {
            y += g.sr;
        } else {
            x += n;
            if (x == g.w) { x = 0; ++y; }
        }
        if (y == g.h) { y = 0; ++b; }
    }
};

template <int MT, int CW, int IW>
__global__ void __launch_bounds__(32 * CW * IW)
k_dw(const __grid_constant__ CUtensorMap zmap, const __grid_constant__ CUtensorMap imap,
     const DwGeom g, long long P, long long per, int cout, int cin, float *__restrict__ part,
     int *err) {
    constexpr int COT = 16 * MT * CW, CIT = 8 * IW;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full[DW_STAGES];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cw = warp % CW, iw = warp / CW;
    const int ci0 = int(blockIdx.x) * CIT, co0 = int(blockIdx.y) * COT, split = int(blockIdx.z);
    const int z_bytes = 2 * MT * CW * g.z_group(), i_bytes = IW * g.i_group();
    const int stage_bytes = (z_bytes + i_bytes + 127) / 128 * 128;
    unsigned char *smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    if (tid == 0) {
        for (int k = 0; k < DW_STAGES; ++k) mbar_init(&full[k], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    const long long q0 = split * per, q1 = min(P, q0 + per);
    DwWalk here(g, q0, q1), ahead(here);
    int loaded = 0;   // by thread 0
    auto load = [&]() {
        const int s = loaded % DW_STAGES;
        mbar_expect_tx(&full[s], uint32_t(z_bytes + i_bytes));
        tma_load_4d(smem + s * stage_bytes, &zmap, ahead.x * 2, ahead.y, co0 / 8, ahead.b,
                    &full[s]);
        tma_load_4d(smem + s * stage_bytes + z_bytes, &imap, ahead.x * 2, ahead.y, ci0 / 8,
                    ahead.b, &full[s]);
        ahead.next(g);
        ++loaded;
    };
    if (tid == 0)
        while (loaded < DW_STAGES - 1 && !ahead.done()) load();

    float acc[MT][9][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int t = 0; t < 9; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[m][t][e] = 0.f;

    // ldmatrix rows: this lane's matrix and pixel.  dz: matrices (channels
    // 0-7, pixels 0-7), (8-15, 0-7), (0-7, 8-15), (8-15, 8-15); input: two
    // taps at a time, pixels 0-7 and 8-15 of each.
    const int mi = lane >> 3, mr = (lane & 7) * 16;
    const int zoff = (2 * MT * cw + (mi & 1)) * g.z_group() + (mi >> 1) * 128 + mr;
    int ioff[5];
#pragma unroll
    for (int u = 0; u < 5; ++u) {
        const int t = min(2 * u + (mi >> 1), 8);
        ioff[u] = z_bytes + iw * g.i_group() + (t / 3) * g.i_row() + (t % 3) * 16 + (mi & 1) * 128 +
                  mr;
    }
    bool ok = true;
    for (int k = 0; !here.done(); ++k) {
        const int s = k % DW_STAGES;
        ok = mbar_wait(&full[s], uint32_t(k / DW_STAGES) & 1);
        // every warp is done with the stage before, which the next load takes
        if (!__syncthreads_and(ok)) { ok = false; break; }
        if (tid == 0 && !ahead.done()) load();
        const unsigned char *st = smem + s * stage_bytes;
        const int steps = here.len(g) / 16;
        int col = 0, pix = 0;   // of the step: column in the row, offset in the patch
        for (int j = 0; j < steps; ++j) {
            unsigned a[MT][4], b[5][4];
#pragma unroll
            for (int m = 0; m < MT; ++m)
                ldsm_x4_t(a[m], st + zoff + 2 * m * g.z_group() + j * 256);
#pragma unroll
            for (int u = 0; u < 5; ++u) ldsm_x4_t(b[u], st + ioff[u] + pix);
#pragma unroll
            for (int t = 0; t < 9; ++t)
#pragma unroll
                for (int m = 0; m < MT; ++m)
                    mma_bf16(acc[m][t], a[m], b[t / 2][2 * (t & 1)], b[t / 2][2 * (t & 1) + 1]);
            col += 16;
            pix += 256;
            if (col == g.sw) { col = 0; pix += 32; }   // past the row's two halo pixels
        }
        here.next(g);
    }
    if (!ok) {
        if (tid == 0) {
            atomicExch(err, 1);
            // copies in flight land (bounded) before shared memory is released
            for (int k = loaded > DW_STAGES ? loaded - DW_STAGES : 0; k < loaded; ++k)
                mbar_wait(&full[k % DW_STAGES], uint32_t(k / DW_STAGES) & 1);
        }
        return;
    }
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int co = co0 + 16 * (MT * cw + m) + (lane >> 2) + 8 * half;
            const int ci = ci0 + 8 * iw + (lane & 3) * 2;
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                float *o = part + (((size_t(split) * cout + co) * 9 + t) * cin + ci);
                *reinterpret_cast<float2 *>(o) =
                    make_float2(acc[m][t][half * 2], acc[m][t][half * 2 + 1]);
            }
        }
}

// Any width: CTA tile MT co x NT ci of one tap, 4 warps (2 x 2), stages of 64
// pixels gathered by cp.async, operands pixel-major for transposing ldmatrix.
template <int MT, int NT>
__global__ void __launch_bounds__(128)
k_dw_any(const bf16 *__restrict__ dz, const bf16 *__restrict__ in, int H, int W, long long P,
         long long per, int cout, int cin, float *__restrict__ part) {
    __shared__ __align__(16) bf16 As[2][DW_PIX][MT + 8];
    __shared__ __align__(16) bf16 Bs[2][DW_PIX][NT + 8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = warp & 1, wn = warp >> 1;
    const int ci0 = blockIdx.x * NT, co0 = blockIdx.y * MT;
    const int splits = int(gridDim.z / 9);
    const int tap = blockIdx.z / splits, split = blockIdx.z - tap * splits;
    const int dy = tap / 3 - 1, dx = tap % 3 - 1;
    const long long q0 = split * per, q1 = min(P, q0 + per);
    const uint4 *z8 = reinterpret_cast<const uint4 *>(dz);
    const uint4 *i8 = reinterpret_cast<const uint4 *>(in);

    auto load = [&](int s, long long pb) {
        constexpr int ACH = MT / 8, BCH = NT / 8;
        auto at = [&](long long p, int &b, int &y, int &x) {
            b = int(p / ((long long)H * W));
            const int rem = int(p - (long long)b * H * W);
            y = rem / W;
            x = rem - y * W;
        };
        int b, y, x;
        for (int c = tid; c < DW_PIX * ACH; c += 128) {
            const int r = c % DW_PIX, h = c / DW_PIX;
            const long long p = pb + r;
            if (p < q1) {
                at(p, b, y, x);
                cp16(&As[s][r][h * 8], z8 + plane8(b, co0 / 8 + h, cout / 8, H, W) + pixel8(y, x, W));
            } else {
                *reinterpret_cast<uint4 *>(&As[s][r][h * 8]) = make_uint4(0, 0, 0, 0);
            }
        }
        for (int c = tid; c < DW_PIX * BCH; c += 128) {
            const int r = c % DW_PIX, h = c / DW_PIX;
            const long long p = pb + r;
            if (p < q1) {
                at(p, b, y, x);
                cp16(&Bs[s][r][h * 8],
                     i8 + plane8(b, ci0 / 8 + h, cin / 8, H, W) + pixel8(y + dy, x + dx, W));
            } else {
                *reinterpret_cast<uint4 *>(&Bs[s][r][h * 8]) = make_uint4(0, 0, 0, 0);
            }
        }
        cp_commit();
    };

    constexpr int MI = MT / 32, NI = NT / 16;  // per warp: MT/2 rows, NT/2 cols
    float acc[MI][NI][4];
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < NI; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;

    const long long nst = q1 > q0 ? (q1 - q0 + DW_PIX - 1) / DW_PIX : 0;
    if (nst > 0) load(0, q0);
    for (long long st = 0; st < nst; ++st) {
        const int s = int(st & 1);
        if (st + 1 < nst) {
            load(s ^ 1, q0 + (st + 1) * DW_PIX);
            cp_wait<1>();
        } else {
            cp_wait<0>();
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < DW_PIX / 16; ++kk) {
            unsigned a[MI][4];
#pragma unroll
            for (int m = 0; m < MI; ++m)
                ldsm_x4_t(a[m], &As[s][kk * 16 + (lane & 7) + ((lane >> 4) << 3)]
                                  [wm * (MT / 2) + m * 16 + ((lane >> 3) & 1) * 8]);
#pragma unroll
            for (int nj = 0; nj < NI / 2; ++nj) {
                unsigned bfr[4];
                ldsm_x4_t(bfr, &Bs[s][kk * 16 + (lane & 7) + ((lane >> 3) & 1) * 8]
                                 [wn * (NT / 2) + nj * 16 + ((lane >> 4) << 3)]);
#pragma unroll
                for (int m = 0; m < MI; ++m) {
                    mma_bf16(acc[m][2 * nj], a[m], bfr[0], bfr[1]);
                    mma_bf16(acc[m][2 * nj + 1], a[m], bfr[2], bfr[3]);
                }
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int m = 0; m < MI; ++m)
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int co = co0 + wm * (MT / 2) + m * 16 + (lane >> 2) + half * 8;
#pragma unroll
            for (int ni = 0; ni < NI; ++ni) {
                const int ci = ci0 + wn * (NT / 2) + ni * 8 + (lane & 3) * 2;
                float *o = part + ((size_t(split) * cout + co) * 9 + tap) * cin + ci;
                *reinterpret_cast<float2 *>(o) =
                    make_float2(acc[m][ni][half * 2], acc[m][ni][half * 2 + 1]);
            }
        }
}

template <int MT, int CW, int IW>
cudaError_t launch_dw(const bf16 *dz, const bf16 *in, int B, const DwGeom &g, int cout, int cin,
                      int splits, long long per, float *part, int *err, cudaStream_t st) {
    auto k = k_dw<MT, CW, IW>;
    const int smem = 128 + DW_STAGES * ((2 * MT * CW * g.z_group() + IW * g.i_group() + 127) / 128 *
                                        128);
    static const cudaError_t attr =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
    if (attr != cudaSuccess) return attr;
    CUtensorMap zmap, imap;
    if (!blocked_map(&zmap, dz, B, cout, g.h, g.w, false, g.sw, g.sr, 2 * MT * CW) ||
        !blocked_map(&imap, in, B, cin, g.h, g.w, true, g.sw + 2, g.sr + 2, IW))
        return cudaErrorNotSupported;
    k<<<dim3(unsigned(cin / (8 * IW)), unsigned(cout / (16 * MT * CW)), unsigned(splits)),
        32 * CW * IW, smem, st>>>(zmap, imap, g, (long long)B * g.h * g.w, per, cout, cin, part,
                                  err);
    return cudaGetLastError();
}

// Output channels 64 (two 32-channel warps), 32 or 16 per CTA times 8 IW
// input channels.
template <int IW>
cudaError_t launch_dw_co(const bf16 *dz, const bf16 *in, int B, const DwGeom &g, int cout, int cin,
                         int splits, long long per, float *part, int *err, cudaStream_t st) {
    if (cout % 64 == 0 && IW == 4)
        return launch_dw<2, 2, IW>(dz, in, B, g, cout, cin, splits, per, part, err, st);
    if (cout % 32 == 0)
        return launch_dw<2, 1, IW>(dz, in, B, g, cout, cin, splits, per, part, err, st);
    return launch_dw<1, 1, IW>(dz, in, B, g, cout, cin, splits, per, part, err, st);
}

// Sums over splits of many arrays: grid.y picks the array.  Many splits of
// few values (tree) are summed as 256 strided partial sums and a binary tree
// over them, 32 values per block; others in order.
__global__ void __launch_bounds__(256) k_sum_splits(const __grid_constant__ SumJobs jobs) {
    __shared__ float red[256][33];
    const SumJob &j = jobs.j[blockIdx.y];
    if (!SumJobs::tree(j)) {
        for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < j.n;
             i += (long long)gridDim.x * blockDim.x) {
            float s = 0.f;
#pragma unroll 8
            for (int k = 0; k < j.splits; ++k) s += j.part[k * j.n + i];
            j.dst[i] = s;
        }
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (long long i0 = blockIdx.x * 32LL; i0 < j.n; i0 += gridDim.x * 32LL) {
        const long long i = i0 + lane;
        const bool in = i < j.n;
#pragma unroll 4
        for (int t = warp; t < 256; t += 8) {
            float s = 0.f;
            if (in)
                for (int k = t; k < j.splits; k += 256) s += j.part[k * j.n + i];
            red[t][lane] = s;
        }
        __syncthreads();
        for (int o = 128; o > 0; o >>= 1) {
            for (int t = warp; t < o; t += 8) red[t][lane] += red[t + o][lane];
            __syncthreads();
        }
        if (warp == 0 && in) j.dst[i] = red[0][lane];
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Elementwise kernels over blocked tensors: a thread takes the eight channels
// of one pixel.  Images fit 32-bit indices (checked where a network is sized).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void ld8f(const float *p, size_t u, float (&v)[8]) {
    const float4 *q = reinterpret_cast<const float4 *>(p) + 2 * u;
    const float4 x = q[0], y = q[1];
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
}

// Bias gradients: a block's pixels are summed per channel in 256 / C phases
// (every 256 / C-th pixel), the phases then in order.
constexpr int ACT_THREADS = 256, ACT_PIX = 512;   // pixels staged at a time

// One block's phase sums of eight channels from staged values.
struct PhaseSum {
    int phases;
    float s = 0.f;
    __device__ explicit PhaseSum(int c) : phases(256 / c) {}
    // n staged pixels, the first of them a multiple of `phases` into the block
    __device__ void add(const float (*v)[8], int n) {
        if (threadIdx.x >= 8 * phases) return;
        const int c = threadIdx.x & 7;
#pragma unroll 8
        for (int p = threadIdx.x >> 3; p < n; p += phases) s += v[p][c];
    }
    // the block's sum of channel threadIdx.x < 8
    __device__ float total(float (*red)[8]) {
        if (threadIdx.x < 8 * phases) red[threadIdx.x >> 3][threadIdx.x & 7] = s;
        __syncthreads();
        float t = 0.f;
        if (threadIdx.x < 8)
            for (int k = 0; k < phases; ++k) t += red[k][threadIdx.x];
        return t;
    }
};

template <GradSource SRC>
__global__ void __launch_bounds__(ACT_THREADS) k_act_back(const ActBack a, unsigned per) {
    __shared__ float stage[ACT_PIX][8];
    __shared__ float red[32][8];
    const int G = a.C / 8, g = int(blockIdx.y);
    const unsigned HW = unsigned(a.H) * unsigned(a.W), P = unsigned(a.B) * HW;
    const unsigned p0 = blockIdx.x * per, p1 = min(P, p0 + per);
    PhaseSum sum(a.C);
    for (unsigned q = p0; q < p1; q += ACT_PIX) {
        const unsigned n = min(p1 - q, unsigned(ACT_PIX));
        for (unsigned k = threadIdx.x; k < n; k += ACT_THREADS) {
            const unsigned p = q + k, b = p / HW, r = p - b * HW;
            const int y = int(r / unsigned(a.W)), x = int(r - unsigned(y) * unsigned(a.W));
            const size_t u = (size_t(b) * G + g) * HW + r;
            float v[8];
            if constexpr (SRC == G_UPSUM) {
                // gradient of nearest upsampling: the four pixels it fed
                const size_t row = size_t(2 * a.W);
                const size_t f = (size_t(b) * G + g) * 4 * HW + size_t(2 * y) * row + 2 * x;
                float c1[8], c2[8], c3[8];
                ld8f(a.a, f, v);
                ld8f(a.a, f + 1, c1);
                ld8f(a.a, f + row, c2);
                ld8f(a.a, f + row + 1, c3);
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = v[j] + c1[j] + c2[j] + c3[j];
            } else {
                ld8f(a.a, u, v);
            }
            if constexpr (SRC == G_POOL) {
                // gradient of the average pooling: a quarter to each of its pixels
                float c[8];
                ld8f(a.b, (size_t(b) * G + g) * (HW / 4) + size_t(y / 2) * (a.W / 2) + x / 2, c);
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] += 0.25f * c[j];
            }
            float s[8];
            unpack8(reinterpret_cast<const uint4 *>(a.y)[plane8(int(b), g, G, a.H, a.W) +
                                                         pixel8(y, x, a.W)], s);
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (s[j] <= 0.f) v[j] *= LEAK;
            put8(reinterpret_cast<uint4 *>(a.dz) + plane8(int(b), g, G, a.H, a.W), y, x, a.H, a.W,
                 pack8(v));
            const float4 lo = make_float4(v[0], v[1], v[2], v[3]);
            const float4 hi = make_float4(v[4], v[5], v[6], v[7]);
            if (a.g_out) {
                float4 *o = reinterpret_cast<float4 *>(a.g_out) + 2 * u;
                o[0] = lo;
                o[1] = hi;
            }
            *reinterpret_cast<float4 *>(&stage[k][0]) = lo;
            *reinterpret_cast<float4 *>(&stage[k][4]) = hi;
        }
        __syncthreads();
        sum.add(stage, int(n));
        __syncthreads();
    }
    const float t = sum.total(red);
    if (threadIdx.x < 8) a.bpart[size_t(blockIdx.x) * a.C + g * 8 + threadIdx.x] = t;
}

__global__ void k_pack_features(const float *__restrict__ f, int B, int H, int W, int feat, int G,
                                bf16 *__restrict__ x) {
    const unsigned HW = unsigned(H) * unsigned(W), P = unsigned(B) * HW;
    for (unsigned p = blockIdx.x * blockDim.x + threadIdx.x; p < P; p += gridDim.x * blockDim.x) {
        const unsigned b = p / HW, r = p - b * HW;
        const int py = int(r / unsigned(W)), px = int(r - unsigned(py) * unsigned(W));
        for (int g = 0; g < G; ++g) {
            float v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                v[j] = 8 * g + j < feat ? f[size_t(p) * feat + 8 * g + j] : 0.f;
            put8(reinterpret_cast<uint4 *>(x) + plane8(int(b), g, G, H, W), py, px, H, W, pack8(v));
        }
    }
}

// Loss: mean over pixels and outputs of (y - t)^2; dz = BF16 of its gradient
// 2 (y - t) / count (the output layer has no activation).
constexpr int MAX_OUT = 8;

__global__ void __launch_bounds__(ACT_THREADS)
k_mse(const float *__restrict__ y, const float *__restrict__ t, int nout, int B, int H, int W,
      unsigned per, int groups, bf16 *__restrict__ dz, double *__restrict__ part,
      float *__restrict__ bpart) {
    __shared__ float stage[ACT_PIX][8];
    __shared__ float red[32][8];
    __shared__ double lred[ACT_THREADS];
    const unsigned HW = unsigned(H) * unsigned(W), P = unsigned(B) * HW;
    const double inv = 1.0 / double((long long)P * nout);
    const unsigned p0 = blockIdx.x * per, p1 = min(P, p0 + per);
    double s = 0.0;
    PhaseSum sum(32);
    for (unsigned q = p0; q < p1; q += ACT_PIX) {
        const unsigned n = min(p1 - q, unsigned(ACT_PIX));
        for (unsigned k = threadIdx.x; k < n; k += ACT_THREADS) {
            const unsigned p = q + k;
            float v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                v[j] = 0.f;
                if (j < nout) {
                    const float d = y[size_t(p) * nout + j] - t[size_t(p) * nout + j];
                    s += double(d) * d;
                    v[j] = float(2.0 * d * inv);
                }
                stage[k][j] = v[j];
            }
            const unsigned b = p / HW, r = p - b * HW;
            const int py = int(r / unsigned(W)), px = int(r - unsigned(py) * unsigned(W));
            put8(reinterpret_cast<uint4 *>(dz) + plane8(int(b), 0, groups, H, W), py, px, H, W,
                 pack8(v));
        }
        __syncthreads();
        sum.add(stage, int(n));
        __syncthreads();
    }
    lred[threadIdx.x] = s;
    const float bs = sum.total(red);
    for (int o = ACT_THREADS / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) lred[threadIdx.x] += lred[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = lred[0] * inv;
    if (threadIdx.x < 8 * groups)
        bpart[size_t(blockIdx.x) * 8 * groups + threadIdx.x] = threadIdx.x < 8 ? bs : 0.f;
}

__global__ void k_loss_final(const double *__restrict__ part, int n, const int *flag, double *out) {
    __shared__ double red[256];
    double s = 0.0;
    for (int k = threadIdx.x; k < n; k += 256) s += part[k];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = red[0];
        out[1] = *flag ? 1.0 : 0.0;
    }
}

// The two BF16 copies of weight i = (co, tap, ci).
__device__ __forceinline__ void put_copies(const LayerParams &l, long long i, float p) {
    const int ci = int(i % l.cin), t = int((i / l.cin) % 9), co = int(i / (9LL * l.cin));
    const bf16 v = __float2bfloat16_rn(p);
    l.wb[((size_t(t) * (l.cin / 8) + ci / 8) * l.cout + co) * 8 + (ci & 7)] = v;
    l.wt[((size_t(8 - t) * (l.cout / 8) + co / 8) * l.cin + ci) * 8 + (co & 7)] = v;
}

__global__ void k_adam(const __grid_constant__ NetParams net, float lr, float b1, float b2,
                       float eps, float c1, float c2, long long step, const int *flag,
                       long long *applied) {
    if (*flag) return;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *applied = step;
    const LayerParams &l = net.l[blockIdx.y];
    const long long nw = 9LL * l.cout * l.cin, n = nw + l.cout;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        const bool isw = k < nw;
        const long long i = isw ? k : k - nw;
        float *p = isw ? l.w : l.b, *m = isw ? l.mw : l.mb, *v = isw ? l.vw : l.vb;
        const float gi = (isw ? l.gw : l.gb)[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        p[i] = pi;
        if (isw) put_copies(l, i, pi);
    }
}

__global__ void k_refresh(const __grid_constant__ NetParams net) {
    const LayerParams &l = net.l[blockIdx.y];
    const long long nw = 9LL * l.cout * l.cin;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nw;
         i += (long long)gridDim.x * blockDim.x)
        put_copies(l, i, l.w[i]);
}

__global__ void k_nhwc_to_blocked(const bf16 *__restrict__ x, int B, int H, int W, int C,
                                  bf16 *__restrict__ o) {
    const int G = C / 8;
    const size_t n = size_t(B) * H * W * G;
    for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n;
         i += size_t(gridDim.x) * blockDim.x) {
        const int g = int(i % G);
        const size_t p = i / G;
        const int xx = int(p % W), y = int(p / W % H), b = int(p / (size_t(W) * H));
        put8(reinterpret_cast<uint4 *>(o) + plane8(b, g, G, H, W), y, xx, H, W,
             reinterpret_cast<const uint4 *>(x)[i]);
    }
}

__global__ void k_blocked_to_nhwc(const float *__restrict__ x, int B, int H, int W, int C,
                                  float *__restrict__ o) {
    const size_t HW = size_t(H) * W, n = size_t(B) * HW * C;
    for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n;
         i += size_t(gridDim.x) * blockDim.x) {
        const int c = int(i % C);
        const size_t p = i / C, b = p / HW;
        o[i] = x[((b * (C / 8) + c / 8) * HW + (p - b * HW)) * 8 + (c & 7)];
    }
}

__global__ void k_block_weights(const bf16 *__restrict__ w, int cout, int cin,
                                bf16 *__restrict__ o) {
    const size_t n = size_t(cout) * 9 * cin;
    for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n;
         i += size_t(gridDim.x) * blockDim.x) {
        const int ci = int(i % cin), t = int(i / cin % 9), co = int(i / (size_t(9) * cin));
        o[((size_t(t) * (cin / 8) + ci / 8) * cout + co) * 8 + (ci & 7)] = w[i];
    }
}

unsigned blocks_for(size_t n) { return unsigned(std::min<size_t>((n + 255) / 256, 8192)); }

}  // namespace

// One split per 4096 pixels, at most 128.
int weight_grad_splits(int B, int H, int W) {
    const long long s = (long long)B * H * W / 4096;
    return int(std::max<long long>(1, std::min<long long>(128, s)));
}

cudaError_t weight_grad(const bf16 *dz, const bf16 *in, int B, int H, int W, int cout, int cin,
                        int splits, float *part, int *err, cudaStream_t st) {
    if (cout % 16 || cin % 16 || splits < 1) return cudaErrorInvalidValue;
    const long long P = (long long)B * H * W;
    long long per = (P + splits - 1) / splits;
    per = (per + DW_PIX - 1) / DW_PIX * DW_PIX;
    if (W % 16 || splits > 65535) {
        if (cout % 32 || cin % 32) return cudaErrorInvalidValue;
        const int mt = cout % 64 == 0 ? 64 : 32, nt = cin % 64 == 0 ? 64 : 32;
        const dim3 grid(unsigned(cin / nt), unsigned(cout / mt), unsigned(9 * splits));
        if (mt == 64 && nt == 64)
            k_dw_any<64, 64><<<grid, 128, 0, st>>>(dz, in, H, W, P, per, cout, cin, part);
        else if (mt == 64)
            k_dw_any<64, 32><<<grid, 128, 0, st>>>(dz, in, H, W, P, per, cout, cin, part);
        else if (nt == 64)
            k_dw_any<32, 64><<<grid, 128, 0, st>>>(dz, in, H, W, P, per, cout, cin, part);
        else
            k_dw_any<32, 32><<<grid, 128, 0, st>>>(dz, in, H, W, P, per, cout, cin, part);
        return cudaGetLastError();
    }
    DwGeom g{W, H, std::min(W, DW_PIX), 1};
    if ((W == 16 || W == 32) && H % (DW_PIX / W) == 0) g.sr = DW_PIX / W;
    // 32 input channels per CTA, fewer where that leaves SMs without one
    // (four warps, or eight with 64 output channels, fill an SM's tensor
    // pipes better than one)
    int sms = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return cudaErrorInvalidDevice;
    auto ctas = [&](int iw) {
        const int cot = cout % 64 == 0 && iw == 4 ? 64 : cout % 32 == 0 ? 32 : 16;
        return (long long)splits * (cout / cot) * (cin / (8 * iw));
    };
    int iw = cin % 32 == 0 ? 4 : 2;
    while (iw > 1 && 2 * ctas(iw) <= sms) iw /= 2;
    if (iw == 4) return launch_dw_co<4>(dz, in, B, g, cout, cin, splits, per, part, err, st);
    if (iw == 2) return launch_dw_co<2>(dz, in, B, g, cout, cin, splits, per, part, err, st);
    return launch_dw_co<1>(dz, in, B, g, cout, cin, splits, per, part, err, st);
}

cudaError_t sum_splits(const SumJobs &jobs, int count, cudaStream_t st) {
    long long most = 1;
    for (int k = 0; k < count; ++k)
        most = std::max(most, jobs.j[k].n * (SumJobs::tree(jobs.j[k]) ? 8 : 1));
    k_sum_splits<<<dim3(unsigned(std::min<long long>((most + 255) / 256, 1024)), unsigned(count)),
                   256, 0, st>>>(jobs);
    return cudaGetLastError();
}

int bias_blocks(int B, int H, int W) {
    const long long P = (long long)B * H * W;
    return int(std::min<long long>(1024, std::max<long long>(1, P / 256)));
}

cudaError_t act_back(const ActBack &a, GradSource src, cudaStream_t st) {
    if (a.C > 256 || 256 % a.C) return cudaErrorInvalidValue;
    const long long P = (long long)a.B * a.H * a.W;
    const int blocks = bias_blocks(a.B, a.H, a.W);
    const unsigned per = unsigned((P + blocks - 1) / blocks);
    const dim3 grid{unsigned(blocks), unsigned(a.C / 8)};
    switch (src) {
    case G_DIRECT: k_act_back<G_DIRECT><<<grid, ACT_THREADS, 0, st>>>(a, per); break;
    case G_UPSUM: k_act_back<G_UPSUM><<<grid, ACT_THREADS, 0, st>>>(a, per); break;
    default: k_act_back<G_POOL><<<grid, ACT_THREADS, 0, st>>>(a, per); break;
    }
    return cudaGetLastError();
}

cudaError_t pack_features(const float *f, int B, int H, int W, int feat, int cpad, bf16 *x,
                          cudaStream_t st) {
    k_pack_features<<<blocks_for(size_t(B) * H * W), 256, 0, st>>>(f, B, H, W, feat, cpad / 8, x);
    return cudaGetLastError();
}

cudaError_t mse(const float *y, const float *t, int nout, int B, int H, int W, int groups, bf16 *dz,
                double *part, float *bpart, cudaStream_t st) {
    if (nout > MAX_OUT) return cudaErrorInvalidValue;
    const int blocks = bias_blocks(B, H, W);
    const unsigned per = unsigned(((long long)B * H * W + blocks - 1) / blocks);
    k_mse<<<blocks, ACT_THREADS, 0, st>>>(y, t, nout, B, H, W, per, groups, dz, part, bpart);
    return cudaGetLastError();
}

cudaError_t loss_final(const double *part, int n, const int *flag, double *out, cudaStream_t st) {
    k_loss_final<<<1, 256, 0, st>>>(part, n, flag, out);
    return cudaGetLastError();
}

cudaError_t adam(const NetParams &p, int layers, float lr, float b1, float b2, float eps, float c1,
                 float c2, long long step, const int *flag, long long *applied, cudaStream_t st) {
    k_adam<<<dim3(592, unsigned(layers)), 256, 0, st>>>(p, lr, b1, b2, eps, c1, c2, step, flag,
                                                        applied);
    return cudaGetLastError();
}

cudaError_t refresh_copies(const NetParams &p, int layers, cudaStream_t st) {
    k_refresh<<<dim3(592, unsigned(layers)), 256, 0, st>>>(p);
    return cudaGetLastError();
}

cudaError_t nhwc_to_blocked(const bf16 *x, int B, int H, int W, int C, bf16 *o, cudaStream_t st) {
    k_nhwc_to_blocked<<<blocks_for(size_t(B) * H * W * (C / 8)), 256, 0, st>>>(x, B, H, W, C, o);
    return cudaGetLastError();
}

cudaError_t blocked_to_nhwc_f32(const float *x, int B, int H, int W, int C, float *o,
                                cudaStream_t st) {
    k_blocked_to_nhwc<<<blocks_for(size_t(B) * H * W * C), 256, 0, st>>>(x, B, H, W, C, o);
    return cudaGetLastError();
}

cudaError_t block_weights(const bf16 *w, int cout, int cin, bf16 *o, cudaStream_t st) {
    k_block_weights<<<blocks_for(size_t(cout) * 9 * cin), 256, 0, st>>>(w, cout, cin, o);
    return cudaGetLastError();
}

}  // namespace surr
