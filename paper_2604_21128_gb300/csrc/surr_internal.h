// Internal declarations of the learned surrogate's kernels.  Not installed.
// Layouts are those of surr_kernels.cuh: "blocked" BF16 tensors have eight
// channels per pixel and a periodic halo, blocked FP32 tensors no halo.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "surr_kernels.cuh"

namespace surr {

// Pixel tile of the contractions: eight columns (one operand row group per
// image row) by sixteen rows.
constexpr int TX = 8, TY = 16, TM = TX * TY;

// Elements of a blocked BF16 tensor of C channels.
inline size_t blocked_elems(int B, int C, int H, int W) {
    return size_t(B) * C * size_t(H + 2) * size_t(W + 2);
}

enum ConvMode {
    EP_ACT,    // act(acc + bias + skip) -> out, and optionally its 2x2 pooling / upsampling
    EP_F32,    // acc -> out_f, blocked FP32
    EP_OUT     // acc + bias, first n_out channels -> out_f[pixel][n_out]
};

struct ConvArgs {
    const bf16 *in;      // blocked, cin channels (16, or a multiple of 32)
    int B, H, W, cin, cout;
    const bf16 *w;       // [tap][cin / 8][cout][8]
    const float *bias;   // [cout]
    const bf16 *skip;    // blocked, cout channels, or null
    bf16 *out;           // blocked
    bf16 *pool;          // blocked, H/2 x W/2, or null
    bf16 *up;            // blocked, 2H x 2W, or null
    float *out_f;
    int n_out;
    int *err;            // raised when one of the launch's mbarrier waits gives up
};

cudaError_t conv3x3(const ConvArgs &a, ConvMode mode, cudaStream_t st);
// Test hook: make one CTA run out a wait, in convolutions of every mode (1) or
// of EP_F32 only (2), as long as the launch's flag is not raised.
cudaError_t conv_tc_stall(int on);

// A tensor map over a blocked BF16 tensor: box of bx pixels x by rows x bg
// channel groups; with the halo, or the interior only (zeros outside).
bool blocked_map(CUtensorMap *map, const bf16 *t, int B, int C, int H, int W, bool halo, int bx,
                 int by, int bg);

// part[split][co][tap][ci] = this split's sum over pixels of dz x shifted in
// (both blocked; cout, cin 16 or multiples of 32).  err: as in ConvArgs.
cudaError_t weight_grad(const bf16 *dz, const bf16 *in, int B, int H, int W, int cout, int cin,
                        int splits, float *part, int *err, cudaStream_t st);
// The network's splits for a level.
int weight_grad_splits(int B, int H, int W);

// Sums over splits, in a fixed order, of up to MAX_JOBS arrays in one launch.
constexpr int MAX_JOBS = 20;
struct SumJob { const float *part; float *dst; int splits; long long n; };
struct SumJobs {
    SumJob j[MAX_JOBS];
    // many splits of few values are summed as a tree (see k_sum_splits)
    static __host__ __device__ bool tree(const SumJob &j) {
        return j.splits >= 64 && j.n <= 65535;
    }
};
cudaError_t sum_splits(const SumJobs &jobs, int count, cudaStream_t st);

// Backward through an activation: g = (source) * act'(y), dz = BF16 g, the
// per-channel sums of g over each of bias_blocks pixel ranges to bpart[range][C].
enum GradSource {
    G_DIRECT,   // a[unit]
    G_UPSUM,    // the four pixels of a (2H x 2W) that the upsampling fed
    G_POOL      // a[unit] + b[half-resolution unit] / 4
};
struct ActBack {
    const float *a, *b;  // blocked FP32
    const bf16 *y;       // blocked activations
    bf16 *dz;
    float *g_out;        // g itself, or null
    float *bpart;
    int B, H, W, C;
};
int bias_blocks(int B, int H, int W);
cudaError_t act_back(const ActBack &a, GradSource src, cudaStream_t st);

// Features [pixel][feat] FP32 -> blocked BF16 of cpad channels.
cudaError_t pack_features(const float *f, int B, int H, int W, int feat, int cpad, bf16 *x,
                          cudaStream_t st);
// Mean-square loss over [pixel][nout]: sums of bias_blocks pixel ranges to
// part, dz (channel group 0 of `groups`) and its bias sums bpart[range][16].
cudaError_t mse(const float *y, const float *t, int nout, int B, int H, int W, int groups, bf16 *dz,
                double *part, float *bpart, cudaStream_t st);
// out[0] = sum of part; out[1] = the wait flag (0 or 1).
cudaError_t loss_final(const double *part, int n, const int *flag, double *out, cudaStream_t st);

// Adam on FP32 master weights [cout][tap][cin] and biases of all layers, and
// the two BF16 copies the convolutions read: wb [tap][cin/8][cout][8] and the
// flipped transpose wt [tap][cout/8][cin][8] (wt[t][co][ci] = w[co][8-t][ci]).
// Skips everything while *flag is raised, else writes `step` to *applied.
// Without Adam (refresh), only the copies are written.
constexpr int MAX_LAYERS = 10;
struct LayerParams {
    float *w, *gw, *mw, *vw, *b, *gb, *mb, *vb;
    bf16 *wb, *wt;
    int cout, cin;
};
struct NetParams { LayerParams l[MAX_LAYERS]; };
cudaError_t adam(const NetParams &p, int layers, float lr, float b1, float b2, float eps, float c1,
                 float c2, long long step, const int *flag, long long *applied, cudaStream_t st);
cudaError_t refresh_copies(const NetParams &p, int layers, cudaStream_t st);

// NHWC BF16 <-> blocked, weights [cout][tap][cin] -> [tap][cin/8][cout][8].
cudaError_t nhwc_to_blocked(const bf16 *x, int B, int H, int W, int C, bf16 *o, cudaStream_t st);
cudaError_t blocked_to_nhwc_f32(const float *x, int B, int H, int W, int C, float *o,
                                cudaStream_t st);
cudaError_t block_weights(const bf16 *w, int cout, int cin, bf16 *o, cudaStream_t st);

}  // namespace surr
