// The learned surrogate: a five-level convolutional operator that maps the
// E_z state and the medium of a lattice to the state K steps later, trained
// on trajectories the library computes, and the routine that uses it with
// plain QLA as fallback and arbiter (declared in qla.h, surr_*).
//
// Network (widths 32, 64, 128, 256, 256; 3x3 periodic convolutions, leaky
// ReLU 0.1, 2x2 average pooling down, nearest 2x upsampling up, additive
// skips):
//   E0 = a(conv(X))            E1 = a(conv(pool E0))  ...  E4 = a(conv(pool E3))
//   D3 = a(conv(up E4) + E3)   D2 = a(conv(up D3) + E2)  ...  D0 = a(conv(up D1) + E0)
//   Y  = conv(D0)              (3 outputs: the change of q2, q3, q4)
// Inputs: q2, q3, q4, n - 1.5, 4 dn/dx, 4 dn/dy (centred differences).
// BF16 weights and activations, FP32 accumulation, FP32 master weights,
// gradients and Adam state.
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>
#include <random>
#include <string>
#include <vector>

#include "qla_internal.h"
#include "surr_internal.h"

using namespace surr;

namespace {

constexpr int LEVELS = 5;
constexpr int WIDTH[LEVELS] = {32, 64, 128, 256, 256};
constexpr int FEAT = 6, NOUT = 3, CPAD = 16;   // inputs and outputs padded to one K step
constexpr int NCONV = 10;

struct ConvSpec {
    int cin, cout, level;   // padded channel counts; level of its output
    int cin_real, cout_real;
    bool act, skip;
};

ConvSpec spec(int i) {
    // 0..4 encoder, 5..8 decoder (levels 3..0), 9 output
    if (i == 0) return {CPAD, WIDTH[0], 0, FEAT, WIDTH[0], true, false};
    if (i < 5) return {WIDTH[i - 1], WIDTH[i], i, WIDTH[i - 1], WIDTH[i], true, false};
    if (i < 9) {
        const int l = 8 - i;  // 3, 2, 1, 0
        return {WIDTH[l + 1], WIDTH[l], l, WIDTH[l + 1], WIDTH[l], true, true};
    }
    return {WIDTH[0], CPAD, 0, WIDTH[0], NOUT, false, false};
}

template <typename T>
T *carve(char *&p, size_t n) {
    T *r = reinterpret_cast<T *>(p);
    p += (n * sizeof(T) + 255) & ~size_t(255);
    return r;
}

}  // namespace

struct surr_net {
    int H = 0, W = 0, maxB = 0;
    cudaStream_t stream = nullptr;
    char *mem = nullptr;
    // parameters, gradients, Adam state and the BF16 copies, by layer
    NetParams prm;
    size_t nw[NCONV];
    // activations (blocked BF16), per level: E, D (l < 4), and the inputs of
    // the convolutions, P = pool E (l >= 1), U = up D (l < 4)
    bf16 *X, *E[LEVELS], *D[LEVELS], *Pl[LEVELS], *U[LEVELS];
    float *Y;                                  // [P0][NOUT]
    // gradients (blocked FP32): of D0, of E through the skips, of P and U
    float *dD0, *dE[LEVELS], *dP[LEVELS], *dU[LEVELS];
    bf16 *dz, *dz9;                            // of a layer, of the output layer
    float *part[NCONV], *bpart[NCONV];         // split sums of weights and biases
    double *lpart;                             // loss partials
    double *lout;                              // loss and wait flag
    double *lhost = nullptr;                   // the same, pinned
    cudaEvent_t ldone = nullptr;
    int *flag;                                 // raised by a wait that ran out
    long long *applied;                        // Adam steps made (device)
    long long step = 0;                        // Adam steps enqueued and not known to be skipped
    std::string err;
};

namespace {

qla_status nfail(surr_net *n, qla_status s, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    if (n) n->err = buf;
    return s;
}

#define NCUDA(n, call, what)                                                        \
    do {                                                                            \
        cudaError_t e_ = (call);                                                    \
        if (e_ != cudaSuccess)                                                      \
            return nfail((n), QLA_ECUDA, "%s: %s", (what), cudaGetErrorString(e_)); \
    } while (0)

// Lays the network out from n->mem (null: only measured); returns the bytes.
size_t carve_all(surr_net *n) {
    char *p = n->mem;
    const int B = n->maxB, H = n->H, W = n->W;
    for (int i = 0; i < NCONV; ++i) {
        const ConvSpec s = spec(i);
        LayerParams &l = n->prm.l[i];
        const size_t nw = size_t(s.cout) * 9 * s.cin;
        n->nw[i] = nw;
        l.cout = s.cout;
        l.cin = s.cin;
        l.w = carve<float>(p, nw);
        l.gw = carve<float>(p, nw);
        l.mw = carve<float>(p, nw);
        l.vw = carve<float>(p, nw);
        l.b = carve<float>(p, s.cout);
        l.gb = carve<float>(p, s.cout);
        l.mb = carve<float>(p, s.cout);
        l.vb = carve<float>(p, s.cout);
        l.wb = carve<bf16>(p, nw);
        l.wt = carve<bf16>(p, nw);
    }
    auto act = [&](int c, int l) { return carve<bf16>(p, blocked_elems(B, c, H >> l, W >> l)); };
    auto grad = [&](int c, int l) {
        return carve<float>(p, size_t(B) * c * size_t(H >> l) * size_t(W >> l));
    };
    size_t dz = 0;
    n->X = act(CPAD, 0);
    for (int l = 0; l < LEVELS; ++l) {
        n->E[l] = act(WIDTH[l], l);
        n->D[l] = l < 4 ? act(WIDTH[l], l) : nullptr;
        n->Pl[l] = l >= 1 ? act(WIDTH[l - 1], l) : nullptr;
        n->U[l] = l < 4 ? act(WIDTH[l + 1], l) : nullptr;
        n->dE[l] = l < 4 ? grad(WIDTH[l], l) : nullptr;
        n->dP[l] = l >= 1 ? grad(WIDTH[l - 1], l) : nullptr;
        n->dU[l] = l < 4 ? grad(WIDTH[l + 1], l) : nullptr;
        dz = std::max(dz, blocked_elems(B, WIDTH[l], H >> l, W >> l));
    }
    n->dD0 = grad(WIDTH[0], 0);
    n->Y = carve<float>(p, size_t(B) * H * W * NOUT);
    n->dz = carve<bf16>(p, dz);
    n->dz9 = act(CPAD, 0);
    for (int i = 0; i < NCONV; ++i) {
        const ConvSpec s = spec(i);
        const int h = H >> s.level, w = W >> s.level;
        // smaller batches never take more splits or chunks
        n->part[i] = carve<float>(p, size_t(weight_grad_splits(B, h, w)) * n->nw[i]);
        n->bpart[i] = carve<float>(p, size_t(bias_blocks(B, h, w)) * s.cout);
    }
    // the lattice checks of surr_advance use 768 doubles of it
    n->lpart = carve<double>(p, size_t(std::max(768, bias_blocks(B, H, W))));
    n->lout = carve<double>(p, 2);
    n->flag = carve<int>(p, 1);
    n->applied = carve<long long>(p, 1);
    return size_t(p - n->mem);
}

// conv layer i: its input and output tensors
const bf16 *conv_input(const surr_net *n, int i) {
    if (i == 0) return n->X;
    if (i < 5) return n->Pl[i];
    if (i < 9) return n->U[8 - i];
    return n->D[0];
}

bf16 *conv_output(surr_net *n, int i) {
    if (i < 5) return n->E[i];
    if (i < 9) return n->D[8 - i];
    return nullptr;
}

// Ten launches: each convolution writes its output and, where the next layer
// reads it pooled (encoder) or upsampled (decoder), that too.
qla_status forward(surr_net *n, int B, float *y) {
    for (int i = 0; i < NCONV; ++i) {
        const ConvSpec s = spec(i);
        const int l = s.level;
        ConvArgs a{};
        a.in = conv_input(n, i);
        a.B = B;
        a.H = n->H >> l;
        a.W = n->W >> l;
        a.cin = s.cin;
        a.cout = s.cout;
        a.w = n->prm.l[i].wb;
        a.bias = n->prm.l[i].b;
        a.skip = s.skip ? n->E[l] : nullptr;
        a.out = conv_output(n, i);
        a.pool = i < 4 ? n->Pl[l + 1] : nullptr;
        a.up = i >= 4 && i < 8 ? n->U[l - 1] : nullptr;
        a.out_f = y;
        a.n_out = NOUT;
        a.err = n->flag;
        NCUDA(n, conv3x3(a, i == 9 ? EP_OUT : EP_ACT, n->stream), "surrogate: conv");
    }
    return QLA_OK;
}

// The weight gradient's split sums of layer i from its dz, and (d_in) the
// gradient of its input.
qla_status conv_backward(surr_net *n, int i, int B, const bf16 *dz, float *d_in, SumJobs &jobs,
                         int &njobs) {
    const ConvSpec s = spec(i);
    const int h = n->H >> s.level, w = n->W >> s.level;
    const LayerParams &l = n->prm.l[i];
    const int splits = weight_grad_splits(B, h, w);
    NCUDA(n, weight_grad(dz, conv_input(n, i), B, h, w, s.cout, s.cin, splits, n->part[i],
                         n->flag, n->stream),
          "surrogate: weight grad");
    jobs.j[njobs++] = {n->part[i], l.gw, splits, (long long)n->nw[i]};
    jobs.j[njobs++] = {n->bpart[i], l.gb, bias_blocks(B, h, w), s.cout};
    if (d_in) {
        ConvArgs a{};
        a.in = dz;
        a.B = B;
        a.H = h;
        a.W = w;
        a.cin = s.cout;
        a.cout = s.cin;
        a.w = l.wt;
        a.out_f = d_in;
        a.err = n->flag;
        NCUDA(n, conv3x3(a, EP_F32, n->stream), "surrogate: input grad");
    }
    return QLA_OK;
}

qla_status backward(surr_net *n, int B) {
    SumJobs jobs{};
    int njobs = 0;
    qla_status r;
    // through layer i's activation: dz from the gradient of its output
    auto through = [&](int i, GradSource src, const float *a, const float *b, float *g_out) {
        const ConvSpec s = spec(i);
        const ActBack args{a, b, conv_output(n, i), n->dz, g_out, n->bpart[i], B,
                           n->H >> s.level, n->W >> s.level, s.cout};
        NCUDA(n, act_back(args, src, n->stream), "surrogate: activation backward");
        return QLA_OK;
    };
    // output convolution (dz9 from the loss) -> dD0
    if ((r = conv_backward(n, 9, B, n->dz9, n->dD0, jobs, njobs)) != QLA_OK) return r;
    // decoder levels 0..3 (layer 8 - l): dD_l -> dU_l, the skip's share to dE_l
    for (int l = 0; l < 4; ++l) {
        const int i = 8 - l;
        if ((r = through(i, l == 0 ? G_DIRECT : G_UPSUM, l == 0 ? n->dD0 : n->dU[l - 1], nullptr,
                         n->dE[l])) != QLA_OK)
            return r;
        if ((r = conv_backward(n, i, B, n->dz, n->dU[l], jobs, njobs)) != QLA_OK) return r;
    }
    // encoder levels 4..0: dE_l (upsampling; skip and pooling below) -> dP_l
    for (int l = 4; l >= 0; --l) {
        if ((r = l == 4 ? through(4, G_UPSUM, n->dU[3], nullptr, nullptr)
                        : through(l, G_POOL, n->dE[l], n->dP[l + 1], nullptr)) != QLA_OK)
            return r;
        if ((r = conv_backward(n, l, B, n->dz, l >= 1 ? n->dP[l] : nullptr, jobs, njobs)) != QLA_OK)
            return r;
    }
    NCUDA(n, sum_splits(jobs, njobs, n->stream), "surrogate: gradient sums");
    return QLA_OK;
}

// A bounded wait of one of this network's kernels ran out (its CTA skipped
// its outputs, so they are not to be trusted).  The flag is cleared once
// nothing enqueued reads it any more; Adam steps that found it raised made no
// update and do not count.
qla_status wait_ran_out(surr_net *n) {
    long long applied = 0;
    NCUDA(n, cudaMemcpyAsync(&applied, n->applied, sizeof applied, cudaMemcpyDeviceToHost,
                             n->stream), "surrogate: step count");
    NCUDA(n, cudaMemsetAsync(n->flag, 0, sizeof(int), n->stream), "surrogate: wait flag");
    NCUDA(n, cudaStreamSynchronize(n->stream), "surrogate: sync");
    n->step = applied;
    return nfail(n, QLA_ETIMEOUT,
                 "surrogate: a tensor-core wait ran out; results of tensor-core launches "
                 "are undefined until the network is rebuilt");
}

qla_status tc_waits_ok(surr_net *n) {
    int flag = 0;
    NCUDA(n, cudaMemcpyAsync(&flag, n->flag, sizeof flag, cudaMemcpyDeviceToHost, n->stream),
          "surrogate: wait flag");
    NCUDA(n, cudaStreamSynchronize(n->stream), "surrogate: sync");
    return flag ? wait_ran_out(n) : QLA_OK;
}

// The loss of n->Y, its gradient into dz9, and loss and wait flag on their
// way to the host.
qla_status loss_begin(surr_net *n, int B, const float *target) {
    NCUDA(n, mse(n->Y, target, NOUT, B, n->H, n->W, CPAD / 8, n->dz9, n->lpart, n->bpart[9],
                 n->stream), "surrogate: loss");
    NCUDA(n, loss_final(n->lpart, bias_blocks(B, n->H, n->W), n->flag, n->lout, n->stream),
          "surrogate: loss sum");
    NCUDA(n, cudaMemcpyAsync(n->lhost, n->lout, 16, cudaMemcpyDeviceToHost, n->stream),
          "surrogate: loss copy");
    NCUDA(n, cudaEventRecord(n->ldone, n->stream), "surrogate: loss event");
    return QLA_OK;
}

// Waits for the loss (not for the work enqueued after it).
qla_status loss_end(surr_net *n, double *out) {
    NCUDA(n, cudaEventSynchronize(n->ldone), "surrogate: sync");
    *out = n->lhost[0];
    return n->lhost[1] != 0.0 ? wait_ran_out(n) : QLA_OK;
}

qla_status pack(surr_net *n, const float *feat, int B) {
    NCUDA(n, pack_features(feat, B, n->H, n->W, FEAT, CPAD, n->X, n->stream), "surrogate: pack");
    return QLA_OK;
}

qla_status check_batch(surr_net *n, int B) {
    if (B < 1 || B > n->maxB) return nfail(n, QLA_EINVAL, "batch %d outside 1..%d", B, n->maxB);
    return QLA_OK;
}

// Forward, loss and backward enqueued.
qla_status enqueue_grad(surr_net *n, const float *feat, const float *target, int B) {
    qla_status s = check_batch(n, B);
    if (s != QLA_OK) return s;
    if ((s = pack(n, feat, B)) != QLA_OK) return s;
    if ((s = forward(n, B, n->Y)) != QLA_OK) return s;
    if ((s = loss_begin(n, B, target)) != QLA_OK) return s;
    return backward(n, B);
}

}  // namespace

// ---------------------------------------------------------------------------
// Lattice side: features, candidate checks, the window loop with fallback.
// ---------------------------------------------------------------------------
namespace {

// Features of an FP32 E_z context (the state with the pending potential
// step applied, and the medium): [ny][nx][6].
__global__ void k_features(const float *__restrict__ q, size_t plane, int nx, int ny, int pitch,
                           bool vin, const uint32_t *__restrict__ midx,
                           const qla::MedRec<float> *__restrict__ table,
                           const double *__restrict__ n, float *__restrict__ f) {
    const size_t N = size_t(nx) * ny;
    for (size_t t = blockIdx.x * size_t(blockDim.x) + threadIdx.x; t < N;
         t += size_t(gridDim.x) * blockDim.x) {
        const int j = int(t / nx), i = int(t - size_t(j) * nx);
        const size_t g = size_t(j) * pitch + i;
        float s[6];
        qla::load_site<float, 3, qla::V_ROTATION>(q, plane, g, vin, midx, table, s);
        const double dnx = 0.5 * (n[size_t(j) * pitch + qla::wrap(i + 1, nx)] -
                                  n[size_t(j) * pitch + qla::wrap(i - 1, nx)]);
        const double dny = 0.5 * (n[size_t(qla::wrap(j + 1, ny)) * pitch + i] -
                                  n[size_t(qla::wrap(j - 1, ny)) * pitch + i]);
        float *o = f + t * FEAT;
        o[0] = s[2];
        o[1] = s[3];
        o[2] = s[4];
        o[3] = float(n[g] - 1.5);
        o[4] = float(4.0 * dnx);
        o[5] = float(4.0 * dny);
    }
}

// candidate q = q(t) (from the features) + y; energy and the change of the
// discrete divergence of B (centred differences) against q(t)'s, as sums.
__global__ void k_candidate(const float *__restrict__ f, const float *__restrict__ y, int nx,
                            int ny, float *__restrict__ cand, double *__restrict__ sums) {
    __shared__ double red[3][256];
    const size_t N = size_t(nx) * ny;
    double e = 0.0, dd = 0.0, gg = 0.0;
    for (size_t t = blockIdx.x * size_t(blockDim.x) + threadIdx.x; t < N;
         t += size_t(gridDim.x) * blockDim.x) {
        const int j = int(t / nx), i = int(t - size_t(j) * nx);
        float c[3];
        for (int k = 0; k < 3; ++k) {
            c[k] = f[t * FEAT + k] + y[t * NOUT + k];
            cand[k * N + t] = c[k];
            e += double(c[k]) * c[k];
        }
        auto at = [&](int ii, int jj, int k) {
            const size_t s = size_t(qla::wrap(jj, ny)) * nx + qla::wrap(ii, nx);
            return double(f[s * FEAT + k]) + double(y[s * NOUT + k]);
        };
        auto at0 = [&](int ii, int jj, int k) {
            const size_t s = size_t(qla::wrap(jj, ny)) * nx + qla::wrap(ii, nx);
            return double(f[s * FEAT + k]);
        };
        // B_x = q3 (index 1), B_y = q4 (index 2)
        const double dbx = 0.5 * (at(i + 1, j, 1) - at(i - 1, j, 1));
        const double dby = 0.5 * (at(i, j + 1, 2) - at(i, j - 1, 2));
        const double d0 = 0.5 * (at0(i + 1, j, 1) - at0(i - 1, j, 1)) +
                          0.5 * (at0(i, j + 1, 2) - at0(i, j - 1, 2));
        const double dv = dbx + dby - d0;
        dd += dv * dv;
        gg += dbx * dbx + dby * dby;
    }
    red[0][threadIdx.x] = e;
    red[1][threadIdx.x] = dd;
    red[2][threadIdx.x] = gg;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o)
            for (int k = 0; k < 3; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int k = 0; k < 3; ++k) sums[blockIdx.x * 3 + k] = red[k][0];
}

// Write a candidate (three contiguous planes q2, q3, q4) as the state.
__global__ void k_store_candidate(const float *__restrict__ cand, int nx, int ny, int pitch,
                                  size_t plane, float *__restrict__ q) {
    const size_t N = size_t(nx) * ny;
    for (size_t t = blockIdx.x * size_t(blockDim.x) + threadIdx.x; t < N;
         t += size_t(gridDim.x) * blockDim.x) {
        const int j = int(t / nx), i = int(t - size_t(j) * nx);
        const size_t g = size_t(j) * pitch + i;
        for (int k = 0; k < 3; ++k) q[k * plane + g] = cand[k * N + t];
    }
}

qla_status ctx_ok(qla_ctx *c) {
    if (!c) return QLA_EINVAL;
    if (c->sticky != QLA_OK) return c->sticky;
    if (c->prec != QLA_FP32 || c->P != 3 || c->vmode != qla::V_ROTATION) return QLA_EINVAL;
    if (!c->has_medium || !c->has_state) return QLA_ESTATE;
    return QLA_OK;
}

}  // namespace

extern "C" {

size_t surr_workspace_bytes(int height, int width, int max_batch) {
    if (height < 16 || width < 16 || height % 16 || width % 16 || max_batch < 1) return 0;
    // the elementwise kernels index the widest level-0 tensor with 32 bits
    if ((long long)max_batch * height * width * 32 >= (1LL << 31)) return 0;
    surr_net n;
    n.H = height;
    n.W = width;
    n.maxB = max_batch;
    return carve_all(&n);
}

qla_status surr_create(surr_net **out, int height, int width, int max_batch,
                       unsigned long long seed, void *cuda_stream, void *workspace,
                       size_t workspace_bytes) {
    if (!out) return QLA_EINVAL;
    *out = nullptr;
    const size_t need = surr_workspace_bytes(height, width, max_batch);
    if (need == 0) return QLA_EINVAL;
    if (!workspace || workspace_bytes < need || (reinterpret_cast<uintptr_t>(workspace) & 255))
        return QLA_EINVAL;
    surr_net *n = new (std::nothrow) surr_net();
    if (!n) return QLA_ENOMEM;
    n->H = height;
    n->W = width;
    n->maxB = max_batch;
    n->stream = static_cast<cudaStream_t>(cuda_stream);
    n->mem = static_cast<char *>(workspace);
    carve_all(n);
    // the output layer's dz keeps zeros in its padded channels
    if (cudaMemsetAsync(n->flag, 0, sizeof(int), n->stream) != cudaSuccess ||
        cudaMemsetAsync(n->applied, 0, sizeof(long long), n->stream) != cudaSuccess ||
        cudaMallocHost(&n->lhost, 16) != cudaSuccess ||
        cudaEventCreateWithFlags(&n->ldone, cudaEventDisableTiming) != cudaSuccess ||
        cudaMemsetAsync(n->dz9, 0, blocked_elems(max_batch, CPAD, height, width) * 2,
                        n->stream) != cudaSuccess) {
        cudaGetLastError();
        surr_destroy(n);
        return QLA_ECUDA;
    }
    // He-style initialisation from a seeded generator (host), zero biases
    std::mt19937_64 rng(seed);
    for (int i = 0; i < NCONV; ++i) {
        const ConvSpec s = spec(i);
        LayerParams &l = n->prm.l[i];
        std::vector<float> w(n->nw[i], 0.f);
        const double fan_in = 9.0 * s.cin_real;
        std::normal_distribution<double> nd(0.0, std::sqrt(2.0 / fan_in) * (i == 9 ? 0.1 : 1.0));
        for (int co = 0; co < s.cout_real; ++co)
            for (int t = 0; t < 9; ++t)
                for (int ci = 0; ci < s.cin_real; ++ci)
                    w[(size_t(co) * 9 + t) * s.cin + ci] = float(nd(rng));
        if (cudaMemcpyAsync(l.w, w.data(), n->nw[i] * 4, cudaMemcpyHostToDevice, n->stream) ||
            cudaMemsetAsync(l.b, 0, s.cout * 4, n->stream) ||
            cudaMemsetAsync(l.mw, 0, n->nw[i] * 4, n->stream) ||
            cudaMemsetAsync(l.vw, 0, n->nw[i] * 4, n->stream) ||
            cudaMemsetAsync(l.mb, 0, s.cout * 4, n->stream) ||
            cudaMemsetAsync(l.vb, 0, s.cout * 4, n->stream) ||
            cudaStreamSynchronize(n->stream)) {
            surr_destroy(n);
            return QLA_ECUDA;
        }
    }
    if (refresh_copies(n->prm, NCONV, n->stream) != cudaSuccess ||
        cudaStreamSynchronize(n->stream) != cudaSuccess) {
        surr_destroy(n);
        return QLA_ECUDA;
    }
    *out = n;
    return QLA_OK;
}

long long surr_param_count(const surr_net *n) {
    (void)n;
    long long c = 0;
    for (int i = 0; i < NCONV; ++i) {
        const ConvSpec s = spec(i);
        c += (long long)s.cout_real * s.cin_real * 9 + s.cout_real;
    }
    return c;
}

// Host layout, per conv layer: weights (cout, cin, 3, 3) then bias (cout),
// real channel counts; ky, kx = dy + 1, dx + 1.
static qla_status params_io(surr_net *n, float *host, bool get, bool grads) {
    if (!n || !host) return QLA_EINVAL;
    int flag = 0;   // read with the last layer
    size_t off = 0;
    for (int i = 0; i < NCONV; ++i) {
        const ConvSpec s = spec(i);
        std::vector<float> w(n->nw[i]), b(s.cout);
        float *dw = grads ? n->prm.l[i].gw : n->prm.l[i].w;
        float *db = grads ? n->prm.l[i].gb : n->prm.l[i].b;
        if (get || true) {
            NCUDA(n, cudaMemcpyAsync(w.data(), dw, n->nw[i] * 4, cudaMemcpyDeviceToHost, n->stream),
                  "surrogate: params");
            NCUDA(n, cudaMemcpyAsync(b.data(), db, s.cout * 4, cudaMemcpyDeviceToHost, n->stream),
                  "surrogate: params");
            if (get && i == NCONV - 1)
                NCUDA(n, cudaMemcpyAsync(&flag, n->flag, sizeof flag, cudaMemcpyDeviceToHost,
                                         n->stream), "surrogate: wait flag");
            NCUDA(n, cudaStreamSynchronize(n->stream), "surrogate: sync");
        }
        for (int co = 0; co < s.cout_real; ++co)
            for (int ci = 0; ci < s.cin_real; ++ci)
                for (int t = 0; t < 9; ++t) {
                    float &d = w[(size_t(co) * 9 + t) * s.cin + ci];
                    float &h = host[off + (size_t(co) * s.cin_real + ci) * 9 + t];
                    if (get) h = d; else d = h;
                }
        off += size_t(s.cout_real) * s.cin_real * 9;
        for (int co = 0; co < s.cout_real; ++co) {
            if (get) host[off + co] = b[co]; else b[co] = host[off + co];
        }
        off += s.cout_real;
        if (!get) {
            NCUDA(n, cudaMemcpyAsync(dw, w.data(), n->nw[i] * 4, cudaMemcpyHostToDevice, n->stream),
                  "surrogate: params");
            NCUDA(n, cudaMemcpyAsync(db, b.data(), s.cout * 4, cudaMemcpyHostToDevice, n->stream),
                  "surrogate: params");
            NCUDA(n, cudaStreamSynchronize(n->stream), "surrogate: sync");
        }
    }
    if (!get) {
        NCUDA(n, refresh_copies(n->prm, NCONV, n->stream), "surrogate: params");
        NCUDA(n, cudaStreamSynchronize(n->stream), "surrogate: sync");
    }
    return flag ? wait_ran_out(n) : QLA_OK;
}

qla_status surr_get_params(surr_net *n, float *host) { return params_io(n, host, true, false); }
qla_status surr_set_params(surr_net *n, const float *host) {
    return params_io(n, const_cast<float *>(host), false, false);
}

qla_status surr_forward(surr_net *n, const float *feat_dev, int B, float *out_dev) {
    if (!n || !feat_dev || !out_dev) return QLA_EINVAL;
    qla_status s = check_batch(n, B);
    if (s != QLA_OK) return s;
    if ((s = pack(n, feat_dev, B)) != QLA_OK) return s;
    return forward(n, B, out_dev);
}

qla_status surr_loss_grad(surr_net *n, const float *feat_dev, const float *target_dev, int B,
                          double *loss_out, float *grad_host) {
    if (!n || !feat_dev || !target_dev) return QLA_EINVAL;
    qla_status s = enqueue_grad(n, feat_dev, target_dev, B);
    if (s != QLA_OK) return s;
    double l = 0.0;
    if ((s = loss_end(n, &l)) != QLA_OK) return s;
    if (loss_out) *loss_out = l;
    if (grad_host) return params_io(n, grad_host, true, true);
    return QLA_OK;
}

// The whole step is enqueued before the host waits for the loss, so the GPU
// does not idle between the loss and the backward pass.  If a wait ran out,
// Adam skips its update: a wait before the loss is reported here, one after
// it by the next call that reads the flag, which takes the step back.
qla_status surr_train_step(surr_net *n, const float *feat_dev, const float *target_dev, int B,
                           float lr, double *loss_out) {
    if (!n || !feat_dev || !target_dev) return QLA_EINVAL;
    qla_status s = enqueue_grad(n, feat_dev, target_dev, B);
    if (s != QLA_OK) return s;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const long long step = n->step + 1;
    const float c1 = float(1.0 - std::pow(0.9, double(step)));
    const float c2 = float(1.0 - std::pow(0.999, double(step)));
    NCUDA(n, adam(n->prm, NCONV, lr, b1, b2, eps, c1, c2, step, n->flag, n->applied, n->stream),
          "surrogate: adam");
    double l = 0.0;
    if ((s = loss_end(n, &l)) != QLA_OK) return s;
    n->step = step;
    if (loss_out) *loss_out = l;
    return QLA_OK;
}

const char *surr_last_error(const surr_net *n) { return n ? n->err.c_str() : "null network"; }

void surr_destroy(surr_net *n) {
    if (!n) return;
    cudaStreamSynchronize(n->stream);
    if (n->ldone) cudaEventDestroy(n->ldone);
    if (n->lhost) cudaFreeHost(n->lhost);
    delete n;
}

qla_status surr_features(qla_ctx *c, float *feat_dev) {
    qla_status s = ctx_ok(c);
    if (s != QLA_OK) return s;
    if (!feat_dev) return QLA_EINVAL;
    const size_t N = size_t(c->nx) * c->ny;
    k_features<<<int(std::min<size_t>((N + 255) / 256, 8192)), 256, 0, c->stream>>>(
        static_cast<const float *>(c->state[c->cur]), c->plane_elems, c->nx, c->ny, c->pitch,
        c->pending_v, c->midx, static_cast<const qla::MedRec<float> *>(c->table), c->n, feat_dev);
    return cudaGetLastError() == cudaSuccess ? QLA_OK : QLA_ECUDA;
}

qla_status surr_advance(qla_ctx *c, surr_net *n, int windows, int K, double energy_tol,
                        double div_tol, float *scratch_dev, int *accepted, double *energies) {
    qla_status s = ctx_ok(c);
    if (s != QLA_OK) return s;
    if (!n || !scratch_dev || windows < 0 || K < 1 || n->H != c->ny || n->W != c->nx)
        return QLA_EINVAL;
    const size_t N = size_t(c->nx) * c->ny;
    float *feat = scratch_dev, *y = feat + N * FEAT, *cand = y + N * NOUT;
    const int blocks = 256;
    double *sums = n->lpart;  // blocks * 3 doubles
    int acc = 0;
    for (int wdx = 0; wdx < windows; ++wdx) {
        double e0 = 0.0;
        if ((s = qla_energy(c, &e0)) != QLA_OK) return s;
        if ((s = surr_features(c, feat)) != QLA_OK) return s;
        if ((s = surr_forward(n, feat, 1, y)) != QLA_OK) return s;
        k_candidate<<<blocks, 256, 0, c->stream>>>(feat, y, c->nx, c->ny, cand, sums);
        std::vector<double> h(size_t(blocks) * 3);
        if (cudaMemcpyAsync(h.data(), sums, h.size() * 8, cudaMemcpyDeviceToHost, c->stream) ||
            cudaStreamSynchronize(c->stream))
            return QLA_ECUDA;
        if ((s = tc_waits_ok(n)) != QLA_OK) return s;
        double e1 = 0.0, dd = 0.0, gg = 0.0;
        for (int b = 0; b < blocks; ++b) {
            e1 += h[b * 3];
            dd += h[b * 3 + 1];
            gg += h[b * 3 + 2];
        }
        const bool ok = std::fabs(e1 / e0 - 1.0) <= energy_tol &&
                        std::sqrt(dd / (gg > 0 ? gg : 1e-300)) <= div_tol;
        if (ok) {
            k_store_candidate<<<int(std::min<size_t>((N + 255) / 256, 8192)), 256, 0, c->stream>>>(
                cand, c->nx, c->ny, c->pitch, c->plane_elems, static_cast<float *>(c->state[c->cur]));
            if (cudaGetLastError() != cudaSuccess) return QLA_ECUDA;
            c->pending_v = false;
            ++acc;
        } else {
            if ((s = qla_step(c, K)) != QLA_OK) return s;
        }
        if (energies && (s = qla_energy(c, energies + wdx)) != QLA_OK) return s;
    }
    if (accepted) *accepted = acc;
    return QLA_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Direct access to the two contraction kernels, for exactness tests: with
// BF16 inputs their only rounding is the FP32 accumulation.
// ---------------------------------------------------------------------------
namespace {
// Stream-ordered scratch, given back on every path.
struct Scratch {
    cudaStream_t st;
    void *p = nullptr;
    explicit Scratch(cudaStream_t s) : st(s) {}
    ~Scratch() { if (p) cudaFreeAsync(p, st); }
    template <typename T> T *get(size_t n) {
        return cudaMallocAsync(&p, n * sizeof(T), st) == cudaSuccess ? static_cast<T *>(p)
                                                                     : nullptr;
    }
};

// Whether the layout conversion can read a tensor's pixels (16 bytes at a time).
bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// Waits for the stream; QLA_ETIMEOUT if a wait of the call's kernels ran out.
qla_status raw_waits_ok(const int *flag_dev, cudaStream_t st) {
    int flag = 0;
    if (cudaMemcpyAsync(&flag, flag_dev, sizeof flag, cudaMemcpyDeviceToHost, st) ||
        cudaStreamSynchronize(st))
        return QLA_ECUDA;
    return flag ? QLA_ETIMEOUT : QLA_OK;
}
}  // namespace

extern "C" qla_status surr_conv3x3_raw(const void *in_bf16, int B, int H, int W, int cin,
                                       const void *w_bf16, int cout, float *out_f32,
                                       void *cuda_stream) {
    if (!in_bf16 || !w_bf16 || !out_f32 || B < 1 || H < 1 || W < 1 || cin % 32 || cout % 32)
        return QLA_EINVAL;
    if (!aligned16(in_bf16)) return QLA_ECUDA;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    Scratch sx(st), sw(st), so(st), sf(st);
    bf16 *x = sx.get<bf16>(blocked_elems(B, cin, H, W));
    bf16 *w = sw.get<bf16>(size_t(cout) * 9 * cin);
    float *o = so.get<float>(size_t(B) * H * W * cout);
    int *flag_dev = sf.get<int>(1);
    if (!x || !w || !o || !flag_dev || cudaMemsetAsync(flag_dev, 0, sizeof(int), st)) {
        cudaGetLastError();
        return QLA_ECUDA;
    }
    ConvArgs a{};
    a.in = x;
    a.B = B;
    a.H = H;
    a.W = W;
    a.cin = cin;
    a.cout = cout;
    a.w = w;
    a.out_f = o;
    a.err = flag_dev;
    if (nhwc_to_blocked(static_cast<const bf16 *>(in_bf16), B, H, W, cin, x, st) != cudaSuccess ||
        block_weights(static_cast<const bf16 *>(w_bf16), cout, cin, w, st) != cudaSuccess ||
        conv3x3(a, EP_F32, st) != cudaSuccess ||
        blocked_to_nhwc_f32(o, B, H, W, cout, out_f32, st) != cudaSuccess)
        return QLA_ECUDA;
    return raw_waits_ok(flag_dev, st);
}

extern "C" qla_status surr_test_stall_conv(int on) {
    return conv_tc_stall(on == 2 ? 2 : on ? 1 : 0) == cudaSuccess ? QLA_OK : QLA_ECUDA;
}

extern "C" qla_status surr_weight_grad_raw(const void *dz_bf16, const void *in_bf16, int B, int H,
                                           int W, int cout, int cin, int splits, float *part,
                                           float *dw_f32, void *cuda_stream) {
    if (!dz_bf16 || !in_bf16 || !part || !dw_f32 || cin % 32 || cout % 32 || splits < 1)
        return QLA_EINVAL;
    if (!aligned16(dz_bf16) || !aligned16(in_bf16)) return QLA_ECUDA;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (B < 1 || H < 1 || W < 1) {   // no pixels: the sums are zero
        const size_t n = size_t(cout) * 9 * cin;
        return cout > 0 && cin > 0 && cudaMemsetAsync(part, 0, splits * n * 4, st) == cudaSuccess &&
                       cudaMemsetAsync(dw_f32, 0, n * 4, st) == cudaSuccess
                   ? QLA_OK : QLA_ECUDA;
    }
    Scratch sz(st), sx(st), sf(st);
    bf16 *z = sz.get<bf16>(blocked_elems(B, cout, H, W));
    bf16 *x = sx.get<bf16>(blocked_elems(B, cin, H, W));
    int *flag_dev = sf.get<int>(1);
    if (!z || !x || !flag_dev || cudaMemsetAsync(flag_dev, 0, sizeof(int), st)) {
        cudaGetLastError();
        return QLA_ECUDA;
    }
    SumJobs jobs{};
    jobs.j[0] = {part, dw_f32, splits, (long long)cout * 9 * cin};
    if (nhwc_to_blocked(static_cast<const bf16 *>(dz_bf16), B, H, W, cout, z, st) != cudaSuccess ||
        nhwc_to_blocked(static_cast<const bf16 *>(in_bf16), B, H, W, cin, x, st) != cudaSuccess ||
        weight_grad(z, x, B, H, W, cout, cin, splits, part, flag_dev, st) != cudaSuccess ||
        sum_splits(jobs, 1, st) != cudaSuccess)
        return QLA_ECUDA;
    // a stream that is being captured cannot be waited for
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) == cudaSuccess && cap != cudaStreamCaptureStatusNone)
        return QLA_OK;
    return raw_waits_ok(flag_dev, st);
}
