// Tile kernel of the QLA step: Eq. 2e14 on any lattice size, FP64 or FP32,
// six planes or the E_z triple, every potential reading, tensor media; one
// step per launch, or, on lattices whose tiles are all resident at once, all
// the steps of a qla_step call in one launch.
//
// A CTA owns a tile of at most 24 x 24 sites and works on the 32 x 32 region
// around it: U_x and U_y each reach four cells along their axis (four of
// their eight layers pair neighbouring sites).  Both are done in registers
// with one site per lane and the neighbour layers' partners by shuffle:
//  * U_x: a warp takes whole region rows, lane = column.  The row comes
//    straight from global memory (with the previous step's V_x, V_y applied
//    where pending); planes that U_y does not touch are final and stored,
//    the others go to shared memory.
//  * U_y: a warp takes region columns, lane = row, read from shared memory
//    (rows padded to 33 sites, so neither direction has bank conflicts) and
//    written back for a coalesced store.
// Two barriers per step instead of one per layer, and a shared-memory round
// trip per direction instead of one per layer.  The region's outer four
// cells on each side are the recomputed halo; lanes outside the lattice's
// tile hold whatever their neighbours give, which reaches halo cells only.
//
// Several steps per launch (n_steps > 1): the CTA keeps its region's
// collision coefficients and record indices in shared memory and waits
// before each step until its eight neighbours have published the step
// before (their outputs are its halo; they have also read the buffer it is
// about to overwrite).  The launch is cooperative, so every tile is
// resident.  Every wait is bounded: one that runs out raises *err, the CTAs
// return, and the host reads QLA_ETIMEOUT at the next synchronising call.
//
// What bounds it: on small lattices latency (barriers, the exchange through
// L2); with many tiles, instruction issue (FP32) or the FP64 pipe, on the
// 1.55 x 576 sites per tile the halo costs.  Measured per step, us (other:
// the marching kernel, or for odd sides and tensor media a tile kernel that
// kept the whole region in shared memory and took one barrier and one round
// trip through it per layer):
//                            other   per-step tiles   resident tiles
//   256^2 FP32 E_z            16.6        6.3              3.4
//   512^2 FP32 E_z            17.8       10.4              6.9
//   512^2 FP32 six planes     43         14.5             10.3
//   256^2 FP64 E_z           166         18.6             15.2
//   640^2 FP64 E_z           166         70                -
//   1023 x 769 FP32 E_z       34         18.8              -
//   1024^2 FP32 tensor       100         48.7              -
//
// For a diagonal index tensor (six planes) each pair class has its own
// coefficient and this step's V is applied before storing; so it is for the
// LCU form of V (Eqs. 2f1-2f7).
#include <algorithm>

#include "qla_march.cuh"
#include "qla_plateau.cuh"

namespace qla {
namespace {

using march::bond_rot;
using march::layer_sign;
using march::shfl_dn1;
using march::shfl_up1;

constexpr int HALO = 4;
constexpr int REG = 32;              // region side (one warp)
constexpr int TILE = REG - 2 * HALO; // largest tile side
constexpr int LINE = REG + 1;        // padded region row in shared memory
constexpr int AREA = REG * LINE;
constexpr int TILE_WARPS = 8, MAX_WARPS = 16;

// Both components of one pair along a line of 32 sites, one per lane, through
// the eight layers of U.  a_m1: the pair's first component is the S1 mover.
template <typename T, bool XDIR, bool AM1, int L>
__device__ __forceinline__ void line_layer(T &a, T &b, const typename Coef<T>::C &k) {
    constexpr Layer ly = layer_of(L);
    const T g = T(layer_sign<XDIR, L>());
    if constexpr (ly.mover == 0) {
        rotate(a, b, k, g);
    } else {
        constexpr bool am = (ly.mover == 1) == AM1;   // a is the moved one
        T &m = am ? a : b;
        T &u = am ? b : a;
        // the bond at this lane's site takes the partner of the neighbouring
        // lane and returns the result to it
        T p = ly.shift < 0 ? shfl_up1(m) : shfl_dn1(m);
        bond_rot(u, p, k, g, am);
        m = ly.shift < 0 ? shfl_dn1(p) : shfl_up1(p);
    }
}

// N independent lines (rows or columns of the same pair), layer by layer.
template <typename T, bool XDIR, bool AM1, int N>
__device__ __forceinline__ void lines_U(T (&a)[N], T (&b)[N],
                                        const typename Coef<T>::C (&k)[N]) {
#define QLA_LAYER(L)                                                          \
    _Pragma("unroll") for (int n = 0; n < N; ++n)                             \
        line_layer<T, XDIR, AM1, L>(a[n], b[n], k[n]);
    QLA_LAYER(0) QLA_LAYER(1) QLA_LAYER(2) QLA_LAYER(3)
    QLA_LAYER(4) QLA_LAYER(5) QLA_LAYER(6) QLA_LAYER(7)
#undef QLA_LAYER
}

// Tiles of one lattice: n_tx x n_ty, of qx columns and qy rows, the first rx
// and ry along each axis one wider.  Two or more tiles along an axis are at
// least 12 wide there, so a halo meets the adjacent tiles only.  (Quotients
// and remainders come from the host: divisions cost each warp of a tile as
// many instructions as several rows of sites.)
struct TileGrid {
    int n_tx, n_ty, qx, rx, qy, ry;
    TileGrid() = default;
    TileGrid(int nx, int ny, int tx, int ty)
        : n_tx(tx), n_ty(ty), qx(nx / tx), rx(nx % tx), qy(ny / ty), ry(ny % ty) {}
};

// i mod n for i within a region of the lattice: at most a few periods away
// on lattices smaller than the region, one otherwise (cheaper than %).
__device__ __forceinline__ int wrap_near(int i, int n) {
    while (i < 0) i += n;
    while (i >= n) i -= n;
    return i;
}

// Wait until the 3 x 3 tiles around (tx, ty) have published `need` steps.
// Gives up after `budget` SM cycles or when another CTA has raised *err.
__device__ __forceinline__ bool tiles_ready(const unsigned *done, int tx, int ty, TileGrid tg,
                                            unsigned need, int *err, long long budget) {
    int bad = 0;
    if (threadIdx.x < 9) {
        int i = tx + int(threadIdx.x) % 3 - 1, j = ty + int(threadIdx.x) / 3 - 1;
        i = i < 0 ? tg.n_tx - 1 : i == tg.n_tx ? 0 : i;
        j = j < 0 ? tg.n_ty - 1 : j == tg.n_ty ? 0 : j;
        const unsigned *f = done + j * tg.n_tx + i;
        const long long t0 = clock64();
        int polls = 0;
        while (march::ld_acquire_gpu(f) < need) {
            if ((++polls & 63) == 0 &&
                (clock64() - t0 > budget || *static_cast<volatile int *>(err) != 0)) {
                bad = 1;
                atomicExch(err, 1);
                break;
            }
        }
    }
    return __syncthreads_or(bad) == 0;
}

// TS: a diagonal index tensor (QLA_ANISOTROPIC, six planes): per-site
// records in ttable, each pair with its own coefficient.
template <typename T, int P, int VM, bool TS>
__global__ void __launch_bounds__(32 * MAX_WARPS)
k_step_tile(T *a, T *b, const uint32_t *__restrict__ midx, const MedRec<T> *__restrict__ table,
            const MedRecT<T> *__restrict__ ttable, int nx, int ny, int pitch, size_t plane_elems,
            TileGrid tg, bool vin0, int n_steps, unsigned *done, int *err, long long budget,
            long long withhold) {
    using C = typename Coef<T>::C;
    // FULL: this step's V is applied before the store, so every plane goes
    // through shared memory; otherwise only the planes of U_y do
    constexpr bool FULL = TS || VM == V_LCU;
    constexpr bool VIN = !FULL && VM != V_NONE;
    constexpr int NP = FULL ? nplanes<P>() : P == 6 ? 4 : 2;
    // plane of amplitude c in shared memory (-1: none)
    auto slot = [](int c) {
        if (plane_of<P>(c) < 0) return -1;
        if (FULL) return slot_of<P>(c);
        if (P == 6) return c == 0 ? 0 : c == 2 ? 1 : c == 3 ? 2 : c == 5 ? 3 : -1;
        return c == 2 ? 0 : c == 3 ? 1 : -1;
    };
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *sc = reinterpret_cast<C *>(smem_raw);              // coefficients (with q2)
    C *sc5 = sc + AREA;                                   // TS: y coefficients with q5
    T *sq = reinterpret_cast<T *>(sc + (TS ? 2 : 1) * AREA);
    uint32_t *sid = reinterpret_cast<uint32_t *>(sq + NP * AREA);

    // the warp index through a shuffle, so that the compiler knows it is
    // uniform: row addresses then live in uniform registers
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0);
    const int tx = int(blockIdx.x) % tg.n_tx, ty = int(blockIdx.x) / tg.n_tx;
    const int x0 = tx * tg.qx + min(tx, tg.rx), w = tg.qx + (tx < tg.rx ? 1 : 0);
    const int y0 = ty * tg.qy + min(ty, tg.ry), h = tg.qy + (ty < tg.ry ? 1 : 0);
    const int rows = h + 2 * HALO;
    const unsigned ux = unsigned(wrap_near(x0 - HALO + lane, nx));
    const bool col_in = lane >= HALO && lane < HALO + w;

    // region rows beyond the tile's halo are read by lanes whose values no
    // output depends on; give them defined values
    for (int t = rows * LINE + int(threadIdx.x); t < AREA; t += int(blockDim.x)) {
        sc[t] = C{};
        if constexpr (TS) sc5[t] = C{};
#pragma unroll
        for (int p = 0; p < NP; ++p) sq[p * AREA + t] = T(0);
    }

    for (int s = 0; s < n_steps; ++s) {
        if (s > 0 && !tiles_ready(done, tx, ty, tg, unsigned(s), err, budget)) return;
        const T *in = (s & 1) ? b : a;
        T *out = (s & 1) ? a : b;
        const bool vin = s > 0 || vin0;

        // U_x, two rows at a time (two independent chains per lane)
        for (int r0 = warp; r0 < rows; r0 += 2 * nw) {
            T q[2][6];
            C k[2], k5[2];
            size_t g[2];
            int row[2];
            uint32_t id[2];
            const bool second = r0 + nw < rows;   // warp-uniform
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                row[n] = n == 0 || second ? r0 + n * nw : r0;
                g[n] = size_t(wrap_near(y0 - HALO + row[n], ny)) * pitch;
#pragma unroll
                for (int c = 0; c < 6; ++c)
                    if (plane_of<P>(c) >= 0)
                        q[n][c] = __ldcg((in + plane_of<P>(c) * plane_elems + g[n]) + ux);
                const int t = row[n] * LINE + lane;
                if constexpr (TS) {
                    k5[n] = (ttable + g[n])[ux].c15;
                    k[n] = s == 0 ? (ttable + g[n])[ux].c2 : sc[t];
                } else {
                    id[n] = s == 0 ? (midx + g[n])[ux] : sid[t];
                    k[n] = s == 0 ? table[id[n]].c : sc[t];
                    k5[n] = k[n];
                }
            }
            if (s == 0) {
#pragma unroll
                for (int n = 0; n < 2; ++n) {
                    if (n > 0 && !second) break;
                    const int t = row[n] * LINE + lane;
                    sc[t] = k[n];
                    if constexpr (TS) sc5[t] = (ttable + g[n])[ux].c05;
                    else sid[t] = id[n];
                }
            }
            if constexpr (VIN) {
                // V is exactly the identity on shared-record sites
#pragma unroll
                for (int n = 0; n < 2; ++n)
                    if (vin && id[n] >= uint32_t(UNIFORM_SLOTS))
                        apply_potential<T, P, VM>(q[n], table[id[n]].v);
            }
            {
                T u[2] = {q[0][2], q[1][2]}, v[2] = {q[0][4], q[1][4]};
                lines_U<T, true, false>(u, v, k);
                q[0][2] = u[0]; q[1][2] = u[1]; q[0][4] = v[0]; q[1][4] = v[1];
            }
            if constexpr (P == 6) {
                T u[2] = {q[0][1], q[1][1]}, v[2] = {q[0][5], q[1][5]};
                lines_U<T, true, true>(u, v, k5);
                q[0][1] = u[0]; q[1][1] = u[1]; q[0][5] = v[0]; q[1][5] = v[1];
            }
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                if (n > 0 && !second) break;
                const bool in_tile = col_in && unsigned(row[n] - HALO) < unsigned(h);
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    if (plane_of<P>(c) < 0) continue;
                    if (slot(c) >= 0) sq[slot(c) * AREA + row[n] * LINE + lane] = q[n][c];
                    else if (in_tile) (out + plane_of<P>(c) * plane_elems + g[n])[ux] = q[n][c];
                }
            }
        }
        __syncthreads();

        // U_y, lane = row: three columns at a time while three are left (24
        // columns over 8 warps), then one
        const bool keep = unsigned(lane - HALO) < unsigned(h);
        auto columns = [&](auto count, int c0) {
            constexpr int N = decltype(count)::value;
            C k[N], k5[N];
            T u[N], v[N];
            const int t0 = lane * LINE + HALO + c0;
#pragma unroll
            for (int n = 0; n < N; ++n) {
                k[n] = sc[t0 + n * nw];
                k5[n] = TS ? sc5[t0 + n * nw] : k[n];
            }
            T *p2 = sq + slot(2) * AREA + t0, *p3 = sq + slot(3) * AREA + t0;
#pragma unroll
            for (int n = 0; n < N; ++n) { u[n] = p2[n * nw]; v[n] = p3[n * nw]; }
            lines_U<T, false, false>(u, v, k);
            if (keep) {
#pragma unroll
                for (int n = 0; n < N; ++n) { p2[n * nw] = u[n]; p3[n * nw] = v[n]; }
            }
            if constexpr (P == 6) {
                T *p0 = sq + slot(0) * AREA + t0, *p5 = sq + slot(5) * AREA + t0;
#pragma unroll
                for (int n = 0; n < N; ++n) { u[n] = p0[n * nw]; v[n] = p5[n * nw]; }
                lines_U<T, false, true>(u, v, k5);
                if (keep) {
#pragma unroll
                    for (int n = 0; n < N; ++n) { p0[n * nw] = u[n]; p5[n * nw] = v[n]; }
                }
            }
        };
        {
            int c0 = warp;
            for (; c0 + 2 * nw < w; c0 += 3 * nw) columns(std::integral_constant<int, 3>{}, c0);
            for (; c0 < w; c0 += nw) columns(std::integral_constant<int, 1>{}, c0);
        }
        __syncthreads();

        if (col_in) {
            for (int r = warp; r < h; r += nw) {
                const int t = (r + HALO) * LINE + lane;
                const size_t g = size_t(y0 + r) * pitch;
                T q[6];
#pragma unroll
                for (int c = 0; c < 6; ++c) q[c] = slot(c) >= 0 ? sq[slot(c) * AREA + t] : T(0);
                if constexpr (TS) {
                    const MedRecT<T> &rec = (ttable + g)[ux];
                    apply_potential_tensor<T, P, VM>(q, rec.vz, rec.vt);   // V_y V_x (Eq. 2e14)
                } else if constexpr (VM == V_LCU) {
                    apply_potential<T, P, VM>(q, table[(midx + g)[ux]].v);   // Eqs. 2f1-2f7
                }
#pragma unroll
                for (int c = 0; c < 6; ++c)
                    if (slot(c) >= 0) (out + plane_of<P>(c) * plane_elems + g)[ux] = q[c];
            }
        }
        if (s + 1 < n_steps) {
            // publish: every thread's stores, then the tile's counter
            __syncthreads();
            if (threadIdx.x == 0 &&
                (long long)s * (tg.n_tx * tg.n_ty) + blockIdx.x != withhold) {
                __threadfence();
                atomicExch(done + blockIdx.x, unsigned(s + 1));
            }
        }
    }
}

template <typename T, int P, int VM, bool TS> struct TileKernel {
    static constexpr int NP = TS || VM == V_LCU ? nplanes<P>() : P == 6 ? 4 : 2;
    static constexpr size_t SMEM = size_t(AREA) * ((TS ? 2 : 1) * sizeof(typename Coef<T>::C) +
                                                   NP * sizeof(T) + (TS ? 0 : 4));
    // resident CTAs per SM with TILE_WARPS and with MAX_WARPS warps
    struct Occ { cudaError_t err; int per_sm, per_sm16; };
    // per instantiation, per process; initialised once (thread-safe)
    static const Occ &occ() {
        static const Occ o = [] {
            auto kern = k_step_tile<T, P, VM, TS>;
            Occ v{cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       int(SMEM)), 0, 0};
            if (v.err == cudaSuccess)
                v.err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v.per_sm, kern,
                                                                      32 * TILE_WARPS, SMEM);
            if (v.err == cudaSuccess)
                v.err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v.per_sm16, kern,
                                                                      32 * MAX_WARPS, SMEM);
            return v;
        }();
        return o;
    }
};

// The tile counts along each axis that give the shortest step with at most
// `cap` tiles: whole waves of tiles over the SMs, each costing its region
// rows and its columns (the warps' work in U_x and U_y).  n_tx = 0 if even
// the largest tiles are more than cap.
TileGrid resident_tiles(int nx, int ny, int num_sms, long long cap) {
    TileGrid best;
    best.n_tx = 0;
    long long best_cost = -1;
    auto lo = [](int n) { return (n + TILE - 1) / TILE; };
    // tiles of 12 or more sites a side, one tile on axes shorter than that
    auto hi = [&](int n) { return std::max(lo(n), n / 12); };
    for (int i = lo(nx); i <= hi(nx); ++i) {
        for (int j = lo(ny); j <= hi(ny); ++j) {
            const long long tiles = (long long)i * j;
            if (tiles > cap) break;
            const long long waves = (tiles + num_sms - 1) / num_sms;
            const long long cost = waves * ((ny + j - 1) / j + 2 * HALO + (nx + i - 1) / i);
            if (best_cost < 0 || cost < best_cost) {
                best = TileGrid(nx, ny, i, j);
                best_cost = cost;
            }
        }
    }
    return best;
}

template <typename T, int P, int VM, bool TS = false>
cudaError_t launch_tile_t(qla_ctx *c, const void *in, void *out, bool vin, long long n_steps,
                          bool *resident) {
    using K = TileKernel<T, P, VM, TS>;
    const auto &occ = K::occ();
    if (occ.err != cudaSuccess) return occ.err;
    auto kern = k_step_tile<T, P, VM, TS>;
    T *a = static_cast<T *>(const_cast<void *>(in)), *b = static_cast<T *>(out);
    const MedRec<T> *table = static_cast<const MedRec<T> *>(c->table);
    const MedRecT<T> *ttable = static_cast<const MedRecT<T> *>(c->ttable);
    if (!resident) {
        const TileGrid tg(c->nx, c->ny, (c->nx + TILE - 1) / TILE, (c->ny + TILE - 1) / TILE);
        kern<<<unsigned(tg.n_tx) * unsigned(tg.n_ty), 32 * TILE_WARPS, K::SMEM, c->stream>>>(
            a, b, c->midx, table, ttable, c->nx, c->ny, c->pitch, c->plane_elems, tg, vin, 1,
            nullptr, nullptr, 0, -1);
        return cudaGetLastError();
    }
    *resident = false;
    // FP64 (pipe-bound) gains nothing from tiles that share an SM for many
    // steps: one tile per SM, the per-step launches beyond (384^2 E_z equal,
    // 512^2 57.6 us per step against 62.6)
    const int per_sm = std::is_same<T, double>::value ? 1 : occ.per_sm;
    TileGrid tg = resident_tiles(
        c->nx, c->ny, c->num_sms,
        std::min<long long>((long long)per_sm * c->num_sms, TILE_COUNTERS));
    if (tg.n_tx == 0) return cudaSuccess;
    // an SM that holds one tile hides its latencies with 16 warps (256^2:
    // FP32 3.4 us per step against 4.0 with 8, FP64 15.2 against 15.8)
    const int warps = tg.n_tx * tg.n_ty <= c->num_sms && occ.per_sm16 > 0 ? MAX_WARPS : TILE_WARPS;
    *resident = true;
    if (n_steps == 1) {   // nothing to wait for: an ordinary launch
        kern<<<unsigned(tg.n_tx * tg.n_ty), 32 * warps, K::SMEM, c->stream>>>(
            a, b, c->midx, table, ttable, c->nx, c->ny, c->pitch, c->plane_elems, tg, vin, 1,
            nullptr, nullptr, 0, -1);
        return cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(c->tile_done, 0, size_t(tg.n_tx) * tg.n_ty * 4, c->stream);
    if (e != cudaSuccess) return e;
    int steps = int(n_steps);
    int *err = c->wait_flag;
    long long budget = c->flow_budget, withhold = c->flow_withhold;
    void *args[] = {&a,  &b,   &c->midx, &table, &ttable,       &c->nx, &c->ny,  &c->pitch,
                    &c->plane_elems, &tg, &vin, &steps, &c->tile_done, &err, &budget, &withhold};
    e = cudaLaunchCooperativeKernel(kern, dim3(unsigned(tg.n_tx * tg.n_ty)), dim3(32 * warps),
                                    args, K::SMEM, c->stream);
    if (e == cudaSuccess) note_waits(c);
    return e;
}

template <typename T>
cudaError_t launch_tensor_vm(qla_ctx *c, const void *in, void *out, long long n, bool *r) {
    switch (c->vmode) {
    case V_ROTATION: return launch_tile_t<T, 6, V_ROTATION, true>(c, in, out, false, n, r);
    case V_LITERAL:  return launch_tile_t<T, 6, V_LITERAL, true>(c, in, out, false, n, r);
    case V_LCU:      return launch_tile_t<T, 6, V_LCU, true>(c, in, out, false, n, r);
    default:         return launch_tile_t<T, 6, V_NONE, true>(c, in, out, false, n, r);
    }
}

template <typename T, int P>
cudaError_t launch_tile_vm(qla_ctx *c, const void *in, void *out, bool vin, long long n,
                           bool *r) {
    switch (c->vmode) {
    case V_ROTATION: return launch_tile_t<T, P, V_ROTATION>(c, in, out, vin, n, r);
    case V_LITERAL:  return launch_tile_t<T, P, V_LITERAL>(c, in, out, vin, n, r);
    case V_LCU:      return launch_tile_t<T, P, V_LCU>(c, in, out, false, n, r);
    default:         return launch_tile_t<T, P, V_NONE>(c, in, out, false, n, r);
    }
}

cudaError_t launch_tiles(qla_ctx *c, const void *in, void *out, bool vin, long long n, bool *r) {
    const bool d = c->prec == QLA_FP64;
    if (c->tensor && c->P == 6)
        return d ? launch_tensor_vm<double>(c, in, out, n, r)
                 : launch_tensor_vm<float>(c, in, out, n, r);
    if (d)
        return c->P == 6 ? launch_tile_vm<double, 6>(c, in, out, vin, n, r)
                         : launch_tile_vm<double, 3>(c, in, out, vin, n, r);
    return c->P == 6 ? launch_tile_vm<float, 6>(c, in, out, vin, n, r)
                     : launch_tile_vm<float, 3>(c, in, out, vin, n, r);
}

}  // namespace

cudaError_t launch_step_tile(qla_ctx *c, const void *in, void *out, bool vin) {
    return launch_tiles(c, in, out, vin, 1, nullptr);
}

// Which steps of an automatic context the tile kernel takes from the
// marching one.  FP32 six planes: 1024^2 34.6 us per step against 45.2,
// 1536^2 equal.  FP32 E_z: resident tiles only; beyond them the march, though
// per-step tiles win up to about 1024^2 (768^2 14.5 / 16.6, 1024^2 22.7 /
// 22.7).  FP64: tiles take 0.152 to 0.170 us per 1000
// sites (E_z 1024^2 to 3072^2, compared as 0.165, which leaves 1024^2, 178 /
// 168, to the march; six planes 0.307 to 0.336, as 0.325), the march 4.2 us (8.1) per row of the items
// that its schedulers hold one of, whatever the lattice: a march has a
// window's rows in sequence, so lattices with few windows pay its latency;
// tiles pay the halo instead (E_z 768^2 98 / 166, 2048^2 655 / 539).
bool tile_steps_pay(const qla_ctx *c) {
    const size_t sites = size_t(c->nx) * c->ny;
    if (c->prec == QLA_FP32) return c->P == 6 && sites <= (size_t(3) << 19);
    const bool te = c->P == 3;
    return double(sites) * (te ? 0.165e-3 : 0.325e-3) < march64_rows(c) * (te ? 4.2 : 8.1);
}

// Calls of every length: FP32 E_z, us per step of calls of one, two and eight
// steps against the march: 512^2 10.3, 9.5, 7.4 / 16.5; 720^2 12.3, 13.4, 11.1
// / 20.6; 1024 x 448 12.3, 13.7, 10.5 / 16.4.
cudaError_t launch_steps_resident(qla_ctx *c, long long n_steps, long long *done) {
    *done = 0;
    const long long n = std::min<long long>(n_steps, 1LL << 24);
    bool resident = false;
    const cudaError_t e = launch_tiles(c, c->state[c->cur], c->state[c->cur ^ 1], c->pending_v, n,
                                       &resident);
    if (e == cudaSuccess && resident) {
        *done = n;
        c->plan_due = c->medium_gen;
    }
    return e;
}

}  // namespace qla
