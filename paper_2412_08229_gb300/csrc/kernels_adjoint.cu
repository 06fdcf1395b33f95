// kernels_adjoint.cu - the hand-written adjoint (vector-Jacobian product) of one fused
// pull-stream + neural-collision step (Sec. II.A-B), FP32 on the CUDA cores.
//
// Forward step t: f_{t+1}[x][i] = C(f_t)[src(x,i)][ip(x,i)] (pull map, a bijection), with
// C(f) = M^-1 m*, m* = m - S_theta(m) (m - m^eq(m)), m = M f (eq. omegatheta).
// Adjoint, per cell y:
//   lam*[y][j] = lam_{t+1}[x][i] for the (x, i) that pulls (y, j)  (push with reflection);
//   mu* = M^-T lam*;                                 cotangent of m*
//   dL/dm = diag(1 - s) mu* + omega_nu (dm^eq/dm)^T mu*_(order 2) + (dtheta-network term);
//   the learned rates omega_n = 1/tau_n(tau~_n), tau~ = (1/48) sum_g Phi(P_g m), get the
//   cotangent -sum_{order(e)=n} mu*_e m_e and are backpropagated through the sigmoid,
//   the group mean and the 48 copies of Phi (weights and inputs);
//   lam_t[y] = M^T dL/dm.
// The 48 elements are taken per axis permutation p: for its 8 sign vectors s the first layer
// is an 8-point Walsh-Hadamard transform of the parity-class partial sums of W1p m (the
// forward kernel's form), and so are the first layer's cotangents: with E[c][j] =
// sum_s (-1)^popcount(s & c) delta h1[s][j], the cotangent of m_t is sum_j W1p[j][t]
// E[c(t)][j] and dW1p[j][t] = sum over cells of m_t E[c(t)][j], c(t) the parity class of
// moment t.
//
// A block has twelve warps (net_f32.cuh) and a tile of 32 cells (two-layer network) or 16
// (third hidden layer). h1 of every column stays in shared memory from the forward to the
// backward part; of the last hidden layer only the signs are kept (20 bits per column), so
// nothing of the forward is computed twice. The weight gradients are outer products summed
// over columns: a lane has 10 x 6 outputs, 60 FMAs for 15 floats read.
//
// lam's arithmetic is that of one thread per cell, bit for bit: the group sum in the order of the
// group (handed from warp to warp), the cotangent of m as the relaxation's part plus 120 products
// one after the other, on small grids in 2, 3 or 6 parts. A sweep of 200 steps turns other
// roundings into up to 3e-5 of the gradient. Sums that end in the gradient are grouped freely.
// (The two sums in order: 32^3 training pass 61.1 -> 63.6 ms.)
//
// A block per SM walks over the tiles and keeps the parameter gradients in FP64 in shared
// memory, so the global atomics come once per block (a block per tile: 32^3 225 us).
//
// What bounds it (32^3, ncu): shared-memory latency and bandwidth between bursts of FMAs
// (wavefronts 50 %, issue 47 %, three warps a scheduler). One step: 32^3 213 us, with the
// third hidden layer 382 us, 16^3 38 and 61 us; before (one thread per cell, the forward
// computed twice, outer products by 40 of 128 threads): 723, 1137, 232 and 359 us.
//
// Observations of the kinetic energy k = (1/2)<|u|^2> at intermediate steps (the loss of
// Sec. IV is a function of k(t)) enter as extra seeds added to lam_t when the reverse
// sweep passes step t: dk/df_i = (1/cells) sum_a u_a (c_ia - u_a) / rho.
#include "cell.cuh"
#include "launch.cuh"
#include "net_f32.cuh"

namespace lbm {

// Gradient accumulator (doubles) in the flat parameter order W1 (printed columns), b1, W2,
// b2, (Wd, bd: third hidden layer), W3, b3.
template <bool DEEP>
struct GradLayout {
    static constexpr int kB1 = kHidden * Q;
    static constexpr int kW2 = kB1 + kHidden;
    static constexpr int kB2 = kW2 + kHidden * kHidden;
    static constexpr int kWd = kB2 + kHidden;
    static constexpr int kBd = kWd + kHidden * kHidden;
    static constexpr int kW3 = DEEP ? kBd + kHidden : kB2 + kHidden;
    static constexpr int kB3 = kW3 + kOut * kHidden;
    static constexpr int kLen = kB3 + kOut;
};
static_assert(GradLayout<false>::kLen == kNumTheta && GradLayout<true>::kLen == kNumThetaDeep, "parameter order");

int adjoint_grad_len(bool deep) { return deep ? GradLayout<true>::kLen : GradLayout<false>::kLen; }

// Column of W1p[p] that printed column k of W1 went to (the moment permutation of the
// element with axis permutation p and no reflection).
struct PermColumns {
    unsigned char t[6][Q];
};
constexpr PermColumns make_perm_columns() {
    PermColumns r{};
    const GroupTables g = make_group();
    for (int p = 0; p < 6; ++p)
        for (int k = 0; k < Q; ++k) r.t[p][k] = static_cast<unsigned char>(g.mperm_t[p * 8][kPrinted.e[k]]);
    return r;
}
__constant__ PermColumns kPermColumns = make_perm_columns();

// Inverse of the pull map: the (x, i) whose pulled value is population j of cell y.
template <int BC>
__device__ __forceinline__ void push_target(int y0, int y1, int y2, int j, const Dims& d, int& i, int& dst) {
    const int c[3] = {cx_of(j), cy_of(j), cz_of(j)};
    const int n[3] = {d.nx, d.ny, d.nz};
    const int y[3] = {y0, y1, y2};
    int x[3], ci[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        int t = y[a] + c[a];
        if (BC == LBM_BC_PERIODIC) {
            t = t < 0 ? t + n[a] : (t >= n[a] ? t - n[a] : t);
            x[a] = t;
            ci[a] = c[a];
        } else if (BC == LBM_BC_TGV_REDUCED) {
            x[a] = t;
            ci[a] = c[a];
        } else {
            const bool out = t < 0 || t >= n[a];
            x[a] = out ? y[a] : t;
            ci[a] = out ? -c[a] : c[a];
        }
    }
    i = 9 * (ci[2] + 1) + 3 * (ci[1] + 1) + (ci[0] + 1);
    if (BC == LBM_BC_TGV_REDUCED) {
        // Appendix A: a population leaving the domain towards the block r of q = y + c_j
        // re-enters as its image under the flow symmetry g_r = (A, t) of that block: at
        // g_r(q) with velocity A c_j. This inverts the pull, which takes the source
        // g_r(x - c_i) for a source outside the domain: g_r is the only symmetry mapping
        // block r onto the domain, so g_r^-1 is the one for the block g_r(domain).
        tgv_reduced_image(d, x[0], x[1], x[2], c[0], c[1], c[2], i);
    }
    dst = (x[2] * d.ny + x[1]) * d.nx + x[0];
}

struct AdjArgs {
    Dims d;
    const void* state;   // stored buffer whose pull image is f_t
    const float* lam_in; // lam_{t+1}: 27 planes
    float* lam_out;      // lam_t: 27 planes
    double* grad;        // GradLayout<DEEP>::kLen accumulators
    float tau;
    const float* force;  // forced step: the force field of step t (3 planes), else null
    int parts;           // SPLIT: parts of the cotangent of m, the axis permutations in 2, 3 or 6 groups
};

constexpr int kAdjThreads = 32 * kNetWarps;
constexpr int kGradBlock = kHidden * kHidden + kHidden;  // dW and db of a 20 x 20 layer

// LANES lanes share a cell, each holding COLS of the half's four sign vectors. SPLIT: the
// cotangent of m in parts.
template <bool DEEP, int LANES, bool SPLIT>
struct AdjShared {
    static constexpr int kCells = 32 / LANES;
    static constexpr int kCols = 4 / LANES;
    static constexpr int kRow = net_row(kCols);
    // per warp: the staged cotangents of one column per lane (32 x 20), and at the end the weight
    // gradients of the hidden layers and of the warp's half of W1p
    static constexpr int kD1 = DEEP ? 2 * kGradBlock : kGradBlock;
    static constexpr int kStage = (kD1 + (Q + 1) * kHalf + 3) / 4 * 4;
    static_assert(kStage >= 32 * kHidden, "stage holds a column per lane");

    NetParams net;
    double grad[GradLayout<DEEP>::kLen];  // the block's parameter gradients, summed over its tiles
    float h1[kNetWarps][net_rows(kCols)];  // h1, then delta h1, then E
    float h2[DEEP ? kNetWarps : 1][32][DEEP ? kRow : 4];  // h2, then delta h2 (third hidden layer)
    float stage[kNetWarps][kStage];
    float m[kCells][28];      // moments (tensor order), 1 (the bias input)
    float mu[kCells][28];     // mu* (class order), then the relaxation's part of dL/dm, then dL/dm
    float hsum[kCells][kHidden];  // group sum of the last hidden layer
    float v3[kCells][kHidden];  // cotangent of the last hidden layer, the same for every group element
    float gbar[kCells][kOut];
    float rates[kCells][kOut];
    // dL/dm of the second to sixth part (the deep network's h2 is free by then)
    float more[SPLIT && !DEEP ? 5 : 1][SPLIT && !DEEP ? kCells : 1][28];
    __device__ __forceinline__ float (*part(int i))[28] {
        if (i == 0) return mu;
        return reinterpret_cast<float(*)[28]>(DEEP ? &h2[0][0][0] : &more[0][0][0]) + (i - 1) * kCells;
    }
    static_assert(!DEEP || 5 * kCells * 28 <= kNetWarps * 32 * kRow, "the parts fit h2");
};

// A cell's 27 values to and from a row in class order.
__device__ __forceinline__ void store_class_order(float* row, const float* v) {
    static_for<Q>([&](auto T) { row[class_pos(decltype(T)::value)] = v[decltype(T)::value]; });
}
__device__ __forceinline__ void load_class_order(float* v, const float* row) {
    static_for<Q>([&](auto T) { v[decltype(T)::value] = row[class_pos(decltype(T)::value)]; });
}

// Classes of the places 4 g, 4 g + 1 (bits 8 g..) and 4 g + 2, 4 g + 3 (bits 8 g + 4..).
constexpr unsigned long long make_class_of_pair() {
    unsigned long long r = 0;
    for (int g = 0; g < 7; ++g)
        for (int i = 0; i < 2; ++i) r |= static_cast<unsigned long long>(class_at(4 * g + 2 * i)) << (8 * g + 4 * i);
    return r;
}
constexpr bool pairs_of_places_share_a_class() {
    for (int k = 0; k < Q - 1; k += 2)
        if (class_at(k) != class_at(k + 1)) return false;
    return true;
}
static_assert(pairs_of_places_share_a_class(), "two places, one class");
constexpr unsigned long long kClassOfPair = make_class_of_pair();

// Outer products summed over columns: a warp's 20 x 21 gradient (W | b) in tiles of 10 x 5
// (and the bias column) over 2 x 4 lanes; the four groups of eight lanes take the rows
// r = 0..31 of a column in turn.
struct OuterTile {
    float a[kHalf][6];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int j = 0; j < kHalf; ++j)
#pragma unroll
            for (int k = 0; k < 6; ++k) a[j][k] = 0.0f;
    }
    // rows r of d (stride ds) times rows r of h (stride hs)
    __device__ __forceinline__ void add(const float* d, int ds, const float* h, int hs, int lane) {
        const int grp = lane >> 3, jt = (lane >> 2) & 1, kt = lane & 3;
        d += grp * ds + jt * kHalf;
        h += grp * hs + kt * 5;
#pragma unroll 1
        for (int r = 0; r < 32; r += 4, d += 4 * ds, h += 4 * hs) {
            float dv[kHalf], hv[5];
#pragma unroll
            for (int j = 0; j < kHalf; j += 2) {
                const float2 t = *reinterpret_cast<const float2*>(d + j);
                dv[j] = t.x;
                dv[j + 1] = t.y;
            }
#pragma unroll
            for (int k = 0; k < 5; ++k) hv[k] = h[k];
#pragma unroll
            for (int j = 0; j < kHalf; ++j) {
#pragma unroll
                for (int k = 0; k < 5; ++k) a[j][k] = fmaf(dv[j], hv[k], a[j][k]);
                a[j][5] += dv[j];
            }
        }
    }
    // sums over the four groups to out: [j][k] (20 x 20), then the bias column
    __device__ __forceinline__ void flush(float* out, int lane) {
        const int jt = (lane >> 2) & 1, kt = lane & 3;
#pragma unroll
        for (int j = 0; j < kHalf; ++j)
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                float v = a[j][k];
                v += __shfl_xor_sync(0xffffffffu, v, 8);
                v += __shfl_xor_sync(0xffffffffu, v, 16);
                if (lane < 8) {
                    if (k < 5) out[(jt * kHalf + j) * kHidden + kt * 5 + k] = v;
                    else if (kt == 0) out[kHidden * kHidden + jt * kHalf + j] = v;
                }
            }
    }
};

// Hands the tile's group sums from warp w - 1 to warp w: a named barrier of the two, the pair's
// own (pair_sync) inside a permutation.
__device__ __forceinline__ int group_sum_barrier(int w) { return w & 1 ? (w >> 1) + 1 : kNetWarps / 2 + (w >> 1); }
__device__ __forceinline__ void group_sum_wait(int w) { asm volatile("bar.sync %0, 64;" ::"r"(group_sum_barrier(w)) : "memory"); }
__device__ __forceinline__ void group_sum_pass(int w) { asm volatile("bar.arrive %0, 64;" ::"r"(group_sum_barrier(w)) : "memory"); }

template <int STORAGE, int BC, bool DEEP, int LANES, bool SPLIT>
__global__ void __launch_bounds__(kAdjThreads, 1) adjoint_step_kernel(const AdjArgs a,
                                                                      const NetParams* __restrict__ net_in, int ntiles) {
    using GL = GradLayout<DEEP>;
    using SH = AdjShared<DEEP, LANES, SPLIT>;
    using At = BySigns<LANES>;
    constexpr int kCells = SH::kCells, C = SH::kCols, kRow = SH::kRow;
    extern __shared__ __align__(16) uint8_t adj_smem_raw[];
    SH& sh = *reinterpret_cast<SH*>(adj_smem_raw);
    const NetParams& net = sh.net;
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int w = __shfl_sync(0xffffffffu, tid >> 5, 0);  // uniform, and seen to be
    const int p = w >> 1, half = w & 1;
    const int l = lane & 15, og = lane >> 4;  // the rows l and l + 16, units [10 og, 10 og + 10)
    const int own = w == 0 ? tid : tid - 32;  // first of a thread's parameters (all warps but 1)
    load_params(&sh.net, net_in, tid, kAdjThreads);
    for (int i = tid; i < GL::kLen; i += kAdjThreads) sh.grad[i] = 0.0;
    overlap_wait();

#pragma unroll 1
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const long long cell0 = static_cast<long long>(tile) * kCells;

        // ---- moments (warp 0) and cotangents in moment space (warp 1) of the tile's cells
        if constexpr (BC == LBM_BC_TGV_REDUCED) {
            // the boundary's branches serialise a warp's 27 loads: spread over the block (into the
            // rows of h1) they run side by side (16^3, third hidden layer: 77 -> 69 us a step;
            // on the other boundaries the extra barrier costs more, 32^3 225 -> 236 us)
            {
                constexpr int kPer = kAdjThreads / kCells;
                float* const raw = sh.h1[0];
                const long long cell = cell0 + tid % kCells;
                const bool valid = cell < a.d.ncell;
                int x = 0, y = 0, z = 0;
                if (valid) cell_coords(cell, a.d, x, y, z);
                using S = Store<STORAGE>;
#pragma unroll
                for (int it = 0; it < (2 * Q + kPer - 1) / kPer; ++it) {
                    const int i = tid / kCells + it * kPer;
                    float v = 0.0f;  // a cell past the end: no cotangent, so it adds nothing
                    if (valid && i < Q) {
                        int ip, src;
                        pull_source<BC>(x, y, z, i, a.d, ip, src);
                        v = S::ld(static_cast<const typename S::T*>(a.state) + static_cast<size_t>(ip) * a.d.ncell + src);
                    } else if (valid && i < 2 * Q) {
                        int ip, dst;
                        push_target<BC>(x, y, z, i - Q, a.d, ip, dst);
                        v = a.lam_in[static_cast<size_t>(ip) * a.d.ncell + dst];
                    }
                    if (i < 2 * Q) raw[i * kCells + tid % kCells] = v;
                }
                __syncthreads();
                if (w < 2 && lane < kCells) {
                    float v[Q];
                    const float* src = raw + w * Q * kCells + lane;
#pragma unroll
                    for (int e = 0; e < Q; ++e) v[e] = src[e * kCells];
                    if (w == 0) {
                        float m[Q];
                        moments_from_dev(v, m);
#pragma unroll
                        for (int e = 0; e < Q; ++e) sh.m[lane][e] = m[e];
                        sh.m[lane][Q] = 1.0f;
                    } else {
                        populations_transpose_inplace(v);  // mu* = M^-T lam*
                        store_class_order(sh.mu[lane], v);
                    }
                }
            }
        } else {
            if (w < 2 && lane < kCells) {
                const long long cell = cell0 + lane;
                float v[Q];
                if (cell < a.d.ncell) {
                    int x, y, z;
                    cell_coords(cell, a.d, x, y, z);
                    if (w == 0) {
                        float df[Q];
                        load_pulled<STORAGE, BC>(a.state, a.d, x, y, z, df);
                        moments_from_dev(df, v);
                    } else {
#pragma unroll
                        for (int j = 0; j < Q; ++j) {
                            int i, dst;
                            push_target<BC>(x, y, z, j, a.d, i, dst);
                            v[j] = a.lam_in[static_cast<size_t>(i) * a.d.ncell + dst];
                        }
                        populations_transpose_inplace(v);  // mu* = M^-T lam*
                    }
                } else {  // a cell past the end: no cotangent, so it adds nothing
#pragma unroll
                    for (int e = 0; e < Q; ++e) v[e] = 0.0f;
                    if (w == 0) v[0] = 1.0f;
                }
                if (w == 0) {
#pragma unroll
                    for (int e = 0; e < Q; ++e) sh.m[lane][e] = v[e];
                    sh.m[lane][Q] = 1.0f;
                } else {
                    store_class_order(sh.mu[lane], v);
                }
            }
        }
        __syncthreads();

        // ---- first layer
        float* const rows = sh.h1[w];
        float* const row = rows + l * kRow;
        {
            float m[2 / LANES][28];
#pragma unroll
            for (int k = 0; k < 2 / LANES; ++k)
#pragma unroll
                for (int e = 0; e < 28; e += 4)
                    *reinterpret_cast<float4*>(&m[k][e]) = *reinterpret_cast<const float4*>(&sh.m[l + 16 * k][e]);
            first_layer<At>(net, p, half, lane, m, sh.h1[2 * p]);
        }
        pair_sync(p);

        // ---- the layers up to the group sum; mask[r][c] keeps which units of the last hidden layer
        // are on in column c of row l + 16 r (unit j in bit 31 - j)
        uint32_t mask[2][C];
        {
            float acc[2][C][kHalf];
            set_bias(net.b2, lane, acc);
            mat_vec<C, 5>(net.W2, lane, acc, RowColumns<C>{row});
            if constexpr (DEEP) {
                float* const row2 = sh.h2[w][l];
                store_relu(row2, lane, acc);
                __syncwarp();
                set_bias(net.bd, lane, acc);
                mat_vec<C, 5>(net.Wd, lane, acc, RowColumns<C>{row2});
            }
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    uint32_t k = 0u;
#pragma unroll
                    for (int o = 0; o < kHalf; ++o) {
                        acc[r][c][o] = fmaxf(acc[r][c][o], 0.0f);
                        k = __funnelshift_l(__float_as_uint(0.0f - acc[r][c][o]), k, 1);  // the sign of -h: h > 0
                    }
                    k <<= og ? 32 - kHidden : 32 - kHalf;
                    mask[r][c] = k | __shfl_xor_sync(0xffffffffu, k, 16);
                }
            // the group sum, element by element in the order of the group (the rates are those of the
            // step, bit for bit): warp after warp adds its sign vectors to it
            if (w > 0) group_sum_wait(w);
#pragma unroll
            for (int k = 0; k < At::kCells; ++k)
#pragma unroll
                for (int o = 0; o < kHalf; o += 2) {
                    float2* const q = reinterpret_cast<float2*>(&sh.hsum[l + 16 * k][og * kHalf + o]);
                    float2 h = w > 0 ? *q : make_float2(0.0f, 0.0f);
#pragma unroll
                    for (int r = k; r < k + LANES; ++r)
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            h.x += acc[r][c][o];
                            h.y += acc[r][c][o + 1];
                        }
                    *q = h;
                }
            if (w + 1 < kNetWarps) group_sum_pass(w + 1);
        }
        __syncthreads();
        if (tid < kOut * kCells) {  // rates and the cotangents of tau~, one (cell, output) per thread
            const int n = tid / kCells, c = tid % kCells;
            float t = 0.0f;
#pragma unroll
            for (int j = 0; j < kHidden; ++j) t = fmaf(net.W3[n][j], sh.hsum[c][j], t);
            t = t * (1.0f / 48.0f) + net.b3[n];
            const float e = expf(t);
            const float tau_n = 0.5f / (1.0f + e) + 0.5f;
            float gw = 0.0f;
            static_for<Q>([&](auto K) {
                constexpr int k = decltype(K)::value, q = class_pos(k);
                if (order_of(k) >= 3 && order_of(k) == n + 3) gw = fmaf(-sh.mu[c][q], sh.m[c][k], gw);
            });
            // d omega / d tau~ = sigma (1 - sigma) / (2 tau_n^2), sigma = 1 / (1 + e^{tau~})
            const float sg = 1.0f / (1.0f + e);
            sh.rates[c][n] = 1.0f / tau_n;
            sh.gbar[c][n] = cell0 + c < a.d.ncell ? gw * sg * (1.0f - sg) / (2.0f * tau_n * tau_n) : 0.0f;
        }
        __syncthreads();
        for (int i = tid; i < kCells * kHidden; i += kAdjThreads) {  // W3^T gbar / 48
            const int c = i / kHidden, j = i % kHidden;
            float v = 0.0f;
#pragma unroll
            for (int n = 0; n < kOut; ++n) v = fmaf(net.W3[n][j], sh.gbar[c][n], v);
            sh.v3[c][j] = v * (1.0f / 48.0f);
        }
        __syncthreads();

        // ---- the relaxation's part of dL/dm, one warp (the others run ahead)
        if (w == kNetWarps - 1 && lane < kCells) {
            const long long cell = cell0 + lane;
            const bool valid = cell < a.d.ncell;
            const float* m = sh.m[lane];
            float mus[Q];
            load_class_order(mus, sh.mu[lane]);
            const float omega_nu = 1.0f / a.tau;
            const float irho = 1.0f / m[0];
            float dm[Q];
#pragma unroll
            for (int e = 0; e < Q; ++e) dm[e] = 0.0f;
#pragma unroll
            for (int e = 0; e < Q; ++e) {
                const int n = order_of(e);
                const float mu = mus[e];
                if (n <= 1) {
                    dm[e] += mu;
                } else if (n == 2) {
                    dm[e] += (1.0f - omega_nu) * mu;
                    // m^eq_e = m_a m_b / m_0 for the axes a, b of component e
                    const int ex = ex_of(e), ey = ey_of(e), ez = ez_of(e);
                    int ia = -1, ib = -1, axa = 0, axb = 0;
                    const int cnt[3] = {ex, ey, ez};
                    const int idx[3] = {1, 3, 9};
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        if (cnt[k] == 2) { ia = idx[k]; ib = idx[k]; axa = axb = k; }
                        if (cnt[k] == 1) {
                            if (ia < 0) { ia = idx[k]; axa = k; }
                            else { ib = idx[k]; axb = k; }
                        }
                    }
                    const float ma = m[ia], mb = m[ib];
                    const float c = omega_nu * mu;
                    dm[ia] += c * mb * irho;
                    dm[ib] += c * ma * irho;
                    dm[0] -= c * ma * mb * irho * irho;
                    if (a.force && valid) {
                        // Kupershtokh source (Sec. II.A) in moment space: its only state-dependent part
                        // is order 2, dm*_ab = 3 ((j + F)_a (j + F)_b - j_a j_b) / rho with m_a = sqrt3 j_a,
                        // i.e. (sqrt3 (m_a F_b + F_a m_b) + 3 F_a F_b) / rho; the force is an input
                        const float Fa = a.force[static_cast<size_t>(axa) * a.d.ncell + cell];
                        const float Fb = a.force[static_cast<size_t>(axb) * a.d.ncell + cell];
                        const float src = (kSqrt3 * (ma * Fb + Fa * mb) + 3.0f * Fa * Fb) * irho;
                        dm[ia] += mu * kSqrt3 * Fb * irho;
                        dm[ib] += mu * kSqrt3 * Fa * irho;
                        dm[0] -= mu * src * irho;
                    }
                } else {
                    dm[e] += (1.0f - sh.rates[lane][n - 3]) * mu;
                }
            }
            store_class_order(sh.mu[lane], dm);
        }
        __syncwarp();

        // units j..j+3 of the last hidden layer's cotangent where they are on: v3 of the cell at a
        // row, and the bits k of a column
        auto masked = [](const float4& v, uint32_t k) {
            return make_float4(static_cast<int>(k) < 0 ? v.x : 0.0f, static_cast<int>(k << 1) < 0 ? v.y : 0.0f,
                               static_cast<int>(k << 2) < 0 ? v.z : 0.0f, static_cast<int>(k << 3) < 0 ? v.w : 0.0f);
        };
        auto v3_at = [&](int r, int j) { return *reinterpret_cast<const float4*>(&sh.v3[r % kCells][j]); };
        auto last_columns = [&](int j, float4(&v)[2][C]) {
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const float4 t = v3_at(l + 16 * r, j);
#pragma unroll
                for (int c = 0; c < C; ++c) v[r][c] = masked(t, mask[r][c] << j);
            }
        };
        // weight gradient of the layer above the columns h: (v3 masked) times h, a column of every
        // row staged at a time
        auto last_layer_grad = [&](const float* h, float* out) {
            OuterTile t;
            t.clear();
            float* const st = sh.stage[w];
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const uint32_t k = og ? mask[1][c] : mask[0][c];
#pragma unroll
                for (int j = 0; j < kHidden; j += 4)
                    *reinterpret_cast<float4*>(st + lane * kHidden + j) = masked(v3_at(lane, j), k << j);
                __syncwarp();
                t.add(st, kHidden, h + c * kHidden, kRow, lane);
                __syncwarp();
            }
            t.flush(out, lane);
        };
        // acc where the unit is on in x replaces x
        auto gate_into = [&](float* x, const float(&acc)[2][C][kHalf]) {
            x += og * kHalf;
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int c = 0; c < C; ++c)
#pragma unroll
                    for (int o = 0; o < kHalf; o += 2) {
                        float2* const q = reinterpret_cast<float2*>(x + 16 * r * kRow + c * kHidden + o);
                        const float2 h = *q;
                        *q = make_float2(h.x > 0.0f ? acc[r][c][o] : 0.0f, h.y > 0.0f ? acc[r][c][o + 1] : 0.0f);
                    }
        };

        // ---- backward through the hidden layers
        if constexpr (DEEP) {
            float* const rows2 = &sh.h2[w][0][0];
            float* const row2 = sh.h2[w][l];
            last_layer_grad(rows2, sh.stage[w]);
            {
                float acc[2][C][kHalf] = {};
                mat_vec<C, 5>(net.WdT, lane, acc, last_columns);
                gate_into(row2, acc);  // delta h2
            }
            __syncwarp();
            {
                OuterTile t;
                t.clear();
#pragma unroll 1
                for (int c = 0; c < C; ++c) t.add(rows2 + c * kHidden, kRow, rows + c * kHidden, kRow, lane);
                t.flush(sh.stage[w] + kGradBlock, lane);
            }
            __syncwarp();
            float acc[2][C][kHalf] = {};
            mat_vec<C, 5>(net.W2T, lane, acc, RowColumns<C>{row2});
            gate_into(row, acc);  // delta h1
        } else {
            last_layer_grad(rows, sh.stage[w]);
            float acc[2][C][kHalf] = {};
            mat_vec<C, 5>(net.W2T, lane, acc, last_columns);
            gate_into(row, acc);  // delta h1
        }
        pair_sync(p);

        // ---- first layer: E of class c in place of delta h1 of sign vector c
        {
            const int j0 = half * kHalf + og * 5;
            float* const q = sh.h1[2 * p] + l * kRow + j0;
#pragma unroll 1
            for (int i = 0; i < 5; ++i)
#pragma unroll
                for (int k = 0; k < At::kCells; ++k) {
                    float e[8];
                    auto at = [&](int s) -> float& {
                        return q[At::half(s, k) * net_rows(C) + At::row(s, k) * kRow + At::col(s, k) * kHidden + i];
                    };
#pragma unroll
                    for (int s = 0; s < 8; ++s) e[s] = at(s);
                    wht<8>(e);
#pragma unroll
                    for (int s = 0; s < 8; ++s) at(s) = e[s];
                }
        }
        pair_sync(p);
        {
            const int t = lane < Q ? lane : Q;
            const int ex = t % 3, ey = (t / 3) % 3, ez = t / 9;
            const int c = t < Q ? ((ex == 1) << 2) | ((ey == 1) << 1) | (ez == 1) : 0;
            // dW1p[j][t] = sum over cells of E[c(t)][j] m_t, lane t (lane 27: db1, the bias input of class 0)
            {
                const float* er = sh.h1[2 * p + At::half(c, 0)] + At::row(c, 0) * kRow + At::col(c, 0) * kHidden + half * kHalf;
                float g[kHalf];
#pragma unroll
                for (int j = 0; j < kHalf; ++j) g[j] = 0.0f;
#pragma unroll 2
                for (int r = 0; r < kCells; ++r) {
                    const float mt = sh.m[r][t];
#pragma unroll
                    for (int j = 0; j < kHalf; j += 2) {
                        const float2 v = *reinterpret_cast<const float2*>(er + r * kRow + j);
                        g[j] = fmaf(v.x, mt, g[j]);
                        g[j + 1] = fmaf(v.y, mt, g[j + 1]);
                    }
                }
                if (lane <= Q) {
#pragma unroll
                    for (int j = 0; j < kHalf; ++j) sh.stage[w][SH::kD1 + t * kHalf + j] = g[j];
                }
            }
            __syncthreads();
            // the network's part of the cotangent of m, W1p[j][t] E[c(t)][j] on top of the relaxation's
            // part, permutation by permutation and unit by unit (a sum whose last bits the sweep carries to
            // the first step), SPLIT in sums of 6 / a.parts permutations each: a lane has a cell and four
            // places of the class order. Warps 0 to 6 have 32 cells each (LANES = 1), or 0 to 3 16 cells
            // and two groups of places
            const int g = LANES == 1 ? w : 2 * w + og, cell = LANES == 1 ? lane : l;
            if (g < 7) {
                const int ca = (kClassOfPair >> (8 * g)) & 7, cb = (kClassOfPair >> (8 * g + 4)) & 7;
                auto e_of = [&](int k) { return sh.h1[At::half(k, 0)] + (At::row(k, 0) + cell) * kRow + At::col(k, 0) * kHidden; };
                const float *ea = e_of(ca), *eb = e_of(cb);
                float4* q = reinterpret_cast<float4*>(&sh.mu[cell][4 * g]);
                float4 dm = *q;
                const int per = SPLIT ? 6 / a.parts : 6;
                int left = per, part = 0;
#pragma unroll 1
                for (int pp = 0; pp < kNetWarps / 2; ++pp, ea += 2 * net_rows(C), eb += 2 * net_rows(C)) {
                    if (SPLIT && left-- == 0) {  // the next part
                        *q = dm;
                        q = reinterpret_cast<float4*>(&sh.part(++part)[cell][4 * g]);
                        dm = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                        left = per - 1;
                    }
#pragma unroll
                    for (int j = 0; j < kHidden; j += 4) {
                        const float4 a4 = *reinterpret_cast<const float4*>(ea + j);
                        const float4 b4 = LANES == 1 && ca == cb ? a4 : *reinterpret_cast<const float4*>(eb + j);
                        auto add = [&](int jj, float a1, float b1) {
                            const float4 wt = *reinterpret_cast<const float4*>(&net.W1p[pp][jj][4 * g]);
                            dm.x = fmaf(wt.x, a1, dm.x);
                            dm.y = fmaf(wt.y, a1, dm.y);
                            dm.z = fmaf(wt.z, b1, dm.z);
                            dm.w = fmaf(wt.w, b1, dm.w);
                        };
                        add(j, a4.x, b4.x);
                        add(j + 1, a4.y, b4.y);
                        add(j + 2, a4.z, b4.z);
                        add(j + 3, a4.w, b4.w);
                    }
                }
                *q = dm;
            }
        }
        __syncthreads();

        if (w == 1) {  // lam_t = M^T dL/dm, by the warp that fills mu again
            const long long cell = cell0 + lane;
            if (lane < kCells && cell < a.d.ncell) {
                float v[Q];
                load_class_order(v, sh.mu[lane]);
                moments_transpose_inplace(v);
                if constexpr (SPLIT) {
#pragma unroll 1
                    for (int i = 1; i < a.parts; ++i) {
                        float more[Q];
                        load_class_order(more, sh.part(i)[lane]);
                        moments_transpose_inplace(more);
#pragma unroll
                        for (int e = 0; e < Q; ++e) v[e] += more[e];
                    }
                }
#pragma unroll
                for (int i = 0; i < Q; ++i) a.lam_out[static_cast<size_t>(i) * a.d.ncell + cell] = v[i];
            }
            continue;  // until the next tile's first barrier it writes nothing that the others still read
        }
        // parameter gradients of the tile, a thread's own: sums over the warps (W1: the six
        // permutations' columns that a printed column went to), added in FP64
        for (int i = own; i < GL::kLen; i += kAdjThreads - 32) {
            float v = 0.0f;
            if (i < GL::kW2) {
                const int j = i < GL::kB1 ? i / Q : i - GL::kB1, k = i < GL::kB1 ? i % Q : Q;
                const int h = j >= kHalf, jo = j - h * kHalf;
#pragma unroll
                for (int q = 0; q < 6; ++q) {
                    const int t = k < Q ? kPermColumns.t[q][k] : Q;
                    v += sh.stage[2 * q + h][SH::kD1 + t * kHalf + jo];
                }
            } else if (i < GL::kW3) {
                // stage: with the third hidden layer (Wd | bd) then (W2 | b2), else (W2 | b2)
                int o = i - GL::kW2;
                if (DEEP) o = o < kGradBlock ? o + kGradBlock : o - kGradBlock;
#pragma unroll
                for (int q = 0; q < kNetWarps; ++q) v += sh.stage[q][o];
            } else {
                const int o = i - GL::kW3;
                const int n = o < kOut * kHidden ? o / kHidden : o - kOut * kHidden;
                for (int c = 0; c < kCells; ++c)
                    v = fmaf(sh.gbar[c][n], o < kOut * kHidden ? sh.hsum[c][o % kHidden] * (1.0f / 48.0f) : 1.0f, v);
            }
            sh.grad[i] += static_cast<double>(v);
        }
    }
    if (w != 1)
        for (int i = own; i < GL::kLen; i += kAdjThreads - 32) atomicAdd(&a.grad[i], sh.grad[i]);
}

// lam[i] (=, or += when accumulate) sum_a g_a (c_ia - u_a) / rho + dL/drho for the state
// whose pull image is f, with g_a = dL/du_a + ke_scale u_a: the cotangent of the
// macroscopic fields, and of the kinetic energy k = (1/2)<|u|^2> with ke_scale =
// (dL/dk) / cells.
template <int STORAGE, int BC>
__global__ void adjoint_seed_kernel(const Dims d, const void* state, const float* __restrict__ du,
                                    const float* __restrict__ drho_in, float ke_scale, int accumulate,
                                    float* lam) {
    const long long cell = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (cell >= d.ncell) return;
    int x, y, z;
    cell_coords(cell, d, x, y, z);
    float df[Q], m[Q];
    load_pulled<STORAGE, BC>(state, d, x, y, z, df);
    const float dr = moments_from_dev(df, m);
    const Macro q = macro_from_moments(m, dr);
    const float gx = (du ? du[cell] : 0.0f) + ke_scale * q.ux;
    const float gy = (du ? du[d.ncell + cell] : 0.0f) + ke_scale * q.uy;
    const float gz = (du ? du[2 * d.ncell + cell] : 0.0f) + ke_scale * q.uz;
    const float gr = drho_in ? drho_in[cell] : 0.0f;
    const float ir = 1.0f / q.rho;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const float v = (gx * (cx_of(i) - q.ux) + gy * (cy_of(i) - q.uy) + gz * (cz_of(i) - q.uz)) * ir + gr;
        float* o = lam + static_cast<size_t>(i) * d.ncell + cell;
        *o = accumulate ? *o + v : v;
    }
}

cudaError_t launch_adjoint_seed(const Dims& d, int storage, int bc, const void* state, const float* du,
                                const float* drho, float ke_scale, bool accumulate, float* lam, cudaStream_t s) {
    const dim3 grid(static_cast<unsigned>((d.ncell + 127) / 128));
    if (storage != LBM_STORE_F32) return cudaErrorInvalidValue;
    const int acc = accumulate ? 1 : 0;
    if (bc == LBM_BC_PERIODIC)
        adjoint_seed_kernel<LBM_STORE_F32, LBM_BC_PERIODIC><<<grid, 128, 0, s>>>(d, state, du, drho, ke_scale, acc, lam);
    else if (bc == LBM_BC_MIRROR)
        adjoint_seed_kernel<LBM_STORE_F32, LBM_BC_MIRROR><<<grid, 128, 0, s>>>(d, state, du, drho, ke_scale, acc, lam);
    else if (bc == LBM_BC_TGV_REDUCED)
        adjoint_seed_kernel<LBM_STORE_F32, LBM_BC_TGV_REDUCED><<<grid, 128, 0, s>>>(d, state, du, drho, ke_scale, acc, lam);
    else
        return cudaErrorInvalidValue;
    return cudaGetLastError();
}

template <int BC, bool DEEP, int LANES, bool SPLIT>
static cudaError_t launch_adjoint_step_t(const AdjArgs& a, const NetParams* net, cudaStream_t s) {
    using SH = AdjShared<DEEP, LANES, SPLIT>;
    constexpr size_t smem = sizeof(SH);
    static_assert(smem <= 227 * 1024, "shared memory budget");
    static std::atomic<unsigned long long> attr{0};  // one set of per-device flags per instantiation
    const auto kernel = adjoint_step_kernel<LBM_STORE_F32, BC, DEEP, LANES, SPLIT>;
    const cudaError_t e = ensure_dynamic_smem(kernel, static_cast<int>(smem), attr);
    if (e != cudaSuccess) return e;
    const int ntiles = static_cast<int>((a.d.ncell + SH::kCells - 1) / SH::kCells);
    const int sms = sm_count();
    return launch_kernel(kernel, static_cast<unsigned>(ntiles < sms ? ntiles : sms), kAdjThreads, smem, s, true, a, net,
                         ntiles);
}

template <int BC, bool SPLIT>
static cudaError_t launch_adjoint_step_d(const AdjArgs& a, bool deep, const NetParams* net, cudaStream_t s) {
    return deep ? launch_adjoint_step_t<BC, true, 2, SPLIT>(a, net, s) : launch_adjoint_step_t<BC, false, 1, SPLIT>(a, net, s);
}

template <int BC>
static cudaError_t launch_adjoint_step_bc(const AdjArgs& a, bool deep, const NetParams* net, cudaStream_t s) {
    return a.parts > 1 ? launch_adjoint_step_d<BC, true>(a, deep, net, s) : launch_adjoint_step_d<BC, false>(a, deep, net, s);
}

cudaError_t launch_adjoint_step(const Dims& d, int storage, int bc, const void* state, const float* lam_in,
                                float* lam_out, double* grad, float tau, const float* force, bool deep,
                                const NetParams* d_net, cudaStream_t s) {
    if (storage != LBM_STORE_F32) return cudaErrorInvalidValue;
    // as many parts as one thread per cell took blocks of 128 cells for grids of fewer of them than
    // SMs: the roundings, and with them the gradient of given inputs, stay the same at every size
    const long long tiles = (d.ncell + 127) / 128, sms = sm_count();
    const int parts = tiles >= sms ? 1 : tiles * 2 >= sms ? 2 : tiles * 3 >= sms ? 3 : 6;
    const AdjArgs a{d, state, lam_in, lam_out, grad, tau, force, parts};
    switch (bc) {
        case LBM_BC_PERIODIC: return launch_adjoint_step_bc<LBM_BC_PERIODIC>(a, deep, d_net, s);
        case LBM_BC_MIRROR: return launch_adjoint_step_bc<LBM_BC_MIRROR>(a, deep, d_net, s);
        case LBM_BC_TGV_REDUCED: return launch_adjoint_step_bc<LBM_BC_TGV_REDUCED>(a, deep, d_net, s);
        default: return cudaErrorInvalidValue;
    }
}

void adjoint_fold_gradient(const double* acc, bool deep, float* out) {
    const int n = adjoint_grad_len(deep);
    for (int i = 0; i < n; ++i) out[i] = static_cast<float>(acc[i]);
}

}  // namespace lbm
