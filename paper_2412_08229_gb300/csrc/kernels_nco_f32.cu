// kernels_nco_f32.cu - the fused neural-collision step (Sec. II.A-B) with the invariant
// network in FP32 on the CUDA cores.
//
// A persistent block per SM takes tiles of 32 cells. Its twelve network warps evaluate one
// (permutation, half of the cells) each (net_f32.cuh) and add their sign vectors to the group sum
// in the order of the group, permutation after permutation; beside them a loader warp pulls the
// next tile's populations and forms its moments, and a finisher warp takes the previous tile's
// group sum, forms the rates, relaxes and stores. The three stages are one tile apart and meet
// at one barrier per tile.
//
// The order of the group sum and of everything after it is that of one thread per cell, bit for
// bit: a long unroll carries a last bit to 1e-5 of its gradient (handing the sum from one
// permutation to the next costs 32^3 50.2 -> 52.9 us, 96^3 1185 -> 1264, starts not overlapped).
//
// What bounds it (32^3, ncu): issue, 53 % of the cycles, in bursts: the twelve warps go through
// their FMA and shared-memory phases nearly together and hand on the group sum one after the
// other; shared-memory wavefronts 40 %. Step of the two-layer network with FP32 storage: 256^3
// 23.8 ms, 48^3 163 us, 32^3 52 us, 16^3 10.8 us; with one thread per cell and the weights in the
// constant bank 26.1 ms, 183, 55 and 47 us (16^3 fills 32 of 152 SMs that way, here 128). Third
// hidden layer: 16^3 15.6 us (70).
// The registers are at their limit of 128 (fourteen warps): the network's loop is sensitive to
// what lives around it (the parameters copied before the first load instead of after: 8 % slower).
#include "cell.cuh"
#include "force.cuh"
#include "launch.cuh"
#include "net_f32.cuh"

namespace lbm {

namespace {

constexpr int kTile = 32;
constexpr int kLoader = kNetWarps, kFinisher = kNetWarps + 1;
constexpr int kThreads = 32 * (kNetWarps + 2);

struct NetShared {
    NetParams net;
    float rows[kNetWarps][net_rows(4)];          // the columns' h1 (then h2)
    float part[2][kTile][kHidden];                     // sums of the last hidden layer over the group, permutation by permutation
    float m[2][kTile][28];                             // moments (tensor order)
    float df[3][Q][kTile];                             // the pulled deviations
    float fh2[kForcedModes * 6];                       // forced steps: 2 F^
    unsigned long long red[frc::kProjValues];          // forced steps: the block's projection sums
};
static_assert(sizeof(NetShared) <= 227 * 1024, "shared memory budget");

// Hands the tile's group sums from the two warps of permutation p - 1 to those of p: a named
// barrier of the four (pair_sync has the ids 1 to 6).
__device__ __forceinline__ void group_sum_wait(int p) { asm volatile("bar.sync %0, 128;" ::"r"(kNetWarps / 2 + p) : "memory"); }
__device__ __forceinline__ void group_sum_pass(int p) { asm volatile("bar.arrive %0, 128;" ::"r"(kNetWarps / 2 + p) : "memory"); }

template <int STORAGE, int BC>
__device__ __forceinline__ void load_tile(const StepArgs& a, long long cell, float (*m)[28], float (*df)[kTile], int lane) {
    float v[Q], mo[Q];
    if (cell < a.d.ncell) {
        int x, y, z;
        cell_coords(cell, a.d, x, y, z);
        load_pulled_offsets<STORAGE, BC>(a.src, a.d, x, y, z, v);
        moments_from_dev(v, mo);
        if (!(mo[0] >= a.rho_min && mo[0] <= a.rho_max)) atomicOr(a.status, 1);
    } else {
#pragma unroll
        for (int e = 0; e < Q; ++e) v[e] = mo[e] = 0.0f;
        mo[0] = 1.0f;
    }
#pragma unroll
    for (int e = 0; e < Q; ++e) {
        df[e][lane] = v[e];
        m[lane][e] = mo[e];
    }
}

// The block's first tile, which nothing overlaps, on the reduced domain, whose branches
// serialise a warp's 27 loads: spread over the network warps.
template <int STORAGE, int BC>
__device__ __forceinline__ void load_first_tile(const StepArgs& a, long long cell, float (*df)[kTile], int w, int lane) {
    using S = Store<STORAGE>;
    int x = 0, y = 0, z = 0;
    const bool valid = cell < a.d.ncell;
    if (valid) cell_coords(cell, a.d, x, y, z);
#pragma unroll
    for (int it = 0; it < (Q + kNetWarps - 1) / kNetWarps; ++it) {
        const int i = w + it * kNetWarps;
        float v = 0.0f;
        if (valid && i < Q) {
            int ip, src;
            pull_source<BC>(x, y, z, i, a.d, ip, src);
            v = S::ld(static_cast<const typename S::T*>(a.src) + static_cast<size_t>(ip) * a.d.ncell + src);
        }
        if (i < Q) df[i][lane] = v;
    }
}

template <int STORAGE, int BC, bool FORCED, bool DEEP>
__global__ void __launch_bounds__(kThreads, 1) step_nco_f32_kernel(const StepArgs a, const NetParams* __restrict__ net_in,
                                                                   const FusedForce ff, int ntiles) {
    extern __shared__ __align__(16) uint8_t smem[];
    NetShared& sh = *reinterpret_cast<NetShared*>(smem);
    const NetParams& net = sh.net;
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int w = __shfl_sync(0xffffffffu, tid >> 5, 0);  // uniform, and seen to be
    const int n = (ntiles - static_cast<int>(blockIdx.x) + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x);
    auto cell_of = [&](int i) {
        return (static_cast<long long>(blockIdx.x) + static_cast<long long>(i) * gridDim.x) * kTile + lane;
    };
    overlap_wait();
    if (FORCED) {
        frc::load_fh2(ff.fhat, sh.fh2);
        if (tid < frc::kProjValues) sh.red[tid] = 0ull;
    }
    if constexpr (BC == LBM_BC_TGV_REDUCED) {
        if (w < kNetWarps) load_first_tile<STORAGE, BC>(a, cell_of(0), sh.df[0], w, lane);
        load_params(&sh.net, net_in, tid, kThreads);
        __syncthreads();
        if (w == kLoader) {
            float v[Q], m[Q];
#pragma unroll
            for (int e = 0; e < Q; ++e) v[e] = sh.df[0][e][lane];
            moments_from_dev(v, m);
            if (cell_of(0) < a.d.ncell && !(m[0] >= a.rho_min && m[0] <= a.rho_max)) atomicOr(a.status, 1);
#pragma unroll
            for (int e = 0; e < Q; ++e) sh.m[0][lane][e] = m[e];
        }
    } else {
        if (w == kLoader) load_tile<STORAGE, BC>(a, cell_of(0), sh.m[0], sh.df[0], lane);
        if (w < kNetWarps) load_params(&sh.net, net_in, tid, 32 * kNetWarps);
    }
    __syncthreads();

    long long pacc[3] = {0, 0, 0};  // forced steps: fixed-point projection sums of the finisher's lane
    int b = 0;                      // i modulo 3: df of tile i; (b + 1) of tile i + 1, (b + 2) of tile i - 1
    for (int i = 0; i <= n; ++i) {
        const int bn = b == 2 ? 0 : b + 1, bp = b == 0 ? 2 : b - 1;
        if (w < kNetWarps) {
            if (i < n) {
                const int p = w >> 1, half = w & 1, l = lane & 15;
                {
                    float m[2][28];
#pragma unroll
                    for (int k = 0; k < 2; ++k)
#pragma unroll
                        for (int e = 0; e < 28; e += 4)
                            *reinterpret_cast<float4*>(&m[k][e]) = *reinterpret_cast<const float4*>(&sh.m[i & 1][l + 16 * k][e]);
                    first_layer<ByCells>(net, p, half, lane, m, sh.rows[2 * p]);
                }
                pair_sync(p);
                float* const row = sh.rows[w] + l * net_row(4);
                float acc[2][4][kHalf];
                set_bias(net.b2, lane, acc);
                mat_vec<4, 1>(net.W2, lane, acc, RowColumns<4>{row});
                if constexpr (DEEP) {  // 27-20-20-20-4: a third hidden layer before the group sum
                    __syncwarp();      // h1 is read before h2 replaces it
                    store_relu(row, lane, acc);
                    __syncwarp();
                    set_bias(net.bd, lane, acc);
                    mat_vec<4, 1>(net.Wd, lane, acc, RowColumns<4>{row});
                }
                // the group sum, element by element in the order of the group: the eight sign vectors of
                // this permutation on top of the permutations before it
                float* const out = &sh.part[i & 1][16 * half + l][(lane >> 4) * kHalf];
                float h[kHalf];
                if (p > 0) {
                    group_sum_wait(p);
#pragma unroll
                    for (int o = 0; o < kHalf; o += 2) {
                        const float2 t = *reinterpret_cast<const float2*>(out + o);
                        h[o] = t.x;
                        h[o + 1] = t.y;
                    }
                } else {
#pragma unroll
                    for (int o = 0; o < kHalf; ++o) h[o] = 0.0f;
                }
#pragma unroll
                for (int r = 0; r < 2; ++r)
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int o = 0; o < kHalf; ++o) h[o] += fmaxf(acc[r][c][o], 0.0f);
#pragma unroll
                for (int o = 0; o < kHalf; o += 2) *reinterpret_cast<float2*>(out + o) = make_float2(h[o], h[o + 1]);
                if (p + 1 < kNetWarps / 2) group_sum_pass(p + 1);
            }
        } else if (w == kLoader) {
            if (i + 1 < n) load_tile<STORAGE, BC>(a, cell_of(i + 1), sh.m[(i + 1) & 1], sh.df[bn], lane);
        } else if (i >= 1) {
            const long long cell = cell_of(i - 1);
            const bool valid = cell < a.d.ncell;
            float h[kHidden];
#pragma unroll
            for (int j = 0; j < kHidden; j += 4) {
                const float4 v = *reinterpret_cast<const float4*>(&sh.part[(i - 1) & 1][lane][j]);
                h[j] = v.x;
                h[j + 1] = v.y;
                h[j + 2] = v.z;
                h[j + 3] = v.w;
            }
            float rates[kOut];
#pragma unroll
            for (int o = 0; o < kOut; ++o) {
                float t = 0.0f;
#pragma unroll
                for (int j = 0; j < kHidden; ++j) t = fmaf(net.W3[o][j], h[j], t);
                rates[o] = rate_from_output(t * (1.0f / 48.0f) + net.b3[o]);
            }
            float df[Q], m[Q];
#pragma unroll
            for (int e = 0; e < Q; ++e) df[e] = sh.df[bp][e][lane];
            // the moments once more, not read back: the compiler then contracts their last products into the
            // relaxation as it does for one thread per cell
            const float drho = moments_from_dev(df, m);
            Macro q = macro_from_moments(m, drho);
            collide_mrt(df, m, q, 1.0f / a.tau, rates);
            if constexpr (FORCED) {  // every lane takes part in the projection, cells past the end with u = 0
                int x = 0, y = 0, z = 0;
                if (valid) cell_coords(cell, a.d, x, y, z);
                frc::Cx ph[kForcedModes];
                frc::cell_phases(x, y, z, a.d, ff.tab, ph);
                if (valid) {
                    float F[3];
                    frc::synth_force(sh.fh2, ph, F);
                    add_kupershtokh(df, q, F[0], F[1], F[2]);
                    store_cell<STORAGE>(a.dst, a.d, cell, df);
                } else {
                    q.ux = q.uy = q.uz = 0.0f;
                }
                if (ff.proj) frc::project_warp(q.ux, q.uy, q.uz, ph, lane, pacc, ff.scale);
            } else if (valid) {
                store_cell<STORAGE>(a.dst, a.d, cell, df);
            }
        }
        __syncthreads();
        b = bn;
    }
    if (FORCED && ff.proj) {
        if (w == kFinisher) frc::proj_to_shared(sh.red, pacc, lane);
        __syncthreads();
        frc::proj_to_global(sh.red, ff.proj);
    }
}

template <int STORAGE, int BC, bool FORCED, bool DEEP>
cudaError_t launch_t(const StepArgs& a, const FusedForce& ff, const NetParams* net, bool overlap, cudaStream_t s) {
    static std::atomic<unsigned long long> attr{0};
    const cudaError_t e = ensure_dynamic_smem(step_nco_f32_kernel<STORAGE, BC, FORCED, DEEP>,
                                              static_cast<int>(sizeof(NetShared)), attr);
    if (e != cudaSuccess) return e;
    const int ntiles = static_cast<int>((a.d.ncell + kTile - 1) / kTile);
    const int sms = sm_count();
    return launch_kernel(step_nco_f32_kernel<STORAGE, BC, FORCED, DEEP>, static_cast<unsigned>(ntiles < sms ? ntiles : sms),
                         kThreads, sizeof(NetShared), s, overlap, a, net, ff, ntiles);
}

template <int STORAGE, int BC, bool FORCED>
cudaError_t launch_d(const StepArgs& a, const FusedForce& ff, bool deep, const NetParams* net, bool overlap, cudaStream_t s) {
    return deep ? launch_t<STORAGE, BC, FORCED, true>(a, ff, net, overlap, s) : launch_t<STORAGE, BC, FORCED, false>(a, ff, net, overlap, s);
}

template <int STORAGE>
cudaError_t launch_s(const StepArgs& a, const FusedForce* ff, int bc, bool deep, const NetParams* net, bool overlap, cudaStream_t s) {
    if (ff) {  // forcing runs on periodic boxes only
        if (bc != LBM_BC_PERIODIC) return cudaErrorInvalidValue;
        return launch_d<STORAGE, LBM_BC_PERIODIC, true>(a, *ff, deep, net, overlap, s);
    }
    const FusedForce none{};
    if (bc == LBM_BC_PERIODIC) return launch_d<STORAGE, LBM_BC_PERIODIC, false>(a, none, deep, net, overlap, s);
    if (bc == LBM_BC_TGV_REDUCED) return launch_d<STORAGE, LBM_BC_TGV_REDUCED, false>(a, none, deep, net, overlap, s);
    return launch_d<STORAGE, LBM_BC_MIRROR, false>(a, none, deep, net, overlap, s);
}

}  // namespace

cudaError_t launch_step_nco_f32(const StepArgs& a, const FusedForce* ff, int storage, int bc, bool deep,
                                const NetParams* d_net, bool overlap, cudaStream_t s) {
    switch (storage) {
        case LBM_STORE_F32: return launch_s<LBM_STORE_F32>(a, ff, bc, deep, d_net, overlap, s);
        case LBM_STORE_F16_DEV: return launch_s<LBM_STORE_F16_DEV>(a, ff, bc, deep, d_net, overlap, s);
        default: return launch_s<LBM_STORE_BF16_DEV>(a, ff, bc, deep, d_net, overlap, s);
    }
}

}  // namespace lbm
