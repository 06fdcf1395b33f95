// kernels_step.cu - the fused pull-stream-collide step (Sec. II.A-B) with the BGK, KBC
// and REG operators, plus state set/get, macroscopic fields and the
// FP64 kinetic-energy reduction.
//
// One thread per cell; consecutive threads take consecutive x, so every one of the 27
// population loads and stores of a warp is a contiguous run of one plane (shifted by
// c_x for the loads). In the pull scheme every stored value is read exactly once per
// step, so there is no reuse for shared-memory staging to capture; the +-1 shift along
// x is absorbed by L1/L2 sectors that neighbouring warps share.
#include <atomic>

#include "force.cuh"
#include "internal.h"
#include "launch.cuh"

namespace lbm {

constexpr int kStepThreads = 128;

// Collision of one cell's pulled deviations df, in place; reports a density outside the
// window and returns the cell's pre-collision macroscopic state.
template <int OP>
__device__ __forceinline__ Macro collide_cell(const StepArgs& a, float* df) {
    Macro q;
    if constexpr (OP == LBM_OP_KBC) {  // needs only rho, u and the second-order moments
        float s2[6];
        q = kbc_moments(df, s2);
        if (!(q.rho >= a.rho_min && q.rho <= a.rho_max)) atomicOr(a.status, 1);
        collide_kbc(df, s2, q, a.tau);
    } else {
        float m[Q];
        const float drho = moments_from_dev(df, m);
        q = macro_from_moments(m, drho);
        if (!(q.rho >= a.rho_min && q.rho <= a.rho_max)) atomicOr(a.status, 1);
        const float omega = 1.0f / a.tau;
        if constexpr (OP == LBM_OP_BGK) {
            collide_bgk(df, q, omega);
        } else {  // REG: orders 3..6 relaxed with rate 1
            const float ones[kOut] = {1.0f, 1.0f, 1.0f, 1.0f};
            collide_mrt(df, m, q, omega, ones);
        }
    }
    return q;
}

template <int OP, int STORAGE, int BC>
__device__ __forceinline__ void step_body(const StepArgs& a) {
    const long long cell = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (cell >= a.d.ncell) return;
    int x, y, z;
    cell_coords(cell, a.d, x, y, z);
    float df[Q];
    load_pulled_offsets<STORAGE, BC>(a.src, a.d, x, y, z, df);
    collide_cell<OP>(a, df);
    store_cell<STORAGE>(a.dst, a.d, cell, df);
}

// The forced step (Sec. II.A source, Sec. II.C force) on a grid that strides over the
// cells: per cell the force F(x) is synthesised from the step's 16 coefficients and the
// phase tables and added as the Kupershtokh source after the collision, and the
// pre-collision velocity is added to the fixed-point projection sums of the next step's
// coefficients (force.cuh). Every lane of a warp takes part in the projection; lanes past
// the last cell contribute zero.
template <int OP, int STORAGE, int BC>
__device__ __forceinline__ void step_body_forced(const StepArgs& a, const FusedForce& ff) {
    __shared__ float fh2[kForcedModes * 6];
    __shared__ unsigned long long red[frc::kProjValues];
    frc::load_fh2(ff.fhat, fh2);
    for (int i = threadIdx.x; i < frc::kProjValues; i += blockDim.x) red[i] = 0ull;
    __syncthreads();
    const bool project = ff.proj != nullptr;
    const int lane = threadIdx.x & 31;
    long long acc[3] = {0, 0, 0};
    for (long long base = static_cast<long long>(blockIdx.x) * blockDim.x; base < a.d.ncell;
         base += static_cast<long long>(gridDim.x) * blockDim.x) {
        const long long cell = base + threadIdx.x;
        const bool valid = cell < a.d.ncell;
        int x = 0, y = 0, z = 0;
        float df[Q];
        Macro q{};
        if (valid) {
            cell_coords(cell, a.d, x, y, z);
            load_pulled_offsets<STORAGE, BC>(a.src, a.d, x, y, z, df);
            q = collide_cell<OP>(a, df);
        }
        frc::Cx p[kForcedModes];
        frc::cell_phases(x, y, z, a.d, ff.tab, p);
        if (valid) {
            float F[3];
            frc::synth_force(fh2, p, F);
            add_kupershtokh(df, q, F[0], F[1], F[2]);
            store_cell<STORAGE>(a.dst, a.d, cell, df);
        }
        if (project) frc::project_warp(q.ux, q.uy, q.uz, p, lane, acc, ff.scale);
    }
    if (project) {
        frc::proj_to_shared(red, acc, lane);
        __syncthreads();
        frc::proj_to_global(red, ff.proj);
    }
}

template <int OP, int STORAGE, int BC, bool FORCED>
__global__ void __launch_bounds__(kStepThreads, OP == LBM_OP_KBC && !FORCED ? 7 : 1)
    step_kernel(const StepArgs a, const FusedForce ff) {
    overlap_wait();
    if constexpr (FORCED) step_body_forced<OP, STORAGE, BC>(a, ff);
    else step_body<OP, STORAGE, BC>(a);
}

// Blocks of a forced launch: as many as are resident at once (the grid strides over the
// cells), at most one per 128 cells.
template <typename K>
static unsigned forced_grid(K kernel, int threads, std::atomic<int>& occ, long long ncell) {
    int n = occ.load(std::memory_order_relaxed);
    if (n == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, 0) != cudaSuccess || n < 1) {
            cudaGetLastError();
            n = 1;
        }
        occ.store(n, std::memory_order_relaxed);
    }
    const long long need = (ncell + threads - 1) / threads;
    const long long res = static_cast<long long>(n) * sm_count();
    return static_cast<unsigned>(need < res ? need : res);
}

template <int OP, int STORAGE, int BC, bool FORCED>
static cudaError_t launch_op(const StepArgs& a, const FusedForce& ff, bool overlap, cudaStream_t s) {
    unsigned grid = static_cast<unsigned>((a.d.ncell + kStepThreads - 1) / kStepThreads);
    if constexpr (FORCED) {
        static std::atomic<int> occ{0};
        grid = forced_grid(step_kernel<OP, STORAGE, BC, true>, kStepThreads, occ, a.d.ncell);
    }
    return launch_kernel(step_kernel<OP, STORAGE, BC, FORCED>, grid, kStepThreads, 0, s, overlap, a, ff);
}

template <int STORAGE, int BC, bool FORCED>
static cudaError_t launch_step_t(const StepArgs& a, const FusedForce& ff, int op, bool overlap, cudaStream_t s) {
    if (op == LBM_OP_BGK) return launch_op<LBM_OP_BGK, STORAGE, BC, FORCED>(a, ff, overlap, s);
    if (op == LBM_OP_KBC) return launch_op<LBM_OP_KBC, STORAGE, BC, FORCED>(a, ff, overlap, s);
    return launch_op<LBM_OP_REG, STORAGE, BC, FORCED>(a, ff, overlap, s);
}

// Forcing runs on periodic boxes only (contexts refuse it on the other boundaries).
template <int STORAGE>
static cudaError_t launch_step_s(const StepArgs& a, const FusedForce* ff, int op, int bc, bool overlap, cudaStream_t s) {
    const FusedForce none{};
    if (ff) {
        if (bc != LBM_BC_PERIODIC) return cudaErrorInvalidValue;
        return launch_step_t<STORAGE, LBM_BC_PERIODIC, true>(a, *ff, op, overlap, s);
    }
    if (bc == LBM_BC_PERIODIC) return launch_step_t<STORAGE, LBM_BC_PERIODIC, false>(a, none, op, overlap, s);
    if (bc == LBM_BC_TGV_REDUCED) return launch_step_t<STORAGE, LBM_BC_TGV_REDUCED, false>(a, none, op, overlap, s);
    return launch_step_t<STORAGE, LBM_BC_MIRROR, false>(a, none, op, overlap, s);
}

cudaError_t launch_step(const StepArgs& a, const FusedForce* ff, int op, int storage, int bc, int net_prec, bool deep,
                        const void* net_weights, int tc_shape, long long wait_cycles, bool overlap, cudaStream_t s) {
    if (op == LBM_OP_NCO && net_prec == LBM_NET_BF16)
        return launch_step_nco_tc(a, ff, storage, bc, deep, tc_shape, wait_cycles, net_weights, s);
    if (op == LBM_OP_NCO && net_prec == LBM_NET_BF16X3)
        return launch_step_nco_tc3(a, ff, storage, bc, deep, net_weights, wait_cycles, s);
    if (op == LBM_OP_NCO)
        return launch_step_nco_f32(a, ff, storage, bc, deep, static_cast<const NetParams*>(net_weights), overlap, s);
    switch (storage) {
        case LBM_STORE_F32: return launch_step_s<LBM_STORE_F32>(a, ff, op, bc, overlap, s);
        case LBM_STORE_F16_DEV: return launch_step_s<LBM_STORE_F16_DEV>(a, ff, op, bc, overlap, s);
        default: return launch_step_s<LBM_STORE_BF16_DEV>(a, ff, op, bc, overlap, s);
    }
}

// ---------------------------------------------------------------------------
// State initialisation and access. The stored buffer holds post-collision values
// f*(x, t-1); the pre-collision state is f_i(x, t) = f*_{ip}(src(x, i)), the pull map.
// Writing a given state scatters through the same map (a bijection), so reading it
// back is exact.
// ---------------------------------------------------------------------------
template <int STORAGE, int BC>
__global__ void init_eq_kernel(const Dims d, const float* __restrict__ rho, const float* __restrict__ u,
                               void* dst) {
    const long long cell = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (cell >= d.ncell) return;
    int x, y, z;
    cell_coords(cell, d, x, y, z);
    Macro q;
    q.rho = rho[cell];
    q.drho = q.rho - 1.0f;
    q.ux = u[cell];
    q.uy = u[d.ncell + cell];
    q.uz = u[2 * d.ncell + cell];
    using S = Store<STORAGE>;
    typename S::T* base = static_cast<typename S::T*>(dst);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        int ip, s;
        pull_source<BC>(x, y, z, i, d, ip, s);
        S::st(base + static_cast<size_t>(ip) * d.ncell + s, feq_dev(i, q));
    }
}

template <int STORAGE, int BC>
__global__ void set_state_kernel(const Dims d, const float* __restrict__ f, void* dst) {
    const long long cell = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (cell >= d.ncell) return;
    int x, y, z;
    cell_coords(cell, d, x, y, z);
    using S = Store<STORAGE>;
    typename S::T* base = static_cast<typename S::T*>(dst);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        int ip, s;
        pull_source<BC>(x, y, z, i, d, ip, s);
        S::st(base + static_cast<size_t>(ip) * d.ncell + s, f[static_cast<size_t>(i) * d.ncell + cell] - wgt(i));
    }
}

template <int STORAGE, int BC>
__global__ void get_state_kernel(const Dims d, const void* src, float* __restrict__ f) {
    const long long cell = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (cell >= d.ncell) return;
    int x, y, z;
    cell_coords(cell, d, x, y, z);
    float df[Q];
    load_pulled<STORAGE, BC>(src, d, x, y, z, df);
#pragma unroll
    for (int i = 0; i < Q; ++i) f[static_cast<size_t>(i) * d.ncell + cell] = wgt(i) + df[i];
}

template <int STORAGE, int BC>
__global__ void macroscopic_kernel(const Dims d, const void* src, float* __restrict__ rho,
                                   float* __restrict__ u) {
    const long long cell = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (cell >= d.ncell) return;
    int x, y, z;
    cell_coords(cell, d, x, y, z);
    float df[Q], m[Q];
    load_pulled<STORAGE, BC>(src, d, x, y, z, df);
    const float drho = moments_from_dev(df, m);
    const Macro q = macro_from_moments(m, drho);
    if (rho) rho[cell] = q.rho;
    if (u) {
        u[cell] = q.ux;
        u[d.ncell + cell] = q.uy;
        u[2 * d.ncell + cell] = q.uz;
    }
}

// k = (1/2) <|u|^2>: per-block FP64 partial sums, then one block adds the partials.
constexpr int kKeThreads = 256;

__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = v;
    __syncthreads();
    v = 0.0;
    if (threadIdx.x < (blockDim.x >> 5)) v = sh[threadIdx.x];
    if (w == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    }
    return v;
}

template <int STORAGE, int BC>
__global__ void __launch_bounds__(kKeThreads) ke_partial_kernel(const Dims d, const void* src,
                                                                double* partials) {
    __shared__ double sh[kKeThreads / 32];
    double acc = 0.0;
    for (long long cell = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; cell < d.ncell;
         cell += static_cast<long long>(gridDim.x) * blockDim.x) {
        int x, y, z;
        cell_coords(cell, d, x, y, z);
        float df[Q], m[Q];
        load_pulled<STORAGE, BC>(src, d, x, y, z, df);
        const float drho = moments_from_dev(df, m);
        const Macro q = macro_from_moments(m, drho);
        acc += 0.5 * (static_cast<double>(q.ux) * q.ux + static_cast<double>(q.uy) * q.uy +
                      static_cast<double>(q.uz) * q.uz);
    }
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = acc;
}

__global__ void __launch_bounds__(kKeThreads) sum_partials_kernel(const double* partials, int n,
                                                                  double scale, double* out) {
    __shared__ double sh[kKeThreads / 32];
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) acc += partials[i];
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) *out = acc * scale;
}

int kinetic_energy_blocks(const Dims& d) {
    const long long need = (d.ncell + kKeThreads - 1) / kKeThreads;
    return static_cast<int>(need < 152 * 8 ? need : 152 * 8);
}

// --- dispatch helpers --------------------------------------------------------
#define LBM_DISPATCH_SB(storage, bc, KERNEL_CALL)                                              \
    do {                                                                                       \
        if (storage == LBM_STORE_F32) {                                                        \
            if (bc == LBM_BC_PERIODIC) { constexpr int S_ = LBM_STORE_F32, B_ = LBM_BC_PERIODIC; KERNEL_CALL; } \
            else if (bc == LBM_BC_TGV_REDUCED) { constexpr int S_ = LBM_STORE_F32, B_ = LBM_BC_TGV_REDUCED; KERNEL_CALL; } \
            else { constexpr int S_ = LBM_STORE_F32, B_ = LBM_BC_MIRROR; KERNEL_CALL; }        \
        } else if (storage == LBM_STORE_F16_DEV) {                                             \
            if (bc == LBM_BC_PERIODIC) { constexpr int S_ = LBM_STORE_F16_DEV, B_ = LBM_BC_PERIODIC; KERNEL_CALL; } \
            else if (bc == LBM_BC_TGV_REDUCED) { constexpr int S_ = LBM_STORE_F16_DEV, B_ = LBM_BC_TGV_REDUCED; KERNEL_CALL; } \
            else { constexpr int S_ = LBM_STORE_F16_DEV, B_ = LBM_BC_MIRROR; KERNEL_CALL; }    \
        } else {                                                                               \
            if (bc == LBM_BC_PERIODIC) { constexpr int S_ = LBM_STORE_BF16_DEV, B_ = LBM_BC_PERIODIC; KERNEL_CALL; } \
            else if (bc == LBM_BC_TGV_REDUCED) { constexpr int S_ = LBM_STORE_BF16_DEV, B_ = LBM_BC_TGV_REDUCED; KERNEL_CALL; } \
            else { constexpr int S_ = LBM_STORE_BF16_DEV, B_ = LBM_BC_MIRROR; KERNEL_CALL; }   \
        }                                                                                      \
    } while (0)

static dim3 cell_grid(const Dims& d, int threads) {
    return dim3(static_cast<unsigned>((d.ncell + threads - 1) / threads));
}

cudaError_t launch_init_eq(const Dims& d, int storage, int bc, const float* rho, const float* u,
                           void* dst, cudaStream_t s) {
    LBM_DISPATCH_SB(storage, bc, (init_eq_kernel<S_, B_><<<cell_grid(d, 128), 128, 0, s>>>(d, rho, u, dst)));
    return cudaGetLastError();
}

cudaError_t launch_set_state(const Dims& d, int storage, int bc, const float* f, void* dst, cudaStream_t s) {
    LBM_DISPATCH_SB(storage, bc, (set_state_kernel<S_, B_><<<cell_grid(d, 128), 128, 0, s>>>(d, f, dst)));
    return cudaGetLastError();
}

cudaError_t launch_get_state(const Dims& d, int storage, int bc, const void* src, float* f, cudaStream_t s) {
    LBM_DISPATCH_SB(storage, bc, (get_state_kernel<S_, B_><<<cell_grid(d, 128), 128, 0, s>>>(d, src, f)));
    return cudaGetLastError();
}

cudaError_t launch_macroscopic(const Dims& d, int storage, int bc, const void* src, float* rho, float* u,
                               cudaStream_t s) {
    LBM_DISPATCH_SB(storage, bc, (macroscopic_kernel<S_, B_><<<cell_grid(d, 128), 128, 0, s>>>(d, src, rho, u)));
    return cudaGetLastError();
}

cudaError_t launch_kinetic_energy(const Dims& d, int storage, int bc, const void* src, double* partials,
                                  int npartials, double* out, cudaStream_t s) {
    LBM_DISPATCH_SB(storage, bc,
                    (ke_partial_kernel<S_, B_><<<npartials, kKeThreads, 0, s>>>(d, src, partials)));
    sum_partials_kernel<<<1, kKeThreads, 0, s>>>(partials, npartials, 1.0 / static_cast<double>(d.ncell), out);
    return cudaGetLastError();
}

}  // namespace lbm
