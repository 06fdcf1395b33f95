// net_f32.cuh - the FP32 invariant network of Sec. II.B (eq. gconv_m) as a block of twelve
// warps evaluates it on the CUDA cores; shared by the step and its adjoint.
//
// The 48 elements of O_h are (axis permutation p, sign vector s). With the columns of W1
// rearranged per p (W1p, built on the host from the group tables) the first layer of element
// (p, s) reads sgn(s, t) m_t, where sgn flips the moments that are odd in a
// reflected axis: sgn(s, t) = (-1)^popcount(s & c(t)) with c(t) the parity class of t (which
// axes t is odd in). Grouping the sum by class, the 8 sign vectors of one permutation are an
// 8-point Walsh-Hadamard transform of the 8 class sums y_c = sum_{t in class c} W1p[:, t] m_t:
// 20 x 27 MAC and 20 x 24 additions per permutation instead of 8 x 20 x 27 MAC.
//
// Warps (p, 0) and (p, 1) evaluate permutation p. Which columns (cell, sign vector) each of them
// has in its 32 rows of shared memory is one of the placements below: by halves of the sign
// vectors (the adjoint) or by halves of the cells (the step, whose group sum runs over the sign
// vectors of a cell in their order).
//
// What bounds it, and the layout: FP32 FMAs need their operands from shared memory at 16 bytes
// a lane per four cycles and SM, the time of four FMAs per lane on each scheduler; weights
// through the constant bank were slower (indexed loads stall, unrolled ones outgrow the
// instruction cache, and a launch starts with the bank cold). So a lane takes ten of the
// twenty units of the rows r and r + 16, and per four inputs reads 10 + 2 C vectors for 80 C
// FMAs (C = 4: 18 for 320).
#pragma once

#include "internal.h"

namespace lbm {

constexpr int kNetWarps = 12;       // two per axis permutation
constexpr int kHalf = kHidden / 2;  // hidden units of the first layer per warp

// Floats of a lane's row for C columns, a multiple of 4 whose quarter is odd: the 16-byte
// accesses of eight lanes to their own rows fall in different banks.
constexpr int net_row(int C) { return C * kHidden + 4; }
static_assert(net_row(4) / 4 % 2 == 1 && net_row(2) / 4 % 2 == 1, "bank-conflict-free rows");

// Floats of a warp's 32 rows: the sixteen at the end shift the second warp of a permutation by
// half the banks, so that the eight classes of a cell are read without conflicts.
constexpr int net_rows(int C) { return 32 * net_row(C) + 16; }

// y[s] <- sum_c (-1)^popcount(s & c) y[c] over N = 4 or 8 values, in place (its own inverse
// up to a factor N)
template <int N>
__device__ __forceinline__ void wht(float* y) {
#pragma unroll
    for (int bit = 1; bit < N; bit <<= 1)
#pragma unroll
        for (int c = 0; c < N; ++c)
            if (!(c & bit)) {
                const float u = y[c], v = y[c | bit];
                y[c] = u + v;
                y[c | bit] = u - v;
            }
}

__device__ __forceinline__ void pair_sync(int p) { asm volatile("bar.sync %0, 64;" ::"r"(p + 1) : "memory"); }

// Place of sign vector (or parity class) s of cell l + 16 k, l = lane % 16: which of the two warps
// of the permutation, how many rows after l, and which of the row's kCols columns.
// By sign vectors: warp (p, half) has [4 half, 4 half + 4) of every cell; a tile of 32 cells has
// a row per cell (LANES = 1), one of 16 cells two rows of two columns (LANES = 2; the second row
// has the sign vectors with bit 1 set).
template <int LANES>
struct BySigns {
    static constexpr int kCells = 2 / LANES, kCols = 4 / LANES;  // cells per lane, columns per row
    static __host__ __device__ constexpr int half(int s, int) { return s >> 2; }
    static __host__ __device__ constexpr int row(int s, int k) { return LANES == 1 ? 16 * k : 16 * ((s >> 1) & 1); }
    static __host__ __device__ constexpr int col(int s, int) { return LANES == 1 ? s & 3 : s & 1; }
};
// By cells: warp (p, half) has all eight of the cells [16 half, 16 half + 16), the first four in
// row l and the others in row l + 16.
struct ByCells {
    static constexpr int kCells = 2, kCols = 4;
    static __host__ __device__ constexpr int half(int, int k) { return k; }
    static __host__ __device__ constexpr int row(int s, int) { return 16 * (s >> 2); }
    static __host__ __device__ constexpr int col(int s, int) { return s & 3; }
};

// The block's copy of the parameters (the caller syncs).
__device__ __forceinline__ void load_params(NetParams* dst, const NetParams* __restrict__ src, int tid, int n) {
    for (int i = tid; i < static_cast<int>(sizeof(NetParams) / 16); i += n)
        reinterpret_cast<uint4*>(dst)[i] = __ldg(reinterpret_cast<const uint4*>(src) + i);
}

// relu(W1p x^(s) + b1) for the eight sign vectors s of permutation p, into the rows of its two
// warps (rows: the first warp's; those of the second follow net_rows floats later) as At places
// them. Of the warp's ten units a lane takes five, for the cells l = lane % 16 (and l + 16); m[k]
// are the moments of its cells in tensor order.
template <typename At>
__device__ __forceinline__ void first_layer(const NetParams& net, int p, int half, int lane, const float (*m)[28],
                                            float* rows) {
    constexpr int NC = At::kCells, C = At::kCols, R = net_row(C);
    const int j0 = half * kHalf + (lane >> 4) * 5;
    float* const out = rows + (lane & 15) * R + j0;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        float w[28];
#pragma unroll
        for (int t = 0; t < 28; t += 4) *reinterpret_cast<float4*>(w + t) = *reinterpret_cast<const float4*>(&net.W1p[p][j0 + i][t]);
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            float y[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) y[c] = 0.0f;
            static_for<Q>([&](auto T) {
                constexpr int t = decltype(T)::value, c = odd_mask(t), q = class_pos(t);
                y[c] = fmaf(w[q], m[k][t], y[c]);
            });
            wht<8>(y);
#pragma unroll
            for (int s = 0; s < 8; ++s)
                out[At::half(s, k) * net_rows(C) + At::row(s, k) * R + At::col(s, k) * kHidden + i] = fmaxf(y[s] + w[Q], 0.0f);
        }
    }
}

// acc[r][c][o] += sum_k W[10 og + o][k] x[r][c][k] for the lane's ten units (og = lane / 16)
// and the columns of the rows l + 16 r; get(k, v) loads v[r][c] = x[r][c][k..k+3]. UNROLL:
// steps of four inputs per loop iteration, all five where registers are left for it (the
// adjoint, 32^3 210 -> 203 us; the step, at its limit of 128, loses 2 %).
template <int C, int UNROLL, typename F>
__device__ __forceinline__ void mat_vec(const float (&W)[kHidden][kHidden], int lane, float (&acc)[2][C][kHalf], F&& get) {
    const float* w0 = &W[(lane >> 4) * kHalf][0];
#pragma unroll UNROLL
    for (int k = 0; k < kHidden; k += 4, w0 += 4) {
        float4 v[2][C];
        get(k, v);
#pragma unroll
        for (int o = 0; o < kHalf; ++o) {
            const float4 w = *reinterpret_cast<const float4*>(w0 + o * kHidden);
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    float a = acc[r][c][o];
                    a = fmaf(w.x, v[r][c].x, a);
                    a = fmaf(w.y, v[r][c].y, a);
                    a = fmaf(w.z, v[r][c].z, a);
                    acc[r][c][o] = fmaf(w.w, v[r][c].w, a);
                }
        }
    }
}

// The columns of a lane's two rows in shared memory, as mat_vec's x.
template <int C>
struct RowColumns {
    const float* x;  // row l
    __device__ __forceinline__ void operator()(int k, float4 (&v)[2][C]) const {
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c)
                v[r][c] = *reinterpret_cast<const float4*>(x + 16 * r * net_row(C) + c * kHidden + k);
    }
};

template <int C>
__device__ __forceinline__ void set_bias(const float* b, int lane, float (&acc)[2][C][kHalf]) {
#pragma unroll
    for (int o = 0; o < kHalf; ++o) {
        const float v = b[(lane >> 4) * kHalf + o];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c) acc[r][c][o] = v;
    }
}

// relu(acc) to the columns of the lane's two rows.
template <int C>
__device__ __forceinline__ void store_relu(float* x, int lane, const float (&acc)[2][C][kHalf]) {
    x += (lane >> 4) * kHalf;
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < C; ++c)
#pragma unroll
            for (int o = 0; o < kHalf; o += 2)
                *reinterpret_cast<float2*>(x + 16 * r * net_row(C) + c * kHidden + o) =
                    make_float2(fmaxf(acc[r][c][o], 0.0f), fmaxf(acc[r][c][o + 1], 0.0f));
}

}  // namespace lbm
