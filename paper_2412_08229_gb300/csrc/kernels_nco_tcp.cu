// kernels_nco_tcp.cu - the fused neural-collision step with the invariant network of
// Sec. II.B (eq. gconv_m) on the tcgen05 tensor cores, pipelined over pairs of group
// elements with every MMA operand A and accumulator in tensor memory (TMEM).
//
// One persistent CTA per SM runs three chains. A chain owns tiles of 128 cells (one cell per
// thread and TMEM lane) and walks the 24 pairs P = (2P, 2P + 1) of elements of O_h:
//   L1  D1[128 x 48] = A1[128 x 32] . B1_P^T  A1 = (m in the printed order, 1, 0, ..) in TMEM,
//                                            B1_P rows (e, j) = ((W1 P_g)[j,:], b1[j]), g = 2P + e;
//   L2  D2[128 x 48] = A2[128 x 48] . B2^T    A2 = (relu(h_a), 1, 0, 0, 0, relu(h_b), 1, 0, 0, 0)
//                                            in BF16, B2 = the block-diagonal pair of (W2 | b2),
//                                            so one chain of three MMAs serves both;
//   L3  on the CUDA cores: h = sum_g relu(D2) in FP32, tau~ = W3 h / 48 + b3 (layer 3 is
//       affine, so the group mean moves inside it).
// A2 is written over the upper half of the D1 it was made from, so a chain needs 160 TMEM
// columns - D1[2], D2, A1 - and three chains fit. Each chain has two warpgroups and a warp:
// the converters load the tile, form the moments and A1 and turn each D1 into A2; the summers
// fold each D2 into the group sum, form the rates, relax and store; the issuer warp does
// nothing but wait and issue MMAs. The next tile's populations are loaded into registers
// half-way through the walk; the moments reach the summers through shared memory,
// double-buffered.
//
// What bounds it (160^3, mixed form, ncu): instruction issue, 66 % of the cycles with 148 warp
// instructions per cell, then the chain's own latency (~840 cycles per pair) and the ALU pipe,
// 55 %; tensor pipe 41 % (five N 48 MMAs of 24.5 cycles per pair and tile), DRAM 7 %. The 256^3
// mixed step takes 3.16 ms, 3.36 ms with two tiles of two warpgroups per SM that both converted and
// summed, waiting for each pair's layer 2 before the next. What each part brought, 256^3, from
// 3.36 ms, each with relu as (b + |b|) / 2: 32-bit offsets and A2 in place with three chains 3.27;
// converters and summers apart 3.16; an issuer warp 3.11; named barriers instead of polls 3.05; D2
// read whole before the sum and layer 1 two pairs ahead 2.97. That relu runs on the FMA pipe where
// max runs on the ALU pipe at half the rate, but turns minus infinity into NaN and overflows above
// half of the largest float: with max, as everywhere else, the step takes 3.16 ms where it took 3.05
// on the same GPU.
//
// Hand-overs, per chain (n = 0..23 of a tile, b = n & 1):
//   a1full            A1 of the tile written (4 converter warps)      -> issuer: layer 1 of pairs 0, 1
//   a2full[b]         A2 of pair n written (4 converter warps)        -> issuer, with
//   d2free            D2 of pair n - 1 read (4 summer warps, who
//                     arrive once before the first tile)              -> issuer: layer 2 of pair n
//   CONV[b]           layer 1 of pair n + 1 complete                  issuer -> converters
//   SUM               layer 2 of pair n complete                      issuer -> summers; layer 1 of
//                     pair n + 2 then goes into buffer b, which that layer 2 has read
// The first three and the MMA commits are mbarriers, polled by the issuer alone; CONV and SUM are
// named barriers, in which warps block without taking issue slots (with every warp polling,
// polls were a third of the instructions). The next phase of each follows a hand-over that its
// waiters make after their wait (two pairs on for those with [b]). The moments go through the
// mbarriers mready[t & 1] / mfree[t & 1], complete by the time they are waited on but for the
// pipeline's start.
// Every poll is bounded in clock cycles. When one of a commit runs out the issuer polls no more
// commits and raises the chain's abort flag; the chain walks through its remaining tiles without storing, the
// issuer commits once more and waits (full limit) for that, and TMEM is released only when all
// have drained. B operands use the K-major, no-swizzle core-matrix layout of tc_ptx.cuh.
#include <cstring>

#include "force.cuh"
#include "tc_common.cuh"

namespace lbm {
using namespace tc;
using namespace tcc;

namespace {

constexpr int kTile = 128;
constexpr int kG = 48;
constexpr int kPairs = kG / 2;  // 24 pairs of group elements
constexpr int kN = 48;          // 2 elements x 20 hidden units + 8 padding rows
constexpr int kK1 = 32;         // 27 moments + bias input + pad
constexpr int kK2 = 48;         // 2 x (20 hidden + bias input + 3 pad)
constexpr int kChains = 3;
constexpr int kPrefetchPair = 12;  // the next tile's loads are issued after this pair
constexpr int kThreads = kChains * 256 + 128;  // converters, summers, one warpgroup of issuers
// registers a thread of each warpgroup holds: together the launch's 72 per thread
constexpr int kConverterRegs = 72, kSummerRegs = 88, kIssuerRegs = 24;
static_assert(kChains * (kConverterRegs + kSummerRegs) + kIssuerRegs == (2 * kChains + 1) * 72, "what one gives another takes");

// weight image = shared-memory image: 24 B1 pairs, the block-diagonal B2, W3 and b3 (floats)
constexpr uint32_t kB1PairBytes = kN * kK1 * 2;  // 3072
constexpr uint32_t kB1Off = 0;
constexpr uint32_t kB2Off = kB1Off + kPairs * kB1PairBytes;  // 73728
constexpr uint32_t kB2Bytes = kN * kK2 * 2;                  // 4608
constexpr uint32_t kW3Off = kB2Off + kB2Bytes;
constexpr uint32_t kB3Off = kW3Off + kOut * kHidden * 4;
constexpr uint32_t kWeightBytes = kB3Off + 16;  // 78672
static_assert(kWeightBytes % 16 == 0, "the weight image is one bulk copy");

// the moments and rho - 1 of two tiles of every chain
constexpr int kMVals = Q + 1;
constexpr uint32_t kMBufFloats = kMVals * kTile;
constexpr uint32_t kMOff = (kWeightBytes + 127) / 128 * 128;
constexpr uint32_t kBarOff = kMOff + kChains * 2 * kMBufFloats * 4;
// mbarriers: the commits of layer 1 per buffer and of layer 2, then the hand-overs
enum { kL1 = 0, kL2 = 2, kA1Full = 3, kA2Full = 4, kD2Free = 6, kMReady = 7, kMFree = 9, kDrain = 11, kBarsPerChain = 12 };
enum { kBarConv = 1, kBarSum = 7 };  // named: + 2 chain + b, + chain
// after the chains' barriers: the weight copy's barrier, the TMEM base, the chains' abort
// flags, then (forced steps) 2 F^ as floats and the block's projection sums
constexpr uint32_t kWBarOff = kBarOff + kChains * kBarsPerChain * 8;
constexpr uint32_t kAbortOff = kWBarOff + 16;
constexpr uint32_t kFhOff = kAbortOff + 16;
constexpr uint32_t kRedOff = (kFhOff + 6 * kForcedModes * 4 + 7) / 8 * 8;
constexpr uint32_t kSmemBytes = kRedOff + frc::kProjValues * 8;
static_assert(kBarOff % 8 == 0 && kSmemBytes <= 227 * 1024, "shared memory budget");

constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kTmemPerChain = 160;
constexpr uint32_t kD1Cols = 48, kD2Col = 96, kA1Col = 144;  // D1[b] at 48 b
constexpr uint32_t kA2InD1 = 24;                              // A2 = the upper half of a D1 buffer
static_assert(kChains * kTmemPerChain <= kTmemCols && kA1Col + 16 == kTmemPerChain, "TMEM budget");

// The populations a cell pulls, as stored (27 registers), from the wrapped offsets of
// load_pulled_offsets.
template <int STORAGE, int BC>
__device__ __forceinline__ void load_raw(const StepArgs& a, long long cell, typename Store<STORAGE>::T* raw) {
    int x, y, z;
    cell_coords(cell, a.d, x, y, z);
    using T = typename Store<STORAGE>::T;
    const T* base = static_cast<const T*>(a.src);
    const uint32_t plane = static_cast<uint32_t>(a.d.ncell);  // 27 planes stay below 2^31 elements
    for_pulled<BC>(a.d, x, y, z, [&](auto Ic, int ip, int src) {
        raw[decltype(Ic)::value] = __ldg(base + (static_cast<uint32_t>(ip) * plane + static_cast<uint32_t>(src)));
    });
}

template <int STORAGE, int BC, bool FORCED, bool BATCHED>
__global__ void __launch_bounds__(kThreads, 1) nco_tcp_kernel(const __grid_constant__ StepArgs a0, const BatchTiles bt,
                                                              const uint8_t* __restrict__ wimg, int ntiles,
                                                              long long limit, const FusedForce ff) {
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // uniform, and seen to be
    // warps 0..11 convert, 12..23 sum, 24..26 issue (27 has no part)
    const bool issuer = warp >= kChains * 8, summer = !issuer && warp >= kChains * 4;
    const int chain = issuer ? warp - kChains * 8 : (warp >> 2) - (summer ? kChains : 0);
    const int wq = warp & 3;  // TMEM lane quarter of this warp
    const int r = tid & 127;  // cell of the tile, TMEM lane
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kBarOff) + chain * kBarsPerChain;
    uint64_t* bar_w = reinterpret_cast<uint64_t*>(smem + kWBarOff);
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + kWBarOff + 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kAbortOff) + chain;
    float* fh2 = reinterpret_cast<float*>(smem + kFhOff);
    unsigned long long* red = reinterpret_cast<unsigned long long*>(smem + kRedOff);

    // ---- set-up: barriers, the weights' bulk copy (in flight until the first layer 1), TMEM
    if (tid == 0) {
        for (int c = 0; c < kChains; ++c) {
            uint64_t* b = reinterpret_cast<uint64_t*>(smem + kBarOff) + c * kBarsPerChain;
            for (int k = 0; k < kBarsPerChain; ++k)
                mbar_init(&b[k], k >= kA1Full && k < kDrain ? 4 : 1);
        }
        for (int c = 0; c < 4; ++c) *(reinterpret_cast<volatile int*>(smem + kAbortOff) + c) = 0;
        mbar_init(bar_w, 1);
        fence_mbar_init();
        mbar_expect_tx(bar_w, kWeightBytes);
        bulk_load(smem_u32(smem), wimg, kWeightBytes, bar_w);
    }
    if (FORCED) {
        frc::load_fh2(ff.fhat, fh2);
        if (tid < frc::kProjValues) red[tid] = 0ull;
    }
    if (warp == 0) tmem_alloc(tmem_holder, kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    // the allocation of all columns starts at column 0: TMEM addresses are constants
    const uint32_t tbase = static_cast<uint32_t>(chain) * kTmemPerChain;
    if (*tmem_holder != 0) *abort_flag = 1;
    const uint32_t lanes = static_cast<uint32_t>(wq * 32) << 16;
    float* mst = reinterpret_cast<float*>(smem + kMOff) + chain * 2 * kMBufFloats + r;
    const int lane_id = tid & 31;
    // bounded wait; one that runs out raises the abort flag
    auto wait = [&](uint64_t* bar, uint32_t parity, long long cycles) {
        if (!mbar_try_wait(bar, parity) && !wait_phase(bar, parity, cycles)) *abort_flag = 1;
    };
    auto args_of = [&bt](int gt, int& tile, const StepArgs*& ap) {
        tile = gt;
        if constexpr (BATCHED) {  // the instance owning this tile
            const int inst = __ldg(&bt.tile_inst[gt]);
            tile = gt - static_cast<int>(__ldg(&bt.tile_begin[inst]));
            ap = bt.inst + inst;
        }
    };
    // tiles in rounds over the SMs, so that a small grid spreads over them before it shares one
    const int stride = static_cast<int>(gridDim.x) * kChains;
    int gtile = static_cast<int>(blockIdx.x + gridDim.x * chain);
    bool drained = true;

    if (issuer) {
        reg_dec<kIssuerRegs>();
        // one copy of the loop per chain, so that every operand but the pair's descriptor is constant
        auto run = [&](auto Cc) {
            constexpr uint32_t base = decltype(Cc)::value * kTmemPerChain;
            constexpr uint32_t idesc = idesc_bf16(128, kN);
            const uint64_t db1 = smem_desc(smem_u32(smem + kB1Off), 128, 128 * kK1 / 8);
            const uint64_t db2 = smem_desc(smem_u32(smem + kB2Off), 128, 128 * kK2 / 8);
            auto issue_l1 = [&](int P, int b) {
#pragma unroll
                for (int kk = 0; kk < kK1 / 16; ++kk)
                    mma_bf16_ta(base + kD1Cols * b, base + kA1Col + 8 * kk, db1 + (P * kB1PairBytes + kk * 256) / 16, idesc, kk);
                mma_commit(&bars[kL1 + b]);
            };
            bool ok = *abort_flag == 0;
            auto poll_mma = [&](uint64_t* bar, uint32_t parity) {
                if (ok && !mbar_try_wait(bar, parity)) {
                    ok = wait_phase(bar, parity, limit);
                    if (!ok) *abort_flag = 1;
                }
                tc_fence_after();
                tc_fence_before();
            };
            auto poll_warps = [&](uint64_t* bar, uint32_t parity) {  // also after an abort: keeps pace with the other warps
                wait(bar, parity, kDefaultWaitCycles);
                tc_fence_after();
            };
            for (int it = 0; gtile < ntiles; gtile += stride, ++it) {
                poll_warps(&bars[kA1Full], static_cast<uint32_t>(it) & 1u);
                if (it == 0 && !mbar_try_wait(bar_w, 0) && !wait_phase(bar_w, 0, kDefaultWaitCycles)) {
                    ok = false;  // the weights have not arrived: waits for them once more before the block ends
                    *abort_flag = 1;
                }
                if (elect_one()) {
                    issue_l1(0, 0);
                    issue_l1(1, 1);
                }
                if (limit <= 0) {  // gives up at the first wait
                    ok = false;
                    *abort_flag = 1;
                }
                poll_mma(&bars[kL1], 0);
                bar_arrive<160>(kBarConv + 2 * chain);
#pragma unroll 1
                for (int n2 = 0; n2 < kPairs; n2 += 2) {
#pragma unroll
                    for (int b = 0; b < 2; ++b) {  // pair n = n2 + b, in buffer b
                        const uint32_t half = static_cast<uint32_t>(n2 >> 1);
                        poll_warps(&bars[kA2Full + b], half & 1u);
                        poll_warps(&bars[kD2Free], b);
                        if (elect_one()) {
#pragma unroll
                            for (int kk = 0; kk < kK2 / 16; ++kk)
                                mma_bf16_ta(base + kD2Col, base + kD1Cols * b + kA2InD1 + 8 * kk, db2 + kk * 16, idesc, kk);
                            mma_commit(&bars[kL2]);
                        }
                        if (b == 0 || n2 + 2 < kPairs) {  // a pair n + 1 follows
                            poll_mma(&bars[kL1 + (b ^ 1)], (half + b) & 1u);
                            bar_arrive<160>(kBarConv + 2 * chain + (b ^ 1));
                        }
                        poll_mma(&bars[kL2], b);
                        bar_arrive<160>(kBarSum + chain);
                        if (n2 + 2 < kPairs && elect_one()) issue_l1(n2 + b + 2, b);
                    }
                }
            }
            if (__any_sync(0xffffffffu, !ok)) {
                // one more commit and a wait, with the full limit, for all this lane issued: no MMA
                // may still use TMEM when it is released
                if (elect_one()) mma_commit(&bars[kDrain]);
                drained = wait_phase(&bars[kDrain], 0) && wait_phase(bar_w, 0);
            }
        };
        if (chain == 0) run(std::integral_constant<int, 0>{});
        else if (chain == 1) run(std::integral_constant<int, 1>{});
        else if (chain == 2) run(std::integral_constant<int, 2>{});
    } else if (!summer) {
        const uint32_t tA1 = tbase + kA1Col;
        typename Store<STORAGE>::T raw[Q];
        auto prefetch = [&](int gt) {
            if (gt >= ntiles) return;
            int tile;
            const StepArgs* ap = &a0;
            args_of(gt, tile, ap);
            const long long cell = static_cast<long long>(tile) * kTile + r;
            if (cell < ap->d.ncell) load_raw<STORAGE, BC>(*ap, cell, raw);
        };
        prefetch(gtile);
        for (int it = 0; gtile < ntiles; gtile += stride, ++it) {
            int tile;
            const StepArgs* ap = &a0;
            args_of(gtile, tile, ap);
            const StepArgs& a = *ap;
            const long long cell = static_cast<long long>(tile) * kTile + r;
            const bool valid = cell < a.d.ncell;
            if (it >= 2) wait(&bars[kMFree + (it & 1)], static_cast<uint32_t>((it >> 1) - 1) & 1u, kDefaultWaitCycles);
            {
                float m[Q];
                float drho = 0.0f;
                if (valid) {
                    float df[Q];
#pragma unroll
                    for (int i = 0; i < Q; ++i) df[i] = Store<STORAGE>::cvt(raw[i]);
                    drho = moments_from_dev(df, m);
                } else {
#pragma unroll
                    for (int e = 0; e < Q; ++e) m[e] = 0.0f;
                    m[0] = 1.0f;
                }
                float* mb = mst + (it & 1) * kMBufFloats;
#pragma unroll
                for (int e = 0; e < Q; ++e) mb[e * kTile] = m[e];
                mb[Q * kTile] = drho;
                // (after the transform: a branch among its sums has the compiler fuse other products
                // in the batched kernel, and an instance has to stay bit-identical to its own steps)
                if (valid && !(m[0] >= a.rho_min && m[0] <= a.rho_max)) atomicOr(a.status, 1);
                uint32_t p[16];  // A1 row r: the raw moments in the printed order of Sec. II.B, then the bias input 1
                static_for<13>([&](auto K) {
                    constexpr int k = decltype(K)::value;
                    p[k] = pack_bf16(m[kPrintedE<2 * k>], m[kPrintedE<2 * k + 1>]);
                });
                p[13] = pack_bf16(m[kPrintedE<26>], 1.0f);
                p[14] = 0u;
                p[15] = 0u;
                tmem_st16(tA1 + lanes, p);
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                mbar_arrive_lane0(&bars[kA1Full], lane_id);
                mbar_arrive_lane0(&bars[kMReady + (it & 1)], lane_id);
            }
            if (FORCED && ff.proj) {  // this tile's velocities into the next step's projection
                float* mb = mst + (it & 1) * kMBufFloats;
                Macro q{};
                int x = 0, y = 0, z = 0;
                if (valid) {
                    cell_coords(cell, a.d, x, y, z);
                    q = macro_from(mb[0], mb[1 * kTile], mb[3 * kTile], mb[9 * kTile], 0.0f);
                }
                frc::Cx ph[kForcedModes];
                frc::cell_phases(x, y, z, a.d, ff.tab, ph);
                long long pacc[3] = {0, 0, 0};
                frc::project_warp(q.ux, q.uy, q.uz, ph, tid & 31, pacc, ff.scale);
                frc::proj_to_shared(red, pacc, tid & 31);
            }
#pragma unroll 1
            for (int n2 = 0; n2 < kPairs; n2 += 2) {
#pragma unroll
                for (int b = 0; b < 2; ++b) {  // pair n = n2 + b, in buffer b
                    bar_sync<160>(kBarConv + 2 * chain + b);
                    tc_fence_after();
                    // D1 of the pair -> relu in BF16 = A2, over the upper half of the same buffer
                    const uint32_t t = tbase + lanes + kD1Cols * b;
                    uint32_t v[kHidden], h[24];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {  // one element of the pair after the other: fewer registers
                        tmem_ld16(t + kHidden * e, v);
                        tmem_ld4(t + kHidden * e + 16, v + 16);
                        tmem_ld_wait();
#pragma unroll
                        for (int k = 0; k < 10; ++k) h[12 * e + k] = pack_bf16_relu(as_f(v[2 * k]), as_f(v[2 * k + 1]));
                    }
                    h[10] = h[22] = kBf16One;
                    h[11] = h[23] = 0u;
#pragma unroll
                    for (int k = 0; k < 24; k += 8) tmem_st8(t + kA2InD1 + k, h + k);
                    tmem_st_wait();
                    tc_fence_before();
                    __syncwarp();
                    mbar_arrive_lane0(&bars[kA2Full + b], lane_id);
                }
                if (n2 == kPrefetchPair) prefetch(gtile + stride);
            }
        }
    } else {
        reg_inc<kSummerRegs>();
        const uint32_t tD2 = tbase + kD2Col + lanes;
        const float4* W3 = reinterpret_cast<const float4*>(smem + kW3Off);
        const float* b3 = reinterpret_cast<const float*>(smem + kB3Off);
        mbar_arrive_lane0(&bars[kD2Free], lane_id);  // D2 is free
        for (int it = 0; gtile < ntiles; gtile += stride, ++it) {
            // relu(h) summed over the even and over the odd pairs
            float acc[2][kHidden];
#pragma unroll
            for (int j = 0; j < kHidden; ++j) acc[0][j] = acc[1][j] = 0.0f;
#pragma unroll 1
            for (int n2 = 0; n2 < kPairs; n2 += 2) {
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    bar_sync<160>(kBarSum + chain);
                    tc_fence_after();
                    uint32_t v[40];
                    tmem_ld16(tD2, v);
                    tmem_ld16(tD2 + 16, v + 16);
                    tmem_ld8(tD2 + 32, v + 32);
                    tmem_ld_wait();
                    tc_fence_before();
                    __syncwarp();
                    mbar_arrive_lane0(&bars[kD2Free], lane_id);  // before the sum: layer 2 of the next pair waits for it
#pragma unroll
                    for (int j = 0; j < kHidden; j += 2) {
                        add2_relu(acc[b][j], acc[b][j + 1], as_f(v[j]), as_f(v[j + 1]));
                        add2_relu(acc[b][j], acc[b][j + 1], as_f(v[kHidden + j]), as_f(v[kHidden + j + 1]));
                    }
                }
            }
            wait(&bars[kMReady + (it & 1)], static_cast<uint32_t>(it >> 1) & 1u, kDefaultWaitCycles);
            if (it == 0) wait(bar_w, 0, kDefaultWaitCycles);  // W3 and b3, before this thread first reads them
            int tile;
            const StepArgs* ap = &a0;
            args_of(gtile, tile, ap);
            const StepArgs& a = *ap;
            const long long cell = static_cast<long long>(tile) * kTile + r;
            if (cell < a.d.ncell && !*abort_flag) {
                float rates[kOut];
#pragma unroll
                for (int j = 0; j < kHidden; ++j) acc[0][j] += acc[1][j];
#pragma unroll
                for (int k = 0; k < kOut; ++k) {
                    float t = 0.0f;
#pragma unroll
                    for (int j = 0; j < kHidden; j += 4) {
                        const float4 w = W3[(k * kHidden + j) / 4];
                        t = fmaf(w.x, acc[0][j], t);
                        t = fmaf(w.y, acc[0][j + 1], t);
                        t = fmaf(w.z, acc[0][j + 2], t);
                        t = fmaf(w.w, acc[0][j + 3], t);
                    }
                    rates[k] = rate_from_output(t * (1.0f / 48.0f) + b3[k]);
                }
                float F[3];
                if (FORCED) {  // F(x) from this step's coefficients
                    int x, y, z;
                    cell_coords(cell, a.d, x, y, z);
                    frc::Cx ph[kForcedModes];
                    frc::cell_phases(x, y, z, a.d, ff.tab, ph);
                    frc::synth_force(fh2, ph, F);
                }
                const float* mb = mst + (it & 1) * kMBufFloats;
                float m[Q];
#pragma unroll
                for (int e = 0; e < Q; ++e) m[e] = mb[e * kTile];
                const float drho = mb[Q * kTile];
                const Macro q = macro_from_moments(m, drho);
                if (BATCHED && a.u_out) {
                    a.u_out[cell] = q.ux;
                    a.u_out[a.d.ncell + cell] = q.uy;
                    a.u_out[2 * a.d.ncell + cell] = q.uz;
                }
                float df[Q];
                relax_to_populations(m, drho, q, 1.0f / a.tau, rates, df);
                if (FORCED) add_kupershtokh(df, q, F[0], F[1], F[2]);
                else if (BATCHED && a.force)
                    add_kupershtokh(df, q, a.force[cell], a.force[a.d.ncell + cell], a.force[2 * a.d.ncell + cell]);
                store_cell<STORAGE>(a.dst, a.d, cell, df);
            }
            __syncwarp();
            mbar_arrive_lane0(&bars[kMFree + (it & 1)], lane_id);
        }
    }
    if (lane_id == 0 && *abort_flag) atomicOr(a0.status, 2);
    tc_fence_before();
    if (!__syncthreads_and(drained)) {
        if (tid == 0) atomicOr(a0.status, 4);  // MMAs still running: TMEM is left allocated
        return;
    }
    if (FORCED && ff.proj && *abort_flag == 0) frc::proj_to_global(red, ff.proj);
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(*tmem_holder, kTmemCols);
    }
}

template <int STORAGE, int BC, bool FORCED, bool BATCHED>
cudaError_t launch_tcp_t(const StepArgs& a, const BatchTiles& bt, const void* w, int ntiles, long long wait,
                         const FusedForce& ff, cudaStream_t s) {
    static std::atomic<unsigned long long> attr{0};
    const cudaError_t e =
        ensure_dynamic_smem(nco_tcp_kernel<STORAGE, BC, FORCED, BATCHED>, static_cast<int>(kSmemBytes), attr);
    if (e != cudaSuccess) return e;
    const int grid = ntiles < sm_count() ? ntiles : sm_count();
    if (grid < 1) return cudaSuccess;
    nco_tcp_kernel<STORAGE, BC, FORCED, BATCHED>
        <<<grid, kThreads, kSmemBytes, s>>>(a, bt, static_cast<const uint8_t*>(w), ntiles, wait, ff);
    return cudaGetLastError();
}

template <int STORAGE>
cudaError_t launch_tcp_b(const StepArgs& a, const FusedForce* ff, int bc, const void* w, long long wait,
                         cudaStream_t s) {
    const int ntiles = static_cast<int>((a.d.ncell + kTile - 1) / kTile);
    const BatchTiles none{nullptr, nullptr, nullptr, 0};
    const FusedForce nf{};
    if (ff) {  // forcing runs on periodic boxes only
        if (bc != LBM_BC_PERIODIC) return cudaErrorInvalidValue;
        return launch_tcp_t<STORAGE, LBM_BC_PERIODIC, true, false>(a, none, w, ntiles, wait, *ff, s);
    }
    if (bc == LBM_BC_TGV_REDUCED)
        return launch_tcp_t<STORAGE, LBM_BC_TGV_REDUCED, false, false>(a, none, w, ntiles, wait, nf, s);
    return bc == LBM_BC_PERIODIC ? launch_tcp_t<STORAGE, LBM_BC_PERIODIC, false, false>(a, none, w, ntiles, wait, nf, s)
                                 : launch_tcp_t<STORAGE, LBM_BC_MIRROR, false, false>(a, none, w, ntiles, wait, nf, s);
}

}  // namespace

size_t nco_tcp_weight_bytes() { return kWeightBytes; }

void nco_tcp_pack_weights(const float* theta, void* out) {
    const float* W1 = theta;  // (20, 27), printed moment order
    const float* b1 = W1 + kHidden * Q;
    const float* W2 = b1 + kHidden;
    const float* b2 = W2 + kHidden * kHidden;
    const float* W3 = b2 + kHidden;
    const float* b3 = W3 + kOut * kHidden;
    uint8_t* img = static_cast<uint8_t*>(out);
    std::memset(img, 0, kWeightBytes);
    auto put = [&](uint32_t base, int row, int k, int K, float v) {
        const uint16_t b = f2bf(v);
        std::memcpy(img + base + kmajor_offset(row, k, K), &b, 2);
    };
    const GroupTables& gt = group_tables();
    for (int g = 0; g < kG; ++g) {
        const uint32_t base = kB1Off + (g / 2) * kB1PairBytes;
        for (int j = 0; j < kHidden; ++j) {
            const int row = (g % 2) * kHidden + j;
            // (W1 P_g m)_j = sum_k W1[j][k] msign[g][k] m[mperm[g][k]] (printed order)
            for (int k = 0; k < Q; ++k) {
                const int e = kPrinted.e[k];
                int kp = 0;
                for (int t = 0; t < Q; ++t)
                    if (kPrinted.e[t] == gt.mperm_t[g][e]) kp = t;
                put(base, row, kp, kK1, W1[j * Q + k] * static_cast<float>(gt.msign_t[g][e]));
            }
            put(base, row, Q, kK1, b1[j]);
        }
    }
    for (int j = 0; j < kHidden; ++j)
        for (int half = 0; half < 2; ++half) {  // block diagonal: element a at K 0..20, element b at K 24..44
            const int row = half * kHidden + j, k0 = half * 24;
            for (int k = 0; k < kHidden; ++k) put(kB2Off, row, k0 + k, kK2, W2[j * kHidden + k]);
            put(kB2Off, row, k0 + kHidden, kK2, b2[j]);
        }
    std::memcpy(img + kW3Off, W3, kOut * kHidden * sizeof(float));
    std::memcpy(img + kB3Off, b3, kOut * sizeof(float));
}

cudaError_t launch_step_nco_tcp_batch(const StepArgs* d_inst, const long long* d_tile_begin, const int* d_tile_inst,
                                      int ninst, long long ntiles, int storage, int* status, const void* w,
                                      cudaStream_t s) {
    StepArgs sa{};
    sa.status = status;
    const BatchTiles bt{d_inst, d_tile_begin, d_tile_inst, ninst};
    const int nt = static_cast<int>(ntiles);
    const FusedForce nf{};
    switch (storage) {
        case LBM_STORE_F32:
            return launch_tcp_t<LBM_STORE_F32, LBM_BC_PERIODIC, false, true>(sa, bt, w, nt, kDefaultWaitCycles, nf, s);
        case LBM_STORE_F16_DEV:
            return launch_tcp_t<LBM_STORE_F16_DEV, LBM_BC_PERIODIC, false, true>(sa, bt, w, nt, kDefaultWaitCycles, nf, s);
        default:
            return launch_tcp_t<LBM_STORE_BF16_DEV, LBM_BC_PERIODIC, false, true>(sa, bt, w, nt, kDefaultWaitCycles, nf, s);
    }
}

cudaError_t launch_step_nco_tcp(const StepArgs& a, const FusedForce* ff, int storage, int bc, const void* w,
                                long long wait_cycles, cudaStream_t s) {
    switch (storage) {
        case LBM_STORE_F32: return launch_tcp_b<LBM_STORE_F32>(a, ff, bc, w, wait_cycles, s);
        case LBM_STORE_F16_DEV: return launch_tcp_b<LBM_STORE_F16_DEV>(a, ff, bc, w, wait_cycles, s);
        default: return launch_tcp_b<LBM_STORE_BF16_DEV>(a, ff, bc, w, wait_cycles, s);
    }
}

}  // namespace lbm
