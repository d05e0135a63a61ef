// Fused coupled fine/coarse Dean--Kawasaki sample kernel for sm_103a.
//
// One launch runs `count` independent samples of one level (Section 3.2: the
// fine path on G_{h_l} and, for l >= 1, the Right-Most NN coupled coarse path
// on G_{h_{l-1}}), each for M fine steps of Eq. (FullyDiscreteDK) with
// b0 = 0, b1 = 1 (Section 7.2), and reduces every sample on the fly to the
// observables (rho^T, I_h phi_k)_h, the quantities P = N (Y_j - Ybar_j)(Y_k -
// Ybar_k) of Eq. (eqn_MLMCLevels) and the FP64 moment sums that the estimator
// of Eq. (MLMCEstimator) and the allocation of Eq. (opt_M_ell) need.
//
// Work decomposition.  A sample's fine grid is cut into bands of FR = 2R fine
// rows; a band is held by LPB <= 32 consecutive lanes of one warp, each lane
// owning an FR x FC block (FC = 2C) of fine cells, i.e. an R x C block of the
// coarse grid, so the coupled coarse increment (the sum over the 2x2 fine
// cells to the right of each coarse point and over the 4 fine steps of one
// coarse step) is accumulated in the lane's registers.  The whole state lives
// in registers for the whole run.  Left/right neighbours come from the
// adjacent lanes by warp shuffles (the periodic wrap is the shuffle's segment
// wrap).  Up/down neighbours come
//   * by shuffles too when the whole sample fits one warp (n <= 32), so those
//     samples run without any barrier or shared memory, or
//   * through shared memory (double-buffered band edge rows, one barrier per
//     fine step) when the sample spans several warps; grids that need more
//     registers than one SM has span a thread-block cluster and read the
//     neighbouring CTA's edge rows through distributed shared memory.
//
// Arithmetic.  The state is 32-bit fixed point q = rho 2^S.  Each fine step
// computes, per cell, the noise transfers G_r = rint(c 2^S sqrt(rho^+) Z_r)
// (c = N^-1/2 sqrt(tau) / (2 h^2)) and, per edge, the diffusion flux
// rint(tau/(2h^2) (q_far - q_near)); the new state adds these integers
// exactly, so sum_x q is invariant bit for bit (the divergence form of the
// scheme) and every rounding error enters in divergence form.  Observables
// and moments are accumulated in FP64.
//
// What bounds it: instruction pipes, not memory.  A fine cell-step needs 7 XU
// operations (log, sine, cosine, two square roots, two conversions: 56 cycles of
// the sub-partition per warp), about 11 wide multiplies (half a Philox4x32-10
// call and the fluxes: 55 cycles of the FMA pipe) and some 50 instructions in
// all.  Hence two cell pairs at a time in packed FP32 (half the FP32
// instructions, the same roundings) and, where the registers allow, the next
// pairs' Philox rounds interleaved with the current pairs' functions (PIPE).
// Per warp of fine cells, 64^2 coupled: 107 cycles before, 89 now (9.47 ms for
// 1151 samples x 832 steps, 11.07 before); 256^2, 59 x 1536: 19.7 ms, 22.8
// before; 32^2 fine only, 1000 x 103: 0.280 ms, 0.316 before.
#include <cooperative_groups.h>

#include <algorithm>

#include "dk_device.cuh"
#include "dk_kernels.h"

namespace cg = cooperative_groups;

namespace dk {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kRedW = 2 * kMaxObs + 2;     // reduced values per sample
constexpr int kMaxStride = 2 + kNSum * 10;  // largest slot stride (4 obs with products)

template <int NF_, int C_, int R_, int CL_, bool COUPLED_, bool FLUCT_ = false, int CHAIN_ = 1, bool SECOND_ = false>
struct Shape {
    static constexpr int NF = NF_, C = C_, R = R_, CL = CL_;
    static constexpr bool COUPLED = COUPLED_;
    // fluctuation state: q holds (rho - rho-bar^m) 2^S, rho-bar^m read from a
    // per-step mean-field table (see KArgs::rbf)
    static constexpr bool FLUCT = FLUCT_;
    // a lane's FP32 projection sums run on through the blocks of CHAIN bands, one
    // below the other: the sums of a shape with CHAIN times the rows per lane
    static constexpr int CHAIN = CHAIN_;
    // the second build of a shape that has two (see Split)
    static constexpr bool SECOND = SECOND_;
    static constexpr int NC = NF / 2;
    static constexpr int FR = 2 * R, FC = 2 * C;
    static constexpr int LPB = NC / C;            // lanes per band
    static constexpr int NB = NC / R;             // bands per sample
    static constexpr int LPS = LPB * NB;          // lanes per sample
    static constexpr bool WARP = LPS <= 32;       // sample resident in one warp
    static constexpr int SPW = WARP ? 32 / LPS : 1;
    static constexpr int THREADS = WARP ? 128 : LPS / CL;
    static constexpr int BPC = WARP ? 1 : NB / CL;   // bands per CTA
    // How a step is laid out in the instruction stream (the arithmetic is the
    // same), by block size and registers per thread; measured, ms at the sizes
    // given (coupled unless said otherwise; "before": scalar FP32 noise, no bound on
    // the registers):
    //   PIPE   the Philox rounds of the next two cell pairs run between the
    //          Box--Muller stages of the current two (FMA and ALU pipes under the
    //          XU pipe), and a row is updated as soon as its transfers are known.
    //          It wants the registers of 8 to 16 warps per SM: one-CTA samples of
    //          several warps (64^2, 1151 samples x 832 steps: 9.6, without 10.5,
    //          before 11.1; 32^2, 4630 x 208: 2.31, 2.52, 2.57), of one warp with 16
    //          cells a lane or a coupled path (16^2, 2 x 2 coarse cells a lane, 1000 x 52
    //          plain: 0.055, without 0.068, before 0.068; 1 x 2 coupled, 10000 x 52:
    //          0.35, 0.37, 0.37), and in clusters blocks of 32 cells (256^2, 59 x 1536:
    //          19.8, 23.5, 22.8) or of one coarse row (128^2 by 4 CTAs, 304 x 64: 3.24,
    //          without 3.83, before 3.54).  With 2 x 2 coarse cells at 128 registers it
    //          spills and loses (128^2, 304 x 1664: 25.0, without 23.7).
    //   REDRAW the sample's Philox counter word is opaque to the compiler, which
    //          then does not keep the step-independent parts of the first rounds in
    //          registers, where those would spill (128^2: 22.7 with, 23.7 without,
    //          25.1 before; 256^2: 19.8 with, 23.0 without).  Fine-only 128^2 does not
    //          spill (40 samples x 384: 1.32 with, 1.27 without, 1.31 before).  One
    //          coarse row: only plain with 4 columns (256^2, 59 x 102: 3.13 with, 3.49
    //          without, 3.72 before).
    //   The fluctuation state needs its mean-field rows in registers as well and
    //   is fastest with neither (128^2, 311 x 1024: 18.6, before 20.2; 64^2, 997 x
    //   256: 2.89, with PIPE 3.28, before 3.13; loading the next step's rows
    //   early: 20.3 at 128^2), but for the plain 32^2 level (1824 x 64: 0.269 with,
    //   0.328 without, before 0.302).
    static constexpr bool PIPE = FLUCT    ? NF == 32 && !COUPLED && SECOND && CHAIN == 1
                                 : CL > 1 ? R == 1 || FR * FC >= 32
                                 : WARP   ? R == 2 && (COUPLED || C == 2)
                                          : !(NF == 16 && C == 1 && R == 1 && !SECOND && CHAIN == 1);
    static constexpr bool REDRAW = !FLUCT && CL > 1 && (R == 1 ? C == 4 && !COUPLED : COUPLED || FR * FC >= 32);
    // Resident warps per SM asked for (a bound on the registers per thread); the
    // figures of the shapes with two builds are at Split.  32^2 fine-only, 1000 x 103:
    // 8 warps 0.288 ms, 12 warps 0.281; 16^2 in one warp, plain, 9250 x 52: 16 warps
    // 0.316, 24 warps 0.306 (before 0.337), coupled, 1000 x 52: 16 warps with PIPE
    // 0.059, 24 warps 0.072 (before 0.062).
    static constexpr int WARPS_MIN =
        FLUCT               ? (NF == 8 ? (SECOND ? 16 : 20) : !SECOND ? 16 : PIPE ? 12 : 8)
        : FR * FC >= 32     ? 8
        : WARP              ? (FR * FC >= 16 ? 8 : FR * FC >= 8 && !COUPLED ? 24 : 16)
        : FR * FC < 8       ? (PIPE ? 12 : 24)
        : PIPE && FR * FC < 16 && NF == 32 && CHAIN == 1 ? (SECOND ? 12 : 16)
        : PIPE              ? (COUPLED && FR * FC >= 16 ? 8 : 12)
                            : 16;
    static constexpr int MINB = WARPS_MIN * 32 / THREADS > 0 ? WARPS_MIN * 32 / THREADS : 1;
    static constexpr int SLOTS_PER_CTA = WARP ? (THREADS / 32) * SPW : 1;
    // Two cell pairs (Philox calls) are worked on together, packed: neighbours
    // along a row (C even), or the same pair of two coarse rows (C = 1, R = 2),
    // or the two rows of a single coarse cell (C = R = 1).
    static constexpr int DPC = C >= 2 ? 1 : 0;                 // offset of the second pair: columns,
    static constexpr int DR = C >= 2 ? 0 : (R >= 2 ? 2 : 1);   // fine rows
    static constexpr bool ZPACK = C >= 2 || R >= 2;            // their coupled sums are two coarse cells'
    static constexpr int NZ = (R * C + 1) / 2;                 // packed coupled sums per component
    static_assert(C % 2 == 0 || (C == 1 && R <= 2), "cell pairs are worked on two at a time");
    static_assert(LPB <= 32 && (LPB & (LPB - 1)) == 0, "a band must be a power-of-two warp segment");
    static_assert(NC % C == 0 && NC % R == 0, "lane blocks must tile the coarse grid");
    static_assert(CHAIN == 1 || (CHAIN == 2 && !WARP && CL == 1 && 32 % (2 * LPB) == 0),
                  "chained bands share a warp");
    static_assert(WARP || (THREADS % 32 == 0 && THREADS <= 1024 && NB % CL == 0), "bad CTA shape");
    static_assert(WARP || CL == 1 || (LPS / CL) % LPB == 0, "bands may not straddle CTAs");
    static constexpr size_t fixed_smem() {
        return WARP ? 0
                    : sizeof(int2) * 2 * 2 * BPC * NF + (COUPLED ? sizeof(int2) * 2 * BPC * NC : 0) +
                          sizeof(double) * (THREADS / 32) * kRedW;
    }
};

template <int N>
__device__ __forceinline__ void load_row(int32_t (&dst)[N], const int32_t* src) {
    if constexpr (N == 1) {
        dst[0] = __ldg(src);
    } else if constexpr (N == 2) {
        const int2 v = __ldg(reinterpret_cast<const int2*>(src));
        dst[0] = v.x; dst[1] = v.y;
    } else {
        static_assert(N % 4 == 0, "");
#pragma unroll
        for (int i = 0; i < N; i += 4) {
            const int4 v = __ldg(reinterpret_cast<const int4*>(src + i));
            dst[i] = v.x; dst[i + 1] = v.y; dst[i + 2] = v.z; dst[i + 3] = v.w;
        }
    }
}

template <int N>
__device__ __forceinline__ void load_row_f(float (&dst)[N], const float* src) {
    if constexpr (N == 1) {
        dst[0] = __ldg(src);
    } else if constexpr (N == 2) {
        const float2 v = __ldg(reinterpret_cast<const float2*>(src));
        dst[0] = v.x; dst[1] = v.y;
    } else {
#pragma unroll
        for (int i = 0; i < N; i += 4) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(src + i));
            dst[i] = v.x; dst[i + 1] = v.y; dst[i + 2] = v.z; dst[i + 3] = v.w;
        }
    }
}

// Store / load the N (q, G1) pairs of one lane's part of a band edge row.
// Lane-interleaved layout: pair chunk k (columns 2k, 2k+1 of the lane) of lane
// `lib` is int4 number k*LPB + lib of the row, so a warp's store or load of one
// chunk is LPB consecutive 16-byte words (no bank conflicts).  N = 1 uses one
// int2 per lane.
template <int N, int LPB>
__device__ __forceinline__ void put_edge(int2* row, int lib, const int32_t (&qv)[N], const int32_t (&gv)[N]) {
    if constexpr (N % 2 == 0) {
        int4* r4 = reinterpret_cast<int4*>(row);
#pragma unroll
        for (int k = 0; k < N / 2; ++k) r4[k * LPB + lib] = make_int4(qv[2 * k], gv[2 * k], qv[2 * k + 1], gv[2 * k + 1]);
    } else {
        static_assert(N == 1, "odd edge chunks other than 1 are not used");
        row[lib] = make_int2(qv[0], gv[0]);
    }
}

template <int N, int LPB>
__device__ __forceinline__ void get_edge(const int2* row, int lib, int32_t (&qv)[N], int32_t (&gv)[N]) {
    if constexpr (N % 2 == 0) {
        const int4* r4 = reinterpret_cast<const int4*>(row);
#pragma unroll
        for (int k = 0; k < N / 2; ++k) {
            const int4 v = r4[k * LPB + lib];
            qv[2 * k] = v.x; gv[2 * k] = v.y; qv[2 * k + 1] = v.z; gv[2 * k + 1] = v.w;
        }
    } else {
        const int2 v = row[lib];
        qv[0] = v.x; gv[0] = v.y;
    }
}

// Index of the cell pair `pc` of a lane's block row at column col0.
template <class S>
__device__ __forceinline__ uint32_t pair_index(int row, int col0, int pc) {
    return static_cast<uint32_t>((row * S::NF + col0 + 2 * pc) >> 1);
}

// Row r's part of the update, with its transfers known and its state (and the
// row above's) old: the horizontal fluxes and transfers, halo columns by
// shuffles from the adjacent lanes, and the vertical flux between rows r - 1
// and r, which completes row r - 1 (all but the first row, which waits for the
// row above the block).  Row by row, only one row's pending change and transfers
// are live at a time.
template <class S>
__device__ __forceinline__ void row_update(int r, int32_t (&q)[S::FR][S::FC], const int32_t (&G1)[S::FR][S::FC],
                                           const int32_t (&G2)[S::FR][S::FC], int32_t (&pend)[2][S::FC],
                                           int32_t (&pend0)[S::FC], int left, int right, int32_t A) {
    constexpr int FC = S::FC;
    const int32_t qL = __shfl_sync(kFull, q[r][FC - 1], left, S::LPB), gL = __shfl_sync(kFull, G2[r][FC - 1], left, S::LPB);
    const int32_t qR = __shfl_sync(kFull, q[r][0], right, S::LPB), gR = __shfl_sync(kFull, G2[r][0], right, S::LPB);
    int32_t (&cur)[FC] = pend[r & 1];
    int32_t h = edge_flux(A, q[r][0] - qL);
#pragma unroll
    for (int c = 0; c < FC; ++c) {
        const int32_t hn = c + 1 < FC ? edge_flux(A, q[r][c + 1] - q[r][c]) : edge_flux(A, qR - q[r][FC - 1]);
        const int32_t g2r = c + 1 < FC ? G2[r][c + 1] : gR, g2l = c > 0 ? G2[r][c - 1] : gL;
        cur[c] = (hn - h) + (g2r - g2l);
        h = hn;
    }
    if (r > 0) {
#pragma unroll
        for (int c = 0; c < FC; ++c) {
            const int32_t v = edge_flux(A, q[r][c] - q[r - 1][c]);
            cur[c] -= v + G1[r - 1][c];
            const int32_t u = pend[(r - 1) & 1][c] + v + G1[r][c];
            if (r == 1) pend0[c] = u;
            else q[r - 1][c] += u;
        }
    }
}

template <class S, class T>
__device__ __forceinline__ const T* peer(const T* local, int rank) {
    if constexpr (S::CL > 1) {
        return cg::this_cluster().map_shared_rank(const_cast<T*>(local), rank);
    } else {
        return local;
    }
}

// The same update in two phases around a split barrier: phase 1 updates the
// interior rows (1 .. RR-2), which need no vertical halo, and keeps the old
// values of rows 1 and RR-2 that the boundary rows' fluxes need; phase 2
// (after the halo arrives) updates rows 0 and RR-1.
template <int RR, int CC>
__device__ __forceinline__ void flux_update_interior(int32_t (&q)[RR][CC], const int32_t (&G1)[RR][CC],
                                                     const int32_t (&G2)[RR][CC], const int32_t (&qL)[RR],
                                                     const int32_t (&gL)[RR], const int32_t (&qR)[RR],
                                                     const int32_t (&gR)[RR], int32_t A, int32_t (&keep1)[CC],
                                                     int32_t (&keep2)[CC]) {
#pragma unroll
    for (int c = 0; c < CC; ++c) {
        keep1[c] = q[1][c];
        keep2[c] = q[RR - 2][c];
    }
    if constexpr (RR >= 3) {
        int32_t V[RR + 1][CC];
#pragma unroll
        for (int c = 0; c < CC; ++c)
#pragma unroll
            for (int r = 1; r < RR; ++r) V[r][c] = edge_flux(A, q[r][c] - q[r - 1][c]);
#pragma unroll
        for (int r = 1; r + 1 < RR; ++r) {
            int32_t H[CC + 1];
            H[0] = edge_flux(A, q[r][0] - qL[r]);
#pragma unroll
            for (int c = 1; c < CC; ++c) H[c] = edge_flux(A, q[r][c] - q[r][c - 1]);
            H[CC] = edge_flux(A, qR[r] - q[r][CC - 1]);
#pragma unroll
            for (int c = 0; c < CC; ++c) {
                const int32_t g2r = (c + 1 < CC) ? G2[r][c + 1] : gR[r];
                const int32_t g2l = (c > 0) ? G2[r][c - 1] : gL[r];
                q[r][c] += (V[r + 1][c] - V[r][c]) + (H[c + 1] - H[c]) + (G1[r + 1][c] - G1[r - 1][c]) + (g2r - g2l);
            }
        }
    }
}

template <int RR, int CC>
__device__ __forceinline__ void flux_update_boundary(int32_t (&q)[RR][CC], const int32_t (&G1)[RR][CC],
                                                     const int32_t (&G2)[RR][CC], const int32_t (&qU)[CC],
                                                     const int32_t (&gU)[CC], const int32_t (&qD)[CC],
                                                     const int32_t (&gD)[CC], const int32_t (&qL)[RR],
                                                     const int32_t (&gL)[RR], const int32_t (&qR)[RR],
                                                     const int32_t (&gR)[RR], int32_t A, const int32_t (&keep1)[CC],
                                                     const int32_t (&keep2)[CC]) {
    // row 0 (its lower neighbour is the old row 1) and row RR-1 (upper neighbour the old row RR-2)
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const int r = side == 0 ? 0 : RR - 1;
        if (side == 1 && RR == 1) break;
        int32_t H[CC + 1];
        H[0] = edge_flux(A, q[r][0] - qL[r]);
#pragma unroll
        for (int c = 1; c < CC; ++c) H[c] = edge_flux(A, q[r][c] - q[r][c - 1]);
        H[CC] = edge_flux(A, qR[r] - q[r][CC - 1]);
#pragma unroll
        for (int c = 0; c < CC; ++c) {
            const int32_t up = (r == 0) ? qU[c] : keep2[c];
            const int32_t dn = (r == RR - 1) ? qD[c] : keep1[c];
            const int32_t g1u = (r == 0) ? gU[c] : G1[r - 1][c];
            const int32_t g1d = (r == RR - 1) ? gD[c] : G1[r + 1][c];
            const int32_t x = q[r][c];
            const int32_t v = edge_flux(A, dn - x) - edge_flux(A, x - up);
            const int32_t g2r = (c + 1 < CC) ? G2[r][c + 1] : gR[r];
            const int32_t g2l = (c > 0) ? G2[r][c - 1] : gL[r];
            q[r][c] = x + v + (H[c + 1] - H[c]) + (g1d - g1u) + (g2r - g2l);
        }
    }
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }

template <class S>
__global__ void __launch_bounds__(S::THREADS, S::MINB) level_kernel(const KArgs a) {
    constexpr int NF = S::NF, NC = S::NC, FR = S::FR, FC = S::FC, R = S::R, C = S::C;
    constexpr int LPB = S::LPB, LPS = S::LPS, CL = S::CL, BPC = S::BPC;
    constexpr bool CPL = S::COUPLED;
    // clusters split the per-step barrier: arrive after publishing the edge
    // rows, update the interior rows, then wait for the neighbours' rows
    constexpr bool SPLIT = !S::WARP && (CL > 1);
    extern __shared__ __align__(16) unsigned char smem_raw[];

    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int lib = lane % LPB;   // lane within its band
    int band, bl = 0, rank = 0, slot_local;
    long long slot, n_slots, base_slot;
    if constexpr (S::WARP) {
        band = (lane % LPS) / LPB;
        slot_local = (tid >> 5) * S::SPW + lane / LPS;
        slot = (long long)blockIdx.x * S::SLOTS_PER_CTA + slot_local;
        n_slots = (long long)gridDim.x * S::SLOTS_PER_CTA;
        base_slot = (long long)blockIdx.x * S::SLOTS_PER_CTA + (tid >> 5) * S::SPW;
    } else {
        if constexpr (CL > 1) rank = (int)cg::this_cluster().block_rank();
        bl = tid / LPB;
        band = rank * BPC + bl;
        slot_local = 0;
        slot = blockIdx.x / CL;
        n_slots = gridDim.x / CL;
        base_slot = slot;
    }
    const int row0 = band * FR, col0 = lib * FC;     // fine block origin
    const int crow0 = band * R, ccol0 = lib * C;      // coarse block origin
    const int left = (lib + LPB - 1) % LPB, right = (lib + 1) % LPB;
    const int up_lane = ((lane % LPS) + LPS - LPB) % LPS, dn_lane = ((lane % LPS) + LPB) % LPS;

    // shared memory: [fine edge rows][coarse edge rows][reduction][slot accumulators]
    unsigned char* sp = smem_raw;
    int2* fx = nullptr;
    int2* cx = nullptr;
    double* red = nullptr;
    if constexpr (!S::WARP) {
        fx = reinterpret_cast<int2*>(sp);
        sp += sizeof(int2) * 2 * 2 * BPC * NF;
        if constexpr (CPL) {
            cx = reinterpret_cast<int2*>(sp);
            sp += sizeof(int2) * 2 * BPC * NC;
        }
        red = reinterpret_cast<double*>(sp);
        sp += sizeof(double) * (S::THREADS / 32) * kRedW;
    }
    double* acc = reinterpret_cast<double*>(sp);
    for (int i = tid; i < S::SLOTS_PER_CTA * a.slot_stride; i += S::THREADS) acc[i] = 0.0;
    __syncthreads();

    const long long iters = a.count > base_slot ? (a.count - base_slot + n_slots - 1) / n_slots : 0;
    unsigned bad = 0;

    for (long long it = 0; it < iters; ++it) {
        const long long idx = slot + it * n_slots;
        const bool active = idx < a.count;
        const long long sid = a.first + (active ? idx : 0);
        uint32_t c2 = static_cast<uint32_t>(sid);
        const uint32_t c3 = a.tag | ((static_cast<uint32_t>(static_cast<unsigned long long>(sid) >> 32) & 0xffffu) << 16);

        int32_t q[FR][FC];
#pragma unroll
        for (int r = 0; r < FR; ++r) load_row<FC>(q[r], a.q0f + (size_t)(row0 + r) * NF + col0);
        int32_t qc[R][C];
        f32x2 zt[S::NZ][2];                 // coupled normal sums, two coarse cells each
        if constexpr (CPL) {
#pragma unroll
            for (int i = 0; i < R; ++i) load_row<C>(qc[i], a.q0c + (size_t)(crow0 + i) * NC + ccol0);
#pragma unroll
            for (int z = 0; z < S::NZ; ++z) zt[z][0] = zt[z][1] = 0ull;
        }

        // Philox words of the two cell pairs drawn next
        uint4 w0 = make_uint4(pair_index<S>(row0, col0, 0), 0u, c2, c3);
        uint4 w1 = make_uint4(pair_index<S>(row0 + S::DR, col0, S::DPC), 0u, c2, c3);
        philox_rounds<0, 10>(w0, w1, a.key0, a.key1);

        for (int m = 0; m < a.M; ++m) {
            // fluctuation state: the noise-free path rho-bar^m of this lane's cells
            float rb[S::FLUCT ? FR : 1][S::FLUCT ? FC : 1];
            if constexpr (S::FLUCT) {
#pragma unroll
                for (int r = 0; r < FR; ++r)
                    load_row_f<FC>(rb[r], a.rbf + (size_t)m * NF * NF + (size_t)(row0 + r) * NF + col0);
            }
            if constexpr (S::REDRAW) asm volatile("" : "+r"(c2));
            // ---- rows of the block in order: noise, transfers, and the row's part of the update
            const bool cstep = CPL && ((m & 3) == 3);
            const int par = m & 1;
            // the coarse path's noise-free row.  A sample in one warp loads it here, ahead of
            // the noise: few samples wait for every load (8^2 x 640 steps, 256 samples: 291 us
            // with scalar noise, whose loads the compiler moved up; packed 325 where it is
            // used, 300 here; 20000 samples 2554, 2331, 2298).  The larger shapes need the
            // registers: 64^2 x 256, 152 samples 435 there, 480 here.
            constexpr bool kEarly = S::FLUCT && CPL && S::WARP;
            float rbc[S::FLUCT && CPL ? R : 1][S::FLUCT && CPL ? C : 1];
            if constexpr (kEarly) {
                if (cstep) {
#pragma unroll
                    for (int i = 0; i < R; ++i)
                        load_row_f<C>(rbc[i], a.rbc + (size_t)(m >> 2) * NC * NC + (size_t)(crow0 + i) * NC + ccol0);
                }
            }
            const f32x2 gf2 = pack2(a.gf, a.gf);
            int32_t G1[FR][FC], G2[FR][FC];
            int32_t pend[2][FC];      // change of the row in hand still to be added (parity of the row)
            int32_t pend0[FC];        // the same for the first row, which waits for the row above it
#pragma unroll
            for (int r = 0; r < FR; ++r) {
                if (S::DR == 0 || !(r & S::DR)) {   // with DR, row r + DR's noise is drawn with row r's
#pragma unroll
                    for (int pa = 0; pa < C; pa += 1 + S::DPC) {
                        const int r2 = r + S::DR, p2 = pa + S::DPC;
                        const auto draw = [&](int row, int pair, int step) {
                            w0 = make_uint4(pair_index<S>(row0 + row, col0, pair), static_cast<uint32_t>(step), c2, c3);
                            w1 = make_uint4(pair_index<S>(row0 + row + S::DR, col0, pair + S::DPC),
                                            static_cast<uint32_t>(step), c2, c3);
                        };
                        if constexpr (!S::PIPE) {
                            draw(r, pa, m);
                            philox_rounds<0, 10>(w0, w1, a.key0, a.key1);
                        }
                        const uint4 x0 = w0, x1 = w1;
                        if constexpr (S::PIPE) {
                            // the two pairs after these (the next step's first after the last)
                            const bool row_end = pa + 1 + S::DPC >= C;
                            int nr = row_end ? r + 1 : r;
                            if (S::DR && (nr & S::DR)) nr += S::DR;
                            const bool last = nr >= FR;
                            draw(last ? 0 : nr, row_end ? 0 : pa + 1 + S::DPC, last ? m + 1 : m);
                        }
                        philox_rounds<0, 3, S::PIPE>(w0, w1, a.key0, a.key1);
                        const f32x2 la = bm_lnu2(x0.x, x1.x), lb = bm_lnu2(x0.z, x1.z);
                        philox_rounds<3, 4, S::PIPE>(w0, w1, a.key0, a.key1);
                        const f32x2 ha = bm_angle2(x0.y, x1.y), hb = bm_angle2(x0.w, x1.w);
                        const f32x2 ca = pack2(cos_normal(lo2(ha)), cos_normal(hi2(ha)));
                        const f32x2 cb = pack2(cos_normal(lo2(hb)), cos_normal(hi2(hb)));
                        philox_rounds<4, 5, S::PIPE>(w0, w1, a.key0, a.key1);
                        const f32x2 ra = pack2(sqrt_approx(lo2(la)), sqrt_approx(hi2(la)));
                        const f32x2 rbb = pack2(sqrt_approx(lo2(lb)), sqrt_approx(hi2(lb)));
                        philox_rounds<5, 6, S::PIPE>(w0, w1, a.key0, a.key1);
                        const f32x2 sa = pack2(sin_normal(lo2(ha)), sin_normal(hi2(ha)));
                        const f32x2 sb = pack2(sin_normal(lo2(hb)), sin_normal(hi2(hb)));
                        philox_rounds<6, 7, S::PIPE>(w0, w1, a.key0, a.key1);
                        f32x2 ta, tb;
                        if constexpr (S::FLUCT) {
                            ta = noise_amp_fluct2(q[r][2 * pa], q[r2][2 * p2], rb[r][2 * pa], rb[r2][2 * p2], a.isf, gf2);
                            tb = noise_amp_fluct2(q[r][2 * pa + 1], q[r2][2 * p2 + 1], rb[r][2 * pa + 1],
                                                  rb[r2][2 * p2 + 1], a.isf, gf2);
                        } else {
                            ta = noise_amp2(q[r][2 * pa], q[r2][2 * p2], gf2);
                            tb = noise_amp2(q[r][2 * pa + 1], q[r2][2 * p2 + 1], gf2);
                        }
                        ta = mul2(ta, ra);
                        tb = mul2(tb, rbb);
                        philox_rounds<7, 8, S::PIPE>(w0, w1, a.key0, a.key1);
                        const f32x2 a1 = mul2(ta, ca), a2 = mul2(ta, sa), b1 = mul2(tb, cb), b2 = mul2(tb, sb);
                        G1[r][2 * pa] = __float2int_rn(lo2(a1));
                        G2[r][2 * pa] = __float2int_rn(lo2(a2));
                        G1[r2][2 * p2] = __float2int_rn(hi2(a1));
                        G2[r2][2 * p2] = __float2int_rn(hi2(a2));
                        philox_rounds<8, 9, S::PIPE>(w0, w1, a.key0, a.key1);
                        G1[r][2 * pa + 1] = __float2int_rn(lo2(b1));
                        G2[r][2 * pa + 1] = __float2int_rn(lo2(b2));
                        G1[r2][2 * p2 + 1] = __float2int_rn(hi2(b1));
                        G2[r2][2 * p2 + 1] = __float2int_rn(hi2(b2));
                        if constexpr (CPL) {
                            if constexpr (S::ZPACK) {
                                const int z = S::DPC ? ((r >> 1) * C + pa) / 2 : 0;
                                zt[z][0] = fma2(rbb, cb, fma2(ra, ca, zt[z][0]));
                                zt[z][1] = fma2(rbb, sb, fma2(ra, sa, zt[z][1]));
                            } else {
                                // one coarse cell: the sum runs over row 0, then row 1
                                float z1 = lo2(zt[0][0]), z2 = lo2(zt[0][1]);
                                z1 = fmaf(lo2(rbb), lo2(cb), fmaf(lo2(ra), lo2(ca), z1));
                                z2 = fmaf(lo2(rbb), lo2(sb), fmaf(lo2(ra), lo2(sa), z2));
                                z1 = fmaf(hi2(rbb), hi2(cb), fmaf(hi2(ra), hi2(ca), z1));
                                z2 = fmaf(hi2(rbb), hi2(sb), fmaf(hi2(ra), hi2(sa), z2));
                                zt[0][0] = pack2(z1, 0.f);
                                zt[0][1] = pack2(z2, 0.f);
                            }
                        }
                        philox_rounds<9, 10, S::PIPE>(w0, w1, a.key0, a.key1);
                    }
                }
                if constexpr (!S::WARP) {
                    if (r == 0) put_edge<FC, LPB>(fx + ((par * 2 + 0) * BPC + bl) * NF, lib, q[0], G1[0]);
                    if (r == FR - 1) put_edge<FC, LPB>(fx + ((par * 2 + 1) * BPC + bl) * NF, lib, q[FR - 1], G1[FR - 1]);
                }
                if constexpr (S::PIPE) row_update<S>(r, q, G1, G2, pend, pend0, left, right, a.Af);
            }
            int32_t Gc1[R][C], Gc2[R][C];
            if constexpr (CPL) {
                if (cstep) {
                    if constexpr (S::FLUCT && !kEarly) {
#pragma unroll
                        for (int i = 0; i < R; ++i)
                            load_row_f<C>(rbc[i], a.rbc + (size_t)(m >> 2) * NC * NC + (size_t)(crow0 + i) * NC + ccol0);
                    }
#pragma unroll
                    for (int i = 0; i < R; ++i)
#pragma unroll
                        for (int j = 0; j < C; ++j) {
                            float s;
                            if constexpr (S::FLUCT) s = noise_amp_fluct(qc[i][j], rbc[i][j], a.isc, a.gc);
                            else s = noise_amp(qc[i][j], a.gc);
                            const int z = (i * C + j) / 2;
                            const bool hi = (i * C + j) & 1;
                            Gc1[i][j] = __float2int_rn(s * (hi ? hi2(zt[z][0]) : lo2(zt[z][0])));
                            Gc2[i][j] = __float2int_rn(s * (hi ? hi2(zt[z][1]) : lo2(zt[z][1])));
                        }
#pragma unroll
                    for (int z = 0; z < S::NZ; ++z) zt[z][0] = zt[z][1] = 0ull;
                    if constexpr (!S::WARP) {
                        put_edge<C, LPB>(cx + bl * NC, lib, qc[0], Gc1[0]);
                        put_edge<C, LPB>(cx + (BPC + bl) * NC, lib, qc[R - 1], Gc1[R - 1]);
                    }
                }
            }
            if constexpr (SPLIT) cluster_arrive();
            else if constexpr (!S::WARP) __syncthreads();

            // ---- horizontal halo by shuffles within the band segment
            int32_t qL[FR], gL[FR], qR[FR], gR[FR];
            if constexpr (!S::PIPE) {
#pragma unroll
                for (int r = 0; r < FR; ++r) {
                    qL[r] = __shfl_sync(kFull, q[r][FC - 1], left, LPB);
                    gL[r] = __shfl_sync(kFull, G2[r][FC - 1], left, LPB);
                    qR[r] = __shfl_sync(kFull, q[r][0], right, LPB);
                    gR[r] = __shfl_sync(kFull, G2[r][0], right, LPB);
                }
            }
            int32_t cqL[R], cgL[R], cqR[R], cgR[R];
            if constexpr (CPL) {
                if (cstep) {
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        cqL[i] = __shfl_sync(kFull, qc[i][C - 1], left, LPB);
                        cgL[i] = __shfl_sync(kFull, Gc2[i][C - 1], left, LPB);
                        cqR[i] = __shfl_sync(kFull, qc[i][0], right, LPB);
                        cgR[i] = __shfl_sync(kFull, Gc2[i][0], right, LPB);
                    }
                }
            }

            // ---- vertical halo
            int32_t qU[FC], gU[FC], qD[FC], gD[FC];
            [[maybe_unused]] int32_t keep1[FC], keep2[FC];
            int32_t cqU[C], cgU[C], cqD[C], cgD[C];
            if constexpr (S::WARP) {
#pragma unroll
                for (int c = 0; c < FC; ++c) {
                    qU[c] = __shfl_sync(kFull, q[FR - 1][c], up_lane, LPS);
                    gU[c] = __shfl_sync(kFull, G1[FR - 1][c], up_lane, LPS);
                    qD[c] = __shfl_sync(kFull, q[0][c], dn_lane, LPS);
                    gD[c] = __shfl_sync(kFull, G1[0][c], dn_lane, LPS);
                }
                if constexpr (CPL) {
                    if (cstep) {
#pragma unroll
                        for (int j = 0; j < C; ++j) {
                            cqU[j] = __shfl_sync(kFull, qc[R - 1][j], up_lane, LPS);
                            cgU[j] = __shfl_sync(kFull, Gc1[R - 1][j], up_lane, LPS);
                            cqD[j] = __shfl_sync(kFull, qc[0][j], dn_lane, LPS);
                            cgD[j] = __shfl_sync(kFull, Gc1[0][j], dn_lane, LPS);
                        }
                    }
                }
            } else {
                int2* const ftop = fx + ((par * 2 + 0) * BPC) * NF;
                int2* const fbot = fx + ((par * 2 + 1) * BPC) * NF;
                int2* const ctop = cx;
                int2* const cbot = cx + BPC * NC;
                if constexpr (SPLIT) {
                    if constexpr (!S::PIPE) flux_update_interior<FR, FC>(q, G1, G2, qL, gL, qR, gR, a.Af, keep1, keep2);
                    cluster_wait();
                }
                const int2* above = (bl > 0) ? fbot + (bl - 1) * NF
                                             : peer<S>(fbot + (BPC - 1) * NF, (rank + CL - 1) % CL);
                const int2* below = (bl + 1 < BPC) ? ftop + (bl + 1) * NF : peer<S>(ftop, (rank + 1) % CL);
                get_edge<FC, LPB>(above, lib, qU, gU);
                get_edge<FC, LPB>(below, lib, qD, gD);
                if constexpr (CPL) {
                    if (cstep) {
                        const int2* cab = (bl > 0) ? cbot + (bl - 1) * NC
                                                   : peer<S>(cbot + (BPC - 1) * NC, (rank + CL - 1) % CL);
                        const int2* cbe = (bl + 1 < BPC) ? ctop + (bl + 1) * NC : peer<S>(ctop, (rank + 1) % CL);
                        get_edge<C, LPB>(cab, lib, cqU, cgU);
                        get_edge<C, LPB>(cbe, lib, cqD, cgD);
                    }
                }
            }

            // ---- first and last row, coarse step
            if constexpr (S::PIPE) {
#pragma unroll
                for (int c = 0; c < FC; ++c) {
                    const int32_t v0 = edge_flux(a.Af, q[0][c] - qU[c]);
                    const int32_t v1 = edge_flux(a.Af, qD[c] - q[FR - 1][c]);
                    q[0][c] += pend0[c] - v0 - gU[c];
                    q[FR - 1][c] += pend[(FR - 1) & 1][c] + v1 + gD[c];
                }
            } else if constexpr (SPLIT) {
                flux_update_boundary<FR, FC>(q, G1, G2, qU, gU, qD, gD, qL, gL, qR, gR, a.Af, keep1, keep2);
            } else {
                flux_update<FR, FC>(q, G1, G2, qU, gU, qD, gD, qL, gL, qR, gR, a.Af);
            }
            if constexpr (CPL) {
                if (cstep) {
                    flux_update<R, C>(qc, Gc1, Gc2, cqU, cgU, cqD, cgD, cqL, cgL, cqR, cgR, a.Ac);
#pragma unroll
                    for (int i = 0; i < R; ++i)
#pragma unroll
                        for (int j = 0; j < C; ++j) bad |= (static_cast<uint32_t>(qc[i][j]) + 0x40000000u) >> 31;
                }
            }
            if ((m & 3) == 3 || m + 1 == a.M) {
#pragma unroll
                for (int r = 0; r < FR; ++r)
#pragma unroll
                    for (int c = 0; c < FC; ++c) bad |= (static_cast<uint32_t>(q[r][c]) + 0x40000000u) >> 31;
            }
        }

        // ---- observables: fluctuation sums against the fixed-point mean field, mass
        double v[kRedW];
        {
            long long mf = 0;
#pragma unroll
            for (int r = 0; r < FR; ++r)
#pragma unroll
                for (int c = 0; c < FC; ++c) mf += q[r][c];
            v[2 * kMaxObs] = static_cast<double>(mf);
            long long mc = 0;
            if constexpr (CPL) {
#pragma unroll
                for (int i = 0; i < R; ++i)
#pragma unroll
                    for (int j = 0; j < C; ++j) mc += qc[i][j];
            }
            v[2 * kMaxObs + 1] = static_cast<double>(mc);
#pragma unroll
            for (int k = 0; k < kMaxObs; ++k) {
                float sf = 0.f, sc = 0.f;
                if (k < a.n_obs) {
                    if constexpr (!CPL && CL == 1 && !S::WARP && FR * FC >= 16) {
                        // (in place: within the lambda below, the registers of these shapes' step
                        // loop are allocated worse: 32^2, 1000 x 103 steps 288 us so, 281 in place;
                        // 64^2, 1151 x 208 2397 and 2345.  Coupled, cluster and small blocks are
                        // the other way round, 64^2 coupled fluctuation state 434 and 480.)
#pragma unroll
                        for (int r = 0; r < FR; ++r) {
                            int32_t qb[FC];
                            float ph[FC];
                            load_row<FC>(qb, a.qbf + (size_t)(row0 + r) * NF + col0);
                            load_row_f<FC>(ph, a.phif + (size_t)k * NF * NF + (size_t)(row0 + r) * NF + col0);
#pragma unroll
                            for (int c = 0; c < FC; ++c) sf = fmaf(__int2float_rn(q[r][c] - qb[c]), ph[c], sf);
                        }
                    } else {
                        const auto project = [&]() {
#pragma unroll
                            for (int r = 0; r < FR; ++r) {
                                int32_t qb[FC];
                                float ph[FC];
                                load_row<FC>(qb, a.qbf + (size_t)(row0 + r) * NF + col0);
                                load_row_f<FC>(ph, a.phif + (size_t)k * NF * NF + (size_t)(row0 + r) * NF + col0);
#pragma unroll
                                for (int c = 0; c < FC; ++c) sf = fmaf(__int2float_rn(q[r][c] - qb[c]), ph[c], sf);
                            }
                            if constexpr (CPL) {
#pragma unroll
                                for (int i = 0; i < R; ++i) {
                                    int32_t qb[C];
                                    float ph[C];
                                    load_row<C>(qb, a.qbc + (size_t)(crow0 + i) * NC + ccol0);
                                    load_row_f<C>(ph, a.phic + (size_t)k * NC * NC + (size_t)(crow0 + i) * NC + ccol0);
#pragma unroll
                                    for (int j = 0; j < C; ++j) sc = fmaf(__int2float_rn(qc[i][j] - qb[j]), ph[j], sc);
                                }
                            }
                        };
                        project();
                        if constexpr (S::CHAIN == 2) {
                            // odd bands continue the sum of the band above, in the same warp
                            const float uf = __shfl_up_sync(kFull, sf, LPB), uc = __shfl_up_sync(kFull, sc, LPB);
                            sf = sc = 0.f;
                            if (band & 1) {
                                sf = uf;
                                sc = uc;
                                project();
                            }
                        }
                    }
                }
                v[k] = static_cast<double>(sf);
                v[kMaxObs + k] = static_cast<double>(sc);
            }
        }
        bool leader;
        if constexpr (S::WARP) {
#pragma unroll
            for (int off = LPS / 2; off >= 1; off >>= 1)
#pragma unroll
                for (int i = 0; i < kRedW; ++i) v[i] += __shfl_xor_sync(kFull, v[i], off, LPS);
            leader = (lane % LPS) == 0;
        } else {
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1)
#pragma unroll
                for (int i = 0; i < kRedW; ++i) v[i] += __shfl_xor_sync(kFull, v[i], off);
            if (lane == 0)
#pragma unroll
                for (int i = 0; i < kRedW; ++i) red[(tid >> 5) * kRedW + i] = v[i];
            __syncthreads();
            if (tid == 0) {
                for (int w = 1; w < S::THREADS / 32; ++w)
#pragma unroll
                    for (int i = 0; i < kRedW; ++i) v[i] += red[w * kRedW + i];
#pragma unroll
                for (int i = 0; i < kRedW; ++i) red[i] = v[i];
            }
            if constexpr (CL > 1) {
                cg::this_cluster().sync();
                if (rank == 0 && tid == 0) {
                    for (int rr = 1; rr < CL; ++rr) {
                        const double* o = peer<S>(red, rr);
#pragma unroll
                        for (int i = 0; i < kRedW; ++i) v[i] += o[i];
                    }
                }
            }
            leader = (tid == 0) && (rank == 0);
        }

        // ---- FP64 quantities and moment sums (one lane per sample)
        if (leader && active) {
            double Df[kMaxObs], Dc[kMaxObs];
#pragma unroll
            for (int k = 0; k < kMaxObs; ++k) {
                Df[k] = a.dscale_f * v[k] + a.delta_f[k];
                Dc[k] = CPL ? a.dscale_c * v[kMaxObs + k] + a.delta_c[k] : 0.0;
            }
            double* A = acc + slot_local * a.slot_stride;
            A[0] += 1.0;
            double merr = fabs(v[2 * kMaxObs] - static_cast<double>(a.mass0_f)) * a.dscale_f;
            if (CPL) merr = fmax(merr, fabs(v[2 * kMaxObs + 1] - static_cast<double>(a.mass0_c)) * a.dscale_c);
            A[1] = fmax(A[1], merr);
            int qi = 0;
            for (int j = 0; j < a.n_obs; ++j) {
                const int kend = a.products ? a.n_obs : j + 1;
                for (int k = j; k < kend; ++k, ++qi) {
                    const double pf = a.N * Df[j] * Df[k];
                    const double pc = CPL ? a.N * Dc[j] * Dc[k] : 0.0;
                    const double dp = pf - pc, dp2 = dp * dp;
                    double* B = A + 2 + kNSum * qi;
                    B[0] += dp; B[1] += dp2; B[2] += dp2 * dp; B[3] += dp2 * dp2;
                    B[4] += pf; B[5] += pf * pf; B[6] += pc; B[7] += pc * pc;
                    B[8] += Df[j]; B[9] += Df[j] * Df[j]; B[10] += Dc[j]; B[11] += Dc[j] * Dc[j];
                }
            }
            if (a.samples) {
                double* o = a.samples + idx * (2 * a.n_obs + 2);
                for (int k = 0; k < a.n_obs; ++k) {
                    o[k] = Df[k];
                    o[a.n_obs + k] = Dc[k];
                }
                o[2 * a.n_obs] = v[2 * kMaxObs] * a.dscale_f + a.mass_off_f;
                o[2 * a.n_obs + 1] = CPL ? v[2 * kMaxObs + 1] * a.dscale_c + a.mass_off_c : 0.0;
            }
        }
    }
    if (bad) atomicOr(a.err, kErrRange);

    // ---- per-slot partial sums to global scratch, entry-major [stride][n_slots]
    __syncthreads();
    if (S::WARP || rank == 0) {
        const long long slot0 = S::WARP ? (long long)blockIdx.x * S::SLOTS_PER_CTA : slot;
        for (int i = tid; i < S::SLOTS_PER_CTA * a.slot_stride; i += S::THREADS) {
            const int s = i / a.slot_stride, e = i % a.slot_stride;
            a.partials[(size_t)e * n_slots + slot0 + s] = acc[i];
        }
    }
    if constexpr (CL > 1) cg::this_cluster().sync();   // peers may still read our shared memory
}

// ------------------------------------------------------------------ dispatch
template <class S>
struct Kern {
    static size_t smem_bytes(int stride) { return S::fixed_smem() + sizeof(double) * S::SLOTS_PER_CTA * stride; }

    static cudaError_t prepare() {
        auto fn = level_kernel<S>;
        const size_t smax = smem_bytes(kMaxStride);
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smax);
        if (e != cudaSuccess || S::CL == 1) return e;
        return cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    }

    static cudaError_t info(int stride, VariantInfo* vi) {
        auto fn = level_kernel<S>;
        cudaError_t e = prepare();
        if (e != cudaSuccess) return e;
        int dev = 0, sms = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        vi->supported = 1;
        vi->threads = S::THREADS;
        vi->cluster = S::CL;
        vi->slots_per_cta = S::SLOTS_PER_CTA;
        vi->smem = smem_bytes(stride);
        if (S::CL == 1) {
            int nb = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, S::THREADS, vi->smem);
            if (e != cudaSuccess) return e;
            vi->max_ctas = nb * sms;
        } else {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(S::CL * sms);
            cfg.blockDim = dim3(S::THREADS);
            cfg.dynamicSmemBytes = vi->smem;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = S::CL;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int ncl = 0;
            e = cudaOccupancyMaxActiveClusters(&ncl, fn, &cfg);
            if (e != cudaSuccess) return e;
            vi->max_ctas = ncl * S::CL;
        }
        return vi->max_ctas > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
    }

    static cudaError_t launch(const KArgs& a, int n_ctas, cudaStream_t st, int priority) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(n_ctas);
        cfg.blockDim = dim3(S::THREADS);
        cfg.dynamicSmemBytes = smem_bytes(a.slot_stride);
        cfg.stream = st;
        cudaLaunchAttribute at[2];
        int na = 0;
        if (S::CL > 1) {
            at[na].id = cudaLaunchAttributeClusterDimension;
            at[na].val.clusterDim.x = S::CL;
            at[na].val.clusterDim.y = 1;
            at[na].val.clusterDim.z = 1;
            ++na;
        }
        if (priority != 0) {
            at[na].id = cudaLaunchAttributePriority;
            at[na].val.priority = priority;
            ++na;
        }
        cfg.attrs = na ? at : nullptr;
        cfg.numAttrs = na;
        return cudaLaunchKernelEx(&cfg, level_kernel<S>, a);
    }
};

// Kernel variants: fine size n, lane block C x R coarse cells (2R x 2C fine),
// cluster size.  Every entry keeps the whole state in registers; the first
// entry for each n is the default, the others are candidates for the tuner.
#define DK_VARIANTS(X) \
    X(4, 1, 1, 1)      \
    X(8, 1, 1, 1)      \
    X(16, 1, 2, 1)     \
    X(16, 2, 2, 1)     \
    X(16, 1, 1, 1)     \
    X(32, 2, 2, 1)     \
    X(32, 1, 2, 1)     \
    X(32, 2, 1, 1)     \
    X(64, 2, 2, 1)     \
    X(64, 4, 2, 1)     \
    X(64, 2, 1, 1)     \
    X(64, 4, 1, 1)     \
    X(128, 2, 2, 2)    \
    X(128, 4, 1, 2)    \
    X(128, 2, 1, 4)    \
    X(256, 4, 2, 8)    \
    X(256, 4, 1, 8)

struct VariantEntry {
    int n, C, R, CL;
    cudaError_t (*info)(bool coupled, int stride, VariantInfo* vi);
    cudaError_t (*launch)(bool coupled, const VariantInfo& vi, const KArgs& a, int* n_ctas, cudaStream_t st, int priority);
};
// The fluctuation-state builds' table.
const VariantEntry* fluct_variants(int* count);

namespace {
// Few samples: the same level on twice the lanes, half the rows each.  Below about
// a warp per scheduler the time of a batch is that of one sample's chain of steps,
// and half the cells per lane shorten it; the sums keep the full shape's order
// (CHAIN).  Measured, us, full shape / twice the lanes: 16^2 x 52 steps, 256 samples
// 43.6 / 25.1, 912 57.8 / 44.1, 1216 56.9 / 65.4; 32^2 x 208 coupled, 152 samples 193 /
// 122, 456 297 / 248, 608 300 / 391; 32^2 plain, 456 282 / 231, 608 283 / 362.  At
// 64^2 the full shape fills an SM's schedulers with one sample and wins (152: 312 / 347).
//
// Two builds of a shape, of which the first holds more samples at once and the
// second has more registers: which is the faster one depends on how full the
// passes over the resident samples are.  Measured, us, first / second build (in
// brackets before the packed noise, with no bound on the registers):
//   fluctuation state, 64^2 x 256 coupled, resident 304 / 152: 152 samples 548 / 436
//     (455), 400 1285 / 1288 (1347), 456 1717 / 1290 (1348), 712 2040 / 2140 (2240), 760
//     2565 / 2145 (2243); plain, 152 samples 461 / 430 (488), 304 794 / 851 (818)
//   fluctuation state, 32^2 x 64 coupled, resident 1216 / 608: 608 samples 139 / 115
//     (115), 912 173 / 215 (217), 1672 318 / 322 (323), 1824 367 / 323 (323), 4256 749 /
//     741 (740); plain, 1216 / 912: 608 113 / 100 (119), 1216 196 / 222 (255), 1824 328 /
//     269 (302), 2432 380 / 396 (445), 20000 3048 / 2846 (3208)
//   fluctuation state, 8^2 x 64 coupled, 6080 / 4864: 2000 samples 55 / 50 (51), 5000
//     87 / 90 (92), 100000 1185 / 1182 (1318)
//   16^2 x 52 on two warps, 1824 / 912: 256 samples 28.8 / 24.7 (28.8), 1200 57 / 65
//     (57), 1824 76 / 76 (78), 5000 202 / 185 (189), 20000 712 / 712 (712)
//   32^2 x 103 on four warps, coupled, 608 / 456: 456 samples 138 / 131 (144), 608 176 /
//     206 (182), 912 290 / 249 (302), 4630 1261 / 1229 (1300)
template <int NF, int C, int R, int CL, bool FL>
struct Split {
    static constexpr bool HALVE = CL == 1 && ((NF == 16 && C == 1 && R == 2) || (NF == 32 && C == 2 && R == 2));
    static constexpr long long HALF_MAX = !HALVE ? 0 : FL ? (NF == 16 ? 456 : 304) : (NF == 16 ? 912 : 456);
    template <bool CPL>
    using half = Shape<NF, C, HALVE ? R / 2 : R, CL, CPL, FL, HALVE ? 2 : 1, true>;
    template <bool CPL>
    using first = Shape<NF, C, R, CL, CPL, FL>;
    template <bool CPL>
    using second = Shape<NF, C, R, CL, CPL, FL, 1, true>;
    static constexpr bool TWO = FL ? NF == 8 || NF == 32 || NF == 64
                                   : CL == 1 && ((NF == 16 && C == 1 && R == 1) || (NF == 32 && C * R == 2));
    // Whether `count` samples run on the second build: `most` and `few` are the
    // samples that the first and the second build hold at once, `rest` the samples of
    // the first build's last pass (one that is at most three quarters of `few` runs
    // alone on its SMs at once, a fuller one two samples to an SM).
    static bool use_second(bool coupled, long long count, long long most, long long few) {
        const long long rest = (count - 1) % most + 1;
        if constexpr (!FL) return count <= few || count > (NF == 32 ? most : 2 * most);
        if constexpr (NF == 8) return count <= few;
        if (!coupled) return NF == 64 ? count <= few : rest <= few || count > 2 * most;
        return count <= few || (rest <= few && 4 * rest > 3 * few && (NF == 64 || count <= 4 * most));
    }
};

template <int NF, int C, int R, int CL, bool FL>
cudaError_t variant_info_fn(bool coupled, int stride, VariantInfo* vi) {
    using SP = Split<NF, C, R, CL, FL>;
    cudaError_t e = cudaSuccess;
    if constexpr (SP::HALVE) {
        // its slots are those of the first build; only the launch attribute (and its code loaded)
        e = coupled ? Kern<typename SP::template half<true>>::prepare() : Kern<typename SP::template half<false>>::prepare();
        if (e != cudaSuccess) return e;
    }
    VariantInfo second{};
    if constexpr (SP::TWO) {
        e = coupled ? Kern<typename SP::template second<true>>::info(stride, &second)
                    : Kern<typename SP::template second<false>>::info(stride, &second);
        if (e != cudaSuccess) return e;
    }
    e = coupled ? Kern<typename SP::template first<true>>::info(stride, vi)
                : Kern<typename SP::template first<false>>::info(stride, vi);
    vi->second_ctas = second.max_ctas;
    return e;
}

template <int NF, int C, int R, int CL, bool FL>
cudaError_t variant_launch_fn(bool coupled, const VariantInfo& vi, const KArgs& a, int* n_ctas, cudaStream_t st,
                              int priority) {
    using SP = Split<NF, C, R, CL, FL>;
    if constexpr (SP::HALVE) {
        // one CTA per sample slot, the same slots
        if (a.count <= SP::HALF_MAX) {
            const int n_slots = *n_ctas * SP::template first<true>::SLOTS_PER_CTA;
            return coupled ? Kern<typename SP::template half<true>>::launch(a, n_slots, st, priority)
                           : Kern<typename SP::template half<false>>::launch(a, n_slots, st, priority);
        }
    }
    if constexpr (SP::TWO) {
        static_assert(CL == 1, "CTAs hold whole samples");
        constexpr int slots = SP::template first<true>::SLOTS_PER_CTA;
        if (SP::use_second(coupled, a.count, (long long)vi.max_ctas * slots, (long long)vi.second_ctas * slots)) {
            *n_ctas = std::min(*n_ctas, vi.second_ctas);
            return coupled ? Kern<typename SP::template second<true>>::launch(a, *n_ctas, st, priority)
                           : Kern<typename SP::template second<false>>::launch(a, *n_ctas, st, priority);
        }
    }
    return coupled ? Kern<typename SP::template first<true>>::launch(a, *n_ctas, st, priority)
                   : Kern<typename SP::template first<false>>::launch(a, *n_ctas, st, priority);
}

#ifdef DK_FLUCT_BUILD
// Fluctuation-state builds: one lane-block shape per grid size up to 128^2
// (the grids of the high-particle-number hierarchies that need them).
#define DK_FLUCT_VARIANTS(X) \
    X(4, 1, 1, 1)            \
    X(8, 1, 1, 1)            \
    X(16, 1, 2, 1)           \
    X(32, 2, 2, 1)           \
    X(64, 2, 2, 1)           \
    X(128, 2, 2, 2)
#define DK_ENTRY(NF, C, R, CL) \
    {NF, C, R, CL, variant_info_fn<NF, C, R, CL, true>, variant_launch_fn<NF, C, R, CL, true>},
const VariantEntry kFluctVariants[] = {DK_FLUCT_VARIANTS(DK_ENTRY)};
#undef DK_ENTRY
}  // namespace

const VariantEntry* fluct_variants(int* count) {
    *count = (int)(sizeof(kFluctVariants) / sizeof(kFluctVariants[0]));
    return kFluctVariants;
}
#else
#define DK_ENTRY(NF, C, R, CL) \
    {NF, C, R, CL, variant_info_fn<NF, C, R, CL, false>, variant_launch_fn<NF, C, R, CL, false>},
const VariantEntry kVariants[] = {DK_VARIANTS(DK_ENTRY)};
#undef DK_ENTRY

const VariantEntry* find_variant(int n, int idx, bool fluct) {
    int count = (int)(sizeof(kVariants) / sizeof(kVariants[0])), k = 0;
    const VariantEntry* tab = fluct ? fluct_variants(&count) : kVariants;
    for (int i = 0; i < count; ++i)
        if (tab[i].n == n && k++ == idx) return &tab[i];
    return nullptr;
}
}  // namespace

int variant_count(int n, bool fluct) {
    int k = 0;
    while (find_variant(n, k, fluct)) ++k;
    return k;
}

cudaError_t variant_info(int n, bool coupled, int stride, int idx, VariantInfo* out, bool fluct) {
    *out = VariantInfo{};
    const VariantEntry* v = find_variant(n, idx, fluct);
    if (!v) return cudaSuccess;   // supported = 0
    cudaError_t e = v->info(coupled, stride, out);
    out->C = v->C;
    out->R = v->R;
    return e;
}

cudaError_t launch_level(int n, bool coupled, int idx, const VariantInfo& vi, const KArgs& a, int* n_ctas,
                         cudaStream_t st, int priority, bool fluct) {
    const VariantEntry* v = find_variant(n, idx, fluct);
    if (!v) return cudaErrorInvalidValue;
    return v->launch(coupled, vi, a, n_ctas, st, priority);
}
#endif  // DK_FLUCT_BUILD

}  // namespace dk
