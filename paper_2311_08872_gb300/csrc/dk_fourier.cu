// Fourier-coupled sample kernel for sm_103a (Section 3.1): the fine path of
// Eq. (FullyDiscreteDK) (b0 = 0, b1 = 1) on an n x n grid and, for a coupled
// level, the coarse path on the (n/3) x (n/3) grid with step 9 tau, whose
// noise carries every Fourier mode of the fine noise that the coarse grid
// resolves.
//
// Noise.  The fine Brownian increments are the cell normals of the explicit
// kernels (same Philox counters); their unitary discrete Fourier coefficients
// are exactly the independent complex-conjugate Fourier Brownian increments
// of Section 3.1.  The coarse increment of one coarse step is the restriction
// P1 S P1^T of the sum S of the 9 fine normal fields inside it, P1 (n/3 x n,
// host-built) keeping the modes -n/6..n/6 per axis, the two fine aliases of
// the coarse Nyquist mode weighted 2^-1/2 each; P1 has orthonormal rows, so
// the coarse normal field (P1 S P1^T / 3) is white with unit variance and the
// coarse path has the law of a stand-alone coarse path (Remark
// distribution_W_ell).  The restriction is linear, so the 9 fine fields are
// summed first (FP32, per fine cell) and restricted once per coarse step: two
// small dense products per component (n x n by n x n/3, then n/3 x n by
// n x n/3), under 10% of the stencil work at n = 54.
//
// Arithmetic as in the explicit kernels: int32 fixed-point state, integer
// noise transfers G = rint(c 2^S sqrt(rho^+) Z) and diffusion fluxes, every
// edge flux computed identically by both of its cells, so the mass is exact.
// With the fluctuation state (FL) the state is q = (rho - rho-bar^m) 2^S
// about the noise-free path and the amplitudes read rho-bar^m from the
// per-step tables (fine: step m; coarse: coarse step m / 9).
//
// Work decomposition.  One CTA per sample.  A thread holds a block of 2 x 6
// fine cells (two rows of 3 Philox cell pairs; one row at 6^2), their transfers and their
// summed normals in registers; its two rows of state and G1 and the end columns
// of G2 pass through shared memory, double buffered by the step's parity, so a
// fine step has one barrier.  Every 9 steps the summed normals go to shared
// memory and are restricted by register tiles: a thread forms 2 x 2 points of
// S P1^T, both components packed, then two points of the coarse field.
//
// Bound by instruction issue and its latencies (issue slots 47% busy with 16 warps;
// fixed-latency waits, the special functions and shared memory lead).  54^2, 607
// samples x 648 steps: 4.08 ms; 5.20 with a 1 x 6 segment of cells per thread, whose
// shared-memory traffic (12 words a cell, here 5, with the summed normals there as
// well) and one-point restriction (two loads per FMA) were half of the time.
#include "dk_device.cuh"
#include "dk_kernels.h"

namespace dk {
namespace {

constexpr unsigned kFullMaskF = 0xffffffffu;
constexpr int kRedF = 2 * kMaxObs + 2;

template <int N_, int R_>
struct FShape {
    static constexpr int N = N_, NC = N / 3;
    static constexpr int R = R_, C = 6;                 // fine cells per thread
    static constexpr int BRW = N / R, BCL = N / C;      // rows / columns of blocks
    static constexpr int FT = BRW * BCL;                // threads that hold fine cells
    static constexpr int THREADS = (FT + 31) / 32 * 32;
    static_assert(N % R == 0 && N % C == 0 && NC == 2 * BCL && NC % 2 == 0, "blocks must cover the grid");
    static constexpr int MINB = 512 / THREADS;          // 16 warps of 128 registers on an SM (two samples at 54^2)
    static constexpr int WARPS = THREADS / 32;
    // words: two exchange buffers (q and G1 of every cell, the end columns of G2),
    // summed normals (2), coarse q (2 buffers), coarse G1, G2, the row-restricted
    // sums T (N x NC x 2), P1 (NC x N)
    static constexpr int XBUF = 2 * N * N + 2 * N * BCL;
    static constexpr int WORDS = 2 * XBUF + 2 * N * N + 2 * NC * NC + 2 * NC * NC + 2 * N * NC + NC * N;
    static size_t smem(int slot_stride) {
        return sizeof(int32_t) * (size_t)((WORDS + 1) / 2 * 2) + sizeof(double) * WARPS * kRedF +
               sizeof(double) * slot_stride;
    }
};

// Explicit step of an NN x NN grid in flux form for the cells of this thread:
// qn(x) = q(x) + diffusion fluxes of its four edges + G1(down) - G1(up) +
// G2(right) - G2(left), every edge flux computed from the same two states by
// both cells of the edge.
template <int NN, int THREADS>
__device__ __forceinline__ void explicit_update(const int32_t* q, const int32_t* G1, const int32_t* G2, int32_t* qn,
                                                int32_t A, unsigned& bad) {
    for (int x = threadIdx.x; x < NN * NN; x += THREADS) {
        const int i1 = x / NN, i2 = x % NN;
        const int up = ((i1 + NN - 1) % NN) * NN + i2, dn = ((i1 + 1) % NN) * NN + i2;
        const int lf = i1 * NN + (i2 + NN - 1) % NN, rt = i1 * NN + (i2 + 1) % NN;
        const int32_t c = q[x];
        const int32_t v = c + (edge_flux(A, q[dn] - c) - edge_flux(A, c - q[up])) +
                          (edge_flux(A, q[rt] - c) - edge_flux(A, c - q[lf])) + (G1[dn] - G1[up]) + (G2[rt] - G2[lf]);
        bad |= (static_cast<uint32_t>(v) + 0x40000000u) >> 31;
        qn[x] = v;
    }
}

template <int N, int ROWS, bool CPL, bool FL>
__global__ void __launch_bounds__(FShape<N, ROWS>::THREADS, FShape<N, ROWS>::MINB)
    fourier_kernel(const KArgs a, const FArgs f) {
    using S = FShape<N, ROWS>;
    constexpr int NC = S::NC, THREADS = S::THREADS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x;
    int32_t* const xbuf = reinterpret_cast<int32_t*>(smem_raw);     // exchange buffers
    f32x2* const Zs = reinterpret_cast<f32x2*>(xbuf + 2 * S::XBUF); // [N*N] summed fine normals, both components
    f32x2* const Tm = Zs + N * N;                                   // [N][NC]
    float* const P1 = reinterpret_cast<float*>(Tm + N * NC);        // [NC][N]
    int32_t* const qcA = reinterpret_cast<int32_t*>(P1 + NC * N);   // coarse state, double buffered
    int32_t* const qcB = qcA + NC * NC;
    int32_t* const Gc1 = qcB + NC * NC;
    int32_t* const Gc2 = Gc1 + NC * NC;
    double* red = reinterpret_cast<double*>(smem_raw + sizeof(int32_t) * (size_t)((S::WORDS + 1) / 2 * 2));
    double* acc = red + S::WARPS * kRedF;
    for (int i = tid; i < a.slot_stride; i += THREADS) acc[i] = 0.0;
    if constexpr (CPL)
        for (int i = tid; i < NC * N; i += THREADS) P1[i] = f.P1[i];

    constexpr int R = S::R, C = S::C, BRW = S::BRW, BCL = S::BCL;
    const bool fine_thread = tid < S::FT;
    const int br = fine_thread ? tid / BCL : 0, bc = fine_thread ? tid % BCL : 0;
    const int fx0 = br * R * N + bc * C;                             // first cell of the block
    const int xup = (br == 0 ? N - 1 : br * R - 1) * N + bc * C;     // cells of the rows above / below
    const int xdn = (br == BRW - 1 ? 0 : (br + 1) * R) * N + bc * C;
    const int lb = (bc + BCL - 1) % BCL, rb = (bc + 1) % BCL;        // blocks left / right

    unsigned bad = 0;
    const long long slot = blockIdx.x, n_slots = gridDim.x;
    const long long iters = a.count > slot ? (a.count - slot + n_slots - 1) / n_slots : 0;
    __syncthreads();

    for (long long it = 0; it < iters; ++it) {
        const long long idx = slot + it * n_slots;
        const long long sid = a.first + idx;
        const uint32_t c2 = static_cast<uint32_t>(sid);
        const uint32_t c3 = a.tag | ((static_cast<uint32_t>(static_cast<unsigned long long>(sid) >> 32) & 0xffffu) << 16);
        int ccur = 0;
        int32_t q[R][C];
        f32x2 Z[R][C];   // summed normals of the coarse step, both components
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c) {
                q[r][c] = a.q0f[fx0 + r * N + c];
                Z[r][c] = pack2(0.f, 0.f);
            }
        if constexpr (CPL)
            for (int y = tid; y < NC * NC; y += THREADS) qcA[y] = a.q0c[y];
        __syncthreads();

        for (int m = 0, m9 = 0; m < a.M; ++m) {
            int32_t* const xq = xbuf + (m & 1) * S::XBUF;   // [N*N] state
            int32_t* const xg = xq + N * N;                 // [N*N] G1
            int32_t* const xl = xg + N * N;                 // [N][BCL] G2 of the blocks' first column
            int32_t* const xr = xl + N * BCL;               // [N][BCL] ... last column
            int32_t G1[R][C], G2[R][C];
            // ---- noise of the block: Philox4x32-10 per horizontal cell pair, Box--Muller, transfers
            if (fine_thread) {
                const f32x2 g2v = pack2(a.gf, a.gf);
#pragma unroll
                for (int r = 0; r < R; ++r) {
#pragma unroll
                    for (int j = 0; j < C / 2; ++j) {
                        const int p = ((fx0 + r * N) >> 1) + j;
                        const uint4 x = philox10(make_uint4(static_cast<uint32_t>(p), static_cast<uint32_t>(m), c2, c3),
                                                 a.key0, a.key1);
                        f32x2 rad, co, si;
                        box_muller_polar2(x.x, x.y, x.z, x.w, rad, co, si);
                        f32x2 t;
                        if constexpr (FL) {
                            const float2 rbar = reinterpret_cast<const float2*>(a.rbf + (size_t)m * N * N)[p];
                            t = noise_amp_fluct2(q[r][2 * j], q[r][2 * j + 1], rbar.x, rbar.y, a.isf, g2v);
                        } else {
                            t = noise_amp2(q[r][2 * j], q[r][2 * j + 1], g2v);
                        }
                        t = mul2(t, rad);
                        const f32x2 t1 = mul2(t, co), t2 = mul2(t, si);
                        G1[r][2 * j] = __float2int_rn(lo2(t1));
                        G1[r][2 * j + 1] = __float2int_rn(hi2(t1));
                        G2[r][2 * j] = __float2int_rn(lo2(t2));
                        G2[r][2 * j + 1] = __float2int_rn(hi2(t2));
                        reinterpret_cast<int2*>(xq)[p] = make_int2(q[r][2 * j], q[r][2 * j + 1]);
                        reinterpret_cast<int2*>(xg)[p] = make_int2(G1[r][2 * j], G1[r][2 * j + 1]);
                        if constexpr (CPL) {
                            const float ra = lo2(rad), rb2 = hi2(rad);
                            Z[r][2 * j] = fma2(pack2(ra, ra), pack2(lo2(co), lo2(si)), Z[r][2 * j]);
                            Z[r][2 * j + 1] = fma2(pack2(rb2, rb2), pack2(hi2(co), hi2(si)), Z[r][2 * j + 1]);
                        }
                    }
                    xl[(br * R + r) * BCL + bc] = G2[r][0];
                    xr[(br * R + r) * BCL + bc] = G2[r][C - 1];
                }
                if constexpr (CPL) {
                    if (m9 == 8) {
#pragma unroll
                        for (int r = 0; r < R; ++r)
#pragma unroll
                            for (int c = 0; c < C; c += 2) {
                                reinterpret_cast<ulonglong2*>(Zs)[(fx0 + r * N + c) / 2] =
                                    make_ulonglong2(Z[r][c], Z[r][c + 1]);
                                Z[r][c] = Z[r][c + 1] = pack2(0.f, 0.f);
                            }
                    }
                }
            }
            __syncthreads();
            // ---- explicit step of the block in flux form (every edge flux computed
            // from the same two states by both of its cells)
            if (fine_thread) {
                int32_t qu[C], qd[C], gu[C], gd[C], ql[R], qr[R], gl[R], gr[R];
#pragma unroll
                for (int j = 0; j < C; j += 2) {
                    const int2 a0 = *reinterpret_cast<const int2*>(xq + xup + j);
                    const int2 a1 = *reinterpret_cast<const int2*>(xq + xdn + j);
                    const int2 b0 = *reinterpret_cast<const int2*>(xg + xup + j);
                    const int2 b1 = *reinterpret_cast<const int2*>(xg + xdn + j);
                    qu[j] = a0.x; qu[j + 1] = a0.y; qd[j] = a1.x; qd[j + 1] = a1.y;
                    gu[j] = b0.x; gu[j + 1] = b0.y; gd[j] = b1.x; gd[j + 1] = b1.y;
                }
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int row = br * R + r;
                    ql[r] = xq[row * N + lb * C + C - 1];
                    qr[r] = xq[row * N + rb * C];
                    gl[r] = xr[row * BCL + lb];
                    gr[r] = xl[row * BCL + rb];
                }
                flux_update<R, C>(q, G1, G2, qu, gu, qd, gd, ql, gl, qr, gr, a.Af);
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int c = 0; c < C; ++c) bad |= (static_cast<uint32_t>(q[r][c]) + 0x40000000u) >> 31;
            }
            if constexpr (CPL) {
                if (m9 == 8) {
                    // ---- coarse noise P1 S P1^T (S = summed fine normals, published by the barrier above):
                    // T = S P1^T, a thread its block's rows and the coarse columns 2 bc, 2 bc + 1
                    if (fine_thread) {
                        const ulonglong2* const z = reinterpret_cast<const ulonglong2*>(Zs + br * R * N);
                        const float2* const w0 = reinterpret_cast<const float2*>(P1 + 2 * bc * N);
                        const float2* const w1 = reinterpret_cast<const float2*>(P1 + (2 * bc + 1) * N);
                        f32x2 s0[R], s1[R];
#pragma unroll
                        for (int r = 0; r < R; ++r) s0[r] = s1[r] = pack2(0.f, 0.f);
#pragma unroll 3
                        for (int x = 0; x < N / 2; ++x) {
                            const float2 p = w0[x], w = w1[x];
                            const f32x2 px = pack2(p.x, p.x), py = pack2(p.y, p.y), wx = pack2(w.x, w.x), wy = pack2(w.y, w.y);
#pragma unroll
                            for (int r = 0; r < R; ++r) {
                                const ulonglong2 u = z[r * (N / 2) + x];
                                s0[r] = fma2(u.y, py, fma2(u.x, px, s0[r]));
                                s1[r] = fma2(u.y, wy, fma2(u.x, wx, s1[r]));
                            }
                        }
#pragma unroll
                        for (int r = 0; r < R; ++r)
                            reinterpret_cast<ulonglong2*>(Tm)[(br * R + r) * (NC / 2) + bc] = make_ulonglong2(s0[r], s1[r]);
                    }
                    __syncthreads();
                    const int32_t* qc = ccur ? qcB : qcA;
                    // two coarse points (y1, y2), (y1 + 1, y2) a thread
                    for (int o = tid; o < NC * NC / 2; o += THREADS) {
                        const int y1 = o / NC * 2, y2 = o % NC;
                        const float2* const w0 = reinterpret_cast<const float2*>(P1 + y1 * N);
                        const float2* const w1 = reinterpret_cast<const float2*>(P1 + (y1 + 1) * N);
                        f32x2 s[2] = {pack2(0.f, 0.f), pack2(0.f, 0.f)};
#pragma unroll 3
                        for (int x = 0; x < N / 2; ++x) {
                            const f32x2 t0 = Tm[2 * x * NC + y2], t1 = Tm[(2 * x + 1) * NC + y2];
                            const float2 p = w0[x], w = w1[x];
                            s[0] = fma2(pack2(p.y, p.y), t1, fma2(pack2(p.x, p.x), t0, s[0]));
                            s[1] = fma2(pack2(w.y, w.y), t1, fma2(pack2(w.x, w.x), t0, s[1]));
                        }
#pragma unroll
                        for (int v = 0; v < 2; ++v) {
                            const int y = (y1 + v) * NC + y2;
                            // gc includes the 1/3 of the 9-step sum
                            const float amp = FL ? noise_amp_fluct(qc[y], a.rbc[(size_t)(m / 9) * NC * NC + y], a.isc, a.gc)
                                                 : noise_amp(qc[y], a.gc);
                            Gc1[y] = __float2int_rn(amp * lo2(s[v]));
                            Gc2[y] = __float2int_rn(amp * hi2(s[v]));
                        }
                    }
                    __syncthreads();
                    explicit_update<NC, THREADS>(qc, Gc1, Gc2, ccur ? qcA : qcB, a.Ac, bad);
                    ccur ^= 1;
                    m9 = -1;   // the next barriers order the coarse state for its next step, 9 fine steps on
                }
                ++m9;
            }
        }
        __syncthreads();

        // ---- observables against FP64 test functions, mass; CTA reduction
        double v[kRedF];
#pragma unroll
        for (int i = 0; i < kRedF; ++i) v[i] = 0.0;
        if (fine_thread) {
            long long mass = 0;
            int32_t d[R][C];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    mass += q[r][c];
                    d[r][c] = q[r][c] - a.qbf[fx0 + r * N + c];
                }
            v[2 * kMaxObs] = static_cast<double>(mass);
#pragma unroll
            for (int k = 0; k < kMaxObs; ++k) {
                if (k < a.n_obs) {
#pragma unroll
                    for (int r = 0; r < R; ++r)
#pragma unroll
                        for (int c = 0; c < C; ++c)
                            v[k] += static_cast<double>(d[r][c]) * f.phif64[(size_t)k * N * N + fx0 + r * N + c];
                }
            }
        }
        if constexpr (CPL) {
            const int32_t* qc = ccur ? qcB : qcA;
            for (int y = tid; y < NC * NC; y += THREADS) {
                v[2 * kMaxObs + 1] += static_cast<double>(qc[y]);
                const double d = static_cast<double>(qc[y] - a.qbc[y]);
#pragma unroll
                for (int k = 0; k < kMaxObs; ++k)
                    if (k < a.n_obs) v[kMaxObs + k] += d * f.phic64[(size_t)k * NC * NC + y];
            }
        }
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1)
#pragma unroll
            for (int i = 0; i < kRedF; ++i) v[i] += __shfl_xor_sync(kFullMaskF, v[i], off);
        if ((tid & 31) == 0)
#pragma unroll
            for (int i = 0; i < kRedF; ++i) red[(tid >> 5) * kRedF + i] = v[i];
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < S::WARPS; ++w)
#pragma unroll
                for (int i = 0; i < kRedF; ++i) v[i] += red[w * kRedF + i];
            double Df[kMaxObs], Dc[kMaxObs];
#pragma unroll
            for (int k = 0; k < kMaxObs; ++k) {
                Df[k] = a.dscale_f * v[k] + a.delta_f[k];
                Dc[k] = CPL ? a.dscale_c * v[kMaxObs + k] + a.delta_c[k] : 0.0;
            }
            acc[0] += 1.0;
            double merr = fabs(v[2 * kMaxObs] - static_cast<double>(a.mass0_f)) * a.dscale_f;
            if (CPL) merr = fmax(merr, fabs(v[2 * kMaxObs + 1] - static_cast<double>(a.mass0_c)) * a.dscale_c);
            acc[1] = fmax(acc[1], merr);
            int qi = 0;
            for (int j = 0; j < a.n_obs; ++j) {
                const int kend = a.products ? a.n_obs : j + 1;
                for (int k = j; k < kend; ++k, ++qi) {
                    const double pf = a.N * Df[j] * Df[k];
                    const double pc = CPL ? a.N * Dc[j] * Dc[k] : 0.0;
                    const double dp = pf - pc, dp2 = dp * dp;
                    double* B = acc + 2 + kNSum * qi;
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
        __syncthreads();
    }
    if (bad) atomicOr(a.err, kErrRange);
    __syncthreads();
    for (int i = tid; i < a.slot_stride; i += THREADS) a.partials[(size_t)i * n_slots + slot] = acc[i];
}

// Two builds at 18^2: few samples run on 1 x 6 cells per thread (two warps per
// sample), which is the faster one for a sample, many on 2 x 6 (one warp).
// 18^2 x 72 steps, us, one row / two rows: 3 samples 62 / 113, 1216 116 / 172; 20000
// samples 2310 (one row, normals in shared memory) / 1680.  At 54^2 with the
// fluctuation state, whose mean-field loads a sample alone on its SM waits for, the
// same: x 243 steps, plain, 152 samples 366 / 437 (before the 2 x 6 blocks 411), coupled
// 500 / 570 (606); without it there is little between them (coupled 332 / 330).
template <int N, bool FL>
constexpr long long kFewF = N == 18 ? 1216 : N == 54 && FL ? 152 : 0;
template <int N>
constexpr int kRows = N == 6 ? 1 : 2;

template <int N, bool CPL, bool FL>
cudaError_t fprepare(int slot_stride, VariantInfo* out) {
    using S = FShape<N, kRows<N>>;
    const size_t smem = S::smem(slot_stride);
    const auto kernel = fourier_kernel<N, kRows<N>, CPL, FL>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if constexpr (kFewF<N, FL> > 0) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fourier_kernel<N, 1, CPL, FL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)FShape<N, 1>::smem(slot_stride));
    }
    if (e != cudaSuccess) return e;
    int per_sm = 0, dev = 0, sms = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, S::THREADS, smem)) != cudaSuccess) return e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    *out = VariantInfo{};
    out->supported = per_sm > 0;
    out->threads = S::THREADS;
    out->cluster = 1;
    out->slots_per_cta = 1;
    out->smem = smem;
    out->max_ctas = per_sm * sms;
    return cudaSuccess;
}

template <int N, int ROWS, bool CPL, bool FL>
cudaError_t flaunch_rows(const KArgs& a, const FArgs& f, int n_ctas, cudaStream_t st, int priority) {
    using S = FShape<N, ROWS>;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(n_ctas);
    cfg.blockDim = dim3(S::THREADS);
    cfg.dynamicSmemBytes = S::smem(a.slot_stride);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    int na = 0;
    if (priority != 0) {
        attr[na].id = cudaLaunchAttributePriority;
        attr[na].val.priority = priority;
        ++na;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    return cudaLaunchKernelEx(&cfg, fourier_kernel<N, ROWS, CPL, FL>, a, f);
}

template <int N, bool CPL, bool FL>
cudaError_t flaunch(const KArgs& a, const FArgs& f, int n_ctas, cudaStream_t st, int priority) {
    if constexpr (kFewF<N, FL> > 0) {
        if (a.count <= kFewF<N, FL>) return flaunch_rows<N, 1, CPL, FL>(a, f, n_ctas, st, priority);
    }
    return flaunch_rows<N, kRows<N>, CPL, FL>(a, f, n_ctas, st, priority);
}

template <bool FL>
cudaError_t fourier_info_fl(int n, bool coupled, int slot_stride, VariantInfo* out) {
    switch (n) {
        case 6: return coupled ? cudaSuccess : fprepare<6, false, FL>(slot_stride, out);   // level 0 only
        case 18: return coupled ? fprepare<18, true, FL>(slot_stride, out) : fprepare<18, false, FL>(slot_stride, out);
        case 54: return coupled ? fprepare<54, true, FL>(slot_stride, out) : fprepare<54, false, FL>(slot_stride, out);
        default: return cudaSuccess;
    }
}

template <bool FL>
cudaError_t launch_fourier_fl(int n, bool coupled, const KArgs& a, const FArgs& f, int n_ctas, cudaStream_t st,
                              int priority) {
    switch (n) {
        case 6: return coupled ? cudaErrorInvalidValue : flaunch<6, false, FL>(a, f, n_ctas, st, priority);
        case 18: return coupled ? flaunch<18, true, FL>(a, f, n_ctas, st, priority)
                                : flaunch<18, false, FL>(a, f, n_ctas, st, priority);
        case 54: return coupled ? flaunch<54, true, FL>(a, f, n_ctas, st, priority)
                                : flaunch<54, false, FL>(a, f, n_ctas, st, priority);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

bool fourier_supported(int n) { return n == 6 || n == 18 || n == 54; }

cudaError_t fourier_variant_info(int n, bool coupled, int slot_stride, VariantInfo* out, bool fluct) {
    *out = VariantInfo{};
    return fluct ? fourier_info_fl<true>(n, coupled, slot_stride, out) : fourier_info_fl<false>(n, coupled, slot_stride, out);
}

cudaError_t launch_fourier(int n, bool coupled, const KArgs& a, const FArgs& f, int n_ctas, cudaStream_t st,
                           int priority, bool fluct) {
    if (fluct && (!a.rbf || (coupled && !a.rbc))) return cudaErrorInvalidValue;
    return fluct ? launch_fourier_fl<true>(n, coupled, a, f, n_ctas, st, priority)
                 : launch_fourier_fl<false>(n, coupled, a, f, n_ctas, st, priority);
}

}  // namespace dk
