// Fourier-coupled sample kernel for grids beyond one CTA (Section 3.1): the
// fine path of Eq. (FullyDiscreteDK) (b0 = 0, b1 = 1) on a 162 x 162 grid and,
// for a coupled level, the coarse path on the 54 x 54 grid with step 9 tau,
// whose noise carries every Fourier mode of the fine noise that the coarse
// grid resolves.  Same noise, arithmetic and restriction as the one-CTA
// Fourier kernel: the cell normals of the explicit kernels (same Philox
// counters), the 9 fine normal fields of a coarse step summed per cell (FP32)
// and restricted once, W = P1 S P1^T (P1: nc x n, orthonormal rows), the
// coarse transfers rint(c 2^S sqrt(rho_c^+) W / 3), integer flux form.
//
// Work decomposition.  A sample's 162^2 fine cells (and their transfers and
// summed normals) need about 630 KB, so a thread-block cluster of CL = 6 CTAs
// carries one sample: CTA `rank` holds the band of fine rows 27 rank ..
// 27 rank + 26 and the coarse rows 9 rank .. 9 rank + 8.  A thread owns a block
// of 3 x 6 fine cells, their transfers and summed normals in registers (three
// rows of 3 Philox cell pairs) and publishes the block's edges in shared memory
// (q and G1 of its first and last row, q and G2 of its first and last column);
// the rows just above and below a band come from the neighbouring CTAs' shared
// memory (distributed shared memory, periodic over the cluster).
//
// Bound by instruction issue and latency with 8 warps of 246 registers on an SM.
// 45 samples x 1458 steps: 9.03 ms; 11.65 with a 1 x 6 segment of cells per thread,
// its summed normals in shared memory and 23 warps, whose exchange moved 12 words a
// cell (here 4) and whose restriction loaded two operands per two FMAs.
//
// Exchanges.  State and transfers are double-buffered by the step's parity,
// so a fine step needs one cluster barrier, split: a thread arrives (release)
// after writing its transfers; the warps of the band's first and last rows,
// which read other CTAs, wait (acquire) at once, the others only before their
// next arrival, after their flux update.  At a coarse step each CTA restricts
// its own rows, T = S_band P1^T (27 x 54 per component), and forms the partial
// product P1[:, band] T (54 x 54); after a cluster barrier each CTA sums the 6
// partials of its coarse rows in rank order, forms the coarse transfers, and
// after a second barrier updates its coarse rows.
#include <cooperative_groups.h>

#include "dk_device.cuh"
#include "dk_kernels.h"

namespace cg = cooperative_groups;

namespace dk {
namespace {

constexpr unsigned kFullMaskX = 0xffffffffu;
constexpr int kRedX = 2 * kMaxObs + 2;

template <int N_, int CL_>
struct XShape {
    static constexpr int N = N_, NC = N / 3, CL = CL_;
    static constexpr int BR = N / CL;               // fine rows per CTA
    static constexpr int CBR = NC / CL;             // coarse rows per CTA
    static constexpr int R = 3, C = 6;              // fine cells per thread
    static constexpr int BRW = BR / R, BCL = N / C; // rows / columns of blocks per CTA
    static constexpr int FT = BRW * BCL;            // threads that hold fine cells
    static constexpr int THREADS = (FT + 31) / 32 * 32;
    static constexpr int WARPS = THREADS / 32;
    static constexpr int BAND = BR * N;             // fine cells per CTA
    static constexpr int CBAND = CBR * NC;          // coarse cells per CTA
    static constexpr int HY = NC / 2;               // coarse column pairs
    static constexpr int WY = 6;                    // coarse rows of a thread's tile of the partial product
    static_assert(N % CL == 0 && NC % CL == 0 && N % C == 0 && BR % R == 0 && NC == 2 * BCL && NC % WY == 0 &&
                      BRW >= 2 && CBR >= 2,
                  "band shape");
    static_assert(NC / WY * HY <= THREADS && THREADS <= 1024, "one task per thread");
    // words: two exchange buffers of edges (q and G1 of the blocks' first and last
    // rows, q and G2 of their first and last columns); for a coupled level the summed
    // normals (2 per cell), P1 (NC x N), T (BR x NC x 2), the partial product (NC x
    // NC x 2), coarse q (two buffers), Gc1, Gc2
    static constexpr int ROWS = BRW * N, COLS = BR * BCL;
    static constexpr int XBUF = 4 * ROWS + 4 * COLS;
    static constexpr int WORDS_F = 2 * XBUF;
    static constexpr int WORDS_C = 2 * BAND + N * NC + 2 * BR * NC + 2 * NC * NC + 4 * CBAND;
    __host__ __device__ static constexpr int words(bool cpl) { return WORDS_F + (cpl ? WORDS_C : 0); }
    static size_t smem(bool cpl, int slot_stride) {
        return sizeof(int32_t) * (size_t)((words(cpl) + 1) / 2 * 2) +
               sizeof(double) * (size_t)(WARPS * kRedX + kRedX + slot_stride);
    }
};

// Split cluster barrier: arrive with release after a write that other CTAs
// read, a CTA barrier for the rest of the CTA, then the wait with acquire at
// once (threads that read other CTAs) or before the thread's next arrival.
struct XPhase {
    bool edge;
    bool pend = false;
    __device__ __forceinline__ explicit XPhase(bool edge_) : edge(edge_) {}
    // the built-in forms (release / acquire), which the compiler keeps convergent: the
    // CTA's last warp holds fine cells in part of its lanes only
    __device__ __forceinline__ static void arrive() { __cluster_barrier_arrive(); }
    __device__ __forceinline__ static void wait() { __cluster_barrier_wait(); }
    __device__ __forceinline__ void settle() {
        if (pend) {
            wait();
            pend = false;
        }
    }
    __device__ __forceinline__ void publish() {
        settle();
        arrive();
        __syncthreads();
        if (edge) wait();
        else pend = true;
    }
    __device__ __forceinline__ void full() {
        settle();
        arrive();
        wait();
    }
};

template <int N, int CL, bool CPL>
__global__ void __launch_bounds__(XShape<N, CL>::THREADS, 1)
    fourier_cluster_kernel(const KArgs a, const FArgs f) {
    using S = XShape<N, CL>;
    constexpr int NC = S::NC, BR = S::BR, CBR = S::CBR, R = S::R, C = S::C, BRW = S::BRW, BCL = S::BCL;
    constexpr int BAND = S::BAND, CBAND = S::CBAND, HY = S::HY, ROWS = S::ROWS, COLS = S::COLS, THREADS = S::THREADS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x;
    const int rank = static_cast<int>(cluster.block_rank());
    int32_t* const words = reinterpret_cast<int32_t*>(smem_raw);
    f32x2* const Zs = reinterpret_cast<f32x2*>(words + S::WORDS_F);        // [BAND] summed normals, both components
    f32x2* const Tm = Zs + BAND;                                           // [BR][NC]
    f32x2* const Wp = Tm + BR * NC;                                        // [NC][NC] partial product
    float* const P1 = reinterpret_cast<float*>(Wp + NC * NC);              // [NC][N]
    int32_t* const qc0 = reinterpret_cast<int32_t*>(P1 + NC * N);        // coarse q buffers at qc0, qc0 + CBAND
    int32_t* const Gc1 = qc0 + 2 * CBAND;
    int32_t* const Gc2 = Gc1 + CBAND;
    double* const red = reinterpret_cast<double*>(smem_raw + sizeof(int32_t) * (size_t)((S::words(CPL) + 1) / 2 * 2));
    double* const tot = red + S::WARPS * kRedX;      // this CTA's band totals
    double* const acc = tot + kRedX;                 // the slot's moment sums (rank 0)
    for (int i = tid; i < a.slot_stride; i += THREADS) acc[i] = 0.0;
    if constexpr (CPL) {
        for (int i = tid; i < N * NC; i += THREADS) P1[i] = f.P1[i];
    }

    // ---- the thread's fine block and its neighbours
    const bool fine_thread = tid < S::FT;
    const int br = fine_thread ? tid / BCL : 0, bc = fine_thread ? tid % BCL : 0;
    const int gx0 = (rank * BR + br * R) * N + bc * C;            // first cell on the whole grid
    const int lb = (bc + BCL - 1) % BCL, rb = (bc + 1) % BCL;     // blocks left / right
    // the block rows above / below: row of blocks and CTA
    const int rup = br > 0 ? br - 1 : BRW - 1, rdn = br < BRW - 1 ? br + 1 : 0;
    const int32_t* const up = br > 0 ? words : cluster.map_shared_rank(words, (rank + CL - 1) % CL);
    const int32_t* const dn = br < BRW - 1 ? words : cluster.map_shared_rank(words, (rank + 1) % CL);
    // the warps holding a block of the band's first or last block row read other CTAs
    // (block rows are not warp-aligned, so the test is per warp: the cluster wait is .aligned)
    const int wf = tid & ~31, wl = min(wf + 31, S::FT - 1);
    XPhase ph(wf < S::FT && (wf / BCL == 0 || wl / BCL == BRW - 1));

    const long long n_slots = (long long)gridDim.x / CL;
    const long long slot = (long long)blockIdx.x / CL;
    const long long iters = a.count > slot ? (a.count - slot + n_slots - 1) / n_slots : 0;
    unsigned bad = 0;
    ph.full();

    for (long long it = 0; it < iters; ++it) {
        const long long idx = slot + it * n_slots;
        const long long sid = a.first + idx;
        const uint32_t c2 = static_cast<uint32_t>(sid);
        const uint32_t c3 = a.tag | ((static_cast<uint32_t>(static_cast<unsigned long long>(sid) >> 32) & 0xffffu) << 16);
        int32_t q[R][C];
        f32x2 Z[R][C];   // summed normals of the coarse step, both components
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c) {
                q[r][c] = a.q0f[gx0 + r * N + c];
                Z[r][c] = pack2(0.f, 0.f);
            }
        int cb = 0;
        if constexpr (CPL) {
            for (int y = tid; y < CBAND; y += THREADS) qc0[y] = a.q0c[rank * CBAND + y];
        }
        ph.full();

        for (int m = 0, m9 = 0; m < a.M; ++m) {
            // the step's exchange buffer: rows [BRW][N] of q top, q bottom, G1 top, G1
            // bottom; columns [BR][BCL] of q first, q last, G2 first, G2 last
            const int xo = (m & 1) * S::XBUF, xc = xo + 4 * ROWS;
            int32_t G1[R][C], G2[R][C];
            // ---- noise of the block: Philox4x32-10 per horizontal cell pair, Box--Muller, transfers
            if (fine_thread) {
                const f32x2 g2v = pack2(a.gf, a.gf);
#pragma unroll
                for (int r = 0; r < R; ++r) {
#pragma unroll
                    for (int j = 0; j < C / 2; ++j) {
                        const int p = ((gx0 + r * N) >> 1) + j;
                        const uint4 x = philox10(make_uint4(static_cast<uint32_t>(p), static_cast<uint32_t>(m), c2, c3),
                                                 a.key0, a.key1);
                        f32x2 rad, co, si;
                        box_muller_polar2(x.x, x.y, x.z, x.w, rad, co, si);
                        const f32x2 t = mul2(noise_amp2(q[r][2 * j], q[r][2 * j + 1], g2v), rad);
                        const f32x2 t1 = mul2(t, co), t2 = mul2(t, si);
                        G1[r][2 * j] = __float2int_rn(lo2(t1));
                        G1[r][2 * j + 1] = __float2int_rn(hi2(t1));
                        G2[r][2 * j] = __float2int_rn(lo2(t2));
                        G2[r][2 * j + 1] = __float2int_rn(hi2(t2));
                        if (r == 0 || r == R - 1) {
                            int32_t* const row = words + xo + (r == 0 ? 0 : ROWS) + br * N + bc * C + 2 * j;
                            *reinterpret_cast<int2*>(row) = make_int2(q[r][2 * j], q[r][2 * j + 1]);
                            *reinterpret_cast<int2*>(row + 2 * ROWS) = make_int2(G1[r][2 * j], G1[r][2 * j + 1]);
                        }
                        if constexpr (CPL) {
                            const float za = lo2(rad), zb = hi2(rad);
                            Z[r][2 * j] = fma2(pack2(za, za), pack2(lo2(co), lo2(si)), Z[r][2 * j]);
                            Z[r][2 * j + 1] = fma2(pack2(zb, zb), pack2(hi2(co), hi2(si)), Z[r][2 * j + 1]);
                        }
                    }
                    int32_t* const col = words + xc + (br * R + r) * BCL + bc;
                    col[0] = q[r][0];
                    col[COLS] = q[r][C - 1];
                    col[2 * COLS] = G2[r][0];
                    col[3 * COLS] = G2[r][C - 1];
                }
                if constexpr (CPL) {
                    if (m9 == 8) {
#pragma unroll
                        for (int r = 0; r < R; ++r)
#pragma unroll
                            for (int c = 0; c < C; c += 2) {
                                reinterpret_cast<ulonglong2*>(Zs)[((br * R + r) * N + bc * C + c) / 2] =
                                    make_ulonglong2(Z[r][c], Z[r][c + 1]);
                                Z[r][c] = Z[r][c + 1] = pack2(0.f, 0.f);
                            }
                    }
                }
            }
            ph.publish();
            // ---- explicit step of the block in flux form (every edge flux computed
            // from the same two states by both of its cells)
            if (fine_thread) {
                int32_t qu[C], qd[C], gu[C], gd[C], ql[R], qr[R], gl[R], gr[R];
                const int32_t* const ru = up + xo + ROWS + rup * N + bc * C;
                const int32_t* const rd = dn + xo + rdn * N + bc * C;
#pragma unroll
                for (int j = 0; j < C; j += 2) {
                    const int2 a0 = *reinterpret_cast<const int2*>(ru + j);
                    const int2 a1 = *reinterpret_cast<const int2*>(rd + j);
                    const int2 b0 = *reinterpret_cast<const int2*>(ru + 2 * ROWS + j);
                    const int2 b1 = *reinterpret_cast<const int2*>(rd + 2 * ROWS + j);
                    qu[j] = a0.x; qu[j + 1] = a0.y; qd[j] = a1.x; qd[j + 1] = a1.y;
                    gu[j] = b0.x; gu[j + 1] = b0.y; gd[j] = b1.x; gd[j + 1] = b1.y;
                }
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int32_t* const col = words + xc + (br * R + r) * BCL;
                    ql[r] = col[COLS + lb];
                    qr[r] = col[rb];
                    gl[r] = col[3 * COLS + lb];
                    gr[r] = col[2 * COLS + rb];
                }
                flux_update<R, C>(q, G1, G2, qu, gu, qd, gd, ql, gl, qr, gr, a.Af);
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int c = 0; c < C; ++c) bad |= (static_cast<uint32_t>(q[r][c]) + 0x40000000u) >> 31;
            }
            if constexpr (CPL) {
                if (m9 == 8) {
                    ph.settle();
                    // ---- T = S_band P1^T (S published by the barrier above): the block's rows,
                    // coarse columns 2 bc and 2 bc + 1, both components packed
                    if (fine_thread) {
                        const float2* const w0 = reinterpret_cast<const float2*>(P1 + 2 * bc * N);
                        const float2* const w1 = reinterpret_cast<const float2*>(P1 + (2 * bc + 1) * N);
                        const ulonglong2* const z = reinterpret_cast<const ulonglong2*>(Zs + br * R * N);
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
                            reinterpret_cast<ulonglong2*>(Tm)[(br * R + r) * HY + bc] = make_ulonglong2(s0[r], s1[r]);
                    }
                    __syncthreads();
                    // ---- the band's part of P1 S P1^T: WY coarse rows of the columns 2 yy, 2 yy + 1
                    if (tid < NC / S::WY * HY) {
                        const int y0 = tid / HY * S::WY, yy = tid % HY;
                        f32x2 w0[S::WY], w1[S::WY];
#pragma unroll
                        for (int v = 0; v < S::WY; ++v) w0[v] = w1[v] = pack2(0.f, 0.f);
#pragma unroll 3
                        for (int x = 0; x < BR; ++x) {
                            const ulonglong2 t = reinterpret_cast<const ulonglong2*>(Tm)[x * HY + yy];
#pragma unroll
                            for (int v = 0; v < S::WY; ++v) {
                                const float p = P1[(y0 + v) * N + rank * BR + x];
                                w0[v] = fma2(pack2(p, p), t.x, w0[v]);
                                w1[v] = fma2(pack2(p, p), t.y, w1[v]);
                            }
                        }
#pragma unroll
                        for (int v = 0; v < S::WY; ++v)
                            reinterpret_cast<ulonglong2*>(Wp)[(y0 + v) * HY + yy] = make_ulonglong2(w0[v], w1[v]);
                    }
                    ph.full();
                    // ---- coarse transfers of the CTA's coarse rows: the partials summed in rank order
                    int32_t* const qc = qc0 + cb * CBAND;
                    for (int y = tid; y < CBAND; y += THREADS) {
                        const int o = rank * CBAND + y;   // coarse point (y1, y2), y1 = rank CBR + y / NC
                        float w0 = 0.f, w1 = 0.f;
#pragma unroll
                        for (int r = 0; r < CL; ++r) {
                            const f32x2* const src = r == rank ? Wp : cluster.map_shared_rank(Wp, r);
                            const f32x2 v = src[o];
                            w0 += lo2(v);
                            w1 += hi2(v);
                        }
                        const float amp = noise_amp(qc[y], a.gc);   // gc includes the 1/3 of the 9-step sum
                        Gc1[y] = __float2int_rn(amp * w0);
                        Gc2[y] = __float2int_rn(amp * w1);
                    }
                    ph.full();
                    // ---- explicit coarse step of the CTA's coarse rows
                    for (int y = tid; y < CBAND; y += THREADS) {
                        // neighbours of the coarse cell: above / below in the neighbouring CTA for
                        // the band's first / last coarse row (periodic over the cluster)
                        const int cl1 = y / NC, cy2 = y % NC;
                        const int cra = cl1 > 0 ? rank : (rank + CL - 1) % CL;
                        const int crb = cl1 < CBR - 1 ? rank : (rank + 1) % CL;
                        const int cia = cl1 > 0 ? y - NC : (CBR - 1) * NC + cy2;
                        const int cib = cl1 < CBR - 1 ? y + NC : cy2;
                        const int clf = cl1 * NC + (cy2 + NC - 1) % NC, crt = cl1 * NC + (cy2 + 1) % NC;
                        const int32_t* const cup = cra == rank ? qc0 : cluster.map_shared_rank(qc0, cra);
                        const int32_t* const cdn = crb == rank ? qc0 : cluster.map_shared_rank(qc0, crb);
                        const int32_t c = qc[y];
                        const int32_t* const gu_p = cra == rank ? Gc1 : cluster.map_shared_rank(Gc1, cra);
                        const int32_t* const gd_p = crb == rank ? Gc1 : cluster.map_shared_rank(Gc1, crb);
                        const int32_t qu = cup[cb * CBAND + cia], qd = cdn[cb * CBAND + cib];
                        const int32_t v = c + (edge_flux(a.Ac, qd - c) - edge_flux(a.Ac, c - qu)) +
                                          (edge_flux(a.Ac, qc[crt] - c) - edge_flux(a.Ac, c - qc[clf])) +
                                          (gd_p[cib] - gu_p[cia]) + (Gc2[crt] - Gc2[clf]);
                        bad |= (static_cast<uint32_t>(v) + 0x40000000u) >> 31;
                        qc0[(cb ^ 1) * CBAND + y] = v;
                    }
                    cb ^= 1;
                    m9 = -1;
                }
                ++m9;
            }
        }

        // ---- observables of the band (fine: registers, coarse: the thread's cell), then the
        // band totals summed on rank 0 in rank order
        double v[kRedX];
#pragma unroll
        for (int i = 0; i < kRedX; ++i) v[i] = 0.0;
        if (fine_thread) {
            long long mf = 0;
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < C; ++c) mf += q[r][c];
            v[2 * kMaxObs] = static_cast<double>(mf);
#pragma unroll
            for (int k = 0; k < kMaxObs; ++k) {
                if (k < a.n_obs) {
                    double s = 0.0;
#pragma unroll
                    for (int r = 0; r < R; ++r)
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            const int x = gx0 + r * N + c;
                            s += static_cast<double>(q[r][c] - a.qbf[x]) * f.phif64[(size_t)k * N * N + x];
                        }
                    v[k] = s;
                }
            }
        }
        if constexpr (CPL) {
            for (int y = tid; y < CBAND; y += THREADS) {
                const int cg1 = rank * CBAND + y;
                const int32_t qv = qc0[cb * CBAND + y];
                v[2 * kMaxObs + 1] += static_cast<double>(qv);
                const double d = static_cast<double>(qv - a.qbc[cg1]);
#pragma unroll
                for (int k = 0; k < kMaxObs; ++k)
                    if (k < a.n_obs) v[kMaxObs + k] += d * f.phic64[(size_t)k * NC * NC + cg1];
            }
        }
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1)
#pragma unroll
            for (int i = 0; i < kRedX; ++i) v[i] += __shfl_xor_sync(kFullMaskX, v[i], off);
        if ((tid & 31) == 0)
#pragma unroll
            for (int i = 0; i < kRedX; ++i) red[(tid >> 5) * kRedX + i] = v[i];
        __syncthreads();
        if (tid < kRedX) {
            double x = 0.0;
            for (int w = 0; w < S::WARPS; ++w) x += red[w * kRedX + tid];
            tot[tid] = x;
        }
        ph.full();
        if (rank == 0 && tid == 0) {
            for (int i = 0; i < kRedX; ++i) {
                double x = 0.0;
                for (int r = 0; r < CL; ++r) x += (r == 0 ? tot : cluster.map_shared_rank(tot, r))[i];
                v[i] = x;
            }
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
                o[2 * a.n_obs] = v[2 * kMaxObs] * a.dscale_f;
                o[2 * a.n_obs + 1] = CPL ? v[2 * kMaxObs + 1] * a.dscale_c : 0.0;
            }
        }
        ph.full();   // the band totals and the state planes are reused by the next sample
    }
    if (bad) atomicOr(a.err, kErrRange);

    // ---- the slot's partial sums (rank 0), entry-major [stride][n_slots]
    __syncthreads();
    if (rank == 0)
        for (int i = tid; i < a.slot_stride; i += THREADS) a.partials[(size_t)i * n_slots + slot] = acc[i];
}

constexpr int kFourierClusterN = 162, kFourierClusterCL = 6;

template <int N, int CL, bool CPL>
cudaError_t xprepare(int slot_stride, VariantInfo* out) {
    using S = XShape<N, CL>;
    const size_t smem = S::smem(CPL, slot_stride);
    cudaError_t e = cudaFuncSetAttribute(fourier_cluster_kernel<N, CL, CPL>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(CL);
    cfg.blockDim = dim3(S::THREADS);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    if ((e = cudaOccupancyMaxActiveClusters(&clusters, fourier_cluster_kernel<N, CL, CPL>, &cfg)) != cudaSuccess)
        return e;
    *out = VariantInfo{};
    out->supported = clusters > 0;
    out->threads = S::THREADS;
    out->cluster = CL;
    out->slots_per_cta = 1;   // one sample slot per cluster
    out->smem = smem;
    out->max_ctas = clusters * CL;
    return cudaSuccess;
}

template <int N, int CL, bool CPL>
cudaError_t xlaunch(const KArgs& a, const FArgs& f, int n_ctas, cudaStream_t st, int priority) {
    using S = XShape<N, CL>;
    if (n_ctas <= 0 || n_ctas % CL != 0) return cudaErrorInvalidValue;
    if (CPL && !f.P1) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(n_ctas);
    cfg.blockDim = dim3(S::THREADS);
    cfg.dynamicSmemBytes = S::smem(CPL, a.slot_stride);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int na = 0;
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = CL;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = 1;
    ++na;
    if (priority != 0) {
        attr[na].id = cudaLaunchAttributePriority;
        attr[na].val.priority = priority;
        ++na;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    return cudaLaunchKernelEx(&cfg, fourier_cluster_kernel<N, CL, CPL>, a, f);
}

}  // namespace

bool fourier_cluster_supported(int n) { return n == kFourierClusterN; }

cudaError_t fourier_cluster_variant_info(int n, bool coupled, int slot_stride, VariantInfo* out) {
    *out = VariantInfo{};
    if (n != kFourierClusterN) return cudaSuccess;
    return coupled ? xprepare<kFourierClusterN, kFourierClusterCL, true>(slot_stride, out)
                   : xprepare<kFourierClusterN, kFourierClusterCL, false>(slot_stride, out);
}

cudaError_t launch_fourier_cluster(int n, bool coupled, const KArgs& a, const FArgs& f, int n_ctas, cudaStream_t st,
                                   int priority) {
    if (n != kFourierClusterN) return cudaErrorInvalidValue;
    return coupled ? xlaunch<kFourierClusterN, kFourierClusterCL, true>(a, f, n_ctas, st, priority)
                   : xlaunch<kFourierClusterN, kFourierClusterCL, false>(a, f, n_ctas, st, priority);
}

}  // namespace dk
