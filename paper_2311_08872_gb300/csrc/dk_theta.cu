// Theta-scheme sample kernel for sm_103a: Eq. (FullyDiscreteDK) with an
// implicit diffusion weight b0 > 0 (b1 = 1 - b0; Definition 2.1, the operator
// A_h of Appendix C), for the NN-coupled pair of Section 3.2 on grids up to
// 128 x 128.
//
// Step.  Subtracting (I - b0 tau/2 Delta_h) rho^(m-1) from both sides of the
// scheme gives the increment
//     rho^m - rho^(m-1) = H (tau/2 Delta_h rho^(m-1) + xi^(m-1)),
//     H = (I - b0 tau/2 Delta_h)^(-1) = (I + alpha L)^(-1),  alpha = b0 tau/(2 h^2),
// with L a = 4 a(x) - sum of the four neighbours (= -h^2 Delta_h) and xi the
// explicit noise divergence.  The bracket is the backward difference of a
// face flux F_r (diffusion flux across the face x -> x + e_r plus the two noise
// transfers G_r(x) + G_r(x + e_r) of the central difference), and H commutes
// with every periodic difference operator, so the increment is the backward
// difference of H F_r = F_r + u_r with (I + alpha L) u_r = -alpha L F_r.
// F_r is exact in fixed point as in the explicit kernels, in 32 bits on the fine
// grid (a flux beyond is a range error) and in 64 on the coarse one, where it may
// leave 32 bits as long as the corrected flux does not; only the
// correction u_r is computed in FP32, by K steps of Chebyshev iteration on the
// spectrum [1, 1 + 8 alpha] of I + alpha L (K fixed on the host from the
// Chebyshev error bound), and rounded once.  Adding the integer face fluxes
// keeps sum_x q invariant bit for bit, as in the explicit kernels.  K = 0
// (b0 = 0) is exactly the explicit step.
//
// Work decomposition.  A thread owns an R x C block of fine cells (and the
// (R/2) x (C/2) coarse cells they couple to, so the coupled increments are
// summed in registers); the state, the face fluxes and the Chebyshev operands
// stay in registers, the two components of a cell packed in one FP32 pair, so
// an iteration is 9 packed operations per cell.  A row of blocks is a segment
// of N/C <= 32 consecutive lanes: left / right neighbours come by warp shuffles
// (the segment wrap is the periodic wrap) and only the blocks' top and bottom
// rows pass through shared memory, one CTA barrier per iteration (two buffers
// in turn).  An exchange costs 4 R shuffles and 8 C shared-memory words per
// block against R C cells of arithmetic: 4 x 4 blocks balance the two (2 x 2
// blocks spent more on the exchange than on the cells) and fit in 255
// registers with 8 warps on an SM.  A sample of up to 16 x 16 cells fits one
// warp (no CTA barrier).
//
// 128 x 128 takes a cluster of 4 CTAs, each a band of 8 block rows (one warp
// each).  A warp of the band's first or last block row sends its edge row to
// the neighbouring CTA's shared memory with asynchronous stores that complete
// on an mbarrier there, and waits on its own: an exchange is one message each
// way between two warps, where a cluster barrier held all 4 CTAs at every
// iteration.  Four message slots in turn need no other handshake: slot n % 4 is
// written again by exchange n + 4, after the sender has received the neighbour's
// message n + 3, which that warp sent after the CTA barriers of its exchanges
// n + 1 and n + 2, before which it read message n.  (Two slots are not enough:
// message n + 1 need not depend on message n, as between the coarse and the next
// fine step, and nothing else orders that read before it.)  Every wait is
// bounded: a thread whose message does not come within kMbarPolls polls records
// kErrTimeout and waits no more, arms no slot any more (an arrival on a slot whose
// last message is still out would be one too many), and the CTA stops stepping at
// the next fine step, for all its samples; the neighbours' waits for it run out in
// turn.  It ends only when what they sent in that last step has had time to land.
//
// Bound by instruction issue and latency: 9 packed operations per cell and iteration
// take two cycles each on the FP32 pipe, and an iteration ends in a barrier.
// Crank--Nicolson (14 iterations), ms, in brackets with 2 x 2 blocks per thread and a
// cluster barrier per iteration: 128^2, 75 samples x 384 steps, 14.0 (29.7), 36
// samples 4.95 (9.90); 64^2, 1000 x 96, 6.2 (8.98), 152 samples 1.03 (1.29); 32^2,
// 20000 x 24, 7.17 (10.4).  With the inner rows of a block after the barrier instead
// of before it, 64^2 took 1.11 (152 samples) and 6.61 (1000).
#include <cooperative_groups.h>

#include <type_traits>

#include "dk_device.cuh"
#include "dk_kernels.h"

namespace dk {
namespace {

namespace cg = cooperative_groups;

constexpr unsigned kFullMask = 0xffffffffu;
constexpr int kRed = 2 * kMaxObs + 2;   // reduced values per sample

// Shapes: fine block R x C per thread, CL CTAs per sample.  (A poll limit and a
// stopping step read at run time cost the 128^2 build 100 to 400 bytes of spills and
// a tenth to a quarter of its speed: only the test's build has them.)
enum Build { kFirst, kDense, kMid };   // see first_build
template <int N_, Build B, bool TEST_ = false>
struct TShape {
    static constexpr int N = N_, NC = N / 2;
    static constexpr bool DENSE = B == kDense;
    static constexpr bool TEST = TEST_;                    // build of the failure-detection test (TArgs)
    static constexpr bool SMALL = N < 32 || (N == 32 && B == kFirst);
    static constexpr int R = SMALL ? 2 : 4, C = N >= 16 && !(N == 32 && !DENSE) ? 4 : 2;
    static constexpr int CL = N >= 128 ? 4 : 1;
    static constexpr int LPR = N / C;                      // lanes per row of blocks
    static constexpr int NBR = N / R / CL;                 // block rows per CTA and sample
    static constexpr int TPS = NBR * LPR;                  // threads per sample and CTA
    static constexpr int THREADS = TPS >= 64 ? TPS : 128;
    static constexpr int SPB = THREADS / TPS;              // samples per CTA
    // Registers per thread: up to 255 (8 warps on an SM), 128 for the 2 x 2 blocks at
    // 32^2, 4 x 2 ones and where DENSE (16 warps; the fluxes and the coarse state of 4 x 4 blocks
    // then spill outside the iteration).  16^2 has 155, or 96 where DENSE (20 warps).
    // 4^2 has 128: 100000 samples x 5 steps 171 us with 150, 164 with 128, 193 with 96.
    static constexpr int MIN_CTAS = N == 16 && DENSE ? 5 : (N == 4 || DENSE || N == 32 ? 512 : 256) / THREADS;
    static_assert(LPR <= 32 && (SPB == 1 || TPS <= 32) && (CL == 1 || LPR == 32), "block layout");
    // per sample: two buffers of the blocks' top and bottom rows, two words a cell;
    // in a cluster also four message slots for the rows above and below the band,
    // their mbarriers, and two words that tell of a wait that ran out
    static constexpr int BUF = 4 * N * NBR;                // words of one buffer
    static constexpr int SLOT = 4 * N;                     // words of one message slot (both sides)
    // (4 x 4: 16 words of padding, so that the two samples of a quarter warp use different
    // banks; 100000 samples x 5 steps 230 us without, 171 with, 209 before these blocks)
    static constexpr int WORDS = 2 * BUF + (CL > 1 ? 4 * SLOT : 0) + (N == 4 ? 16 : 0);
    static constexpr size_t SAMPLE_BYTES = sizeof(int32_t) * WORDS + (CL > 1 ? 10 * sizeof(uint64_t) : 0);
    static size_t smem(int slot_stride) {
        return SAMPLE_BYTES * SPB + sizeof(double) * ((THREADS + 31) / 32) * kRed + sizeof(double) * kRed +
               sizeof(double) * SPB * slot_stride;
    }
};

__device__ __forceinline__ int32_t edge_flux64(long long A, int32_t d) {
    return static_cast<int32_t>((A * static_cast<long long>(d) + 0x80000000LL) >> 32);
}

__device__ __forceinline__ float as_f(int32_t v) { return __int_as_float(v); }
__device__ __forceinline__ int32_t as_i(float v) { return __float_as_int(v); }

__device__ __forceinline__ f32x2 pack2i(int32_t lo, int32_t hi) { return pack2(as_f(lo), as_f(hi)); }
__device__ __forceinline__ int32_t lo2i(f32x2 v) { return as_i(lo2(v)); }
__device__ __forceinline__ int32_t hi2i(f32x2 v) { return as_i(hi2(v)); }

// The larger of two values, NaN if one is (fmaxf drops it).
__device__ __forceinline__ float max_nan(float a, float b) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

constexpr unsigned kMbarPolls = 1u << 22;   // polls of one wait before it gives up

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// The exchange of the blocks' top and bottom rows, two words a cell: buffer
// n % 2 of exchange n holds [top, bottom][row of blocks][C/2][lane] vectors of two
// cells (16 bytes, conflict-free).  In a cluster, slot n % 4 takes the rows that the
// CTAs above and below sent, guarded by mbarriers up[n % 4] and dn[n % 4].
template <class S>
struct Exchange {
    float* buf;
    uint64_t* bars = nullptr;              // [up, dn][4]
    uint32_t rup = 0, rdn = 0;             // shared::cluster address of `buf` in the CTA above / below
    unsigned* err;
    unsigned polls;                        // limit of every wait (TEST)
    int br, bc;
    unsigned n = 0;
    bool dead = false;
    __device__ __forceinline__ Exchange(float* b, int br_, int bc_, int rank, unsigned* err_, unsigned polls_)
        : buf(b), err(err_), polls(polls_), br(br_), bc(bc_) {
        if constexpr (S::CL > 1) {
            bars = reinterpret_cast<uint64_t*>(b + S::WORDS);
            rup = mapa(smem_u32(b), (rank + S::CL - 1) % S::CL);
            rdn = mapa(smem_u32(b), (rank + 1) % S::CL);
            if (threadIdx.x == 0) {
                for (int i = 0; i < 8; ++i)
                    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bars + i)) : "memory");
                gone()[0] = gone()[1] = 0;
                asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            }
        }
    }
    __device__ __forceinline__ static uint32_t mapa(uint32_t a, int r) {
        uint32_t v;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(v) : "r"(a), "r"(r));
        return v;
    }
    // word offset of vector h (of two cells, or of one cell where W = 1) of a row:
    // side 0 top, 1 bottom; row NBR: the row from above (side 0) / below (side 1)
    template <int W>
    __device__ __forceinline__ int at(int side, int row, int h) const {
        constexpr int V = W == 1 ? 2 : 4, H = W == 1 ? 1 : W / 2;
        return (row < S::NBR ? static_cast<int>(n & 1) * S::BUF + ((side * S::NBR + row) * H + h) * (S::LPR * V)
                             : 2 * S::BUF + static_cast<int>(n & 3) * S::SLOT + (side * H + h) * (S::LPR * V)) +
               bc * V;
    }
    // Send this thread's part of row v to buffer row NBR, side `side`, of the CTA at `base`.
    template <int W>
    __device__ __forceinline__ void send(uint32_t base, int side, const f32x2 (&v)[W]) const {
        const uint32_t bar = base + 4u * S::WORDS + 8u * (4 * side + (n & 3));
#pragma unroll
        for (int h = 0; h < (W + 1) / 2; ++h) {
            const uint32_t dst = base + 4u * at<W>(side, S::NBR, h);
            if constexpr (W == 1)
                asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(dst),
                             "l"(v[0]), "r"(bar)
                             : "memory");
            else
                asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(dst),
                             "l"(v[2 * h]), "l"(v[2 * h + 1]), "r"(bar)
                             : "memory");
        }
    }
    template <int W>
    __device__ __forceinline__ void store(int side, const f32x2 (&v)[W]) const {
#pragma unroll
        for (int h = 0; h < (W + 1) / 2; ++h) {
            float* o = buf + at<W>(side, br, h);
            if constexpr (W == 1) *reinterpret_cast<f32x2*>(o) = v[0];
            else *reinterpret_cast<ulonglong2*>(o) = make_ulonglong2(v[2 * h], v[2 * h + 1]);
        }
    }
    template <int W>
    __device__ __forceinline__ void load(int side, int row, f32x2 (&v)[W]) const {
#pragma unroll
        for (int h = 0; h < (W + 1) / 2; ++h) {
            const float* o = buf + at<W>(side, row, h);
            if constexpr (W == 1) v[0] = *reinterpret_cast<const f32x2*>(o);
            else {
                const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(o);
                v[2 * h] = x.x;
                v[2 * h + 1] = x.y;
            }
        }
    }
    // Words that a thread whose wait ran out sets, word e % 2 at exchange e.
    __device__ __forceinline__ volatile int* gone() const { return reinterpret_cast<volatile int*>(bars + 8); }
    // Whether to stop before exchange n, the same for the whole CTA: word n % 2 was last
    // set at exchange n - 2 or before, ahead of the barrier of exchange n - 1, and is
    // not set again before that of exchange n.
    __device__ __forceinline__ bool stopped() const { return S::CL > 1 && gone()[n & 1]; }
    // The message of this exchange on side `side` (all lanes of the warp).
    template <int W>
    __device__ __forceinline__ void receive(int side) {
        const uint32_t bar = smem_u32(bars + 4 * side + (n & 3));
        if (bc == 0 && !dead)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(S::LPR * W * 8)
                         : "memory");
        const uint32_t parity = (n >> 2) & 1;
        for (unsigned i = 0; i < (S::TEST ? polls : kMbarPolls) && !dead; ++i) {
            uint32_t ok;
            asm volatile(
                "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                : "=r"(ok)
                : "r"(bar), "r"(parity)
                : "memory");
            if (ok) return;
        }
        if (!dead) atomicOr(err, kErrTimeout);
        dead = true;
        gone()[n & 1] = 1;
    }
    // Hand out the block's first and last row ...
    template <int W>
    __device__ __forceinline__ void publish(const f32x2 (&top)[W], const f32x2 (&bot)[W]) const {
        if (S::CL > 1 && br == 0) send<W>(rup, 1, top);
        else store<W>(0, top);
        if (S::CL > 1 && br == S::NBR - 1) send<W>(rdn, 0, bot);
        else store<W>(1, bot);
    }
    // ... and take the rows above and below it.
    template <int W>
    __device__ __forceinline__ void collect(f32x2 (&up)[W], f32x2 (&dn)[W]) {
        const bool first = br == 0, last = br == S::NBR - 1;
        if constexpr (S::TPS <= 32) __syncwarp();
        else __syncthreads();
        if (!first) load<W>(1, br - 1, up);
        else if constexpr (S::CL == 1) load<W>(1, S::NBR - 1, up);
        if (!last) load<W>(0, br + 1, dn);
        else if constexpr (S::CL == 1) load<W>(0, 0, dn);
        if constexpr (S::CL > 1) {
            if (first) {
                receive<W>(0);
                load<W>(0, S::NBR, up);
            }
            if (last) {
                receive<W>(1);
                load<W>(1, S::NBR, dn);
            }
        }
        ++n;
    }
    __device__ __forceinline__ int32_t left(int32_t v) const {
        return __shfl_sync(kFullMask, v, (bc + S::LPR - 1) % S::LPR, S::LPR);
    }
    __device__ __forceinline__ int32_t right(int32_t v) const {
        return __shfl_sync(kFullMask, v, (bc + 1) % S::LPR, S::LPR);
    }
    __device__ __forceinline__ f32x2 left2(f32x2 v) const { return pack2i(left(lo2i(v)), left(hi2i(v))); }
    __device__ __forceinline__ f32x2 right2(f32x2 v) const { return pack2i(right(lo2i(v)), right(hi2i(v))); }
};

// Exchange of a block field a; f(r, c, up, down, left, right) for every cell, the
// inner rows before the barrier and the neighbours' messages are waited for.
template <int R, int C, class S, class F>
__device__ __forceinline__ void neighbours(f32x2 (&a)[R][C], Exchange<S>& x, F&& f) {
    x.template publish<C>(a[0], a[R - 1]);
    f32x2 l[R], rt[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        l[r] = x.left2(a[r][C - 1]);
        rt[r] = x.right2(a[r][0]);
    }
    const auto row = [&](int r, const f32x2 (&up)[C], const f32x2 (&dn)[C]) {
#pragma unroll
        for (int c = 0; c < C; ++c)
            f(r, c, up[c], dn[c], c > 0 ? a[r][c > 0 ? c - 1 : 0] : l[r], c + 1 < C ? a[r][c + 1 < C ? c + 1 : 0] : rt[r]);
    };
#pragma unroll
    for (int r = 1; r + 1 < R; ++r) row(r, a[r - 1], a[r + 1]);
    f32x2 up[C], dn[C];
    x.template collect<C>(up, dn);
    if constexpr (R == 1) {
        row(0, up, dn);
    } else {
        row(0, up, a[1]);
        row(R - 1, a[R - 2], dn);
    }
}

// One theta step of an R x C block of a periodic grid of LPR C columns (the
// fine grid, or the coarse one with COARSE: the four neighbours are added in
// another order there, in one CTA the recurrence rounds its other product, and
// the face fluxes have 64 bits).
template <int R, int C, bool COARSE, class S>
__device__ __forceinline__ void theta_step(int32_t (&q)[R][C], const int32_t (&G1)[R][C], const int32_t (&G2)[R][C],
                                           long long A, const TArgs& t, unsigned& bad, Exchange<S>& x) {
    // ---- exact face fluxes across the lower and the right edge of every cell
    using Flux = std::conditional_t<COARSE, long long, int32_t>;
    Flux F1[R][C], F2[R][C];
    {
        f32x2 top[C], bot[C], up[C], dn[C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            top[c] = pack2i(q[0][c], G1[0][c]);
            bot[c] = pack2i(q[R - 1][c], G1[R - 1][c]);
        }
        x.template publish<C>(top, bot);
        x.template collect<C>(up, dn);
        const auto face = [&](int32_t near, int32_t far, int32_t gn, int32_t gf) {
            const long long f = (long long)edge_flux64(A, far - near) + gn + gf;
            if constexpr (!COARSE) bad |= (unsigned)(f != (long long)(int32_t)f);
            return static_cast<Flux>(f);
        };
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int32_t qr = x.right(q[r][0]), gr = x.right(G2[r][0]);
#pragma unroll
            for (int c = 0; c < C; ++c) {
                F1[r][c] = face(q[r][c], r + 1 < R ? q[r + 1 < R ? r + 1 : 0][c] : lo2i(dn[c]), G1[r][c],
                                r + 1 < R ? G1[r + 1 < R ? r + 1 : 0][c] : hi2i(dn[c]));
                F2[r][c] = face(q[r][c], c + 1 < C ? q[r][c + 1 < C ? c + 1 : 0] : qr, G2[r][c],
                                c + 1 < C ? G2[r][c + 1 < C ? c + 1 : 0] : gr);
            }
        }
    }
    f32x2 u[R][C];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < C; ++c) u[r][c] = pack2(0.f, 0.f);
    if (t.K > 0) {
        // ---- right-hand side -alpha L F and the first Chebyshev direction
        const f32x2 minus1 = pack2(-1.f, -1.f), nalpha = pack2(-t.alpha, -t.alpha);
        f32x2 res[R][C], d[R][C];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c)
                d[r][c] = pack2(static_cast<float>(static_cast<int32_t>(F1[r][c])),
                                static_cast<float>(static_cast<int32_t>(F2[r][c])));
        if constexpr (COARSE) {
            // (the conversion from 64 bits, like the one to 64 bits below, is the slow one)
            bool wide = false;
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < C; ++c)
                    wide |= (F1[r][c] != (int32_t)F1[r][c]) | (F2[r][c] != (int32_t)F2[r][c]);
            if (wide) {
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int c = 0; c < C; ++c)
                        d[r][c] = pack2(static_cast<float>(F1[r][c]), static_cast<float>(F2[r][c]));
            }
        }
        neighbours<R, C, S>(d, x, [&](int r, int c, f32x2 up, f32x2 dn, f32x2 l, f32x2 rt) {
            f32x2 v = mul2(pack2(4.f, 4.f), d[r][c]);
            if constexpr (COARSE) v = fma2(rt, minus1, fma2(l, minus1, fma2(dn, minus1, fma2(up, minus1, v))));
            else v = fma2(add2(add2(up, dn), add2(l, rt)), minus1, v);
            res[r][c] = mul2(nalpha, v);
        });
        const f32x2 inv = pack2(t.inv_theta, t.inv_theta);
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c) d[r][c] = mul2(res[r][c], inv);
        // ---- K steps u += d, r -= (I + alpha L) d, d <- ca d + cb r; the last needs u only
        const f32x2 diag = pack2(1.f + 4.f * t.alpha, 1.f + 4.f * t.alpha);
#pragma unroll 1
        for (int k = 0; k + 1 < t.K; ++k) {
            neighbours<R, C, S>(d, x, [&](int r, int c, f32x2 up, f32x2 dn, f32x2 l, f32x2 rt) {
                f32x2 s;
                if constexpr (COARSE) s = add2(add2(add2(up, dn), l), rt);
                else s = add2(add2(up, dn), add2(l, rt));
                const f32x2 e = fma2(diag, d[r][c], mul2(nalpha, s));
                res[r][c] = fma2(e, minus1, res[r][c]);
            });
            const f32x2 ca = pack2(t.c1[k], t.c1[k]), cb = pack2(t.c2[k], t.c2[k]);
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    u[r][c] = add2(u[r][c], d[r][c]);
                    if constexpr (COARSE && S::CL == 1) d[r][c] = fma2(cb, res[r][c], mul2(ca, d[r][c]));
                    else d[r][c] = fma2(ca, d[r][c], mul2(cb, res[r][c]));
                }
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c) u[r][c] = add2(u[r][c], d[r][c]);
    }
    // ---- corrected fluxes, rounded once; the update adds integer face fluxes.
    // Corrections fit 32 bits in every sane state: the conversion to 64 bits, which
    // runs on the FP64 pipe (two per cell were a seventh of the step), is kept for a
    // block that has one beyond, or a NaN, which that conversion makes a range error.
    float big = 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < C; ++c) big = max_nan(big, max_nan(fabsf(lo2(u[r][c])), fabsf(hi2(u[r][c]))));
    int32_t H1[R][C], H2[R][C];
    const auto correct = [&](auto round) {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const long long h1 = (long long)F1[r][c] + round(lo2(u[r][c]));
                const long long h2 = (long long)F2[r][c] + round(hi2(u[r][c]));
                bad |= (unsigned)((h1 != (long long)(int32_t)h1) | (h2 != (long long)(int32_t)h2));
                H1[r][c] = static_cast<int32_t>(h1);
                H2[r][c] = static_cast<int32_t>(h2);
            }
    };
    if (big < 2147483648.f) correct([](float v) { return (long long)__float2int_rn(v); });
    else correct([](float v) { return __float2ll_rn(v); });
    f32x2 top[C], bot[C], up[C], dn[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
        top[c] = pack2i(H1[0][c], 0);
        bot[c] = pack2i(H1[R - 1][c], 0);
    }
    x.template publish<C>(top, bot);
    x.template collect<C>(up, dn);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int32_t hl = x.left(H2[r][C - 1]);
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int32_t ha = r > 0 ? H1[r > 0 ? r - 1 : 0][c] : lo2i(up[c]), hb = c > 0 ? H2[r][c > 0 ? c - 1 : 0] : hl;
            const long long v = (long long)q[r][c] + ((long long)H1[r][c] - ha) + ((long long)H2[r][c] - hb);
            bad |= (unsigned)((v >= (1LL << 30)) | (v <= -(1LL << 30)));
            q[r][c] = static_cast<int32_t>(v);
        }
    }
}

// Barrier of all threads of a sample.
template <class S>
__device__ __forceinline__ void sample_barrier() {
    if constexpr (S::CL > 1) cg::this_cluster().sync();
    else __syncthreads();
}

template <int N, bool CPL, Build B, bool TEST = false>
__global__ void __launch_bounds__(TShape<N, B>::THREADS, TShape<N, B>::MIN_CTAS)
    theta_kernel(const KArgs a, const TArgs t) {
    using S = TShape<N, B, TEST>;
    constexpr int NC = S::NC, TPS = S::TPS, SPB = S::SPB, THREADS = S::THREADS, R = S::R, C = S::C, CL = S::CL;
    constexpr int RC = R / 2, CC = C / 2;       // coarse block
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x;
    const int sl = tid / TPS, lt = tid % TPS;   // sample slot in the CTA, thread within the sample
    int rank = 0;
    if constexpr (CL > 1) rank = static_cast<int>(cg::this_cluster().block_rank());
    double* red = reinterpret_cast<double*>(smem_raw + S::SAMPLE_BYTES * SPB);
    double* tot = red + ((THREADS + 31) / 32) * kRed;   // this CTA's band total (clusters)
    double* acc = tot + kRed;                           // moment sums of the CTA's slots (rank 0)
    for (int i = tid; i < SPB * a.slot_stride; i += THREADS) acc[i] = 0.0;

    const int br = lt / S::LPR, bc = lt % S::LPR;
    const int i0 = (rank * S::NBR + br) * R, j0 = bc * C;   // the block's first fine cell
    Exchange<S> x(reinterpret_cast<float*>(smem_raw + S::SAMPLE_BYTES * sl), br, bc, rank, a.err, t.wait_polls);

    const long long n_slots = (long long)gridDim.x * SPB / CL;
    const long long cta_slot0 = (long long)(blockIdx.x / CL) * SPB;
    const long long slot = cta_slot0 + sl;
    const long long iters = a.count > cta_slot0 ? (a.count - cta_slot0 + n_slots - 1) / n_slots : 0;
    unsigned bad = 0;
    sample_barrier<S>();

    for (long long it = 0; it < iters; ++it) {
        const long long idx = slot + it * n_slots;
        const bool active = idx < a.count;
        const long long sid = a.first + (active ? idx : 0);
        const uint32_t c2 = static_cast<uint32_t>(sid);
        const uint32_t c3 = a.tag | ((static_cast<uint32_t>(static_cast<unsigned long long>(sid) >> 32) & 0xffffu) << 16);

        int32_t q[R][C], qc[RC][CC];
        float zt0[RC][CC], zt1[RC][CC];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c) q[r][c] = a.q0f[(i0 + r) * N + j0 + c];
#pragma unroll
        for (int r = 0; r < RC; ++r)
#pragma unroll
            for (int c = 0; c < CC; ++c) {
                zt0[r][c] = zt1[r][c] = 0.f;
                qc[r][c] = CPL ? a.q0c[(i0 / 2 + r) * NC + j0 / 2 + c] : 0;
            }

        const auto step = [&](int m) { return x.stopped() || (S::TEST && m == t.stall_step && rank == 0) ? a.M : m; };
        for (int m = step(0); m < a.M; m = step(m + 1)) {
            {
                // ---- noise of the fine block: Philox4x32-10 per horizontal cell pair, Box--Muller
                int32_t G1[R][C], G2[R][C];
                const f32x2 g2 = pack2(a.gf, a.gf);
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int p = 0; p < C / 2; ++p) {
                        const uint32_t pair = static_cast<uint32_t>(((i0 + r) * N + j0) / 2 + p);
                        const uint4 w = philox10(make_uint4(pair, static_cast<uint32_t>(m), c2, c3), a.key0, a.key1);
                        f32x2 rad, co, si;
                        box_muller_polar2(w.x, w.y, w.z, w.w, rad, co, si);
                        const f32x2 ta = mul2(noise_amp2(q[r][2 * p], q[r][2 * p + 1], g2), rad);
                        const f32x2 t1 = mul2(ta, co), t2 = mul2(ta, si);
                        G1[r][2 * p] = __float2int_rn(lo2(t1));
                        G1[r][2 * p + 1] = __float2int_rn(hi2(t1));
                        G2[r][2 * p] = __float2int_rn(lo2(t2));
                        G2[r][2 * p + 1] = __float2int_rn(hi2(t2));
                        if constexpr (CPL) {
                            float &z0 = zt0[r / 2][p], &z1 = zt1[r / 2][p];
                            z0 = fmaf(hi2(rad), hi2(co), fmaf(lo2(rad), lo2(co), z0));
                            z1 = fmaf(hi2(rad), hi2(si), fmaf(lo2(rad), lo2(si), z1));
                        }
                    }
                theta_step<R, C, false, S>(q, G1, G2, t.Af64, t, bad, x);
            }
            if constexpr (CPL) {
                if ((m & 3) == 3) {
                    // coupled coarse step: 1/4 of the 16 summed fine normals
                    int32_t H1[RC][CC], H2[RC][CC];
#pragma unroll
                    for (int r = 0; r < RC; ++r)
#pragma unroll
                        for (int c = 0; c < CC; ++c) {
                            const float s = noise_amp(qc[r][c], a.gc);
                            H1[r][c] = __float2int_rn(s * zt0[r][c]);
                            H2[r][c] = __float2int_rn(s * zt1[r][c]);
                            zt0[r][c] = zt1[r][c] = 0.f;
                        }
                    theta_step<RC, CC, true, S>(qc, H1, H2, t.Ac64, t, bad, x);
                }
            }
        }

        // ---- observables: fluctuation sums against the fixed-point mean field (FP64), mass
        double v[kRed];
        {
            long long mf = 0, mc = 0;
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < C; ++c) mf += q[r][c];
#pragma unroll
            for (int r = 0; r < RC; ++r)
#pragma unroll
                for (int c = 0; c < CC; ++c) mc += qc[r][c];
            v[2 * kMaxObs] = static_cast<double>(mf);
            v[2 * kMaxObs + 1] = CPL ? static_cast<double>(mc) : 0.0;
#pragma unroll
            for (int k = 0; k < kMaxObs; ++k) {
                double sf = 0.0, sc = 0.0;
                if (k < a.n_obs) {
#pragma unroll
                    for (int r = 0; r < R; ++r)
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            const int f = (i0 + r) * N + j0 + c;
                            sf += static_cast<double>(q[r][c] - a.qbf[f]) * t.phif64[(size_t)k * N * N + f];
                        }
                    if constexpr (CPL) {
#pragma unroll
                        for (int r = 0; r < RC; ++r)
#pragma unroll
                            for (int c = 0; c < CC; ++c) {
                                const int g = (i0 / 2 + r) * NC + j0 / 2 + c;
                                sc += static_cast<double>(qc[r][c] - a.qbc[g]) * t.phic64[(size_t)k * NC * NC + g];
                            }
                    }
                }
                v[k] = sf;
                v[kMaxObs + k] = sc;
            }
        }
        constexpr int SEG = TPS < 32 ? TPS : 32;
#pragma unroll
        for (int off = SEG / 2; off >= 1; off >>= 1)
#pragma unroll
            for (int i = 0; i < kRed; ++i) v[i] += __shfl_xor_sync(kFullMask, v[i], off, SEG);
        bool leader = lt == 0;
        if constexpr (TPS > 32) {
            if ((tid & 31) == 0)
#pragma unroll
                for (int i = 0; i < kRed; ++i) red[(tid >> 5) * kRed + i] = v[i];
            __syncthreads();
            if constexpr (CL == 1) {
                if (leader)
                    for (int w = 1; w < TPS / 32; ++w)
#pragma unroll
                        for (int i = 0; i < kRed; ++i) v[i] += red[w * kRed + i];
            } else {
                // the band totals, then their sum on rank 0 in rank order
                if (tid < kRed) {
                    double s = 0.0;
                    for (int w = 0; w < THREADS / 32; ++w) s += red[w * kRed + tid];
                    tot[tid] = s;
                }
                sample_barrier<S>();
                leader = rank == 0 && tid == 0;
                if (leader)
                    for (int i = 0; i < kRed; ++i) {
                        double s = 0.0;
                        for (int r = 0; r < CL; ++r) s += cg::this_cluster().map_shared_rank(tot, r)[i];
                        v[i] = s;
                    }
            }
        }

        // ---- FP64 quantities and moment sums (one thread per sample)
        if (leader && active) {
            double Df[kMaxObs], Dc[kMaxObs];
#pragma unroll
            for (int k = 0; k < kMaxObs; ++k) {
                Df[k] = a.dscale_f * v[k] + a.delta_f[k];
                Dc[k] = CPL ? a.dscale_c * v[kMaxObs + k] + a.delta_c[k] : 0.0;
            }
            double* A = acc + sl * a.slot_stride;
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
                o[2 * a.n_obs] = v[2 * kMaxObs] * a.dscale_f;
                o[2 * a.n_obs + 1] = CPL ? v[2 * kMaxObs + 1] * a.dscale_c : 0.0;
            }
        }
        sample_barrier<S>();   // the reduction scratch is reused by the next sample
    }
    if (bad) atomicOr(a.err, kErrRange);
    if constexpr (CL > 1) {
        // after a timeout, in some CTA of the cluster: messages that nobody waited for may be
        // on their way to this CTA (all sent before the cluster barrier above; about a
        // microsecond): stay for a millisecond
        if (ld_volatile(a.err) & kErrTimeout)
            for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    }

    // ---- per-slot partial sums to global scratch, entry-major [stride][n_slots]
    __syncthreads();
    if (rank == 0)
        for (int i = tid; i < SPB * a.slot_stride; i += THREADS) {
            const int s = i / a.slot_stride, e = i % a.slot_stride;
            a.partials[(size_t)e * n_slots + cta_slot0 + s] = acc[i];
        }
}

template <class S>
void launch_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&attr)[2], int n_ctas, int slot_stride,
                   cudaStream_t st, int priority) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(n_ctas);
    cfg.blockDim = dim3(S::THREADS);
    cfg.dynamicSmemBytes = S::smem(slot_stride);
    cfg.stream = st;
    int na = 0;
    if constexpr (S::CL > 1) {
        attr[na].id = cudaLaunchAttributeClusterDimension;
        attr[na].val.clusterDim.x = S::CL;
        attr[na].val.clusterDim.y = 1;
        attr[na].val.clusterDim.z = 1;
        ++na;
    }
    if (priority != 0) {
        attr[na].id = cudaLaunchAttributePriority;
        attr[na].val.priority = priority;
        ++na;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
}

// From 16 x 16 on there are two builds (32 x 32: three), chosen by the number of samples: one for
// few, which is the faster one for a sample, and a DENSE one for the GPU's
// throughput.  FEW is the number of samples that the first holds at once.
// Measured, ms, first build / DENSE: 128^2 x 384 steps, 36 samples 5.1 / 6.7, 150
// samples 25.3 / 22.6; 64^2 x 96, 152 samples 1.03 / 1.15, 304 2.2 / 1.8, 1000 7.7 /
// 6.2; 32^2 x 24 (2 x 2 blocks / 4 x 4), 3 samples 0.10 / 0.22, 304 0.160 / 0.25.
// 32^2 has 4 x 2 blocks between the two, for as many samples as those hold (608; two
// to four samples to an SM are too few warps of 4 x 4 blocks): 83 steps, plain, 2 x 2 /
// 4 x 2 / 4 x 4, 304 samples 145 / 165 / 229, 456 250 / 171 / 231 (206 before these
// blocks), 912 - / 363 / 317; coupled, 456 - / 190 / 254 (325).
// 16^2 holds 1824 samples at once in the first build, 3040 in the DENSE one; the
// first keeps the sizes that it finishes in as many passes, or in a short one more
// (coupled, 77 steps, us; in brackets one warp per 2 x 2 blocks and no bound, 2128 at
// once): 256 samples 364 / 370 (386), 2000 970 / 1010 (934), 2432 1212 / 1010 (1123),
// 3648 1495 / 1690 (1690), 5000 2232 / 2180 (2180), 20000 8140 / 8030 (8720).
template <int N>
constexpr long long kFew = N == 32 ? 304 : N == 64 ? 152 : N == 128 ? 36 : 0;
constexpr long long kMid32 = 608;
template <int N>
constexpr bool first_build(long long count) {
    if (N == 16) return count <= 2128 || (count > 3040 && count <= 3648);
    return N < 16 || count <= kFew<N>;
}

template <int N, bool CPL>
cudaError_t prepare(int slot_stride, VariantInfo* out) {
    constexpr Build B = N >= 16 ? kDense : kFirst;   // the build that holds the most samples
    using S = TShape<N, B>;
    const size_t smem = S::smem(slot_stride);
    const auto kernel = theta_kernel<N, CPL, B>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess && N >= 16)
        e = cudaFuncSetAttribute(theta_kernel<N, CPL, kFirst>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)TShape<N, kFirst>::smem(slot_stride));
    if constexpr (N == 32)
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(theta_kernel<N, CPL, kMid>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)TShape<N, kMid>::smem(slot_stride));
    if (e != cudaSuccess) return e;
    *out = VariantInfo{};
    out->threads = S::THREADS;
    out->cluster = S::CL;
    out->slots_per_cta = S::SPB;   // clusters: one sample slot per cluster
    out->smem = smem;
    if constexpr (S::CL > 1) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr[2];
        launch_config<S>(cfg, attr, S::CL, slot_stride, nullptr, 0);
        int clusters = 0;
        if ((e = cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg)) != cudaSuccess) return e;
        out->max_ctas = clusters * S::CL;
    } else {
        int per_sm = 0, dev = 0, sms = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, S::THREADS, smem)) != cudaSuccess ||
            (e = cudaGetDevice(&dev)) != cudaSuccess ||
            (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
            return e;
        out->max_ctas = per_sm * sms;
        if constexpr (N == 16) {
            // the first build also runs batches of several passes, on its own residency
            const auto few = theta_kernel<N, CPL, kFirst>;
            if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, few, TShape<N, kFirst>::THREADS, smem)) != cudaSuccess)
                return e;
            out->second_ctas = per_sm * sms;
        }
    }
    out->supported = out->max_ctas > 0;
    return cudaSuccess;
}

template <int N, bool CPL, Build B, bool TEST = false>
cudaError_t launch_build(const KArgs& a, const TArgs& t, int n_ctas, cudaStream_t st, int priority) {
    using S = TShape<N, B>;
    if (n_ctas % S::CL != 0) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    launch_config<S>(cfg, attr, n_ctas, a.slot_stride, st, priority);
    return cudaLaunchKernelEx(&cfg, theta_kernel<N, CPL, B, TEST>, a, t);
}

template <int N, bool CPL>
cudaError_t launch_n(const VariantInfo& vi, const KArgs& a, const TArgs& t, int* n_ctas, cudaStream_t st, int priority) {
    // (the builds of a grid size have the same sample slots per CTA or cluster)
    static_assert(TShape<N, kFirst>::SPB == TShape<N, (N >= 16 ? kDense : kFirst)>::SPB &&
                      (N != 32 || TShape<32, kMid>::SPB == 1), "slots");
    if constexpr (N == 32)
        if (a.count > kFew<N> && a.count <= kMid32) return launch_build<N, CPL, kMid>(a, t, *n_ctas, st, priority);
    if constexpr (N >= 16)
        if (!first_build<N>(a.count)) return launch_build<N, CPL, kDense>(a, t, *n_ctas, st, priority);
    if (vi.second_ctas > 0 && vi.second_ctas < *n_ctas) *n_ctas = vi.second_ctas;
    return launch_build<N, CPL, kFirst>(a, t, *n_ctas, st, priority);
}

// f(std::integral_constant<int, N>) for the grid sizes with a kernel.
template <class F>
bool for_grid(int n, F&& f) {
    switch (n) {
        case 4: f(std::integral_constant<int, 4>{}); return true;
        case 8: f(std::integral_constant<int, 8>{}); return true;
        case 16: f(std::integral_constant<int, 16>{}); return true;
        case 32: f(std::integral_constant<int, 32>{}); return true;
        case 64: f(std::integral_constant<int, 64>{}); return true;
        case 128: f(std::integral_constant<int, 128>{}); return true;
        default: return false;
    }
}

}  // namespace

bool theta_supported(int n) {
    return for_grid(n, [](auto) {});
}

cudaError_t theta_variant_info(int n, bool coupled, int slot_stride, VariantInfo* out) {
    *out = VariantInfo{};   // supported = 0 for other grids
    cudaError_t e = cudaSuccess;
    for_grid(n, [&](auto N) { e = coupled ? prepare<N.value, true>(slot_stride, out) : prepare<N.value, false>(slot_stride, out); });
    return e;
}

cudaError_t launch_theta_wait_test(const KArgs& a, const TArgs& t, int n_ctas, cudaStream_t st) {
    if (t.K < 0 || t.K > kMaxCheb) return cudaErrorInvalidValue;
    constexpr int N = 128;
    static_assert(TShape<N, kDense>::SAMPLE_BYTES < 45000, "no shared-memory attribute needed");
    return first_build<N>(a.count) ? launch_build<N, true, kFirst, true>(a, t, n_ctas, st, 0)
                                   : launch_build<N, true, kDense, true>(a, t, n_ctas, st, 0);
}

cudaError_t launch_theta(int n, bool coupled, const VariantInfo& vi, const KArgs& a, const TArgs& t, int* n_ctas,
                         cudaStream_t st, int priority) {
    if (t.K < 0 || t.K > kMaxCheb) return cudaErrorInvalidValue;
    cudaError_t e = cudaErrorInvalidValue;
    for_grid(n, [&](auto N) {
        e = coupled ? launch_n<N.value, true>(vi, a, t, n_ctas, st, priority)
                    : launch_n<N.value, false>(vi, a, t, n_ctas, st, priority);
    });
    return e;
}

}  // namespace dk
