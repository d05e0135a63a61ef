// Streamed-state kernels for grids too large to keep a sample in registers
// (n >= 512: the finest levels of the low-density and large workloads).
//
// The state of `S` samples in flight lives in global memory (sized to stay in
// L2): the fine fixed-point state q and the coarse state qc (both double
// buffered) and the coupled coarse normal sums zt.  The scheme is the same as
// the register kernels' (Eq. FullyDiscreteDK with b0 = 0, b1 = 1; NN coupling
// of Section 3.2), in the same integer flux form and with the same FP32
// expressions for the transfers and the coupled sums, so the fine and coarse
// states agree with theirs bit for bit.
//
// One launch per fine step m: a CTA loads q^m on its tile and a one-cell halo,
// draws the normals of step m for the tile and for the halo cells (one extra
// Philox call per halo cell pair, so the transfers G^m never go to memory),
// and writes q^{m+1} and, for coupled samples, the running coarse sums zt.
// After the fourth fine step of a coarse step the coarse transfers are formed
// from qc and zt (tile and halo) and qc is updated, by extra CTAs of the next
// fine step's launch (zt is double buffered by coarse step) or, after the last
// fine step, by a launch of its own.  Kernel boundaries order all reads and
// writes; in the default build the fine steps are programmatic dependent
// launches that draw their noise before waiting for the previous kernel.
//
// Fine-step CTAs: 16 x 16 threads on a 32 x 64 tile, each thread a 2 x 4 block
// of fine cells (two coarse cells); two builds, for 4 or 5 resident CTAs per
// SM (at most 64 or 48 registers per thread), picked by the autotuner.
// Neighbouring blocks exchange the state and transfer of their edge cells:
// columns by shuffles, rows and the halo's cells through shared memory.
// The coarse step and the observables use 32 x 32 tiles.
//
// What bounds it: the same XU and FMA pipes as the register kernels, plus the
// halo's noise (128 extra pairs per 1024) and the tile's loads and stores.  The
// state of the samples in flight stays in L2.  The coarse step had a launch of
// its own every fourth step, which waited for the fine step's last wave and was
// waited for: 512^2, 7 samples x 2048 steps 17.8 ms, now 15.6; 1024^2, 5 x 1024:
// 21.1 ms, now 19.6 (packed FP32 noise, one component drawn in the halo and
// only edge rows in shared memory, 17.9 KB instead of 29.4, included).
#include <cstdint>

#include "dk_device.cuh"
#include "dk_kernels.h"

namespace dk {

namespace {

constexpr int kTile = 32;            // fine cells per tile side
constexpr int kTc = kTile / 2;       // coarse cells per tile side (= threads per side)
constexpr int kThreads = kTc * kTc;  // 256
// fine-step tiles: FR x kFC fine cells, thread rows of two fine rows
constexpr int kFC = 64;
constexpr int kFR = 32;
constexpr int kStreamVariants = 6;
__host__ __device__ constexpr int fine_threads(int fr) { return 8 * fr; }
// words of shared memory of a fine tile: state and transfer of the first and
// the last row of every thread row (FR/2 + 1 each: with the row below and the
// row above the tile), and of the columns left and right of the tile
__host__ __device__ constexpr int fine_words(int fr) { return 4 * (fr / 2 + 1) * kFC + 4 * fr; }
// the same for a coarse tile, one cell row per thread row
constexpr int kCoarseWords = 4 * (kTile + 1) * kTile + 4 * kTile;
__host__ __device__ constexpr int fine_smem(int fr) {
    return (int)sizeof(int32_t) * (fine_words(fr) > kCoarseWords ? fine_words(fr) : kCoarseWords);
}

__device__ __forceinline__ int wrapi(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

__device__ __forceinline__ uint4 pair_words(const SArgs& a, uint32_t p, int m, uint32_t c2, uint32_t c3) {
    return philox10(make_uint4(p, static_cast<uint32_t>(m), c2, c3), a.key0, a.key1);
}

// Box--Muller radii and directions of four cells of a row (two cell pairs):
// packed cells 0 and 2 (a) and cells 1 and 3 (b).
struct RowNormals {
    f32x2 ra, ca, sa, rb, cb, sb;
};

__device__ __forceinline__ RowNormals row_normals(uint4 x, uint4 y) {
    RowNormals z;
    box_muller_polar2(x.x, x.y, y.x, y.y, z.ra, z.ca, z.sa);
    box_muller_polar2(x.z, x.w, y.z, y.w, z.rb, z.cb, z.sb);
    return z;
}

// A halo pair's normals of one component: radius and cosine (rows) or sine
// (columns) of its first and second cell.
struct HaloNormals {
    float ra, da, rb, db;
};

__device__ __forceinline__ HaloNormals halo_normals(uint4 x, bool rows) {
    HaloNormals h;
    float ca, sa, cb, sb;
    box_muller_polar(x.x, x.y, h.ra, ca, sa);
    box_muller_polar(x.z, x.w, h.rb, cb, sb);
    h.da = rows ? ca : sa;
    h.db = rows ? cb : sb;
    return h;
}

// Makes the normals exist at this point of the program (an empty asm
// statement that reads and writes them): the compiler keeps their arithmetic
// before a later volatile asm statement such as the grid dependency wait.
__device__ __forceinline__ void pin(RowNormals& z) {
    asm volatile("" : "+l"(z.ra), "+l"(z.ca), "+l"(z.sa), "+l"(z.rb), "+l"(z.cb), "+l"(z.sb));
}
__device__ __forceinline__ void pin(HaloNormals& z) {
    asm volatile("" : "+f"(z.ra), "+f"(z.da), "+f"(z.rb), "+f"(z.db));
}

__device__ __forceinline__ void sample_counter(const SArgs& a, int s, uint32_t& c2, uint32_t& c3) {
    const long long sid = a.sid0 + s;
    c2 = static_cast<uint32_t>(sid);
    c3 = a.tag | ((static_cast<uint32_t>(static_cast<unsigned long long>(sid) >> 32) & 0xffffu) << 16);
}

}  // namespace

// Initial state.
__global__ void __launch_bounds__(kThreads) stream_init_kernel(const SArgs a) {
    const int s = blockIdx.y;
    if (s >= a.count) return;
    const int tpr = a.n / kTile;
    const int T1 = blockIdx.x / tpr, T2 = blockIdx.x % tpr;
    const int tx = threadIdx.x % kTc, ty = threadIdx.x / kTc;
    const int I = T1 * kTc + ty, J = T2 * kTc + tx;            // coarse cell
    const int r0 = 2 * I, c0 = 2 * J;
    const size_t base = (size_t)s * a.n * a.n;
#pragma unroll
    for (int i = 0; i < 2; ++i)
        *reinterpret_cast<int2*>(a.q[0] + base + (size_t)(r0 + i) * a.n + c0) =
            *reinterpret_cast<const int2*>(a.q0f + (size_t)(r0 + i) * a.n + c0);
    if (a.coupled) a.qc[0][(size_t)s * a.nc * a.nc + (size_t)I * a.nc + J] = a.q0c[(size_t)I * a.nc + J];
}

// Loads of the state: through L1 (one launch per step: kernel boundaries
// order every access), or from L2 only (persistent launch: tiles of other
// CTAs change between this CTA's items).
template <bool CG, typename T>
__device__ __forceinline__ T ldg(const T* p) {
    if constexpr (CG) return __ldcg(p);
    else return *p;
}

// Four words of shared memory.
__device__ __forceinline__ void ld4(int32_t (&v)[4], const int32_t* p) {
    const int4 x = *reinterpret_cast<const int4*>(p);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
}

// Fine step m of the FR x 64 tile at (R0, C0) of sample s: noise of step m on
// the tile and its halo, then q^{m+1}.  Thread (tx, ty) of the 16 x FR/2
// threads owns the 2 x 4 fine block at (R0 + 2 ty, C0 + 4 tx) = 2 coarse cells.
// The barrier between the shared-memory writes and reads also decides, in the
// persistent kernel, whether any warp's wait timed out (`stop`): then no thread
// stores and the function returns true.
// With PDL (one launch per step, launched as a programmatic dependent of the
// previous kernel in the stream) the normals of the tile and its halo, which
// depend on no state, are drawn before the wait for the previous step: CTAs
// that start while the previous step's last wave still runs do that part of
// their work in its shadow.
template <int FR, bool PERSIST, bool PDL = false>
__device__ __forceinline__ bool fine_tile(const SArgs& a, int s, int R0, int C0, int m, int32_t* smem, int stop) {
    constexpr int kHaloPairs = 64 + 2 * FR;   // 2 x 32 pairs in the halo rows, one per row in the halo columns
    static_assert(!(PDL && PERSIST), "the persistent launch has no previous grid to wait for");
    static_assert(kHaloPairs <= fine_threads(FR), "one halo pair per thread");
    const int n = a.n;
    const int t = threadIdx.x;
    const int tx = t % 16, ty = t / 16;
    const int r0 = R0 + 2 * ty, c0 = C0 + 4 * tx;
    const size_t base = (size_t)s * n * n;
    const int32_t* qin = a.q[m & 1] + base;
    int32_t* qout = a.q[(m + 1) & 1] + base;
    uint32_t c2, c3;
    sample_counter(a, s, c2, c3);
    // halo cell pair of this thread (t < kHaloPairs): row halo (t < 64, whole
    // warps) or column halo
    const bool has_halo = t < kHaloPairs, row_halo = t < 64;
    int hr = 0, hc = 0;
    if (has_halo) {
        if (row_halo) {
            hr = wrapi((t >> 5) ? R0 + FR : R0 - 1, n);
            hc = C0 + 2 * (t & 31);
        } else {
            const int u = t - 64;
            hr = R0 + u % FR;
            hc = wrapi(u / FR ? C0 + kFC : C0 - 2, n);
        }
    }
    const uint32_t hp = static_cast<uint32_t>((hr * n + hc) >> 1);
    RowNormals w[2];
    HaloNormals hw{};
    if constexpr (PDL) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint32_t p = static_cast<uint32_t>(((r0 + i) * n + c0) >> 1);
            w[i] = row_normals(pair_words(a, p, m, c2, c3), pair_words(a, p + 1, m, c2, c3));
        }
        if (has_halo) hw = halo_normals(pair_words(a, hp, m, c2, c3), row_halo);
#pragma unroll
        for (int i = 0; i < 2; ++i) pin(w[i]);
        pin(hw);
        wait_previous_grid();
    }

    // first rows (q, G1; row FR/2: the row below the tile), last rows (row 0: the
    // row above it), columns left and right of it (q, G2)
    int32_t (*tq)[kFC] = reinterpret_cast<int32_t (*)[kFC]>(smem);
    int32_t (*tg)[kFC] = tq + FR / 2 + 1;
    int32_t (*bq)[kFC] = tg + FR / 2 + 1;
    int32_t (*bg)[kFC] = bq + FR / 2 + 1;
    int2* const sl = reinterpret_cast<int2*>(bg + FR / 2 + 1);   // [FR]
    int2* const sr = sl + FR;                                    // [FR]

    // own 2x4 block: state, normals of step m, transfers; coupled sums of its
    // two coarse cells in the register kernels' order
    int32_t q[2][4], G1[2][4], G2[2][4];
    float4* const zp = reinterpret_cast<float4*>(a.zt[(m >> 2) & 1] + (size_t)s * a.nc * a.nc +
                                                 (size_t)(r0 >> 1) * a.nc + (c0 >> 1));
    f32x2 z1 = 0ull, z2 = 0ull;
    if (a.coupled && (m & 3) != 0) {
        const float4 v = ldg<PERSIST>(zp);
        z1 = pack2(v.x, v.z);
        z2 = pack2(v.y, v.w);
    }
    const f32x2 gf2 = pack2(a.gf, a.gf);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int4 v = ldg<PERSIST>(reinterpret_cast<const int4*>(qin + (size_t)(r0 + i) * n + c0));
        q[i][0] = v.x; q[i][1] = v.y; q[i][2] = v.z; q[i][3] = v.w;
        if constexpr (!PDL) {
            const uint32_t p = static_cast<uint32_t>(((r0 + i) * n + c0) >> 1);
            w[i] = row_normals(pair_words(a, p, m, c2, c3), pair_words(a, p + 1, m, c2, c3));
        }
        const f32x2 ta = mul2(noise_amp2(v.x, v.z, gf2), w[i].ra), tb = mul2(noise_amp2(v.y, v.w, gf2), w[i].rb);
        const f32x2 a1 = mul2(ta, w[i].ca), a2 = mul2(ta, w[i].sa), b1 = mul2(tb, w[i].cb), b2 = mul2(tb, w[i].sb);
        G1[i][0] = __float2int_rn(lo2(a1)); G1[i][1] = __float2int_rn(lo2(b1));
        G1[i][2] = __float2int_rn(hi2(a1)); G1[i][3] = __float2int_rn(hi2(b1));
        G2[i][0] = __float2int_rn(lo2(a2)); G2[i][1] = __float2int_rn(lo2(b2));
        G2[i][2] = __float2int_rn(hi2(a2)); G2[i][3] = __float2int_rn(hi2(b2));
        z1 = fma2(w[i].rb, w[i].cb, fma2(w[i].ra, w[i].ca, z1));
        z2 = fma2(w[i].rb, w[i].sb, fma2(w[i].ra, w[i].sa, z2));
    }
    // halo: rows R0-1 and R0+FR (32 pairs each, both cells, component 1) and
    // columns C0-1 and C0+kFC (one pair per row, the cell next to the tile,
    // component 2)
    int2 hv = make_int2(0, 0), hg = make_int2(0, 0);
    if (has_halo) {
        hv = ldg<PERSIST>(reinterpret_cast<const int2*>(qin + (size_t)hr * n + hc));
        if constexpr (!PDL) hw = halo_normals(pair_words(a, hp, m, c2, c3), row_halo);
        hg.x = __float2int_rn(noise_amp(hv.x, a.gf) * hw.ra * hw.da);
        hg.y = __float2int_rn(noise_amp(hv.y, a.gf) * hw.rb * hw.db);
    }
    // in the persistent kernel shared memory is free once every warp has finished the previous item
    if constexpr (PERSIST) __syncthreads();
    *reinterpret_cast<int4*>(&tq[ty][4 * tx]) = make_int4(q[0][0], q[0][1], q[0][2], q[0][3]);
    *reinterpret_cast<int4*>(&tg[ty][4 * tx]) = make_int4(G1[0][0], G1[0][1], G1[0][2], G1[0][3]);
    *reinterpret_cast<int4*>(&bq[ty + 1][4 * tx]) = make_int4(q[1][0], q[1][1], q[1][2], q[1][3]);
    *reinterpret_cast<int4*>(&bg[ty + 1][4 * tx]) = make_int4(G1[1][0], G1[1][1], G1[1][2], G1[1][3]);
    if (has_halo) {
        if (row_halo) {
            const bool above = t < 32;
            *reinterpret_cast<int2*>((above ? bq[0] : tq[FR / 2]) + 2 * (t & 31)) = hv;
            *reinterpret_cast<int2*>((above ? bg[0] : tg[FR / 2]) + 2 * (t & 31)) = hg;
        } else {
            const int u = t - 64;
            if (u < FR) sl[u] = make_int2(hv.y, hg.y);
            else sr[u - FR] = make_int2(hv.x, hg.x);
        }
    }
    // columns: the neighbouring lanes of the 16-lane thread row
    int32_t ql[2], qr[2], gl[2], gr[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        ql[i] = __shfl_up_sync(0xffffffffu, q[i][3], 1, 16);
        gl[i] = __shfl_up_sync(0xffffffffu, G2[i][3], 1, 16);
        qr[i] = __shfl_down_sync(0xffffffffu, q[i][0], 1, 16);
        gr[i] = __shfl_down_sync(0xffffffffu, G2[i][0], 1, 16);
    }
    if constexpr (PERSIST) {
        if (__syncthreads_or(stop)) return true;
    } else {
        __syncthreads();
    }

    if (tx == 0) {
        const int4 v = *reinterpret_cast<const int4*>(sl + 2 * ty);
        ql[0] = v.x; gl[0] = v.y; ql[1] = v.z; gl[1] = v.w;
    }
    if (tx == 15) {
        const int4 v = *reinterpret_cast<const int4*>(sr + 2 * ty);
        qr[0] = v.x; gr[0] = v.y; qr[1] = v.z; gr[1] = v.w;
    }
    int32_t up[4], dn[4], gu[4], gd[4];
    ld4(up, &bq[ty][4 * tx]);
    ld4(gu, &bg[ty][4 * tx]);
    ld4(dn, &tq[ty + 1][4 * tx]);
    ld4(gd, &tg[ty + 1][4 * tx]);
    // each edge flux once per block, as in the register kernels
    flux_update<2, 4>(q, G1, G2, up, gu, dn, gd, ql, gl, qr, gr, a.Af);
    unsigned bad = 0;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
#pragma unroll
        for (int j = 0; j < 4; ++j) bad |= (static_cast<uint32_t>(q[i][j]) + 0x40000000u) >> 31;
        *reinterpret_cast<int4*>(qout + (size_t)(r0 + i) * n + c0) = make_int4(q[i][0], q[i][1], q[i][2], q[i][3]);
    }
    if (a.coupled) *zp = make_float4(lo2(z1), lo2(z2), hi2(z1), hi2(z2));
    if (bad) atomicOr(a.err, kErrRange);
    return false;
}

// Coarse step cn (after fine step 4 cn + 3) of the 32 x 32 coarse tile
// (T1, T2) of sample s: transfers from qc^cn and the coupled sums on the tile
// and its halo (no corners: the stencil does not use them), then qc^{cn+1}.
// Thread (tx, ty) of the 8 x 32 threads owns four cells of row ty; the 128 halo
// cells belong to the first 128 threads.
template <bool PERSIST>
__device__ __forceinline__ void coarse_tile(const SArgs& a, int s, int T1, int T2, int cn, int32_t* smem) {
    static_assert(kThreads == 8 * kTile && 4 * kTile <= kThreads, "8 x 32 threads, one halo cell each");
    const int nc = a.nc;
    const size_t base = (size_t)s * nc * nc;
    const int32_t* qin = a.qc[cn & 1] + base;
    int32_t* qout = a.qc[(cn + 1) & 1] + base;
    const float2* zt = a.zt[cn & 1] + base;
    int32_t (*tq)[kTile] = reinterpret_cast<int32_t (*)[kTile]>(smem);
    int32_t (*tg)[kTile] = tq + kTile + 1;
    int32_t (*bq)[kTile] = tg + kTile + 1;
    int32_t (*bg)[kTile] = bq + kTile + 1;
    int2* const sl = reinterpret_cast<int2*>(bg + kTile + 1);
    int2* const sr = sl + kTile;
    const int t = threadIdx.x, tx = t % 8, ty = t / 8;
    const int R0 = T1 * kTile, C0 = T2 * kTile;
    const size_t x = (size_t)(R0 + ty) * nc + C0 + 4 * tx;
    const int4 qv = ldg<PERSIST>(reinterpret_cast<const int4*>(qin + x));
    const float4 za = ldg<PERSIST>(reinterpret_cast<const float4*>(zt + x));
    const float4 zb = ldg<PERSIST>(reinterpret_cast<const float4*>(zt + x) + 1);
    int32_t q[1][4] = {{qv.x, qv.y, qv.z, qv.w}}, G1[1][4], G2[1][4];
    const float w1[4] = {za.x, za.z, zb.x, zb.z}, w2[4] = {za.y, za.w, zb.y, zb.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float amp = noise_amp(q[0][j], a.gc);
        G1[0][j] = __float2int_rn(amp * w1[j]);
        G2[0][j] = __float2int_rn(amp * w2[j]);
    }
    // one row: first and last row of the block are the same words
    const int4 g1v = make_int4(G1[0][0], G1[0][1], G1[0][2], G1[0][3]);
    *reinterpret_cast<int4*>(&tq[ty][4 * tx]) = qv;
    *reinterpret_cast<int4*>(&tg[ty][4 * tx]) = g1v;
    *reinterpret_cast<int4*>(&bq[ty + 1][4 * tx]) = qv;
    *reinterpret_cast<int4*>(&bg[ty + 1][4 * tx]) = g1v;
    if (t < 4 * kTile) {
        const int side = t / kTile, k = t % kTile;   // rows above, below; columns left, right
        const int r = side < 2 ? wrapi(side ? R0 + kTile : R0 - 1, nc) : R0 + k;
        const int c = side < 2 ? C0 + k : wrapi(side == 3 ? C0 + kTile : C0 - 1, nc);
        const int32_t v = ldg<PERSIST>(qin + (size_t)r * nc + c);
        const float2 z = ldg<PERSIST>(zt + (size_t)r * nc + c);
        const int32_t g = __float2int_rn(noise_amp(v, a.gc) * (side < 2 ? z.x : z.y));
        if (side == 0) {
            bq[0][k] = v;
            bg[0][k] = g;
        } else if (side == 1) {
            tq[kTile][k] = v;
            tg[kTile][k] = g;
        } else {
            (side == 2 ? sl : sr)[k] = make_int2(v, g);
        }
    }
    int32_t ql[1] = {__shfl_up_sync(0xffffffffu, q[0][3], 1, 8)}, gl[1] = {__shfl_up_sync(0xffffffffu, G2[0][3], 1, 8)};
    int32_t qr[1] = {__shfl_down_sync(0xffffffffu, q[0][0], 1, 8)}, gr[1] = {__shfl_down_sync(0xffffffffu, G2[0][0], 1, 8)};
    __syncthreads();
    if (tx == 0) {
        ql[0] = sl[ty].x;
        gl[0] = sl[ty].y;
    }
    if (tx == 7) {
        qr[0] = sr[ty].x;
        gr[0] = sr[ty].y;
    }
    int32_t up[4], dn[4], gu[4], gd[4];
    ld4(up, &bq[ty][4 * tx]);
    ld4(gu, &bg[ty][4 * tx]);
    ld4(dn, &tq[ty + 1][4 * tx]);
    ld4(gd, &tg[ty + 1][4 * tx]);
    flux_update<1, 4>(q, G1, G2, up, gu, dn, gd, ql, gl, qr, gr, a.Ac);
    *reinterpret_cast<int4*>(qout + x) = make_int4(q[0][0], q[0][1], q[0][2], q[0][3]);
    unsigned bad = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) bad |= (static_cast<uint32_t>(q[0][j]) + 0x40000000u) >> 31;
    if (bad) atomicOr(a.err, kErrRange);
}

// One launch per fine step m (PDL: launched as a programmatic dependent of the
// previous kernel, which it waits for after drawing its normals).  The CTAs
// past the samples' (blockIdx.z >= count, launched for the first fine step of a
// coarse step but the first) do the coarse step that ended with the previous
// fine step: its state and sums are other buffers than the fine step's, so the
// two share the launch instead of following one another.
template <int FR, int MINB, bool PDL>
__global__ void __launch_bounds__(fine_threads(FR), MINB) stream_fine_kernel(const SArgs a, int m) {
    if constexpr (PDL) launch_dependents();
    extern __shared__ __align__(16) int32_t smem_fine[];
    if (blockIdx.z >= a.count) {
        if constexpr (PDL) wait_previous_grid();
        const int k = ((blockIdx.z - a.count) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        const int tpr = a.nc / kTile, s = k / (tpr * tpr), r = k - s * tpr * tpr;
        if (s < a.count) coarse_tile<false>(a, s, r / tpr, r % tpr, (m >> 2) - 1, smem_fine);
        return;
    }
    fine_tile<FR, false, PDL>(a, blockIdx.z, blockIdx.y * FR, blockIdx.x * kFC, m, smem_fine, 0);
}

// The last coarse step, after the last fine step.
__global__ void __launch_bounds__(kThreads) stream_coarse_kernel(const SArgs a, int cn) {
    const int s = blockIdx.y;
    if (s >= a.count) return;
    __shared__ __align__(16) int32_t smem_coarse[kCoarseWords];
    const int tpr = a.nc / kTile;
    coarse_tile<false>(a, s, blockIdx.x / tpr, blockIdx.x % tpr, cn, smem_coarse);
}

// ---------------------------------------------------------------------------
// Persistent launch: all fine and coarse steps of a wave in one grid of
// resident CTAs.  Work items are taken in a fixed order from a counter:
//   for every coarse step cn: fine steps 4cn .. 4cn+3 (each: every tile of
//   every sample), then the coarse step cn (every coarse tile of every sample)
// (uncoupled: the fine steps only).  An item waits until the items it reads
// from are done, which are always earlier items: a fine tile at step m needs
// itself and its four neighbours at step m (their step m-1 done: q^m written
// and q^{m-1}, which step m overwrites, read); at m = 4cn+4 also the coarse
// tiles whose halo reads its coupled sums done with step cn (the sums that step m
// overwrites, two buffers in turn, are those of coarse step cn-1, so waiting for
// that one would do).  A coarse tile at
// step cn needs the fine tiles under it and its halo done with fine step
// 4cn+3, and itself and its four neighbours done with coarse step cn-1.
// Every earlier item is held by a running CTA, so the waits end; each is
// still bounded (`wait_polls` polls), after which the kernel records
// kErrTimeout, every CTA stops at its next item, and the host reports it.
// Progress: fdone[s][tile] = 8 x fine steps done, cdone[s][ctile] = 8 x coarse
// steps done: each of an item's 8 warps adds 1 with a release after its own
// stores, so no CTA-wide barrier ends an item.  Shared memory is reused only
// after a barrier that follows the next item's noise (every warp is then past
// the previous item's reads).
// ---------------------------------------------------------------------------
constexpr unsigned kItemWarps = fine_threads(kFR) / 32;   // warps of a persistent CTA (also the coarse tiles')
static_assert(fine_threads(kFR) == kThreads, "coarse tiles run on the fine-step CTAs");

struct ItemMap {
    int tr, tc;              // fine tiles per column / row of the grid (n/FR, n/64)
    int ct;                  // coarse tiles per side (nc/32)
    long long F, C, P;       // fine items per step, coarse items per coarse step, items per period
};

__device__ __forceinline__ ItemMap item_map(const SArgs& a, int fr) {
    ItemMap im;
    im.tr = a.n / fr;
    im.tc = a.n / kFC;
    im.ct = a.coupled ? a.nc / kTile : 0;
    im.F = (long long)a.count * im.tr * im.tc;
    im.C = (long long)a.count * im.ct * im.ct;
    im.P = a.coupled ? 4 * im.F + im.C : im.F;
    return im;
}

// Item k -> kind (0 fine, 1 coarse), sample, tile coordinates, step.
struct Item {
    int kind, s, i, j, step;
};

__device__ __forceinline__ Item decode_item(const ItemMap& im, long long k, bool coupled) {
    Item it;
    const long long p = k / im.P, r = k - p * im.P;
    if (!coupled || r < 4 * im.F) {
        const long long q = coupled ? r / im.F : 0, f = coupled ? r - q * im.F : r;
        it.kind = 0;
        it.step = coupled ? (int)(4 * p + q) : (int)p;
        const long long per = (long long)im.tr * im.tc;
        it.s = (int)(f / per);
        const int t = (int)(f - it.s * per);
        it.i = t / im.tc;
        it.j = t - it.i * im.tc;
    } else {
        const long long c = r - 4 * im.F, per = (long long)im.ct * im.ct;
        it.kind = 1;
        it.step = (int)p;
        it.s = (int)(c / per);
        const int t = (int)(c - it.s * per);
        it.i = t / im.ct;
        it.j = t - it.i * im.ct;
    }
    return it;
}

__device__ __forceinline__ int wrapt(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

// Dependency d (0 .. 12) of an item: the counter to read and the value it must
// reach; false when the item has fewer dependencies.  Fine tiles are FR = 32
// rows high, so fine tile rows 2I and 2I+1 lie under coarse tile row I.
__device__ __forceinline__ bool item_dep(const SArgs& a, const ItemMap& im, const Item& it, int d,
                                         const unsigned*& ptr, unsigned& target) {
    const unsigned* fd = a.fdone + (size_t)it.s * im.tr * im.tc;
    const unsigned* cd = a.cdone + (size_t)it.s * im.ct * im.ct;
    if (it.kind == 0) {
        if (d < 5) {
            const int di = d == 1 ? -1 : (d == 2 ? 1 : 0), dj = d == 3 ? -1 : (d == 4 ? 1 : 0);
            ptr = fd + (size_t)wrapt(it.i + di, im.tr) * im.tc + wrapt(it.j + dj, im.tc);
            target = kItemWarps * (unsigned)it.step;
            return true;
        }
        if (!a.coupled || it.step < 4 || (it.step & 3) != 0 || d >= 9) return false;
        const int I = it.i >> 1, J = it.j;
        int ci = I, cj = J;
        if (d == 6) cj = wrapt(J - 1, im.ct);
        else if (d == 7) cj = wrapt(J + 1, im.ct);
        else if (d == 8) ci = wrapt((it.i & 1) ? I + 1 : I - 1, im.ct);
        ptr = cd + (size_t)ci * im.ct + cj;
        target = kItemWarps * (unsigned)(it.step >> 2);
        return true;
    }
    if (d < 8) {
        // fine tiles: rows 2I-1 .. 2I+2 in column J (d = 0..3), rows 2I, 2I+1
        // in column J-1 (d = 4, 5) and in column J+1 (d = 6, 7)
        const int dr = d < 4 ? d - 1 : (d & 1), dc = d < 4 ? 0 : (d < 6 ? -1 : 1);
        ptr = fd + (size_t)wrapt(2 * it.i + dr, im.tr) * im.tc + wrapt(it.j + dc, im.tc);
        target = kItemWarps * (unsigned)(4 * it.step + 4);
        return true;
    }
    if (d < 13) {
        const int e = d - 8;
        const int di = e == 1 ? -1 : (e == 2 ? 1 : 0), dj = e == 3 ? -1 : (e == 4 ? 1 : 0);
        ptr = cd + (size_t)wrapt(it.i + di, im.ct) * im.ct + wrapt(it.j + dj, im.ct);
        target = kItemWarps * (unsigned)it.step;
        return true;
    }
    return false;
}

template <int FR, int MINB>
__global__ void __launch_bounds__(fine_threads(FR), MINB) stream_persist_kernel(const SArgs a) {
    static_assert(FR == 32, "coarse tiles cover two fine tile rows");
    extern __shared__ __align__(16) int32_t smem_fine[];
    __shared__ long long s_item[2];
    const ItemMap im = item_map(a, FR);
    const long long total = a.coupled ? (long long)(a.M / 4) * im.P : (long long)a.M * im.P;
    const int lane = threadIdx.x & 31;
    // the last thread takes items from the counter: its warp has no halo
    // cells, so the atomic's latency falls where that warp waits anyway
    const bool taker = threadIdx.x == blockDim.x - 1;
    if (taker) s_item[0] = (long long)atomicAdd(a.head, 1ull);
    __syncthreads();
    for (int iter = 0;; ++iter) {
        const long long k = s_item[iter & 1];
        if (k >= total) break;
        // the next item, taken now so that its latency hides behind this one
        if (taker) {
            const long long nk = (long long)atomicAdd(a.head, 1ull);
            const unsigned err = ld_volatile(a.err);
            s_item[(iter + 1) & 1] = (err & kErrTimeout) ? total : nk;
        }
        const Item it = decode_item(im, k, a.coupled != 0);
        // every warp waits for the item's dependencies itself (lane d polls
        // dependency d), so its loads are ordered after the acquires
        int stop = 0;
        {
            const unsigned* ptr = nullptr;
            unsigned target = 0;
            bool ok = true;
            if (item_dep(a, im, it, lane, ptr, target)) {
                ok = false;
                for (unsigned poll = 0; poll < a.wait_polls; ++poll) {
                    if (static_cast<int>(ld_acquire(ptr) - target) >= 0) {
                        ok = true;
                        break;
                    }
                    if ((poll & 63u) == 63u && (ld_volatile(a.err) & kErrTimeout)) break;
                    __nanosleep(64);
                }
                if (!ok) atomicOr(a.err, kErrTimeout);
            }
            stop = __any_sync(0xffffffffu, !ok) ? 1 : 0;
            __syncwarp();
        }
        if (it.kind == 0) {
            if (fine_tile<FR, true>(a, it.s, it.i * FR, it.j * kFC, it.step, smem_fine, stop)) break;
        } else {
            if (__syncthreads_or(stop)) break;   // also frees shared memory
            coarse_tile<true>(a, it.s, it.i, it.j, it.step, smem_fine);
        }
        // this warp's stores are done: report them (the failure-detection test
        // withholds step 1 of one tile of sample 0)
        __syncwarp();
        const bool stall = it.kind == 0 && a.stall_tile >= 0 && it.step == 1 && it.s == 0 &&
                           it.i * im.tc + it.j == a.stall_tile;
        if (lane == 0 && !stall) {
            unsigned* ctr = it.kind == 0 ? a.fdone + (size_t)it.s * im.tr * im.tc + (size_t)it.i * im.tc + it.j
                                         : a.cdone + (size_t)it.s * im.ct * im.ct + (size_t)it.i * im.ct + it.j;
            red_release_add(ctr, 1u);
        }
    }
}

// Per-tile partial observables: sums of (q - qbar) phi_k (fine, coarse), masses.
__global__ void __launch_bounds__(kThreads) stream_observe_kernel(const SArgs a) {
    const int s = blockIdx.y;
    if (s >= a.count) return;
    const int n = a.n, nc = a.nc;
    const int tpr = n / kTile;
    const int T1 = blockIdx.x / tpr, T2 = blockIdx.x % tpr;
    const int tx = threadIdx.x % kTc, ty = threadIdx.x / kTc;
    const int I = T1 * kTc + ty, J = T2 * kTc + tx;
    const int r0 = 2 * I, c0 = 2 * J;
    const int32_t* q = a.q[a.M & 1] + (size_t)s * n * n;
    double v[2 * kMaxObs + 2];
#pragma unroll
    for (int i = 0; i < 2 * kMaxObs + 2; ++i) v[i] = 0.0;
    long long mf = 0, mc = 0;
    // FP64 products and sums against FP64 test functions (the integer
    // fluctuations are exact in FP64): the projection of a rough fluctuation on
    // a smooth phi is small, and FP32 rounding of phi or of the partial sums,
    // uncorrelated with the noise, would reach 1e-5 of it on fine grids
    double sf[kMaxObs] = {0.0, 0.0, 0.0, 0.0}, sc[kMaxObs] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const size_t x = (size_t)(r0 + i) * n + c0 + j;
            const int32_t qv = q[x];
            mf += qv;
            for (int k = 0; k < a.n_obs; ++k)
                sf[k] = fma(static_cast<double>(qv - a.qbf[x]), a.phif64[(size_t)k * n * n + x], sf[k]);
        }
    if (a.coupled) {
        const size_t xc = (size_t)I * nc + J;
        const int32_t qv = a.qc[(a.M >> 2) & 1][(size_t)s * nc * nc + xc];
        mc = qv;
        for (int k = 0; k < a.n_obs; ++k)
            sc[k] = static_cast<double>(qv - a.qbc[xc]) * a.phic64[(size_t)k * nc * nc + xc];
    }
#pragma unroll
    for (int k = 0; k < kMaxObs; ++k) {
        v[k] = sf[k];
        v[kMaxObs + k] = sc[k];
    }
    v[2 * kMaxObs] = static_cast<double>(mf);
    v[2 * kMaxObs + 1] = static_cast<double>(mc);
    // block reduction in a fixed order: warp shuffles, then warp 0
    __shared__ double red[kThreads / 32][2 * kMaxObs + 2];
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1)
#pragma unroll
        for (int i = 0; i < 2 * kMaxObs + 2; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], off);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < 2 * kMaxObs + 2; ++i) red[w][i] = v[i];
    __syncthreads();
    if (threadIdx.x < 2 * kMaxObs + 2) {
        double t = 0.0;
        for (int ww = 0; ww < kThreads / 32; ++ww) t += red[ww][threadIdx.x];
        const int tiles = gridDim.x;
        a.tile_part[((size_t)s * tiles + blockIdx.x) * (2 * kMaxObs + 2) + threadIdx.x] = t;
    }
}

// Per sample: tiles reduced in order, then the FP64 quantities and moment sums
// of the sample added to its slot (slot = position in the wave).
__global__ void stream_finish_kernel(const SArgs a, const KArgs k, int tiles, int n_slots) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= a.count) return;
    constexpr int W = 2 * kMaxObs + 2;
    double v[W];
    for (int i = 0; i < W; ++i) v[i] = 0.0;
    for (int t = 0; t < tiles; ++t)
        for (int i = 0; i < W; ++i) v[i] += a.tile_part[((size_t)s * tiles + t) * W + i];
    double Df[kMaxObs], Dc[kMaxObs];
    for (int q = 0; q < kMaxObs; ++q) {
        Df[q] = k.dscale_f * v[q] + k.delta_f[q];
        Dc[q] = a.coupled ? k.dscale_c * v[kMaxObs + q] + k.delta_c[q] : 0.0;
    }
    // entry-major slot partials: partials[e * n_slots + s]
    auto P = [&](int e) -> double& { return k.partials[(size_t)e * n_slots + s]; };
    P(0) += 1.0;
    double merr = fabs(v[2 * kMaxObs] - static_cast<double>(k.mass0_f)) * k.dscale_f;
    if (a.coupled) merr = fmax(merr, fabs(v[2 * kMaxObs + 1] - static_cast<double>(k.mass0_c)) * k.dscale_c);
    P(1) = fmax(P(1), merr);
    int qi = 0;
    for (int j = 0; j < k.n_obs; ++j) {
        const int kend = k.products ? k.n_obs : j + 1;
        for (int l = j; l < kend; ++l, ++qi) {
            const double pf = k.N * Df[j] * Df[l];
            const double pc = a.coupled ? k.N * Dc[j] * Dc[l] : 0.0;
            const double dp = pf - pc, dp2 = dp * dp;
            const int b = 2 + kNSum * qi;
            P(b + 0) += dp; P(b + 1) += dp2; P(b + 2) += dp2 * dp; P(b + 3) += dp2 * dp2;
            P(b + 4) += pf; P(b + 5) += pf * pf; P(b + 6) += pc; P(b + 7) += pc * pc;
            P(b + 8) += Df[j]; P(b + 9) += Df[j] * Df[j]; P(b + 10) += Dc[j]; P(b + 11) += Dc[j] * Dc[j];
        }
    }
    if (k.samples) {
        double* o = k.samples + (a.sid0 - k.first + s) * (2 * k.n_obs + 2);
        for (int q = 0; q < k.n_obs; ++q) {
            o[q] = Df[q];
            o[k.n_obs + q] = Dc[q];
        }
        o[2 * k.n_obs] = v[2 * kMaxObs] * k.dscale_f;
        o[2 * k.n_obs + 1] = a.coupled ? v[2 * kMaxObs + 1] * k.dscale_c : 0.0;
    }
}

__global__ void zero_kernel(double* p, size_t count) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
        p[i] = 0.0;
}

// Progress counters of the persistent launch: fdone [S][fine tiles], cdone
// [S][coarse tiles], then the item counter (8 bytes).
static size_t counter_bytes(int n, int S) {
    const size_t ft = (size_t)(n / kFR) * (n / kFC), ct = (size_t)(n / 2 / kTile) * (n / 2 / kTile);
    return (((size_t)S * (ft + ct) * sizeof(unsigned) + 15) & ~(size_t)15) + 16;
}

// Bytes that the steps of one sample work on: of the two buffers of coupled
// sums, one at a time.
static size_t sample_working_set(int n) {
    const size_t nc = n / 2, tiles = (size_t)(n / kTile) * (n / kTile);
    return (size_t)n * n * 2 * sizeof(int32_t) + nc * nc * (2 * sizeof(int32_t) + sizeof(float2)) +
           tiles * (2 * kMaxObs + 2) * sizeof(double) + counter_bytes(n, 1);
}

size_t stream_bytes(int n, int S) {
    const size_t nc = n / 2, tiles = (size_t)(n / kTile) * (n / kTile);
    return (size_t)S * ((size_t)n * n * 2 * sizeof(int32_t) + nc * nc * 2 * (sizeof(int32_t) + sizeof(float2)) +
                        tiles * (2 * kMaxObs + 2) * sizeof(double)) +
           counter_bytes(n, S);
}

int stream_variant_count() { return kStreamVariants; }
int stream_default_variant() { return 4; }   // one programmatic dependent launch per step, 4 CTAs per SM

// Variants: 0, 1 one launch per step, 2, 3 the persistent launch, 4, 5 one
// launch per step as programmatic dependent launches; even: at most 64
// registers per thread (4 resident CTAs per SM), odd: 48 (5 CTAs).
static bool persistent_variant(int variant) { return variant == 2 || variant == 3; }
static bool pdl_variant(int variant) { return variant >= 4; }

template <typename K>
static cudaError_t fine_attr_occ(K kernel, int* per_sm) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, fine_smem(kFR));
    if (e != cudaSuccess) return e;
    return per_sm ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kernel, fine_threads(kFR), fine_smem(kFR))
                  : cudaSuccess;
}

static cudaError_t fine_attr(int variant, int* per_sm = nullptr) {
    switch (variant) {
        case 0: return fine_attr_occ(stream_fine_kernel<kFR, 4, false>, per_sm);
        case 1: return fine_attr_occ(stream_fine_kernel<kFR, 5, false>, per_sm);
        case 2: return fine_attr_occ(stream_persist_kernel<kFR, 4>, per_sm);
        case 3: return fine_attr_occ(stream_persist_kernel<kFR, 5>, per_sm);
        case 4: return fine_attr_occ(stream_fine_kernel<kFR, 4, true>, per_sm);
        case 5: return fine_attr_occ(stream_fine_kernel<kFR, 5, true>, per_sm);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t stream_variant_info(int n, int variant, VariantInfo* out) {
    if (variant < 0 || variant >= kStreamVariants) return cudaErrorInvalidValue;
    const int fr = kFR;
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e;
    if ((e = fine_attr(variant, &per_sm)) != cudaSuccess) return e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return e;
    *out = VariantInfo{};
    out->supported = (n % kFC == 0 && n % fr == 0 && per_sm > 0) ? 1 : 0;
    out->threads = fine_threads(fr);
    out->cluster = 1;
    out->slots_per_cta = 0;
    out->smem = fine_smem(fr);
    out->max_ctas = sms * per_sm;
    out->C = 2;        // coarse cells per thread along a row
    out->R = 1;
    out->tile_rows = fr;
    out->persistent = persistent_variant(variant) ? 1 : 0;
    out->pdl = pdl_variant(variant) ? 1 : 0;
    return cudaSuccess;
}

int stream_inflight(int n, size_t budget, int variant) {
    // the largest count that fits the budget, lowered while a smaller count
    // fills the last wave of fine-step CTAs clearly better
    const int s_max = (int)std::max<size_t>(1, budget / sample_working_set(n));
    VariantInfo vi{};
    if (stream_variant_info(n, variant, &vi) != cudaSuccess || !vi.supported) return s_max;
    const long long resident = vi.max_ctas, ctas = (long long)(n / kFC) * (n / vi.tile_rows);
    if (vi.persistent) return s_max;   // no waves: CTAs take tiles as they free up
    int best = s_max;
    double best_eff = 0.0;
    for (int S = s_max; S >= std::max(1, s_max / 2); --S) {
        const long long c = S * ctas, waves = (c + resident - 1) / resident;
        const double eff = (double)c / (double)(waves * resident);
        if (eff > best_eff + 0.01) {
            best = S;
            best_eff = eff;
        }
    }
    return best;
}

void stream_carve(SArgs* a, void* buf, int n, int S) {
    unsigned char* p = static_cast<unsigned char*>(buf);
    const size_t cf = (size_t)S * n * n, cc = (size_t)S * (n / 2) * (n / 2);
    a->q[0] = reinterpret_cast<int32_t*>(p); p += cf * sizeof(int32_t);
    a->q[1] = reinterpret_cast<int32_t*>(p); p += cf * sizeof(int32_t);
    a->qc[0] = reinterpret_cast<int32_t*>(p); p += cc * sizeof(int32_t);
    a->qc[1] = reinterpret_cast<int32_t*>(p); p += cc * sizeof(int32_t);
    a->zt[0] = reinterpret_cast<float2*>(p); p += cc * sizeof(float2);
    a->zt[1] = reinterpret_cast<float2*>(p); p += cc * sizeof(float2);
    a->tile_part = reinterpret_cast<double*>(p);
    p += (size_t)S * (n / kTile) * (n / kTile) * (2 * kMaxObs + 2) * sizeof(double);
    a->counters = p;
    a->counter_bytes = counter_bytes(n, S);
    const size_t ft = (size_t)(n / kFR) * (n / kFC);
    a->fdone = reinterpret_cast<unsigned*>(p);
    a->cdone = a->fdone + (size_t)S * ft;
    a->head = reinterpret_cast<unsigned long long*>(p + a->counter_bytes - 16);
}

cudaError_t stream_run(const KArgs& k, SArgs a, int S, int variant, cudaStream_t st) {
    // k.partials holds S slots (entry-major, [stride][S]); zero them, run the
    // waves of S samples, accumulate per slot, then the caller reduces.
    const int n = a.n;
    if (variant < 0 || variant >= kStreamVariants) return cudaErrorInvalidValue;
    const int fr = kFR;
    if (n % kFC != 0 || n % fr != 0 || (a.coupled && (a.nc % kTile != 0 || a.M % 4 != 0))) return cudaErrorInvalidValue;
    const int tiles = (n / kTile) * (n / kTile);
    const int ctiles = a.coupled ? (a.nc / kTile) * (a.nc / kTile) : 0;
    int per_sm = 0, dev = 0, sms = 0;
    cudaError_t e = fine_attr(variant, &per_sm);
    if (e != cudaSuccess) return e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    if (a.wait_polls == 0) a.wait_polls = 1u << 24;
    zero_kernel<<<64, 256, 0, st>>>(k.partials, (size_t)k.slot_stride * S);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    for (long long done = 0; done < k.count; done += S) {
        a.sid0 = k.first + done;
        a.count = (int)std::min<long long>(S, k.count - done);
        const dim3 grid(tiles, a.count), cgrid(ctiles, a.count);
        // CTAs of fine step m: the samples' fine tiles, and after them the coarse
        // tiles of the coarse step that ended before it
        const int ftiles = (n / kFC) * (n / fr);
        auto step_grid = [&](int m) {
            const int extra = a.coupled && m > 0 && (m & 3) == 0 ? (int)((a.count * (long long)ctiles + ftiles - 1) / ftiles) : 0;
            return dim3(n / kFC, n / fr, a.count + extra);
        };
        stream_init_kernel<<<grid, kThreads, 0, st>>>(a);
        if (persistent_variant(variant)) {
            // one grid of resident CTAs (at most one per item) takes the items in order
            if ((e = cudaMemsetAsync(a.counters, 0, a.counter_bytes, st)) != cudaSuccess) return e;
            const long long items = (long long)a.count * (n / fr) * (n / kFC) * a.M +
                                    (a.coupled ? (long long)a.count * ctiles * (a.M / 4) : 0);
            const int ctas = (int)std::min<long long>((long long)sms * per_sm, items);
            if (variant == 2)
                stream_persist_kernel<kFR, 4><<<ctas, fine_threads(kFR), fine_smem(kFR), st>>>(a);
            else
                stream_persist_kernel<kFR, 5><<<ctas, fine_threads(kFR), fine_smem(kFR), st>>>(a);
        } else if (pdl_variant(variant)) {
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[0].val.programmaticStreamSerializationAllowed = 1;
            cudaLaunchConfig_t cfg{};
            cfg.blockDim = dim3(fine_threads(kFR));
            cfg.dynamicSmemBytes = fine_smem(kFR);
            cfg.stream = st;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            for (int m = 0; m < a.M; ++m) {
                cfg.gridDim = step_grid(m);
                e = variant == 4 ? cudaLaunchKernelEx(&cfg, stream_fine_kernel<kFR, 4, true>, a, m)
                                 : cudaLaunchKernelEx(&cfg, stream_fine_kernel<kFR, 5, true>, a, m);
                if (e != cudaSuccess) return e;
            }
        } else {
            for (int m = 0; m < a.M; ++m) {
                if (variant == 0)
                    stream_fine_kernel<kFR, 4, false><<<step_grid(m), fine_threads(kFR), fine_smem(kFR), st>>>(a, m);
                else
                    stream_fine_kernel<kFR, 5, false><<<step_grid(m), fine_threads(kFR), fine_smem(kFR), st>>>(a, m);
            }
        }
        if (a.coupled && !persistent_variant(variant))
            stream_coarse_kernel<<<cgrid, kThreads, 0, st>>>(a, (a.M >> 2) - 1);
        stream_observe_kernel<<<grid, kThreads, 0, st>>>(a);
        stream_finish_kernel<<<(a.count + 63) / 64, 64, 0, st>>>(a, k, tiles, S);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace dk
