// 3D temporally-blocked Jacobi sweep, contracted arithmetic, partial sums along z.
//
// Method (arXiv 1802.00438): 2D spatial blocking in x and y with streaming along z (Sec. 3.1),
// overlapped tiles with halos of width >= rad*T (Eq. 2), a chain of T stages where stage s
// computes time step s+1 (Sec. 3.2), redundant halo computation with only the compute block
// written (Sec. 3.2), trailing stages forwarding when a pass fuses fewer than T steps (Sec. 3.2),
// clamped boundaries at every stage (Sec. 5.1).
//
// GPU mapping: tile 32*VX x NW*VY cells incl. halos; a thread owns VX adjacent x cells of VY
// consecutive rows, a warp spans the tile's width, warps are stacked along y.
//   A stage keeps two partial sums per cell instead of a three-plane window: when plane z of its
//   input (time s) arrives it
//     finishes output plane z-1:   out = P + ca*d
//     starts   output plane z:     P   = Q + cc*d + cw*w + ce*e + cs*s + cn*n (+ sdc*p(z))
//     starts   output plane z+1:   Q   = cb*d (+ ca*amb)
//   Stage s works two planes behind stage s-1: the plane a stage emits in one iteration is the
//   next stage's input in the next one.  So the T stages of an iteration are independent of each
//   other (their shuffles, loads and multiply-adds interleave), and the rows above and below a
//   warp's rows, which come from its neighbour warps through a shared-memory exchange
//   (alternating buffers), need ONE barrier per plane for all stages together instead of one
//   per stage; a segment pays T-1 more iterations to drain.
//   Arithmetic is on packed float32 pairs (fma.rn.f32x2): a packed operation holds the FMA pipe
//   for two cycles but takes one issue slot, and issue is what bounds these kernels.  A pair is
//   cells p and p + VX/2 of a row (VX = 2: the two adjacent cells): its west and east neighbours
//   are the pairs p-1 and p+1, only the outermost pairs mix halves; its y and z neighbours are
//   pairs as they lie, and with VX = 2 loads, stores and the exchange move whole pairs.
//   Clamped z boundaries: at z = 0 the missing plane z-1 is plane 0 itself (Q is started from
//   d before it is used); on arrival of plane nz-1 a stage completes P with ca*d (the missing
//   plane nz is plane nz-1), and emits it unchanged one iteration later.
//   Tile columns of one pass are streamed in step (see segments.h).
//   Measured (GB300), kernel with one barrier per stage and scalar arithmetic -> this one: 512^3
//   diffusion 1022 -> 1330 GCell/s, 512^2 x 256 Hotspot 837 -> 1033, 187 x 141 x 93 diffusion 172
//   -> 304.  What bounds it now (ncu, 512^2 x 256, T = 3): issue 57 % active with 275
//   instructions per thread and plane (115 of them multiply-adds, the other half shuffles,
//   exchange, ring and store addressing), FMA pipe 41 %, shared memory 50 %, DRAM 3.2 TB/s; the
//   warps run the shuffle phase and the multiply-add phase of a plane together.  Tried and not
//   kept: neighbour flags instead of the barrier (1054 against 1265 at the time: polling costs
//   more than the barrier's wait), 16 cells per thread in 8 warps (1172 against 1287).
//   Input planes arrive in a shared-memory ring, PF planes ahead; every stage reads its power
//   plane from a second ring (Hotspot 3D), so each value is read from HBM once per pass.
#pragma once
#include <type_traits>
#include "common.cuh"
#include "internal.h"

namespace stn {

template <int KIND, int T, int VX, int VY, int NW>
struct TB3F {
    static constexpr int NT = 32 * NW;
    static constexpr int BX = 32 * VX;
    static constexpr int BY = NW * VY;
    static constexpr int H = VX / 2;             // pairs per row of a thread
    static constexpr int HX = (T + 3) / 4 * 4;   // 16-byte aligned tile origins
    static constexpr int HY = T;
    static constexpr int CX = BX - 2 * HX;
    static constexpr int CY = BY - 2 * HY;
    static constexpr int PLANE = BX * BY;
    static constexpr uint32_t PLANE_B = 4u * PLANE;
    static constexpr uint32_t ROWB = 4u * BX;
    // exchange of stages 1 .. T-1: [buffer][stage][2*NW + 2 rows], warp w's top row at 2w + 1,
    // its bottom row at 2w + 2 (the outermost rows are never written: they only feed halo rows)
    static constexpr uint32_t XROWS = 2 * NW + 2;
    static constexpr uint32_t XSTAGE = XROWS * ROWB;
    static constexpr uint32_t XBUF = (T - 1) * XSTAGE;
    // power planes an iteration reads: stage s reads plane Z0 - 2s
    static constexpr int PWIN = 2 * T - 1;
    // shared memory with PF planes in flight and xb exchange buffers: one row of padding at
    // either end (a tile's first row looks one row up, its last row one row down), the field
    // ring, the power ring, the exchange, one mbarrier per field slot
    static constexpr size_t smem_for(int pf, int xb)
    {
        return 2 * ROWB + (size_t)((pf + 1) + (KIND == KTHERM ? PWIN + pf : 0)) * PLANE_B +
               (size_t)xb * XBUF + 8 * (pf + 1);
    }
    // blocks of up to 8 warps run two per SM, larger ones one
    static constexpr int MINB = NT <= 256 ? 2 : 1;
    // (1 KiB of each block's share is reserved by the hardware)
    static constexpr size_t BUDGET = MINB == 2 ? 113 * 1024 : 227 * 1024;
    // alternating exchange buffers where they fit with at least one plane in flight, else one
    // buffer and a second barrier per plane; then the deepest prefetch (up to 4 planes) that fits
    static constexpr int XB = smem_for(1, 2) <= BUDGET ? 2 : 1;
    static constexpr int PF = smem_for(4, XB) <= BUDGET ? 4 : smem_for(3, XB) <= BUDGET ? 3
                            : smem_for(2, XB) <= BUDGET ? 2 : 1;
    static constexpr int NBF = PF + 1;
    static constexpr int NBP = KIND == KTHERM ? PWIN + PF : 0;
    static constexpr size_t SMEM = smem_for(PF, XB);
    static_assert(CX > 0 && CY > 0, "tile smaller than its halos");
    static_assert(VX == 2 || VX == 4, "cells per lane");
    static_assert(VX * VY <= 32, "store mask");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

// Per-thread context of one tile column.
struct CtxF3 {
    const float *__restrict__ in;
    float *__restrict__ out;
    const float *__restrict__ pw;
    int nx, ny, nz, tsteps, vec, vec_pw;
    long long ld_in, ld_out, ld_pw;           // row pitches, floats
    long long plane_in, plane_out, plane_pw;  // plane pitches, floats
    int x0, y0;            // tile origin
    int gx, gy;            // my first cell
    int z_start, last_plane, z0, z1;
    bool edge_y;           // warp touches a domain edge in y
    bool lx0;              // my cell 0 is x = 0
    unsigned rxm;          // bit j: my cell j is x = nx-1 (a mask, not an index: a compare of
                           // the index per cell would become an indexed store to memory)
    unsigned ym0, ymn;     // bit k: my row k is y = 0 / y = ny-1
    unsigned st_mask;      // bit (k*VX + j): my cell (row k, x j) is stored
    unsigned st_rows;      // bit k: my row k is stored whole
    bool st_fast;          // vector stores: every row whole or empty, aligned rows
    long long st_off;      // gy * ld_out + gx
    int tid, lane, wid;
};

// Coefficients as pairs of equal values, the operands of the packed float32 operations.
struct Coef3 {
    float2 cc, cw, ce, cs, cn, cb, ca, sdc, ca_amb;
};

// a thread's row of VX cells as pairs: (x, y) of v[p] are cells p and p + VX/2
template <int VX>
__device__ __forceinline__ void lds_pairs(uint32_t a, float2 (&v)[VX / 2])
{
    if constexpr (VX == 2) {
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];\n" : "=f"(v[0].x), "=f"(v[0].y) : "r"(a));
    } else {
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n"
                     : "=f"(v[0].x), "=f"(v[1].x), "=f"(v[0].y), "=f"(v[1].y)
                     : "r"(a));
    }
}

// exchange rows stay in pair order
template <int VX>
__device__ __forceinline__ void lds_xch(uint32_t a, float2 (&v)[VX / 2])
{
#pragma unroll
    for (int p = 0; p < VX / 2; p++)
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];\n"
                     : "=f"(v[p].x), "=f"(v[p].y)
                     : "r"(a + 256u * p));
}

template <int VX>
__device__ __forceinline__ void sts_xch(uint32_t a, const float2 (&v)[VX / 2])
{
#pragma unroll
    for (int p = 0; p < VX / 2; p++)
        asm volatile("st.shared.v2.f32 [%0], {%1, %2};\n" ::"r"(a + 256u * p), "f"(v[p].x), "f"(v[p].y)
                     : "memory");
}

template <int H>
__device__ __forceinline__ float cell3(const float2 (&v)[H], int j)
{
    return j < H ? v[j < H ? j : 0].x : v[j < H ? 0 : j - H].y;
}

template <int H>
__device__ __forceinline__ void set_cell3(float2 (&v)[H], int j, float x)
{
    if (j < H) v[j < H ? j : 0].x = x;
    else v[j < H ? 0 : j - H].y = x;
}

__device__ __forceinline__ void cpa16(uint32_t dst, const void *src, int nbytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(nbytes)
                 : "memory");
}

__device__ __forceinline__ void cpa4(uint32_t dst, const void *src, int nbytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(dst), "l"(src), "r"(nbytes)
                 : "memory");
}

// ---- tensor-map bulk copies completing on an mbarrier ---------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, int count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                 " selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok)
                 : "r"(bar), "r"(parity)
                 : "memory");
    return ok != 0;
}

// Wait for phase `parity` of the barrier; gives up (false) after a bounded number of polls
// (each poll may suspend the thread for a while), so a lost copy cannot hang the GPU.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity)
{
    for (int n = 0; n < (1 << 22); n++)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

__device__ __forceinline__ void tma_plane(uint32_t dst, const CUtensorMap *m, int x, int y, int z,
                                          uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

// Stage the tile's window of one plane (z-plane base `src`, rows ld apart) into the slot at
// `dst` by per-thread copies; cells outside the domain arrive as zeros.
template <int BX, int BY, int NT>
__device__ __forceinline__ void tbf3_load(const CtxF3 &c, const float *src, long long ld, int vec,
                                          uint32_t dst)
{
    constexpr int CH = BX / 4;
    constexpr int NCH = CH * BY;
#pragma unroll
    for (int qq = 0; qq < (NCH + NT - 1) / NT; qq++) {
        const int q = c.tid + qq * NT;
        if (NCH % NT == 0 || q < NCH) {
            const int row = q / CH, ch = q % CH;
            const int y = c.y0 + row, x = c.x0 + 4 * ch;
            const uint32_t d = dst + 4u * (row * BX + 4 * ch);
            const bool yok = (y >= 0 && y < c.ny);
            const float *rs = src + (long long)(yok ? y : 0) * ld;
            if (vec) {
                const int nb = (yok && x >= 0 && x < c.nx) ? min(16, 4 * (c.nx - x)) : 0;
                cpa16(d, nb ? rs + x : src, nb);
            } else {
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const int xx = x + j;
                    const int nb = (yok && xx >= 0 && xx < c.nx) ? 4 : 0;
                    cpa4(d + 4u * j, nb ? rs + xx : src, nb);
                }
            }
        }
    }
}

// Clamped x and y edges of a plane d with its outer rows nt and sb and the values wl, er from the
// neighbour lanes, in a warp that touches an edge: the out-of-domain cell next to each edge cell
// (a ghost: its own value is never used) takes the edge cell's value, inside my cells (d, in
// place) or in the value that arrives from another lane or warp.  The neighbours stay pure
// renames of d, so the common path keeps no second copy of them.
// (every index stays in range even in code the unrolling discards: an out-of-range constant
// index, even in a dead branch, makes the compiler keep the array in memory)
// Which edges an instance handles (a tile column runs one that covers what it touches).
enum : int {
    E3X = 1,   // x = 0 or x = nx-1
    E3Y = 2,   // y = 0 or y = ny-1
};

template <int VX, int VY, int EDGE>
__device__ __forceinline__ void edge3(const CtxF3 &c, float2 (&d)[VY][VX / 2], float2 (&nt)[VX / 2],
                                      float2 (&sb)[VX / 2], float (&wl)[VY], float (&er)[VY])
{
    constexpr int H = VX / 2;
    if ((EDGE & E3Y) && c.edge_y) {
        // y = 0 at my row k: ghost row k-1 (or the row above, nt) := row k; likewise below
#pragma unroll
        for (int p = 0; p < H; p++) {
            nt[p].x = (c.ym0 & 1u) ? d[0][p].x : nt[p].x;
            nt[p].y = (c.ym0 & 1u) ? d[0][p].y : nt[p].y;
            sb[p].x = ((c.ymn >> (VY - 1)) & 1u) ? d[VY - 1][p].x : sb[p].x;
            sb[p].y = ((c.ymn >> (VY - 1)) & 1u) ? d[VY - 1][p].y : sb[p].y;
        }
#pragma unroll
        for (int k = 1; k < VY; k++) {
            const bool g = (c.ym0 >> k) & 1u;
#pragma unroll
            for (int p = 0; p < H; p++) {
                d[k - 1][p].x = g ? d[k][p].x : d[k - 1][p].x;
                d[k - 1][p].y = g ? d[k][p].y : d[k - 1][p].y;
            }
        }
#pragma unroll
        for (int k = 0; k < VY - 1; k++) {
            const bool g = (c.ymn >> k) & 1u;
#pragma unroll
            for (int p = 0; p < H; p++) {
                d[k + 1][p].x = g ? d[k][p].x : d[k + 1][p].x;
                d[k + 1][p].y = g ? d[k][p].y : d[k + 1][p].y;
            }
        }
    }
    if (EDGE & E3X) {
        // x = 0 is always my cell 0 (tile origins are multiples of 4); x = nx-1 is my cell j
#pragma unroll
        for (int k = 0; k < VY; k++) {
            wl[k] = c.lx0 ? d[k][0].x : wl[k];
            er[k] = ((c.rxm >> (VX - 1)) & 1u) ? d[k][H - 1].y : er[k];
#pragma unroll
            for (int j = 1; j < VX; j++) {
                const float e = cell3(d[k], j - 1), own = cell3(d[k], j);
                set_cell3(d[k], j, ((c.rxm >> (j - 1)) & 1u) ? e : own);
            }
        }
    }
}

// my cells of the compute block; dst: my first cell of the plane
template <int VX, int VY>
__device__ __forceinline__ void tbf3_store(const CtxF3 &c, float *dst, const float2 (&v)[VY][VX / 2])
{
    if (c.st_fast) {
        // every row of mine is stored whole or not at all, with aligned vector stores
#pragma unroll
        for (int k = 0; k < VY; k++) {
            if ((c.st_rows >> k) & 1u) {
                if constexpr (VX == 2)
                    *reinterpret_cast<float2 *>(dst) = v[k][0];
                else
                    *reinterpret_cast<float4 *>(dst) =
                        make_float4(v[k][0].x, v[k][VX / 2 - 1].x, v[k][0].y, v[k][VX / 2 - 1].y);
            }
            dst += c.ld_out;
        }
    } else {
#pragma unroll
        for (int k = 0; k < VY; k++) {
#pragma unroll
            for (int j = 0; j < VX; j++)
                if ((c.st_mask >> (VX * k + j)) & 1u) dst[j] = cell3(v[k], j);
            dst += c.ld_out;
        }
    }
}

template <int N>
__device__ __forceinline__ int slot_back(int s, int k)   // (s - k) mod N for 0 <= k <= N
{
    const int r = s - k;
    return r < 0 ? r + N : r;
}

// One iteration: stage s receives plane Z0 - 2s of time s (stage 0 from the ring slot at `field`,
// the others in D[s-1]) and emits plane Z0 - 2s - 1 of time s+1 into D[s], the last stage into
// the output (dst: my first cell there).  p0: ring slot of power plane Z0; xr / xw: exchange
// buffers read and written.
template <int KIND, int T, int VX, int VY, int NW, bool SPECIAL, int EDGE>
__device__ __forceinline__ void tbf3_iter(const CtxF3 &c, const Coef3 &k, uint32_t field,
                                          uint32_t spw, int p0, uint32_t xr, uint32_t xw, float *dst,
                                          float2 (&P)[T][VY][VX / 2], float2 (&Q)[T][VY][VX / 2],
                                          float2 (&D)[T][VY][VX / 2], int Z0)
{
    using C = TB3F<KIND, T, VX, VY, NW>;
    constexpr int H = VX / 2;
    const uint32_t own = C::ROWB * (c.wid * VY) + 4u * VX * c.lane;   // my row 0, cell 0 of a plane
    const uint32_t xo = C::ROWB * (2 * c.wid + 1) + 8u * c.lane;      // my top row in the exchange
    float2 xn[T][H], xs[T][H];
    if constexpr (C::XB == 1 && T > 1) {   // one buffer: every read before the first write
#pragma unroll
        for (int s = 1; s < T; s++) {
            lds_xch<VX>(xr + (s - 1) * C::XSTAGE + xo - C::ROWB, xn[s]);
            lds_xch<VX>(xr + (s - 1) * C::XSTAGE + xo + 2 * C::ROWB, xs[s]);
        }
        __syncthreads();
    }
    float2 res[VY][H];   // the last stage's plane
#pragma unroll
    for (int s = T - 1; s >= 0; s--) {
        const int zc = Z0 - 2 * s;   // the plane that arrives
        float2 d[VY][H], nt[H], sb[H], o[VY][H];
        if (s == 0) {
#pragma unroll
            for (int r = 0; r < VY; r++) lds_pairs<VX>(field + own + r * C::ROWB, d[r]);
        } else {
#pragma unroll
            for (int r = 0; r < VY; r++)
#pragma unroll
                for (int p = 0; p < H; p++) d[r][p] = D[s > 0 ? s - 1 : 0][r][p];
        }
        if (SPECIAL && s >= c.tsteps) {
            // forwarding stage: one plane of delay, no arithmetic
#pragma unroll
            for (int r = 0; r < VY; r++)
#pragma unroll
                for (int p = 0; p < H; p++) {
                    o[r][p] = P[s][r][p];
                    P[s][r][p] = d[r][p];
                }
        } else {
            if (s == 0) {
                lds_pairs<VX>(field + own - C::ROWB, nt);
                lds_pairs<VX>(field + own + VY * C::ROWB, sb);
            } else if constexpr (C::XB == 1) {
#pragma unroll
                for (int p = 0; p < H; p++) {
                    nt[p] = xn[s][p];
                    sb[p] = xs[s][p];
                }
            } else {
                lds_xch<VX>(xr + (s - 1) * C::XSTAGE + xo - C::ROWB, nt);
                lds_xch<VX>(xr + (s - 1) * C::XSTAGE + xo + 2 * C::ROWB, sb);
            }
            // (before the shuffles: the power value is the first term after the pipeline's own --
            // it is small, and added after the large terms it would round by their ulp)
            float2 pv[VY][H];
            if (KIND == KTHERM) {
                const uint32_t ap = spw + slot_back<C::NBP ? C::NBP : 1>(p0, 2 * s) * C::PLANE_B + own;
#pragma unroll
                for (int r = 0; r < VY; r++) lds_pairs<VX>(ap + r * C::ROWB, pv[r]);
            }
            float wl[VY], er[VY];
#pragma unroll
            for (int r = 0; r < VY; r++) {
                wl[r] = __shfl_sync(0xffffffffu, d[r][H - 1].y, (c.lane + 31) & 31);
                er[r] = __shfl_sync(0xffffffffu, d[r][0].x, (c.lane + 1) & 31);
            }
            if (EDGE) edge3<VX, VY, EDGE>(c, d, nt, sb, wl, er);
            const bool first = SPECIAL && zc == 0;          // clamp: plane -1 is plane 0
            const bool last = SPECIAL && zc == c.nz - 1;    // clamp: plane nz is plane nz-1
            const bool past = SPECIAL && zc == c.nz;        // plane nz-1 is complete
            // term by term over all the thread's pairs: consecutive operations are independent
            // (a chain per cell would wait out the latency of each of its links)
#define STN_PAIRS                                                                                  \
    _Pragma("unroll") for (int r = 0; r < VY; r++) _Pragma("unroll") for (int p = 0; p < H; p++)
            float2 t[VY][H];
            if (first) {   // Q of plane 0: plane -1 is plane 0
                STN_PAIRS Q[s][r][p] = KIND == KTHERM ? __ffma2_rn(k.cb, d[r][p], k.ca_amb) : __fmul2_rn(k.cb, d[r][p]);
            }
            STN_PAIRS o[r][p] = past ? P[s][r][p] : __ffma2_rn(k.ca, d[r][p], P[s][r][p]);
            STN_PAIRS t[r][p] = KIND == KTHERM ? __ffma2_rn(k.sdc, pv[r][p], Q[s][r][p]) : Q[s][r][p];
            STN_PAIRS t[r][p] = __ffma2_rn(k.cc, d[r][p], t[r][p]);
            STN_PAIRS Q[s][r][p] = KIND == KTHERM ? __ffma2_rn(k.cb, d[r][p], k.ca_amb) : __fmul2_rn(k.cb, d[r][p]);
            STN_PAIRS t[r][p] = __ffma2_rn(k.cn, r > 0 ? d[r > 0 ? r - 1 : 0][p] : nt[p], t[r][p]);
            STN_PAIRS t[r][p] = __ffma2_rn(k.cs, r < VY - 1 ? d[r < VY - 1 ? r + 1 : r][p] : sb[p], t[r][p]);
            // the outermost pairs take one half from a neighbour lane: their halves are added one
            // by one (building the pair would cost as many register moves)
            STN_PAIRS t[r][p] = p == H - 1
                ? make_float2(__fmaf_rn(k.ce.x, d[r][0].y, t[r][p].x), __fmaf_rn(k.ce.x, er[r], t[r][p].y))
                : __ffma2_rn(k.ce, d[r][p < H - 1 ? p + 1 : p], t[r][p]);
            STN_PAIRS t[r][p] = p == 0
                ? make_float2(__fmaf_rn(k.cw.x, wl[r], t[r][p].x), __fmaf_rn(k.cw.x, d[r][H - 1].x, t[r][p].y))
                : __ffma2_rn(k.cw, d[r][p > 0 ? p - 1 : 0], t[r][p]);
            if (last) STN_PAIRS t[r][p] = __ffma2_rn(k.ca, d[r][p], t[r][p]);
            STN_PAIRS P[s][r][p] = t[r][p];
#undef STN_PAIRS
        }
        if (s == T - 1) {
#pragma unroll
            for (int r = 0; r < VY; r++)
#pragma unroll
                for (int p = 0; p < H; p++) res[r][p] = o[r][p];
        } else {
#pragma unroll
            for (int r = 0; r < VY; r++)
#pragma unroll
                for (int p = 0; p < H; p++) D[s][r][p] = o[r][p];
            sts_xch<VX>(xw + s * C::XSTAGE + xo, o[0]);
            sts_xch<VX>(xw + s * C::XSTAGE + xo + C::ROWB, o[VY - 1]);
        }
    }
    const int R = Z0 - 2 * T + 1;
    if (R >= c.z0 && R < c.z1) tbf3_store<VX, VY>(c, dst, res);
}

template <int KIND, int T, int VX, int VY, int NW>
__global__ void __launch_bounds__(32 * NW, (TB3F<KIND, T, VX, VY, NW>::MINB))
    k_tb3f(const Pass3D p, const __grid_constant__ CUtensorMap tin,
           const __grid_constant__ CUtensorMap tpw)
{
    using C = TB3F<KIND, T, VX, VY, NW>;
    extern __shared__ __align__(128) float smem[];
    const uint32_t sring = smem_u32(smem) + C::ROWB;
    const uint32_t spw = sring + C::NBF * C::PLANE_B;
    const uint32_t sxch = spw + C::NBP * C::PLANE_B;
    const uint32_t sbar = sxch + C::XB * C::XBUF;   // NBF mbarriers, 8 bytes each
    const bool tma = p.use_tma != 0;
    if (tma) {
        if (threadIdx.x == 0) {
            for (int b = 0; b < C::NBF; b++) mbar_init(sbar + 8u * b, 1);
            asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        }
        __syncthreads();
    }
    uint32_t f0 = 0, fpar = 0;   // field slot of the next plane to arrive, its parity
    bool bad = false;       // a bounded wait of mine gave up: no further copies, no further waits
    CtxF3 c;
    c.in = p.in;
    c.out = p.out;
    c.pw = p.pw;
    c.nx = p.nx;
    c.ny = p.ny;
    c.nz = p.nz;
    c.ld_in = p.ld_in;
    c.ld_out = p.ld_out;
    c.ld_pw = p.ld_pw;
    c.plane_in = p.ld_in * p.ny;
    c.plane_out = p.ld_out * p.ny;
    c.plane_pw = p.ld_pw * p.ny;
    c.tsteps = p.tsteps;
    c.vec = p.vec;
    c.vec_pw = p.vec_pw;
    c.tid = threadIdx.x;
    c.lane = threadIdx.x & 31;
    c.wid = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
    Coef3 k;
    auto pair = [&](int i) { return make_float2(p.k[i], p.k[i]); };
    k.cc = pair(0);
    k.cw = pair(1);
    k.ce = pair(2);
    k.cs = pair(3);
    k.cn = pair(4);
    k.cb = pair(5);
    k.ca = pair(6);
    k.sdc = pair(7);
    const float ca_amb = KIND == KTHERM ? __fmul_rn(p.k[6], p.k[8]) : 0.f;
    k.ca_amb = make_float2(ca_amb, ca_amb);

    float2 P[T][VY][C::H], Q[T][VY][C::H], D[T][VY][C::H];
#pragma unroll
    for (int s = 0; s < T; s++)
#pragma unroll
        for (int r = 0; r < VY; r++)
#pragma unroll
            for (int q = 0; q < C::H; q++) P[s][r][q] = Q[s][r][q] = D[s][r][q] = make_float2(0.f, 0.f);

    // (broadcasts, so that the compiler knows the segment's bounds to be uniform across the warp
    // and keeps them, and what follows from them, in uniform registers)
    const int si_end = __shfl_sync(0xffffffffu, __ldg(p.seg_first + blockIdx.x + 1), 0);
    for (int si = __shfl_sync(0xffffffffu, __ldg(p.seg_first + blockIdx.x), 0); si < si_end; si++) {
        const int4 seg = __ldg(p.segs + si);
        const int col = __shfl_sync(0xffffffffu, seg.x, 0);
        const int z0 = __shfl_sync(0xffffffffu, seg.y, 0), z1 = __shfl_sync(0xffffffffu, seg.z, 0);
        const int ty = col / p.ntx, tx = col - ty * p.ntx;

        c.z0 = z0;
        c.z1 = z1;
        c.x0 = tx * C::CX - C::HX;
        c.y0 = ty * C::CY - C::HY;
        c.gx = c.x0 + VX * c.lane;
        c.gy = c.y0 + c.wid * VY;
        c.z_start = max(0, z0 - c.tsteps);
        c.last_plane = min(c.nz - 1, z1 - 1 + c.tsteps);
        c.lx0 = (c.gx == 0);
        const int rxj = (c.gx <= c.nx - 1 && c.nx - 1 < c.gx + VX) ? (c.nx - 1 - c.gx) : -1;
        c.rxm = rxj >= 0 ? (1u << rxj) : 0u;
        const int ky0 = (c.gy <= 0 && 0 < c.gy + VY) ? -c.gy : -1;
        const int kyn = (c.gy <= c.ny - 1 && c.ny - 1 < c.gy + VY) ? (c.ny - 1 - c.gy) : -1;
        c.ym0 = ky0 >= 0 ? (1u << ky0) : 0u;
        c.ymn = kyn >= 0 ? (1u << kyn) : 0u;
        c.edge_y = __any_sync(0xffffffffu, ky0 >= 0 || kyn >= 0);
        {
            const int xl = max(c.x0 + C::HX, 0), xh = min(c.x0 + C::HX + C::CX, c.nx);
            const int yl = max(c.y0 + C::HY, 0), yh = min(c.y0 + C::HY + C::CY, c.ny);
            unsigned msk = 0;
#pragma unroll
            for (int k = 0; k < VY; k++)
#pragma unroll
                for (int j = 0; j < VX; j++) {
                    const int x = c.gx + j, y = c.gy + k;
                    if (x >= xl && x < xh && y >= yl && y < yh) msk |= 1u << (VX * k + j);
                }
            c.st_mask = msk;
            constexpr unsigned ALL = (1u << VX) - 1u;
            unsigned rows = 0;
            bool fast = p.vec_out != 0;
#pragma unroll
            for (int k = 0; k < VY; k++) {
                const unsigned b = (msk >> (VX * k)) & ALL;
                if (b == ALL) rows |= 1u << k;
                else if (b != 0) fast = false;
            }
            c.st_rows = rows;
            c.st_fast = fast;
            c.st_off = (long long)c.gy * c.ld_out + c.gx;
        }
        const int n_it = z1 + 2 * T - 1 - c.z_start;   // the last stage emits plane z1-1 last
        const int bot_i = c.nz - 1 - c.z_start;   // stage 0 meets plane nz-1 first
        const bool top = (c.z_start == 0);
        const bool partial = (c.tsteps < T);

        // queue plane z into field slot `fs` (and power slot `ps`): by tensor-map copies on
        // barrier fs (one elected thread), else by per-thread cp.async (one group)
        auto load = [&](int z, uint32_t fs, uint32_t ps) {
            if (tma) {
                if (threadIdx.x == 0 && z <= c.last_plane && !bad) {
                    const uint32_t bar = sbar + 8u * fs;
                    mbar_expect_tx(bar, (KIND == KTHERM ? 2u : 1u) * C::PLANE_B);
                    tma_plane(sring + fs * C::PLANE_B, &tin, c.x0, c.y0, z, bar);
                    if (KIND == KTHERM) tma_plane(spw + ps * C::PLANE_B, &tpw, c.x0, c.y0, z, bar);
                }
            } else {
                if (z <= c.last_plane) {
                    tbf3_load<C::BX, C::BY, C::NT>(c, c.in + (long long)z * c.plane_in, c.ld_in, c.vec,
                                                   sring + fs * C::PLANE_B);
                    if (KIND == KTHERM)
                        tbf3_load<C::BX, C::BY, C::NT>(c, c.pw + (long long)z * c.plane_pw, c.ld_pw,
                                                       c.vec_pw, spw + ps * C::PLANE_B);
                }
                cp_async_commit();
            }
        };
        // the field ring goes on where the previous segment left it (slot f0 with parity fpar
        // takes this segment's first plane); slots advance with the planes that are loaded
        {
            uint32_t fs = f0;
#pragma unroll 1
            for (int j = 0; j < C::PF; j++) {
                load(c.z_start + j, fs, KIND == KTHERM ? j : 0);
                fs = fs + 1 == C::NBF ? 0 : fs + 1;
            }
        }
        uint32_t p0 = 0;                                         // slot of power plane Z0
        uint32_t xr = sxch, xw = sxch + (C::XB - 1) * C::XBUF;   // exchange read / written
        float *dst = c.out + c.st_off + ((long long)c.z_start - (2 * T - 1)) * c.plane_out;
        if (!tma) cp_async_wait<C::PF - 1>();
        __syncthreads();
        // one plane
        auto step = [&](auto special_tag, auto edge_tag, int i) {
            const int Z0 = c.z_start + i;
            // the slot refilled here was last read in the previous iteration, before its barrier
            load(Z0 + C::PF, f0 == 0 ? C::NBF - 1 : f0 - 1,
                 KIND == KTHERM ? (p0 + C::PF >= C::NBP ? p0 + C::PF - C::NBP : p0 + C::PF) : 0);
            const bool in = Z0 <= c.last_plane;
            if (tma && in && !bad && !mbar_wait_bounded(sbar + 8u * f0, fpar)) {
                bad = true;   // flag it and carry on: every later wait and copy is skipped
                atomicExch(p.err, 1);
            }
            tbf3_iter<KIND, T, VX, VY, NW, decltype(special_tag)::value, decltype(edge_tag)::value>(
                c, k, sring + f0 * C::PLANE_B, spw, p0, xr, xw, dst, P, Q, D, Z0);
            dst += c.plane_out;
            if (in) {
                f0++;
                if (f0 == C::NBF) {
                    f0 = 0;
                    fpar ^= 1u;
                }
            }
            if (KIND == KTHERM) p0 = p0 + 1 == C::NBP ? 0 : p0 + 1;
            const uint32_t t = xr;
            xr = xw;
            xw = t;
            if (!tma) cp_async_wait<C::PF - 1>();   // (plane Z0 + 1, made visible by the barrier)
            __syncthreads();
        };
        // the planes that need z-boundary handling (the first and last of the grid, and all of a
        // pass that forwards trailing stages) run in loops of their own: a loop that chose per
        // plane would have to merge the partial sums of both bodies, with register copies, in
        // every iteration
        const int i_a = partial ? n_it : (top ? min(2 * T - 1, n_it) : 0);
        const int i_b = partial ? n_it : max(i_a, min(n_it, bot_i));
        // A tile column runs the instance that handles the edges it touches (interior ones none):
        // the fix-ups' in-place updates of the plane otherwise cost register copies on every path.
        auto run = [&](auto edge_tag) {
            int i = 0;
#pragma unroll 1
            for (; i < i_a; i++) step(std::true_type{}, edge_tag, i);
#pragma unroll 1
            for (; i < i_b; i++) step(std::false_type{}, edge_tag, i);
#pragma unroll 1
            for (; i < n_it; i++) step(std::true_type{}, edge_tag, i);
        };
        const int touch = (c.x0 <= 0 || c.x0 + C::BX >= c.nx ? E3X : 0) |
                          (c.y0 <= 0 || c.y0 + C::BY >= c.ny ? E3Y : 0);   // block-uniform
        if (touch == 0) run(std::integral_constant<int, 0>{});
        else if (touch == E3Y) run(std::integral_constant<int, E3Y>{});
        else run(std::integral_constant<int, E3X | E3Y>{});
        if (!tma) cp_async_wait<0>();
        if (__syncthreads_or(bad)) {
            // give whatever may still be in flight a bounded chance to land, then leave
            for (int b = 0; b < C::NBF; b++) {
                (void)mbar_wait_bounded(sbar + 8u * b, 0);
                (void)mbar_wait_bounded(sbar + 8u * b, 1);
            }
            return;
        }
    }
}

}  // namespace stn
