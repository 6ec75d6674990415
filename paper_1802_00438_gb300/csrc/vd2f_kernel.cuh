// 2D diffusion with per-cell coefficients (Table 2 row 1, coefficients as arrays, Sec. 5.1),
// contracted arithmetic: one pass advances the grid by `tsteps` (<= T) steps.
//
// The blocking of the contracted kernel (tb2f_kernel.cuh): one-warp tiles, 128 cells wide incl.
// halos, streamed along y through T stages that keep two partial rows each,
//   out(y-1) = P + cs(y-1)*d,   P' = Q + cc(y)*d + cw(y)*w + ce(y)*e,   Q' = cn(y+1)*d,
// on packed float32 pairs (here of adjacent cells, as the coefficients lie in memory; the west and
// east terms go cell by cell).  A coefficient row is used by one stage after the other in
// successive iterations, so its window of T rows is held in registers, and the row loop is
// unrolled T times so that the window turns by renaming: a coefficient crosses shared memory
// once per pass, not once per stage.  cs rows run one row behind the field rows, cn rows one
// ahead: stage s then uses the rows that arrived s iterations ago, of every plane.
//
// What bounds it: the pass reads 24 and writes 4 bytes per cell, so T = 4 steps cost at least 7
// bytes each.  The three-row-window kernel (tb2d_kernel.cuh), which every other shape runs, read
// five coefficient rows per stage from shared memory and waited for it (47 % issue active, 9
// warps per SM).  Measured on GB300, that kernel -> this one, T = 4: 4096^2 x 100 3024 -> 2366 us,
// 8192^2 10952 -> 8800, 4097^2 3928 -> 2685, 1024^2 525 -> 369, 512^2 x 60 224 -> 164; T = 2:
// 8192^2 20519 -> 18017, 4096^2 4798 -> 4735.  At 763 GCell/s an 8192^2 pass moves 5.3 TB/s of
// field and coefficients, 79 % of the copy bandwidth.
#pragma once
#include "tb2f_kernel.cuh"

namespace stn {

template <int T>
struct VD2F {
    static constexpr int V = 4;
    static constexpr int BX = 32 * V;
    static constexpr int H = (T + V - 1) / V * V;
    static constexpr int CX = BX - 2 * H;
    static constexpr int PF = 4;
    static constexpr int NB = PF + 1;                  // ring rows: field and five planes
    static constexpr int ROWB = BX * 4;
    static constexpr size_t SMEM = (size_t)6 * NB * ROWB;
    static_assert(CX > 0, "tile narrower than its halos");
};

struct CtxV {
    const float *in, *w;        // field, coefficient planes
    float *out;
    long long ld_in, ld_out, plane;
    uint32_t sring;
    int nx, ny, tsteps, x0, xt, y_start, last_row, s0, s1, lane;
    unsigned lmask, rmask;
    int st_lo, st_hi, edge;
    bool st_full, st_any, vec_in, vec_w;
    int nb, col;                // my chunk: bytes inside the grid, column to copy from
};

// my four cells of ring row `row`, as two pairs of adjacent cells
__device__ __forceinline__ void vd_row(uint32_t row, int lane, float2 (&v)[2])
{
    const float4 t = lds128(row + 16u * lane);
    v[0] = make_float2(t.x, t.y);
    v[1] = make_float2(t.z, t.w);
}

// my cells of coefficient row y straight from the plane (boundary rows only)
__device__ __forceinline__ void vd_gmem(const CtxV &c, int plane, int y, float2 (&v)[2])
{
    float q[4];
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const int x = c.xt + j;
        q[j] = x >= 0 && x < c.nx ? __ldg(c.w + plane * c.plane + (long long)y * c.nx + x) : 0.f;
    }
    v[0] = make_float2(q[0], q[1]);
    v[1] = make_float2(q[2], q[3]);
}

// One stage on the arrival of row y (values d, time s): emits row y-1 of time s+1.
// k: the window's rows for this stage (cc, cw, ce of row y, cs of row y-1, cn of row y+1).
template <int MODE>
__device__ __forceinline__ void vd_stage(const CtxV &c, int y, bool fwd, const float2 (&cc)[2],
                                         const float2 (&cw)[2], const float2 (&ce)[2],
                                         const float2 (&cs)[2], const float2 (&cn)[2], float2 (&P)[2],
                                         float2 (&Q)[2], float2 (&d)[2], float2 (&out)[2])
{
    constexpr bool SP = MODE == MODE_SPECIAL;
    if (SP && (fwd || y == c.ny)) {   // row ny-1 is complete; forwarding stages pass rows on
#pragma unroll
        for (int p = 0; p < 2; p++) {
            out[p] = P[p];
            P[p] = d[p];
        }
        return;
    }
    float w_in = __shfl_sync(0xffffffffu, d[1].y, (c.lane + 31) & 31);
    float e_in = __shfl_sync(0xffffffffu, d[0].x, (c.lane + 1) & 31);
    if (MODE != MODE_PLAIN) {
        // x = 0 is always a lane's cell 0; the cell beyond x = nx-1 takes its value
        w_in = (c.lmask & 1u) ? d[0].x : w_in;
        e_in = (c.rmask & 8u) ? d[1].y : e_in;
        if (MODE != MODE_EDGE) {
            d[1].y = (c.rmask & 4u) ? d[1].x : d[1].y;
            d[1].x = (c.rmask & 2u) ? d[0].y : d[1].x;
            d[0].y = (c.rmask & 1u) ? d[0].x : d[0].y;
        }
    }
    if (SP && y == 0) {   // the row above row 0 is row 0
        float2 k[2];
        vd_gmem(c, 4, 0, k);
#pragma unroll
        for (int p = 0; p < 2; p++) Q[p] = __fmul2_rn(k[p], d[p]);
    }
#pragma unroll
    for (int p = 0; p < 2; p++) out[p] = __ffma2_rn(cs[p], d[p], P[p]);
    float2 t[2];
#pragma unroll
    for (int p = 0; p < 2; p++) t[p] = __ffma2_rn(cc[p], d[p], Q[p]);
#pragma unroll
    for (int p = 0; p < 2; p++) Q[p] = __fmul2_rn(cn[p], d[p]);
    t[0].y = __fmaf_rn(cw[0].y, d[0].x, t[0].y);
    t[1].x = __fmaf_rn(cw[1].x, d[0].y, t[1].x);
    t[1].y = __fmaf_rn(cw[1].y, d[1].x, t[1].y);
    t[0].x = __fmaf_rn(cw[0].x, w_in, t[0].x);
    t[0].y = __fmaf_rn(ce[0].y, d[1].x, t[0].y);
    t[1].x = __fmaf_rn(ce[1].x, d[1].y, t[1].x);
    t[0].x = __fmaf_rn(ce[0].x, d[0].y, t[0].x);
    t[1].y = __fmaf_rn(ce[1].y, e_in, t[1].y);
    if (SP && y == c.ny - 1) {   // the row below row ny-1 is row ny-1: complete it now
        float2 k[2];
        vd_gmem(c, 3, y, k);
#pragma unroll
        for (int p = 0; p < 2; p++) t[p] = __ffma2_rn(k[p], d[p], t[p]);
    }
#pragma unroll
    for (int p = 0; p < 2; p++) P[p] = t[p];
}

// Queue ring slot `slot` with what iteration i needs: field, cc, cw and ce row y = y_start + i, cs
// row y-1, cn row y+1 (rows outside the loaded range are left as they are: no valid row uses them).
template <int T>
__device__ __forceinline__ void vd_queue(const CtxV &c, int i, int slot)
{
    using C = VD2F<T>;
    const int y = c.y_start + i;
    if (y <= c.last_row) {
        const uint32_t dst = c.sring + slot * C::ROWB + 16u * c.lane;
        const int dy[6] = {0, 0, 0, 0, -1, 1};
#pragma unroll
        for (int a = 0; a < 6; a++) {
            const int yy = y + dy[a];
            if (yy < 0 || yy >= c.ny) continue;
            const float *row = a == 0 ? c.in + (long long)yy * c.ld_in
                                      : c.w + (a - 1) * c.plane + (long long)yy * c.nx;
            const uint32_t d = dst + a * C::NB * C::ROWB;
            if (a == 0 ? c.vec_in : c.vec_w) {
                cp16(d, row + c.col, c.nb);
            } else {
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const int n = 4 * j < c.nb ? 4 : 0;
                    cp4(d + 4 * j, row + (n ? c.col + j : 0), n);
                }
            }
        }
    }
    cp_async_commit();
}

// One row; PH: the window slot the new rows go to (the row s iterations ago is at PH - s mod T).
// SHIFT: PH = 0, the window is moved on by register copies instead of by naming.
template <int T, int MODE, int PH, bool SHIFT>
__device__ __forceinline__ void vd_iter(const CtxV &c, float2 (&W)[5][T][2], float2 (&P)[T][2],
                                        float2 (&Q)[T][2], int i, int &slot, float *&gO, int i_store)
{
    using C = VD2F<T>;
    static_assert(T == 2 || T == 4, "window phases");
    cp_async_wait<C::PF - 1>();
    __syncwarp();
    const uint32_t row = c.sring + slot * C::ROWB;
    float2 d[2], out[2];
    vd_row(row, c.lane, out);
    if (SHIFT) {
#pragma unroll
        for (int a = 0; a < 5; a++)
#pragma unroll
            for (int t = 1; t < T; t++)
#pragma unroll
                for (int q = 0; q < 2; q++) W[a][t][q] = W[a][(t + 1) % T][q];
    }
#pragma unroll
    for (int a = 0; a < 5; a++) vd_row(row + (a + 1) * C::NB * C::ROWB, c.lane, W[a][PH]);
    const int R0 = c.y_start + i;
#pragma unroll
    for (int s = 0; s < T; s++) {
        if (MODE == MODE_HEAD && i < 2 * s) break;   // its first valid row comes at i = 2s
        constexpr int kT = T;
        const int q = (PH + kT - s) % kT;
        d[0] = out[0];
        d[1] = out[1];
        vd_stage<MODE>(c, R0 - s, s >= c.tsteps, W[0][q], W[1][q], W[2][q], W[3][q], W[4][q], P[s], Q[s],
                       d, out);
    }
    if (i >= i_store) {
        if (c.st_full) {
            *reinterpret_cast<float4 *>(gO) = make_float4(out[0].x, out[0].y, out[1].x, out[1].y);
        } else if (c.st_any) {
            const float v[4] = {out[0].x, out[0].y, out[1].x, out[1].y};
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (j >= c.st_lo && j < c.st_hi) gO[j] = v[j];
        }
        gO += c.ld_out;
    }
    __syncwarp();
    vd_queue<T>(c, i + C::PF, slot == 0 ? C::NB - 1 : slot - 1);
    slot = slot + 1 == C::NB ? 0 : slot + 1;
}

// (at most 168 registers: three warps per scheduler)
template <int T>
__global__ void __launch_bounds__(32, 12) k_vd2f(const Pass2D p)
{
    using C = VD2F<T>;
    extern __shared__ __align__(16) float smem[];
    CtxV c;
    c.in = p.in;
    c.out = p.out;
    c.w = p.pw;
    c.ld_in = p.ld_in;
    c.ld_out = p.ld_out;
    c.plane = p.pw_plane;
    c.sring = smem_u32(smem);
    c.nx = p.nx;
    c.ny = p.ny;
    c.tsteps = p.tsteps;
    c.lane = threadIdx.x;
    c.vec_in = p.vec_in != 0;
    c.vec_w = p.vec_pw != 0 && p.pw_plane % 4 == 0;
    float2 W[5][T][2], P[T][2], Q[T][2];
#pragma unroll
    for (int t = 0; t < T; t++)
#pragma unroll
        for (int q = 0; q < 2; q++) {
            P[t][q] = Q[t][q] = make_float2(0.f, 0.f);
#pragma unroll
            for (int a = 0; a < 5; a++) W[a][t][q] = make_float2(0.f, 0.f);
        }
    // (broadcasts: uniform registers, see k_tb2f)
    const int seg_end = __shfl_sync(0xffffffffu, __ldg(p.seg_first + blockIdx.x + 1), 0);
#pragma unroll 1
    for (int si = __shfl_sync(0xffffffffu, __ldg(p.seg_first + blockIdx.x), 0); si < seg_end; si++) {
        const int4 seg = __ldg(p.segs + si);
        const int tx = __shfl_sync(0xffffffffu, seg.x, 0);
        c.s0 = __shfl_sync(0xffffffffu, seg.y, 0);
        c.s1 = __shfl_sync(0xffffffffu, seg.z, 0);
        c.x0 = tx * C::CX - C::H;
        c.xt = c.x0 + 4 * c.lane;
        c.y_start = max(0, c.s0 - c.tsteps);
        c.last_row = min(c.ny - 1, c.s1 - 1 + c.tsteps);
        const int rcl = (c.xt <= c.nx - 1 && c.nx - 1 < c.xt + 4) ? (c.nx - 1 - c.xt) : -1;
        c.lmask = c.xt == 0 ? 1u : 0u;
        c.rmask = rcl >= 0 ? (1u << rcl) : 0u;
        c.edge = __any_sync(0xffffffffu, rcl >= 0 && rcl < 3) ? 2
                 : __any_sync(0xffffffffu, c.xt == 0 || rcl == 3) ? 1 : 0;
        const int lo = max(c.x0 + C::H, 0), hi = min(c.x0 + C::H + C::CX, c.nx);
        c.st_lo = min(max(lo - c.xt, 0), 4);
        c.st_hi = min(max(hi - c.xt, 0), 4);
        c.st_full = p.vec_out && c.st_lo == 0 && c.st_hi == 4;
        c.st_any = c.st_hi > c.st_lo;
        c.nb = (c.xt >= 0 && c.xt < c.nx) ? min(16, 4 * (c.nx - c.xt)) : 0;
        c.col = c.nb ? c.xt : 0;
        float *gO = c.out + (long long)c.s0 * c.ld_out + c.xt;
        int slot = 0;
        const int n_it = c.s1 + T - c.y_start, i_store = c.s0 - c.y_start + T;
#pragma unroll 1
        for (int j = 0; j < C::PF; j++) vd_queue<T>(c, j, j);
        const bool partial = c.tsteps < T;
        const int i_a = partial ? n_it : (c.y_start == 0 ? min(T, n_it) : 0);
        const int i_b = partial ? n_it : max(i_a, min(n_it, c.ny - 1 - c.y_start));
        const int i_h = (partial || c.y_start == 0) ? 0 : min(2 * T - 2, i_b);
        int i = 0;
        // the loops of few rows shift the window: their bodies, one each, are cold code that every
        // block fetches anew (with a body per window phase a pass cost 16 us more: 4096^2 x 100 3110 -> 2373 us)
#pragma unroll 1
        for (; i < i_h; i++) vd_iter<T, MODE_HEAD, 0, true>(c, W, P, Q, i, slot, gO, i_store);
#pragma unroll 1
        for (int part = 0; part < 2; part++) {
            const int end = part == 0 ? i_a : n_it;
#pragma unroll 1
            for (; i < end; i++) vd_iter<T, MODE_SPECIAL, 0, true>(c, W, P, Q, i, slot, gO, i_store);
            if (part == 1) break;
            auto rows = [&](auto mode) {
                constexpr int M = decltype(mode)::value;
#pragma unroll 1
                for (; i + T <= i_b; i += T) {
                    vd_iter<T, M, 1, false>(c, W, P, Q, i, slot, gO, i_store);
                    if constexpr (T == 4) {
                        vd_iter<T, M, 2, false>(c, W, P, Q, i + 1, slot, gO, i_store);
                        vd_iter<T, M, 3, false>(c, W, P, Q, i + 2, slot, gO, i_store);
                    }
                    vd_iter<T, M, 0, false>(c, W, P, Q, i + T - 1, slot, gO, i_store);
                }
            };
            if (c.edge == 0) rows(std::integral_constant<int, MODE_PLAIN>{});
            else if (c.edge == 1) rows(std::integral_constant<int, MODE_EDGE>{});
#pragma unroll 1
            for (; i < i_b; i++) vd_iter<T, MODE_GHOST, 0, true>(c, W, P, Q, i, slot, gO, i_store);
        }
        cp_async_wait<0>();
        __syncwarp();
    }
}

}  // namespace stn
