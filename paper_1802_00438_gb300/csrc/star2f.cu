// Star diffusion of radius 2 in 2D (9 points, Eqs. 1-2 of arXiv 1802.00438 with rad = 2),
// contracted arithmetic: one pass advances the grid by `tsteps` (<= T) steps.
//
// The blocking of the first-order contracted kernel (tb2f_kernel.cuh): a tile 256 cells wide incl.
// halos streamed along y through a chain of T stages by one warp, 8 cells per thread as 4 packed
// pairs (cells p and p + 4), field rows through a cp.async ring, rows of tile columns dealt as
// segments, the fill rows' idle stages skipped, clamped boundary (Sec. 5.1) at every stage.
//
// A stage keeps four pending rows.  When row y of time s arrives it
//   finishes row y-2:   out = A0 + cs2*d
//   row y-1:            A0' = A1 + cs1*d                      (missing its second south term)
//   row y:              A1' = A2 + cc*d + cw1*w1 + ce1*e1 + cw2*w2 + ce2*e2
//   row y+1:            A2' = A3 + cn1*d
//   row y+2:            A3' = cn2*d
// -- each pending row moves one place up as its next term is added, so the shift costs nothing.
// Nine operations per cell and step; a stage runs two rows behind the one before it.
//
// Why this and not tiles in shared memory (star2d.cuh, which exact plans and radii 3 and 4 run): a
// step there reads every cell's column and both side chunks from shared memory and is bound by it
// (2304 of its cycles per 128 x 128 step); here a row crosses shared memory once per pass, the
// neighbours of a stage come from registers and four shuffles per 8 cells, and the halo wastes
// 16 of 256 cells instead of 16 of 128 in both directions.  Measured on GB300 (T = 4), tiles ->
// here: 8192^2 x 64 steps 4026 -> 2327 us, 8191^2 5919 -> 2523, 4096^2 1244 -> 741, 2048^2 637 ->
// 340, 1024^2 310 -> 242, 512^2 x 32 143 -> 112: faster over the whole range, so contracted plans
// of radius 2 run this unless a tile is asked for.  It is bound by issue and latency with two
// warps per scheduler, like the first-order kernel.
#include "tb2f_kernel.cuh"

namespace stn {
namespace {

constexpr int kV = 8, kHV = kV / 2;
// halo 8 = 2T rounded to the cells per thread for every T <= 4: the first-order kernel's T = 8 ring
using RingS = TB2F<KDIFF, 8, kV, STOR_F32>;

struct CoefS {
    float2 cc, w1, e1, s1, n1, w2, e2, s2, n2;
};

#define STN_P _Pragma("unroll") for (int p = 0; p < kHV; p++)

// One stage on the arrival of row y (values d): emits row y-2 in out.
template <int MODE>
__device__ __forceinline__ void star_stage(const CtxF &c, const CoefS &k, int y, bool fwd,
                                           float2 (&A0)[kHV], float2 (&A1)[kHV], float2 (&A2)[kHV],
                                           float2 (&A3)[kHV], float2 (&d)[kHV], float2 (&out)[kHV])
{
    constexpr bool SP = MODE == MODE_SPECIAL;
    constexpr int L = kHV - 1;
    // rows past the grid complete on the arrival of its last row, and a stage beyond this pass's
    // step count passes rows on unchanged, two rows later like the others
    if (SP && (fwd || y >= c.ny)) {
        STN_P out[p] = A0[p];
        STN_P A0[p] = A1[p];
        if (fwd) { STN_P A1[p] = d[p]; }
        return;
    }
    float l1 = __shfl_sync(0xffffffffu, d[L].y, (c.lane + 31) & 31);       // cell -1
    float l2 = __shfl_sync(0xffffffffu, d[L - 1].y, (c.lane + 31) & 31);   // cell -2
    float r1 = __shfl_sync(0xffffffffu, d[0].x, (c.lane + 1) & 31);        // cell 8
    float r2 = __shfl_sync(0xffffffffu, d[1].x, (c.lane + 1) & 31);        // cell 9
    if (MODE != MODE_PLAIN) {
        // x = 0 is always a lane's cell 0; the cells beyond an edge take the edge cell's value
        l1 = (c.lmask & 1u) ? d[0].x : l1;
        l2 = (c.lmask & 1u) ? d[0].x : l2;
        const bool last = (c.rmask >> (kV - 1)) & 1u;
        r1 = last ? d[L].y : r1;
        r2 = last ? d[L].y : r2;
        if (MODE != MODE_EDGE) {   // x = nx-1 inside a lane: its two ghost cells
            r1 = ((c.rmask >> (kV - 2)) & 1u) ? d[L - 1].y : r1;
            r2 = ((c.rmask >> kV) & 1u) ? r1 : r2;   // x = nx-1 is the next lane's cell 0
#pragma unroll
            for (int j = kV - 2; j >= 0; j--) {
                const bool g = (c.rmask >> j) & 1u;
                const float edge = cell(d, j);
#pragma unroll
                for (int t = 1; t <= 2; t++) {
                    const int q = j + t;
                    if (q >= kV) continue;
                    if (q < kHV) d[q < kHV ? q : 0].x = g ? edge : d[q < kHV ? q : 0].x;
                    else d[q < kHV ? 0 : q - kHV].y = g ? edge : d[q < kHV ? 0 : q - kHV].y;
                }
            }
        }
    }
    if (SP && y == 0) {   // rows -1 and -2 are row 0
        STN_P A3[p] = __fmul2_rn(k.n2, d[p]);
        STN_P A2[p] = __ffma2_rn(k.n1, d[p], A3[p]);
    }
    STN_P out[p] = __ffma2_rn(k.s2, d[p], A0[p]);
    STN_P A0[p] = __ffma2_rn(k.s1, d[p], A1[p]);
    // the pairs that mix a lane's halves (each used at distance 1 and 2)
    const float2 m1 = make_float2(l1, d[L].x), m2 = make_float2(l2, d[L - 1].x);
    const float2 p1 = make_float2(d[0].y, r1), p2 = make_float2(d[1].y, r2);
    float2 t[kHV];
    STN_P t[p] = __ffma2_rn(k.cc, d[p], A2[p]);
    STN_P t[p] = __ffma2_rn(k.w1, p > 0 ? d[p > 0 ? p - 1 : 0] : m1, t[p]);
    STN_P t[p] = __ffma2_rn(k.e1, p < L ? d[p < L ? p + 1 : p] : p1, t[p]);
    STN_P t[p] = __ffma2_rn(k.w2, p > 1 ? d[p > 1 ? p - 2 : 0] : p == 1 ? m1 : m2, t[p]);
    STN_P A1[p] = __ffma2_rn(k.e2, p < L - 1 ? d[p < L - 1 ? p + 2 : p] : p == L - 1 ? p1 : p2, t[p]);
    STN_P A2[p] = __ffma2_rn(k.n1, d[p], A3[p]);
    STN_P A3[p] = __fmul2_rn(k.n2, d[p]);
    if (SP && y == c.ny - 1) {   // rows ny and ny+1 are row ny-1: complete rows ny-2 and ny-1
        STN_P A0[p] = __ffma2_rn(k.s2, d[p], A0[p]);
        STN_P A1[p] = __ffma2_rn(k.s1, d[p], A1[p]);
        STN_P A1[p] = __ffma2_rn(k.s2, d[p], A1[p]);
    }
}

// One row: stage s receives row R0 - 2s of time s and emits row R0 - 2s - 2 of time s+1.
template <int T, int MODE>
__device__ __forceinline__ void star_row(const CtxF &c, const CoefS &k, float2 (&A)[T][4][kHV], int i,
                                         RowF &r)
{
    using C = RingS;
    cp_async_wait<C::PF - 1>();
    __syncwarp();
    float2 d[kHV], out[kHV];
    lds_row<kV, false>(c.sF + r.rf * C::ROWB, c, out);
    const int R0 = c.y_start + i;
#pragma unroll
    for (int s = 0; s < T; s++) {
        if (MODE == MODE_HEAD && i < 4 * s) break;   // its first valid row comes at i = 4s
        STN_P d[p] = out[p];
        star_stage<MODE>(c, k, R0 - 2 * s, s >= c.tsteps, A[s][0], A[s][1], A[s][2], A[s][3], d, out);
    }
    if (i >= r.i_store) {
        st_cells<kV>(c, r.gO, out);
        r.gO += c.ld_out;
    }
    __syncwarp();
    tbf_queue<KDIFF, 8, kV, STOR_F32>(c, r, i < r.i_load_end, false, r.rf == 0 ? C::NBF - 1 : r.rf - 1, 0, 0);
    cp_async_commit();
    r.rf = (r.rf + 1 == C::NBF) ? 0 : r.rf + 1;
}

#undef STN_P

template <int T>
__global__ void __launch_bounds__(32) k_star2f(const Pass2D p, const StarCoef2 ks)
{
    using C = RingS;
    extern __shared__ __align__(16) float smem[];
    CtxF c;
    c.in = p.in;
    c.out = p.out;
    c.ld_in = p.ld_in;
    c.ld_out = p.ld_out;
    c.sF = smem_u32(smem);
    c.sP = c.sF;
    c.nx = p.nx;
    c.ny = p.ny;
    c.tsteps = p.tsteps;
    c.vec_in = p.vec_in;
    c.vec_out = p.vec_out;
    c.lane = threadIdx.x;
#pragma unroll
    for (int q = 0; q < 2; q++) {
        c.oq[q] = 16u * ring_pos(2 * c.lane + q);
        c.wq[q] = 16u * ring_pos(c.lane + 32 * q);
    }
    auto pr = [&](int i) { return make_float2(ks.k[i], ks.k[i]); };   // cc, per distance w e s n
    const CoefS k{pr(0), pr(1), pr(2), pr(3), pr(4), pr(5), pr(6), pr(7), pr(8)};
    float2 A[T][4][kHV];
#pragma unroll
    for (int s = 0; s < T; s++)
#pragma unroll
        for (int a = 0; a < 4; a++)
#pragma unroll
            for (int q = 0; q < kHV; q++) A[s][a][q] = make_float2(0.f, 0.f);
    // (broadcasts: uniform registers, see k_tb2f)
    const int seg_end = __shfl_sync(0xffffffffu, __ldg(p.seg_first + blockIdx.x + 1), 0);
#pragma unroll 1
    for (int si = __shfl_sync(0xffffffffu, __ldg(p.seg_first + blockIdx.x), 0); si < seg_end; si++) {
        const int4 seg = __ldg(p.segs + si);
        const int tx = __shfl_sync(0xffffffffu, seg.x, 0);
        c.s0 = __shfl_sync(0xffffffffu, seg.y, 0);
        c.s1 = __shfl_sync(0xffffffffu, seg.z, 0);
        c.x0 = tx * C::CX - C::H;
        c.xt = c.x0 + c.lane * kV;
        c.y_start = max(0, c.s0 - 2 * c.tsteps);
        c.last_row = min(c.ny - 1, c.s1 - 1 + 2 * c.tsteps);
        const int lcl = c.xt == 0 ? 0 : -1;
        // my cell that is x = nx-1, or kV when that is the next lane's cell 0
        const int rcl = (c.xt <= c.nx - 1 && c.nx - 1 <= c.xt + kV) ? (c.nx - 1 - c.xt) : -1;
        c.lmask = lcl >= 0 ? 1u : 0u;
        c.rmask = rcl >= 0 ? (1u << rcl) : 0u;
        c.edge = __any_sync(0xffffffffu, rcl >= 0 && rcl != kV - 1) ? 2
                 : __any_sync(0xffffffffu, lcl >= 0 || rcl >= 0) ? 1 : 0;
        const int lo = max(c.x0 + C::H, 0), hi = min(c.x0 + C::H + C::CX, c.nx);
        c.st_lo = min(max(lo - c.xt, 0), kV);
        c.st_hi = min(max(hi - c.xt, 0), kV);
        c.st_full = c.vec_out && c.st_lo == 0 && c.st_hi == kV;
        c.st_any = c.st_hi > c.st_lo;
        RowF r;
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const int x = c.x0 + 4 * (c.lane + 32 * q);   // chunk q of my lane
            r.nbq[q] = (x >= 0 && x < c.nx) ? min(16, 4 * (c.nx - x)) : 0;
            r.colq[q] = r.nbq[q] ? x : 0;
        }
        r.gF = c.in + (long long)c.y_start * c.ld_in;
        r.rf = 0;
        r.gO = c.out + (long long)c.s0 * c.ld_out + c.xt;
        const int n_it = c.s1 + 2 * T - c.y_start;    // the last stage emits row s1-1 last
        r.i_store = c.s0 - c.y_start + 2 * T;          // it emits row s0 at this iteration
        r.i_load_end = c.last_row - c.y_start - C::PF + 1;
#pragma unroll 1
        for (int j = 0; j < C::PF; j++) {
            tbf_queue<KDIFF, 8, kV, STOR_F32>(c, r, c.y_start + j <= c.last_row, false, j, 0, 0);
            cp_async_commit();
        }
        // stage s meets row 0 at i = 2s when the segment starts at the top, rows ny-1 and on from
        // i = ny-1 - y_start + 2s; a pass that forwards trailing stages runs the special loop only
        const bool partial = c.tsteps < T;
        const int i_a = partial ? n_it : (c.y_start == 0 ? min(2 * T - 1, n_it) : 0);
        const int i_b = partial ? n_it : max(i_a, min(n_it, c.ny - 1 - c.y_start));
        const int i_h = (partial || c.y_start == 0) ? 0 : min(4 * T - 4, i_b);
        int i = 0;
        // (one body for the special rows of the top and the bottom: cold code, see tb2f_kernel.cuh)
#pragma unroll 1
        for (; i < i_h; i++) star_row<T, MODE_HEAD>(c, k, A, i, r);
#pragma unroll 1
        for (int part = 0; part < 2; part++) {
            const int end = part == 0 ? i_a : n_it;
#pragma unroll 1
            for (; i < end; i++) star_row<T, MODE_SPECIAL>(c, k, A, i, r);
            if (part == 1) break;
            auto rows = [&](auto mode) {
#pragma unroll 1
                for (; i < i_b; i++) star_row<T, decltype(mode)::value>(c, k, A, i, r);
            };
            if (c.edge == 0) rows(std::integral_constant<int, MODE_PLAIN>{});
            else if (c.edge == 1) rows(std::integral_constant<int, MODE_EDGE>{});
            else rows(std::integral_constant<int, MODE_GHOST>{});
        }
        cp_async_wait<0>();
        __syncwarp();
    }
}

const void *star2f_fn(int T)
{
    switch (T) {
    case 1: return reinterpret_cast<const void *>(&k_star2f<1>);
    case 2: return reinterpret_cast<const void *>(&k_star2f<2>);
    case 4: return reinterpret_cast<const void *>(&k_star2f<4>);
    default: return nullptr;
    }
}

}  // namespace

int star2f_tile_width() { return RingS::BX; }
int star2f_compute_width() { return RingS::CX; }

cudaError_t star2f_prepare(int T, int *blocks_per_sm)
{
    const void *fn = star2f_fn(T);
    if (!fn) return cudaErrorInvalidValue;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fn, 32, RingS::SMEM);
}

cudaError_t star2f_launch(int T, const Pass2D &p, const StarCoef2 &k, cudaStream_t st)
{
    const void *fn = star2f_fn(T);
    if (!fn) return cudaErrorInvalidValue;
    void *args[] = {const_cast<Pass2D *>(&p), const_cast<StarCoef2 *>(&k)};
    return cudaLaunchKernel(fn, dim3(p.ctas), dim3(32), args, RingS::SMEM, st);
}

}  // namespace stn
