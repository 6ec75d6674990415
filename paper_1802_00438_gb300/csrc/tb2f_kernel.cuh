// 2D temporally-blocked Jacobi sweep, contracted arithmetic (fused multiply-adds): one pass
// advances the grid by `tsteps` (<= T) steps.
//
// Same blocking as the exact kernel (tb2d_kernel.cuh; arXiv 1802.00438 Sec. 3.1-3.2, Eq. 2):
// an overlapped x-tile streamed along y through a chain of T stages, stage s computing time
// step s+1 one row behind stage s-1, halos computed redundantly, only the compute block stored,
// trailing stages forwarding when the pass fuses fewer than T steps, clamped boundary
// (Sec. 5.1) at every stage.
//
// What differs is how a stage holds its window.  When row y of time s reaches stage s it
// completes row y-1 and starts rows y and y+1:
//   out(y-1) = P + cs * d                      (the only operation on the stage-to-stage path)
//   P'       = Q + cc * d + cw * d_w + ce * d_e  (row y, missing only its south term)
//   Q'       = cn * d                           (row y+1's north term)
// Hotspot 2D, c + sdc*(p + (n+s-2c)*Ry + (e+w-2c)*Rx + (amb-c)*Rz), uses the same split of its
// expansion cc*c + cx*(e+w) + cy*(n+s) - cz*c + src (cx = sdc*Rx, cy = sdc*Ry, cz = sdc*Rz,
// cc = 1 - 2cx - 2cy exact in float32, src = sdc*(p + amb*Rz) a per-cell map built once per run):
//   out(y-1) = P + cy * d
//   P'       = Q + cx * (d_e + d_w) + cc * d - cz * d
//   Q'       = cy * d + src(y+1)
// P' accumulates on top of Q and Q' is written where P was, so the two partial rows trade
// places every row: the row loop is unrolled twice with the roles swapped and every update is
// in place (no register copies).  Counted work per cell is unchanged (Table 2: 9 and 15 flops,
// issued as 5 and 6 operations; the plain-power Hotspot instances of the allocation-free entry
// point issue 9).
//
// Packed arithmetic: every operation works on a pair of cells (fma.rn.f32x2 and its add and
// multiply; each half is rounded like the scalar operation, so the results are the same bits).
// The kernel is bound by instruction issue, not by the FMA pipe: a packed operation holds the
// pipe for two cycles but takes one issue slot, and leaves the other to the shuffles, loads and
// integer work.  A pair is cells p and p + V/2 of a thread, not neighbours: then the west and
// east neighbours of a pair are the pairs p-1 and p+1 as they lie, and only the two outermost
// pairs mix halves (pairs of adjacent cells would need ten register moves per eight cells and
// stage).  Field rows, read once per pass from the ring, are paired by register moves; the
// source map, read again by every stage, is stored in pair order (src_pos), so that a 16-byte
// load yields two pairs.  Stage 0 keeps partial rows like the others: it reads one ring row per
// iteration (the direct form read three, and would have to pair each).
// Measured (GB300), scalar kernel on even ranges -> this one on dealt segments: 16384^2 Hotspot
// 2928 -> 3200 GCell/s, diffusion 3753 -> 4466, 8192^2 Hotspot with bf16 storage 2032 -> 2580,
// 3001 x 2003 Hotspot 1053 -> 1545, 3000 x 2000 diffusion 1907.
// What bounds it now (ncu, 6144^2): Hotspot FMA pipe 58 % busy, issue 57 %, shared memory 64 %
// (every stage reads its source row), two warps per scheduler; diffusion 58 / 52 / 30 %.
//
// GPU mapping: one warp per block; a tile is BX = 32*V cells wide incl. halos of
// H = roundup(T, V) cells per side; thread = V consecutive cells; x-neighbours of a thread's
// edge cells by shuffle (the warp edge is the tile edge, inside the halo).  Field and power
// rows arrive through shared-memory rings filled by cp.async PF rows ahead.  The power ring
// keeps a mirrored copy of its first PW-1 slots, so the PW = T + 1 power rows an iteration may
// read are consecutive slots: one base address per row, constant offsets per stage.  The power
// rows run one row ahead of the field rows (receiving row y, a stage starts row y+1).
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "tb2d_kernel.cuh"

namespace stn {

enum { STOR_F32 = 0, STOR_BF16 = 1, STOR_F16 = 2 };
// Flag added to STOR (Hotspot): the power ring holds the source map sdc*(p + amb*Rz) instead of
// p, and the coefficients are the expanded weights (hot_coeffs_src), so a stage issues six
// operations per cell instead of nine.  Float32 plans stage a map built once per run; 16-bit
// plans code the map itself in place of the power map.
__host__ __device__ constexpr int stor_fmt(int s) { return s & 3; }
__host__ __device__ constexpr bool stor_src(int s) { return (s & STOR_SRC) != 0; }
__host__ __device__ constexpr bool stor_all(int s) { return (s & STOR_ALL) != 0; }

template <int KIND, int T, int V, int STOR = STOR_F32>
struct TB2F {
    static constexpr int BX = 32 * V;
    // a multiple of V: tile origins and x = 0 then fall on a lane's first cell, and the source
    // map's V-cell groups (pair order) on lanes, for every T of a plan
    static constexpr int H = (T + V - 1) / V * V;
    static constexpr int CX = BX - 2 * H;
    static constexpr int PF = 4;                                    // rows requested ahead
    // 16-bit storage: the rows in flight wait in the staging rings and are decoded on arrival,
    // a field row into registers, a power row into the float ring; float32 rows land in the
    // float rings directly
    static constexpr bool Q16 = stor_fmt(STOR) != STOR_F32;
    static constexpr int NBF = Q16 ? 0 : PF + 1;                    // field rows i .. i+PF
    static constexpr int PW = T + 1;                                // power rows in use:
                                                                    // i-T+1 .. i+1
    static constexpr int NBP = (KIND == KTHERM) ? (Q16 ? PW : PW + PF) : 0;       // power ring
    static constexpr int NBPX = (KIND == KTHERM) ? (NBP + PW - 1) : 0;  // incl. mirror
    static constexpr int NS = T;                                    // partial-sum stages
    static constexpr int HV = V / 2;                                // packed pairs per thread
    // the power ring holds the source map with each V-cell group in pair order (src_pos), so
    // a 16-byte load yields two packed pairs; plain-power rows and float32 field rows arrive in
    // grid order
    static constexpr bool PPAIR = stor_src(STOR);
    static constexpr int ROWB = BX * 4;                             // bytes per ring row
    // 16-bit storage: rows arrive raw (32-byte header of block codes + 2 bytes per cell) in a
    // staging ring of PF+1 rows per input and are decoded into the float rings once
    static constexpr int NBR = Q16 ? PF + 1 : 0;
    static constexpr int RAWB = 32 + 2 * BX;
    static constexpr size_t SMEM = (size_t)(NBF + NBPX) * ROWB +
                                   (size_t)NBR * RAWB * (KIND == KTHERM ? 2 : 1);
    static_assert(V % 4 == 0 && V <= 8, "V must be 4 or 8");
    static_assert(CX > 0, "tile narrower than its halos");
};

// Coefficients as pairs of equal values, the operands of the packed float32 operations.
struct CoefF {
    // diffusion: cc, cw, ce, cs, cn; Hotspot: sdc, Rx, Ry, Rz, amb, sdc*Ry, -2*Ry; source-map
    // Hotspot kernels (STOR_SRC): cc, cx, cy, -cz, amb, cy, 0 (host-made, hot_coeffs_src)
    float2 a0, a1, a2, a3, a4, a5, a6;
};

__device__ __forceinline__ float4 lds128(uint32_t a)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(a));
    return v;
}

__device__ __forceinline__ float lds32(uint32_t a)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];\n" : "=f"(v) : "r"(a));
    return v;
}

// Ring rows are stored with their 16-byte chunks rotated inside each 128-byte group: chunk g
// (cells 4g .. 4g+3) sits at chunk position ring_pos(g).  A warp's 16-byte accesses are served
// eight lanes at a time, so they are conflict-free when those eight lanes hit eight different
// 16-byte bank groups.  The copies into a row (lane L writes chunk L + 32q) and, with V = 8,
// the reads of a thread's own cells (lane L reads chunks 2L and 2L + 1) would otherwise meet
// only four bank groups per eight lanes; with the rotation both meet all eight.
__host__ __device__ constexpr uint32_t ring_pos(uint32_t g)
{
    return (g & ~7u) | ((g + (g >> 3)) & 7u);
}

// byte offset of cell x in a ring row
__host__ __device__ constexpr uint32_t ring_cell(uint32_t x)
{
    return 16u * ring_pos(x >> 2) + 4u * (x & 3u);
}

__device__ __forceinline__ void cp16(uint32_t dst, const void *src, int nbytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(nbytes)
                 : "memory");
}

__device__ __forceinline__ void cp4(uint32_t dst, const void *src, int nbytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(dst), "l"(src), "r"(nbytes)
                 : "memory");
}

__device__ __forceinline__ void cp8(uint32_t dst, const void *src, int nbytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(dst), "l"(src), "r"(nbytes)
                 : "memory");
}

__device__ __forceinline__ uint2 lds64u(uint32_t a)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];\n" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}

__device__ __forceinline__ void sts128(uint32_t a, float x, float y, float z, float w)
{
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"r"(a), "f"(x), "f"(y), "f"(z),
                 "f"(w)
                 : "memory");
}

// 16-bit codes: bf16 / fp16 bit patterns of q in [-1, 1]
template <int STOR>
__device__ __forceinline__ float q2f(unsigned q)
{
    if (stor_fmt(STOR) == STOR_BF16) return __uint_as_float(q << 16);
    return __half2float(__ushort_as_half((unsigned short)q));
}

// two codes packed in one word (first argument in the low half), each rounded to nearest even
template <int STOR>
__device__ __forceinline__ unsigned f2q2(float a, float b)
{
    if (stor_fmt(STOR) == STOR_BF16) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        return *reinterpret_cast<const unsigned *>(&h);
    }
    // fp16 stops at 65504: a block whose cells lie further than that from its offset
    // saturates instead of storing an infinity
    const __half2 h = __floats2half2_rn(fminf(fmaxf(a, -65504.f), 65504.f),
                                        fminf(fmaxf(b, -65504.f), 65504.f));
    return *reinterpret_cast<const unsigned *>(&h);
}

struct CtxF {
    const float *__restrict__ in;
    float *__restrict__ out;
    const float *__restrict__ pw;
    long long ld_in, ld_out, ld_pw;
    uint32_t sF, sP;       // shared byte addresses of the field and power rings
    int nx, ny, tsteps;
    int x0, xt;
    int y_start, last_row, s0, s1;
    unsigned lmask, rmask;
    int st_lo, st_hi;
    bool st_full, st_any;
    int edge;              // clamped x edges of my tile: 0 none, 1 lane-aligned ones, 2 any
    int vec_in, vec_out, vec_pw;
    int lane;
    uint32_t oq[2];        // byte offsets in a ring row of my cells' 16-byte chunks
    uint32_t wq[2];        // byte offsets of the chunks I copy into a ring row
    // 16-bit storage
    uint32_t sRF, sRP;     // staging rings (raw field / raw power rows)
    const uint16_t *qin, *qpw;
    uint16_t *qout;
    const float2 *min_, *mpw;   // block codes (offset, scale) per (row, tile column)
    float2 *mout;
    long long ld_q;        // row pitch of 16-bit grids (cells)
    int ntx, tx;           // tile columns; my tile column
    int msel;              // which of the three blocks of a loaded row my cells belong to
    float *st_states;      // trajectory passes (STOR_ALL): where step t's rows go
    long long st_stride;
};

// my V cells of the ring row at byte address row, as pairs: (x, y) of v[p] are cells p and
// p + V/2.  PAIR: the row is stored in pair order, each 16-byte load is two pairs as they are.
template <int V, bool PAIR>
__device__ __forceinline__ void lds_row(uint32_t row, const CtxF &c, float2 (&v)[V / 2])
{
    const float4 a = lds128(row + c.oq[0]);
    if (V == 8) {
        const float4 b = lds128(row + c.oq[1]);
        if (PAIR) {
            v[0] = make_float2(a.x, a.y);
            v[1] = make_float2(a.z, a.w);
            v[V / 2 - 2] = make_float2(b.x, b.y);
            v[V / 2 - 1] = make_float2(b.z, b.w);
        } else {
            v[0] = make_float2(a.x, b.x);
            v[1] = make_float2(a.y, b.y);
            v[V / 2 - 2] = make_float2(a.z, b.z);
            v[V / 2 - 1] = make_float2(a.w, b.w);
        }
    } else {
        v[0] = PAIR ? make_float2(a.x, a.y) : make_float2(a.x, a.z);
        v[1] = PAIR ? make_float2(a.z, a.w) : make_float2(a.y, a.w);
    }
}

// cell j of a thread's packed row
template <int H>
__device__ __forceinline__ float cell(const float2 (&v)[H], int j)
{
    return j < H ? v[j].x : v[j - H].y;
}

// Clamped edges of a packed row, before its neighbours are formed: in a warp that holds
// x = nx-1 the ghost cell to its right takes the edge cell's value (a ghost's own value is
// never used), or e_in when the edge is the lane's last cell; x = 0 is always a lane's cell 0
// (tile origins are multiples of V), whose west value is its own.
// GHOST = false: for warps whose only edges are x = 0 and an x = nx-1 on a lane's last cell.
template <int V, bool GHOST>
__device__ __forceinline__ void edge_fix(const CtxF &c, float2 (&d)[V / 2], float &w_in, float &e_in)
{
    constexpr int H = V / 2;
    e_in = ((c.rmask >> (V - 1)) & 1u) ? d[H - 1].y : e_in;
    w_in = (c.lmask & 1u) ? d[0].x : w_in;
    if (!GHOST) return;
#pragma unroll
    for (int j = V - 2; j >= 0; j--) {
        const bool g = (c.rmask >> j) & 1u;
        const float edge = cell(d, j);
        if (j + 1 < H) d[j + 1 < H ? j + 1 : 0].x = g ? edge : d[j + 1 < H ? j + 1 : 0].x;
        else d[j + 1 < H ? 0 : j + 1 - H].y = g ? edge : d[j + 1 < H ? 0 : j + 1 - H].y;
    }
}

// Start row y+1: Xq = its north term (+ its power for Hotspot), written over the finished P.
template <int KIND, int V, bool PPAIR>
__device__ __forceinline__ void qf(const CtxF &c, const CoefF &k, const float2 (&d)[V / 2],
                                   uint32_t p_next, float2 (&Xq)[V / 2])
{
    if (KIND == KDIFF) {
#pragma unroll
        for (int j = 0; j < V / 2; j++) Xq[j] = __fmul2_rn(k.a4, d[j]);
    } else {
        float2 p[V / 2];
        lds_row<V, PPAIR>(p_next, c, p);
#pragma unroll
        for (int j = 0; j < V / 2; j++) Xq[j] = __ffma2_rn(k.a2, d[j], p[j]);
    }
}

// One stage on the arrival of row y (values d, time s).  Xp holds P (row y-1, all but its
// south term), Xq holds Q (row y's north term).  Emits out = row y-1 at time s+1, leaves
// row y's P in Xq and row y+1's Q in Xp.
// SWAP = true: P' is built on top of Q in Xq and Q' is written to Xp (the caller alternates the
// arrays every row).  SWAP = false: P' goes back to Xp and Q' to Xq (no alternation; the
// register allocator decides whether that needs copies).
template <int KIND, int V, int MODE, bool SWAP, int STOR>
__device__ __forceinline__ void stf(const CtxF &c, const CoefF &k, int y, bool fwd,
                                    float2 (&Xp)[V / 2], float2 (&Xq)[V / 2], float2 (&d)[V / 2],
                                    uint32_t p_y, uint32_t p_next, float2 (&out)[V / 2])
{
    constexpr int H = V / 2;
    constexpr bool SP = MODE == MODE_SPECIAL;
    constexpr bool ED = MODE != MODE_PLAIN;
    constexpr bool PPAIR = stor_src(STOR);
    if (SP && fwd) {   // beyond this pass's step count: row y-1 of time s passes unchanged
#pragma unroll
        for (int j = 0; j < H; j++) {
            out[j] = Xp[j];
            if (SWAP) Xq[j] = d[j];   // becomes "P" of the next row: forwarded one row later
            else Xp[j] = d[j];
        }
        return;
    }
    const float2 cs = (KIND == KDIFF) ? k.a3 : k.a5;
#pragma unroll
    for (int j = 0; j < H; j++) out[j] = __ffma2_rn(cs, d[j], Xp[j]);
    if (SP && y == c.ny) {   // row ny-1 was completed on arrival (its south is itself)
#pragma unroll
        for (int j = 0; j < H; j++) out[j] = Xp[j];
    }
    if (SP && y == 0) qf<KIND, V, PPAIR>(c, k, d, p_y, Xq);   // top: the row above row 0 is row 0
    // x-neighbours: west of pair p is pair p-1, east of pair p is pair p+1; only the outermost
    // pairs take a value from the neighbour lane and one across the halves
    float w_in = __shfl_sync(0xffffffffu, d[H - 1].y, (c.lane + 31) & 31);
    float e_in = __shfl_sync(0xffffffffu, d[0].x, (c.lane + 1) & 31);
    if (ED) edge_fix<V, MODE != MODE_EDGE>(c, d, w_in, e_in);
    float2(&Pn)[H] = SWAP ? Xq : Xp;   // where row y's P goes
    float2(&Qn)[H] = SWAP ? Xp : Xq;   // where row y+1's Q goes
#pragma unroll
    for (int j = 0; j < H; j++) {
        constexpr int L = H - 1;
        const float2 dw = j > 0 ? d[j > 0 ? j - 1 : 0] : make_float2(w_in, d[L].x);
        const float2 de = j < L ? d[j < L ? j + 1 : j] : make_float2(d[0].y, e_in);
        if (KIND == KDIFF) {
            float2 t = __ffma2_rn(k.a0, d[j], Xq[j]);
            t = __ffma2_rn(k.a1, dw, t);
            Pn[j] = __ffma2_rn(k.a2, de, t);
        } else {
            // the outermost pairs add their halves one by one: building a pair for the packed
            // addition would cost as many register moves (16384^2 Hotspot 2967 -> 3045 GCell/s)
            float2 ew;
            if (j == 0 || j == L)
                ew = make_float2(__fadd_rn(de.x, dw.x), __fadd_rn(de.y, dw.y));
            else
                ew = __fadd2_rn(de, dw);
            if (stor_src(STOR)) {
                // Q (cy*n + src) + cx*(e + w) + cc*c - cz*c: the expanded weights, cc exact
                float2 t = __ffma2_rn(k.a1, ew, Xq[j]);
                t = __ffma2_rn(k.a0, d[j], t);
                Pn[j] = __ffma2_rn(k.a3, d[j], t);
            } else {
                const float2 t2 = __ffma2_rn(make_float2(-2.0f, -2.0f), d[j], ew);
                float2 t = __ffma2_rn(t2, k.a1, Xq[j]);
                const float2 t3 = __ffma2_rn(make_float2(-1.0f, -1.0f), d[j], k.a4);   // amb - c
                t = __ffma2_rn(t3, k.a3, t);
                t = __ffma2_rn(k.a6, d[j], t);
                Pn[j] = __ffma2_rn(k.a0, t, d[j]);
            }
        }
    }
    qf<KIND, V, PPAIR>(c, k, d, p_next, Qn);
    if (SP && y == c.ny - 1) {   // bottom: complete row ny-1 now with south = itself
#pragma unroll
        for (int j = 0; j < H; j++) Pn[j] = __ffma2_rn(cs, d[j], Pn[j]);
    }
}

// Per-thread, per-segment state of the row loop.
struct RowF {
    const float *gF, *gP;   // field / power pointers at column x0 + 4*lane of the next row to load
    float *gO;              // output pointer at my first cell of the next row to store
    int colq[2];            // per 16-byte chunk: column offset to copy from (0 when off-grid)
    int nbq[2];             // per chunk: bytes inside the grid (0..16)
    int colp[2], nbp[2];    // the same for source-map rows (pair order, padded rows)
    int rf, rp;             // ring slots of field row i / of power row i
    int i_store;            // first iteration that stores a row
    int i_load_end;         // iterations i < i_load_end queue row i+PF
    // 16-bit storage
    const uint16_t *qF, *qP;     // raw rows of the next row to load (at column x0)
    const float2 *mF, *mP;       // block-code rows of the next row to load
    uint16_t *qO;                // raw output at my first cell of the next row to store
    float2 *mO;                  // block-code row of the next row to store
    int rr;                      // staging slot of row i
    int nbr;                     // my raw bytes inside the grid (0 .. 2V), colr: my column
    int colr;
};

// my cells of the compute block to g (row-major, cell 0 at g)
template <int V>
__device__ __forceinline__ void st_cells(const CtxF &c, float *g, const float2 (&v)[V / 2])
{
    if (c.st_full) {
#pragma unroll
        for (int q = 0; q < V / 4; q++)
            *reinterpret_cast<float4 *>(g + 4 * q) = make_float4(
                cell(v, 4 * q), cell(v, 4 * q + 1), cell(v, 4 * q + 2), cell(v, 4 * q + 3));
    } else if (c.st_any) {
#pragma unroll
        for (int j = 0; j < V; j++)
            if (j >= c.st_lo && j < c.st_hi) g[j] = cell(v, j);
    }
}

// Trajectory passes: the row `row` of step t+1 of the pass (stage t's output) into state t,
// for the steps before the pass's last (whose rows go to the pass output) and the rows of
// this segment, compute-block cells only.
template <int V>
__device__ __forceinline__ void tbf_store_state(const CtxF &c, int t, int row,
                                                const float2 (&v)[V / 2])
{
    if (t >= c.tsteps - 1 || row < c.s0 || row >= c.s1) return;
    float *g = c.st_states + (long long)t * c.st_stride + (long long)row * c.ld_out + c.xt;
    st_cells<V>(c, g, v);
}

// One row iteration.  PH selects which of A/B holds P (PH = 0: A) for every stage.  Stage s
// receives row R0-s of time s (stage 0: row R0 in `out`) and emits row R0-s-1 of time s+1 in
// `out`; pbase is the slot of power row R0+1, row R0+1-t sits t slots below it.
template <int KIND, int T, int V, int MODE, int PH, bool SWAP, int STOR>
__device__ __forceinline__ void tbf_iter(const CtxF &c, const CoefF &k,
                                         float2 (&A)[TB2F<KIND, T, V>::NS][V / 2],
                                         float2 (&B)[TB2F<KIND, T, V>::NS][V / 2], int i,
                                         float2 (&out)[V / 2], uint32_t pbase, float *gO,
                                         const RowF &r, bool store)
{
    using C = TB2F<KIND, T, V, STOR>;
    const int R0 = c.y_start + i;
    float2 d[V / 2];
#pragma unroll
    for (int s = 0; s < T; s++) {
        // pipeline fill of a segment that starts inside the grid: stage s gets its first valid
        // row at i = 2s (row y_start + s), before that it and the stages behind it have nothing
        // to do
        if (MODE == MODE_HEAD && i < 2 * s) break;
#pragma unroll
        for (int j = 0; j < V / 2; j++) d[j] = out[j];
        stf<KIND, V, MODE, SWAP, STOR>(c, k, R0 - s, s >= c.tsteps, PH == 0 ? A[s] : B[s],
                                       PH == 0 ? B[s] : A[s], d, pbase - (s + 1) * C::ROWB,
                                       pbase - s * C::ROWB, out);
        if (stor_all(STOR) && s < T - 1) tbf_store_state<V>(c, s, R0 - s - 1, out);
    }
    if (store) {
        if (stor_fmt(STOR) == STOR_F32) {
            st_cells<V>(c, gO, out);
        } else {
            // encode the row segment of this tile as q = x - offset with the offset the value of
            // the block's first cell (tile column tx*CX: lane H/V, its cell 0, in the grid for
            // every tile) and scale 1.  bf16 and fp16 are floating-point formats, so q keeps 8
            // (11) significant bits of each cell's distance from the offset at any magnitude:
            // the error per cell is at most half an ulp of |x - offset| <= the block's spread,
            // and no block-wide minimum and maximum are needed
            const float mid = __shfl_sync(0xffffffffu, out[0].x, C::H / V);
            unsigned q2[V / 2];   // pairs of codes, cell 2i in the low half
#pragma unroll
            for (int j = 0; j < V / 2; j++) 
                q2[j] = f2q2<STOR>(cell(out, 2 * j) - mid, cell(out, 2 * j + 1) - mid);
            if (c.st_full) {
#pragma unroll
                for (int t = 0; t < V / 4; t++)
                    *reinterpret_cast<uint2 *>(r.qO + 4 * t) = make_uint2(q2[2 * t], q2[2 * t + 1]);
            } else if (c.st_any) {
#pragma unroll
                for (int j = 0; j < V; j++)
                    if (j >= c.st_lo && j < c.st_hi)
                        r.qO[j] = (uint16_t)((j & 1) ? (q2[j / 2] >> 16) : (q2[j / 2] & 0xffffu));
            }
            if (c.lane == 0) r.mO[c.tx] = make_float2(mid, 1.0f);
        }
    }
}

// Decode my V cells of a staged raw row (header: codes of the blocks tx-1, tx, tx+1).
template <int V, int STOR>
__device__ __forceinline__ void tbf_decode(const CtxF &c, uint32_t raw, float2 (&x)[V / 2])
{
    const uint2 cw = lds64u(raw + 8u * c.msel);
    const float2 mid = make_float2(__uint_as_float(cw.x), __uint_as_float(cw.x));
    const float2 sc = make_float2(__uint_as_float(cw.y), __uint_as_float(cw.y));
    constexpr int H = V / 2;
    float q[V];
#pragma unroll
    for (int t = 0; t < V / 4; t++) {
        const uint2 w = lds64u(raw + 32u + 2u * V * c.lane + 8u * t);
        q[4 * t] = q2f<STOR>(w.x & 0xffffu);
        q[4 * t + 1] = q2f<STOR>(w.x >> 16);
        q[4 * t + 2] = q2f<STOR>(w.y & 0xffffu);
        q[4 * t + 3] = q2f<STOR>(w.y >> 16);
    }
#pragma unroll
    for (int j = 0; j < H; j++) x[j] = __ffma2_rn(sc, make_float2(q[j], q[j + H]), mid);
}

// ... into a power ring row in pair order (and into its mirror when mirror != 0)
template <int V, int STOR>
__device__ __forceinline__ void tbf_decode_ring(const CtxF &c, uint32_t raw, uint32_t dst,
                                                uint32_t mirror)
{
    float2 x[V / 2];
    tbf_decode<V, STOR>(c, raw, x);
#pragma unroll
    for (int t = 0; t < V / 4; t++) {
        sts128(dst + c.oq[t], x[2 * t].x, x[2 * t].y, x[2 * t + 1].x, x[2 * t + 1].y);
        if (mirror) sts128(mirror + c.oq[t], x[2 * t].x, x[2 * t].y, x[2 * t + 1].x, x[2 * t + 1].y);
    }
}

// Queue the next field row (pointers in r, if f) into field slot lf and the next power row
// (if pw) into power slot lp plus its mirror; with 16-bit storage, both into staging slot lr
// instead.  The power rows run one row ahead of the field rows (a stage that receives row y
// starts row y+1).  Advances the row pointers.
template <int KIND, int T, int V, int STOR>
__device__ __forceinline__ void tbf_queue(const CtxF &c, RowF &r, bool f, bool pw, int lf, int lp,
                                          int lr)
{
    using C = TB2F<KIND, T, V, STOR>;
    if (stor_fmt(STOR) != STOR_F32) {
#pragma unroll
        for (int in = 0; in < (KIND == KTHERM ? 2 : 1); in++) {
            if (!(in == 0 ? f : pw)) continue;
            const uint32_t dr = (in == 0 ? c.sRF : c.sRP) + lr * C::RAWB;
            const uint16_t *src = in == 0 ? r.qF : r.qP;
            const float2 *m = in == 0 ? r.mF : r.mP;
#pragma unroll
            for (int t = 0; t < V / 4; t++) {
                const int nb = max(0, min(8, r.nbr - 8 * t));
                cp8(dr + 32u + 2u * V * c.lane + 8u * t, nb ? src + r.colr + 4 * t : src, nb);
            }
            if (c.lane < 6) {
                const int b = min(max(c.tx - 1 + (c.lane >> 1), 0), c.ntx - 1);
                cp4(dr + 4u * c.lane, reinterpret_cast<const float *>(m + b) + (c.lane & 1), 4);
            }
            if (in == 0) {
                r.qF += c.ld_q;
                r.mF += c.ntx;
            } else {
                r.qP += c.ld_q;
                r.mP += c.ntx;
            }
        }
        return;
    }
    const uint32_t df = c.sF + lf * C::ROWB;
    const uint32_t dp = c.sP + lp * C::ROWB;
    if (f) {
        if (c.vec_in) {
#pragma unroll
            for (int q = 0; q < V / 4; q++) cp16(df + c.wq[q], r.gF + r.colq[q], r.nbq[q]);
        } else {   // rows not 16-byte aligned: element-wise copies
#pragma unroll
            for (int q = 0; q < V / 4; q++)
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const int nb = (4 * j < r.nbq[q]) ? 4 : 0;
                    cp4(df + c.wq[q] + 4 * j, r.gF + (nb ? r.colq[q] + j : 0), nb);
                }
        }
        r.gF += c.ld_in;
    }
    if (KIND == KTHERM && pw) {
        // source-map rows are padded to 32 cells, every chunk of a group that reaches into the
        // grid is whole (pair order puts the group's cells in both of its chunks)
        if (C::PPAIR || c.vec_pw) {
#pragma unroll
            for (int q = 0; q < V / 4; q++) {
                const int nb = C::PPAIR ? r.nbp[q] : r.nbq[q];
                const float *src = r.gP + (C::PPAIR ? r.colp[q] : r.colq[q]);
                cp16(dp + c.wq[q], src, nb);
                if (lp < C::PW - 1) cp16(dp + C::NBP * C::ROWB + c.wq[q], src, nb);
            }
        } else {
#pragma unroll
            for (int q = 0; q < V / 4; q++)
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const int nb = (4 * j < r.nbq[q]) ? 4 : 0;
                    const float *src = r.gP + (nb ? r.colq[q] + j : 0);
                    cp4(dp + c.wq[q] + 4 * j, src, nb);
                    if (lp < C::PW - 1) cp4(dp + C::NBP * C::ROWB + c.wq[q] + 4 * j, src, nb);
                }
        }
        r.gP += c.ld_pw;
    }
}

// One row: wait for row i, run the stages, queue row i+PF, advance pointers and rings.
template <int KIND, int T, int V, int MODE, int PH, bool SWAP, int STOR>
__device__ __forceinline__ void tbf_step(const CtxF &c, const CoefF &k,
                                         float2 (&A)[TB2F<KIND, T, V>::NS][V / 2],
                                         float2 (&B)[TB2F<KIND, T, V>::NS][V / 2], int i, RowF &r)
{
    using C = TB2F<KIND, T, V, STOR>;
    cp_async_wait<C::PF - 1>();   // field row i and power row i+1 have landed
    __syncwarp();
    float2 row[V / 2];
    if (C::Q16) {
        if (KIND == KTHERM)   // (for STOR_SRC the coded map is the source map itself)
            tbf_decode_ring<V, STOR>(c, c.sRP + r.rr * C::RAWB, c.sP + r.rp * C::ROWB,
                                     r.rp < C::PW - 1 ? c.sP + (C::NBP + r.rp) * C::ROWB : 0u);
        tbf_decode<V, STOR>(c, c.sRF + r.rr * C::RAWB, row);
        __syncwarp();
    } else {
        lds_row<V, false>(c.sF + r.rf * C::ROWB, c, row);
    }
    const uint32_t pbase = c.sP + ((KIND == KTHERM && r.rp < C::PW - 1) ? C::NBP + r.rp : r.rp) * C::ROWB;
    const bool store = i >= r.i_store;
    tbf_iter<KIND, T, V, MODE, PH, SWAP, STOR>(c, k, A, B, i, row, pbase, r.gO, r, store);
    if (store) {
        if (stor_fmt(STOR) == STOR_F32) r.gO += c.ld_out;
        else {
            r.qO += c.ld_q;
            r.mO += c.ntx;
        }
    }
    __syncwarp();
    int lf = 0, lp = 0, lr = 0;   // slots of rows i+PF (field), i+PF+1 (power), or the staging slot
    if (!C::Q16) {
        lf = r.rf == 0 ? C::NBF - 1 : r.rf - 1;   // row i-1's slot (NBF = PF + 1)
        if (KIND == KTHERM) {
            lp = r.rp + C::PF;
            lp -= (lp >= C::NBP) ? C::NBP : 0;
        }
    } else {
        lr = r.rr == 0 ? C::NBR - 1 : r.rr - 1;
    }
    tbf_queue<KIND, T, V, STOR>(c, r, i < r.i_load_end, i + 1 < r.i_load_end, lf, lp, lr);
    cp_async_commit();
    if (!C::Q16) r.rf = (r.rf + 1 == C::NBF) ? 0 : r.rf + 1;
    if (KIND == KTHERM) r.rp = (r.rp + 1 == C::NBP) ? 0 : r.rp + 1;
    if (C::Q16) r.rr = (r.rr + 1 == C::NBR) ? 0 : r.rr + 1;
}

// Rows [s0, s1) of tile column tx of one grid's pass.
template <int KIND, int T, int V, bool SWAP, int STOR>
__device__ __forceinline__ void tbf_segment(const Pass2D &p, const int tx, const int s0, const int s1,
                                          float2 (&A)[TB2F<KIND, T, V>::NS][V / 2],
                                          float2 (&B)[TB2F<KIND, T, V>::NS][V / 2], float *smem)
{
    using C = TB2F<KIND, T, V, STOR>;
    CtxF c;
    c.in = p.in;
    c.out = p.out;
    c.pw = p.pw;
    c.ld_in = p.ld_in;
    c.ld_out = p.ld_out;
    c.ld_pw = p.ld_pw;
    c.sF = smem_u32(smem);
    c.sP = c.sF + C::NBF * C::ROWB;
    c.sRF = c.sP + C::NBPX * C::ROWB;
    c.sRP = c.sRF + C::NBR * C::RAWB;
    c.qin = static_cast<const uint16_t *>(p.qin);
    c.qpw = static_cast<const uint16_t *>(p.qpw);
    c.qout = static_cast<uint16_t *>(p.qout);
    c.min_ = p.min_;
    c.mpw = p.mpw;
    c.mout = p.mout;
    c.ld_q = p.ld_q;
    c.ntx = p.ntx;
    c.nx = p.nx;
    c.ny = p.ny;
    c.tsteps = p.tsteps;
    c.vec_in = p.vec_in;
    c.vec_out = p.vec_out;
    c.vec_pw = p.vec_pw;
    c.lane = threadIdx.x;
#pragma unroll
    for (int q = 0; q < 2; q++) {
        c.oq[q] = 16u * ring_pos(min(V / 4 * c.lane + q, V / 4 * c.lane + V / 4 - 1));
        c.wq[q] = 16u * ring_pos(c.lane + 32 * min(q, V / 4 - 1));
    }
    CoefF k;
    const float a3 = stor_src(STOR) ? -p.kf[3] : p.kf[3];
    k.a0 = make_float2(p.kf[0], p.kf[0]);
    k.a1 = make_float2(p.kf[1], p.kf[1]);
    k.a2 = make_float2(p.kf[2], p.kf[2]);
    k.a3 = make_float2(a3, a3);
    k.a4 = make_float2(p.kf[4], p.kf[4]);
    k.a5 = make_float2(p.kf[5], p.kf[5]);   // Hotspot: sdc * Ry
    k.a6 = make_float2(p.kf[6], p.kf[6]);   // Hotspot: -2 Ry (source-map kernels: unused)
    c.st_states = p.states;
    c.st_stride = p.state_stride;

    {
        c.s0 = s0;
        c.s1 = s1;
        c.x0 = tx * C::CX - C::H;
        c.xt = c.x0 + c.lane * V;
        c.y_start = max(0, s0 - c.tsteps);
        c.last_row = min(c.ny - 1, s1 - 1 + c.tsteps);
        {
            const int lcl = (c.xt <= 0 && 0 < c.xt + V) ? -c.xt : -1;
            const int rcl = (c.xt <= c.nx - 1 && c.nx - 1 < c.xt + V) ? (c.nx - 1 - c.xt) : -1;
            c.lmask = lcl >= 0 ? (1u << lcl) : 0u;
            c.rmask = rcl >= 0 ? (1u << rcl) : 0u;
            c.edge = __any_sync(0xffffffffu, rcl >= 0 && rcl < V - 1) ? 2
                     : __any_sync(0xffffffffu, lcl >= 0 || rcl >= 0) ? 1 : 0;
        }
        {
            const int lo = max(c.x0 + C::H, 0), hi = min(c.x0 + C::H + C::CX, c.nx);
            c.st_lo = min(max(lo - c.xt, 0), V);
            c.st_hi = min(max(hi - c.xt, 0), V);
            c.st_full = c.vec_out && c.st_lo == 0 && c.st_hi == V;
            c.st_any = c.st_hi > c.st_lo;
        }
        RowF r;
#pragma unroll
        for (int q = 0; q < V / 4; q++) {
            const int x = c.x0 + 4 * (c.lane + 32 * q);   // chunk q of my lane
            r.nbq[q] = (x >= 0 && x < c.nx) ? min(16, 4 * (c.nx - x)) : 0;
            r.colq[q] = r.nbq[q] ? x : 0;
            const bool in = x >= 0 && (x & ~(V - 1)) < c.nx;   // the chunk's group holds a grid cell
            r.nbp[q] = in ? 16 : 0;
            r.colp[q] = in ? x : 0;
        }
        c.tx = tx;
        c.msel = (c.xt < tx * C::CX) ? 0 : ((c.xt >= (tx + 1) * C::CX) ? 2 : 1);
        if (stor_fmt(STOR) != STOR_F32) {
            r.qF = c.qin + (long long)c.y_start * c.ld_q;
            r.mF = c.min_ + (long long)c.y_start * c.ntx;
            r.qP = (KIND == KTHERM) ? c.qpw + (long long)c.y_start * c.ld_q : nullptr;
            r.mP = (KIND == KTHERM) ? c.mpw + (long long)c.y_start * c.ntx : nullptr;
            r.qO = c.qout + (long long)s0 * c.ld_q + c.xt;
            r.mO = c.mout + (long long)s0 * c.ntx;
            r.rr = 0;
            r.colr = (c.xt >= 0 && c.xt < c.nx) ? c.xt : 0;
            r.nbr = (c.xt >= 0 && c.xt < c.nx) ? 2 * min(V, c.nx - c.xt) : 0;
        }
        r.gF = c.in + (long long)c.y_start * c.ld_in;
        r.gP = (KIND == KTHERM) ? c.pw + (long long)c.y_start * c.ld_pw : nullptr;
        r.rf = 0;
        const int n_it = s1 + T - c.y_start;           // the last stage emits row s1-1 last
        r.i_store = s0 - c.y_start + T;                 // it emits row s0 at this iteration
        r.gO = c.out + (long long)s0 * c.ld_out + c.xt;
        r.i_load_end = c.last_row - c.y_start - C::PF + 1;

        // queue the first PF field rows, and power rows 0 .. PF (row 0 with group 0: it enters
        // only where the segment starts at the grid's top)
        r.rp = KIND == KTHERM ? 1 : 0;   // slot of power row i+1 at i = 0
#pragma unroll 1
        for (int j = 0; j < C::PF; j++) {
            const int y = c.y_start + j;
            if (KIND == KTHERM && j == 0) tbf_queue<KIND, T, V, STOR>(c, r, false, true, 0, 0, C::PF);
            tbf_queue<KIND, T, V, STOR>(c, r, y <= c.last_row, y + 1 <= c.last_row, j, j + 1, j);
            cp_async_commit();
        }
        if (KIND == KTHERM && C::Q16) {   // decode power row 0
            cp_async_wait<C::PF - 1>();
            __syncwarp();
            tbf_decode_ring<V, STOR>(c, c.sRP + C::PF * C::RAWB, c.sP, c.sP + C::NBP * C::ROWB);
        }

        // the fill rows of a segment inside the grid run a loop that skips the idle stages (T^2 of
        // the segment's (rows + 2T) T stage rows, a fifth of them on a 3001 x 2003 grid, whose
        // blocks have 30 rows each: with the dealt segments 692 -> 622 us for 150 steps);
        // rows that need boundary handling: the grid's top rows (for every stage), its bottom
        // rows, and every row of a pass that forwards trailing stages
        const bool partial = (c.tsteps < T);
        const int i_a = partial ? n_it : ((c.y_start == 0) ? min(T, n_it) : 0);
        // (stage s meets row 0 at i = s when the segment starts at the top, and rows ny-1 / ny
        // from i = ny-1 - y_start on)
        const int i_b = partial ? n_it : max(i_a, min(n_it, c.ny - 1 - c.y_start));
        const int i_h = (partial || c.y_start == 0) ? 0 : min(2 * T - 2, i_b);
        int i = 0;
        // Every loop but the two of ordinary rows has one body, with the partial rows updated in
        // place: these bodies are cold code that every block fetches anew (a body per array phase
        // cost a pass several us: see kCal2D in api.cu).  With float32 rows and two sets of
        // partial rows the special rows of the top and the bottom share theirs, too (16384^2
        // diffusion 4253 -> 4469 GCell/s); the other instances are faster with one each (8192^2
        // bf16 Hotspot 5397 -> 5225 us for 200 steps).
        constexpr bool kShare = SWAP && !C::Q16;
#pragma unroll 1
        for (; i < i_h; i++) tbf_step<KIND, T, V, MODE_HEAD, 0, false, STOR>(c, k, A, B, i, r);
        auto special = [&](int end) {
#pragma unroll 1
            for (; i < end; i++) tbf_step<KIND, T, V, MODE_SPECIAL, 0, false, STOR>(c, k, A, B, i, r);
        };
        auto ordinary = [&]() {
            auto rows = [&](auto mode) {
                constexpr int M = decltype(mode)::value;
                if constexpr (SWAP) {
#pragma unroll 1
                    for (; i + 1 < i_b; i += 2) {
                        tbf_step<KIND, T, V, M, 0, true, STOR>(c, k, A, B, i, r);
                        tbf_step<KIND, T, V, M, 1, true, STOR>(c, k, A, B, i + 1, r);
                    }
                } else {
#pragma unroll 1
                    for (; i < i_b; i++) tbf_step<KIND, T, V, M, 0, false, STOR>(c, k, A, B, i, r);
                }
            };
            if (c.edge == 0) rows(std::integral_constant<int, MODE_PLAIN>{});
            else if (c.edge == 1) rows(std::integral_constant<int, MODE_EDGE>{});
#pragma unroll 1
            for (; i < i_b; i++) tbf_step<KIND, T, V, MODE_GHOST, 0, false, STOR>(c, k, A, B, i, r);
        };
        if constexpr (kShare) {
#pragma unroll 1
            for (int part = 0; part < 2; part++) {   // one copy of the special body for both ends
                special(part == 0 ? i_a : n_it);
                if (part == 1) break;
                ordinary();
            }
        } else {
            special(i_a);
            ordinary();
            special(n_it);
        }
        cp_async_wait<0>();
        __syncwarp();
    }
}


template <int KIND, int T, int V, bool SWAP, int STOR>
__global__ void __launch_bounds__(32) k_tb2f(const Pass2D p)
{
    using C = TB2F<KIND, T, V, STOR>;
    extern __shared__ __align__(16) float smem[];
    float2 A[C::NS][V / 2], B[C::NS][V / 2];
#pragma unroll
    for (int s = 0; s < C::NS; s++)
#pragma unroll
        for (int j = 0; j < V / 2; j++) A[s][j] = B[s][j] = make_float2(0.f, 0.f);
    // segments from the plan's list, or (no list) an even share of the (tile column, row) units.
    // The bounds are broadcast so that the compiler knows them, and what follows from them, to
    // be uniform across the warp and keeps it in uniform registers.
    const bool listed = p.segs != nullptr;
    long long f = listed ? __ldg(p.seg_first + blockIdx.x) : (long long)blockIdx.x * p.rows_per_cta;
    const long long fend = listed ? __ldg(p.seg_first + blockIdx.x + 1)
                                  : min(f + p.rows_per_cta, p.total_rows);
#pragma unroll 1
    while (__shfl_sync(0xffffffffu, f < fend ? 1 : 0, 0)) {
        int tx, s0, s1;
        if (listed) {
            const int4 q = __ldg(p.segs + f);
            tx = q.x;
            s0 = q.y;
            s1 = q.z;
            f++;
        } else {
            tx = (int)(f / p.ny);
            s0 = (int)(f - (long long)tx * p.ny);
            s1 = (int)min((long long)p.ny, s0 + (fend - f));
            f += s1 - s0;
        }
        tbf_segment<KIND, T, V, SWAP, STOR>(p, __shfl_sync(0xffffffffu, tx, 0),
                                            __shfl_sync(0xffffffffu, s0, 0),
                                            __shfl_sync(0xffffffffu, s1, 0), A, B, smem);
    }
}

}  // namespace stn
