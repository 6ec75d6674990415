// Host runtime of the stencil engine: plans, parameter choice, pass scheduling, validation.
//
// A run of `steps` Jacobi steps is ceil(steps / T) passes over device memory (Eq. 8 of
// arXiv 1802.00438), each pass one launch of a temporally-blocked kernel that fuses up to T
// steps; the last pass fuses the remainder (Sec. 3.2).  Passes ping-pong between the caller's
// output buffer and one plan-owned scratch grid (Sec. 2.1's second buffer), ordered so that
// the last pass lands in the output.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/stencil.h"
#include "internal.h"
#include "segments.h"

using namespace stn;

namespace {

struct PassCfg2D {
    Shape2D shape;
    int ntx = 0;
    long long total = 0, rows_per_cta = 0;
    int ctas = 0;
    int seg_off = 0;        // ints before the segments
    void *segs = nullptr;   // contracted kernel, device: [first segment of each block | segments]
    bool ready = false;
};

struct PassCfg3D {
    Shape3D shape;
    int ntx = 0, nty = 0;
    long long cols = 0, planes_per_cta = 0;
    int ctas = 0;
    int seg_off = 0;        // ints before the segments
    void *segs = nullptr;   // partial-sum kernel, device: [first segment of each block | segments]
    bool ready = false;
};

}  // namespace

struct stencil_plan_s {
    stencil_desc d;
    cudaStream_t stream = nullptr;
    int device = 0, sms = 0;
    float *scratch = nullptr;
    float *scratch2 = nullptr;  // second scratch grid, where the caller's rows are unaligned
    long long ld_scratch = 0;   // row pitch of the scratch grids, floats
    size_t scratch_bytes = 0;
    int T = 1;
    // 2D
    int V = 4, W = 4;
    std::vector<PassCfg2D> cfg2;   // indexed by kernel T
    // 3D
    int VY = 8, NW = 8, alg3 = 0, VX3 = 2;
    int *err = nullptr;   // device flag set by a kernel whose bounded wait gave up
    double model = 0.0;   // calibrated model's prediction for this plan (1000 steps), GCell/s
    int tuned = 0;        // configuration taken from the tuning cache
    PassCfg2D traj;       // trajectory passes (stencil_run_trajectory)
    float *src = nullptr;   // contracted float32 Hotspot 2D: the source map sdc*(p + amb*Rz);
                            // Hotspot 3D, unaligned rows: the power map with padded rows
    long long ld_src = 0;   // its row pitch, floats
    int ntx_star = 0, nty_star = 0;   // star diffusion (rad > 1): tiles along x and y
    int nseg_star = 1, zseg_star = 0; // 3D star: z-segments per tile column, their length
    int star_rows = 0;                // 2D star streamed by one-warp blocks (contracted, radius 2)
    std::vector<PassCfg3D> cfg3;
    // timing
    bool timing = false;
    std::vector<cudaEvent_t> ev;   // pairs, reused
    size_t ev_used = 0;
    double ms_acc = 0.0;
    long long launches = 0;
    int sticky = ST_OK;
    // 16-bit storage (2D contracted plans): ping-pong grids and block codes, coded power map
    int stor = 0;
    long long ld_q = 0;
    int cx = 0, ntx = 0;
    void *q[2] = {nullptr, nullptr};
    float2 *qm[2] = {nullptr, nullptr};
    void *qp = nullptr;
    float2 *qpm = nullptr;
    // resident tiles (2D): the whole grid on chip for the run, one cooperative launch
    int res = 0, res_vx = 4, res_nw = 0, res_nbx = 0, res_nby = 0, res_cw = 0, res_ch = 0, res_hx = 0;
    float *res_xg = nullptr;      // two exchange grids, rows of res_ld floats
    long long res_ld = 0;
    int *res_flags = nullptr;     // per block: epochs published (grow across runs)
    int res_epoch = 0;            // epoch base of the next run: no counter is above it
    int res_captured = 0;         // most epochs of a captured run: what a replay leaves counted
    long long res_wait_ns = 1000000000LL;
    int res_hold_block = -1, res_hold_epoch = -1;
};

namespace {

const int kTcand[] = {1, 2, 3, 4, 6, 8, 12, 16};

int map_cuda(cudaError_t e)
{
    if (e == cudaSuccess) return ST_OK;
    if (e == cudaErrorMemoryAllocation) return ST_ERR_OOM;
    return ST_ERR_CUDA;
}

long long cells_of(const stencil_desc &d) { return (long long)d.nx * d.ny * d.nz; }

int ncoef(const stencil_desc &d)
{
    if (d.kind == ST_DIFFUSION_VAR) return 0;   // per-cell coefficient planes on the device
    if (d.rad > 1) return 1 + (d.ndim == 2 ? 4 : 6) * d.rad;
    if (d.ndim == 2) return 5;
    return d.kind == ST_DIFFUSION ? 7 : 9;
}

bool stor_src_bits(int stor) { return (stor & STOR_SRC) != 0; }

// storage bits of a plan's 2D kernel shape: the format, plus STOR_SRC for contracted Hotspot
// kernels (they stage p + amb*Rz instead of the power map)
int shape_stor(const stencil_plan_s *p)
{
    return p->stor | ((p->d.kind == ST_THERMAL && !p->d.exact) ? STOR_SRC : 0);
}

bool available(const stencil_plan_s *p, int T)
{
    if (p->d.ndim == 2)
        return tb2d_available(Shape2D{p->d.kind, p->d.exact ? 1 : 0, T, p->V, p->W, shape_stor(p)});
    return tb3d_available(Shape3D{p->d.kind, p->d.exact ? 1 : 0, T, p->VY, p->NW, p->alg3, p->VX3});
}

// ---- parameter choice seeded by the GPU restatement of the paper's model (Eqs. 3-9) -------
//
// Calibration of the contracted 2D kernels (GB300): a pass takes a * (cell steps computed, fill
// included) / (SMs * 128 lanes * clock) + b, per compiled (kind, T, V, variant) with a in cycles
// per lane and cell step and b what a pass costs besides (launch, first rows, drain: the fewer
// warps share a scheduler the more).  Fitted on 16384^2 and 3000 x 2000; within 5 % on 8000^2 and
// 4096^2, 10 % on 1600^2, 25 % on 1000 x 600.
struct Cal2D { int kind, T, V, W; double a, b_us; };
const Cal2D kCal2D[] = {
    {0, 4, 4, 1, 13.1, 4.7},  {0, 8, 4, 1, 9.7, 7.5},   {0, 12, 4, 1, 9.7, 13.4},  {0, 4, 8, 1, 12.1, 6.2},
    {0, 6, 8, 1, 10.5, 7.2},  {0, 8, 8, 1, 8.1, 11.7},  {0, 8, 8, 0, 9.4, 9.0},    {0, 12, 4, 0, 9.9, 8.8},
    {1, 4, 4, 1, 22.7, 1.7},  {1, 8, 4, 1, 11.8, 8.3},  {1, 12, 4, 1, 11.3, 22.8}, {1, 4, 8, 1, 20.5, 3.4},
    {1, 6, 8, 1, 13.4, 10.1}, {1, 8, 8, 1, 11.4, 19.8}, {1, 8, 8, 0, 11.9, 11.4},  {1, 12, 4, 0, 12.3, 12.8},
};

struct Cand2D { int T, V, W; };

// 2D: rows of fill a segment costs, per fused step (2T rows with the idle stages skipped)
constexpr double kFill2 = 1.25;
// 2D: relative cost of a row of an edge tile column (see segments_2d)
constexpr double kEdge2 = 1.05, kGhost2 = 1.45;
// 2D: how far the oldest (youngest) block of a scheduler is ahead (behind): see segments_2d
constexpr double kAhead2 = 0.04;
// 2D: rows a segment that starts or ends at the grid's top or bottom costs besides, per fused step
// (8 and 4 cells per thread)
constexpr double kTop2V8 = 3.0, kTop2V4 = 1.5;

// seg_rows = 0: the plan's own launch geometry; > 0: a batch launch, whose segments hold about
// seg_rows rows across all its grids and whose launch cost the grids share
double model_gcells_2d(const stencil_desc &d, int sms, const Cand2D &k, int bps, int steps,
                       int seg_rows = 0)
{
    double ops = 14.0 + 32.0 / k.T, fixed = 8e-6;   // forced (T, V) without a calibration
    for (const Cal2D &c : kCal2D)
        if (c.kind == d.kind && c.T == k.T && c.V == k.V && c.W == k.W) {
            ops = c.a;
            fixed = c.b_us * 1e-6;
        }
    // one-warp blocks, as many as are resident, over the rows of every tile column
    const int halo = (k.T + k.V - 1) / k.V * k.V;   // tb2d_halo
    const long long cx = 32LL * k.V - 2 * halo;
    const double units = (double)((d.nx + cx - 1) / cx) * d.ny;
    const double rows = seg_rows > 0 ? seg_rows : std::max(1.0, units / ((double)sms * bps));
    stencil_gpu_model_in m = {};
    m.ndim = 2;
    m.nx = d.nx;
    m.ny = d.ny;
    m.nz = 1;
    m.steps = steps > 0 ? steps : 1000;
    m.T = k.T;
    m.bx = 32 * k.V;
    m.halo_x = halo;
    m.sms = sms;
    m.sm_hz = 2.07e9;
    m.hbm_gbs = 6800.0;
    m.bytes_per_cell = d.kind == ST_DIFFUSION ? 8.0 : 12.0;
    m.ops_per_cell = ops;
    m.issue_eff = 1.0;
    m.hbm_eff = 0.90;
    m.stream_overhead = kFill2 * k.T / rows;
    m.launch_s = seg_rows > 0 ? 0.0 : fixed;
    stencil_gpu_model_out r;
    if (stencil_model_gpu(&m, &r) != ST_OK) return 0.0;
    return r.gcells;
}

// relative cost of a plane of each tile column (kWX3, kWY3: see prepare3)
constexpr double kWX3 = 1.4, kWY3 = 1.2;

std::vector<double> column_weights(int ntx, int nty)
{
    std::vector<double> w((size_t)ntx * nty, 1.0);
    for (int ty = 0; ty < nty; ty++)
        for (int tx = 0; tx < ntx; tx++) {
            double &x = w[(size_t)ty * ntx + tx];
            if (tx == 0 || tx == ntx - 1) x *= kWX3;
            if (ty == 0 || ty == nty - 1) x *= kWY3;
        }
    return w;
}

// 3D partial-sum kernel: the same restatement.  Issue-equivalent work per computed cell update
// including halos, by T: 16 / 13.5 / 11.2 / 13 operations (Diffusion, T = 1 .. 4; T = 4 spills
// registers), 18.6 / 15.7 / 12.9 / 13.7 (Hotspot), at an issue efficiency of 0.61 for one 16-warp
// block per SM, x1.04 for two 8-warp blocks, x0.80 for 32-warp blocks of 2 x 2 cells (twice the y
// exchange per cell).  A pass costs 9 us besides (launch, first planes, drain).  Device memory:
// with the columns streamed in step most halo re-reads hit L2: three tenths of the tile fit's
// excess reads, at 90 % of the copy bandwidth.  Calibrated on GB300 over 512^3, 512^2 x 256,
// 256^3, 300 x 200 x 400 and 187 x 141 x 93, both kinds, T = 2 .. 4, 64- and 32-row tiles.
// `bound`: an upper bound instead, with segments dealt at no loss (no bisection)
double model_gcells_3d(const stencil_desc &d, int sms, int T, int VX, int VY, int NW,
                       bool bound = false)
{
    stencil_gpu_model_in m = {};
    m.ndim = 3;
    m.nx = d.nx;
    m.ny = d.ny;
    m.nz = d.nz;
    m.steps = 1000;
    m.T = T;
    m.bx = 32 * VX;
    m.by = VY * NW;
    m.halo_x = (T + 3) / 4 * 4;
    m.halo_y = T;
    m.sms = sms;
    m.sm_hz = 2.07e9;
    m.hbm_gbs = 6800.0;
    const double cx = m.bx - 2.0 * m.halo_x, cy = m.by - 2.0 * m.halo_y;
    if (cx < 1 || cy < 1) return 0.0;
    const long long cols = (long long)std::ceil(d.nx / cx) * (long long)std::ceil(d.ny / cy);
    double rf = std::ceil(d.nx / cx) * m.bx * std::ceil(d.ny / cy) * m.by / ((double)d.nx * d.ny);
    // the segments prepare3 will take
    const long long slots = (long long)sms * (NW <= 8 ? 2 : 1);
    const double seg_cost =
        bound ? 0.0
              : SegmentDealer(d.nz, (int)slots, 3.0 * T - 1, 0.0,
                              column_weights((int)std::ceil(d.nx / cx), (int)std::ceil(d.ny / cy)))
                    .best(0.02 * cols * d.nz / slots + 0.5, nullptr);
    const double alg = d.kind == ST_DIFFUSION ? 8.0 : 12.0;
    const double read = alg - 4.0;   // field (and power) in; the field out is written once
    m.bytes_per_cell = alg;
    m.hbm_eff = 0.90 * alg / (read * (1.0 + 0.3 * (rf - 1.0)) + 4.0);
    const double ops[2][5] = {{0, 16.0, 13.5, 11.2, 13.0}, {0, 18.6, 15.7, 12.9, 13.7}};
    m.ops_per_cell = ops[d.kind == ST_DIFFUSION ? 0 : 1][std::min(std::max(T, 1), 4)];
    m.issue_eff = 0.61 * (NW <= 8 ? 1.04 : NW >= 32 ? 0.80 : 1.0);
    // plane-times per block beyond an even share of the planes (fill, edge columns)
    m.stream_overhead = std::max(0.0, seg_cost * slots / ((double)cols * d.nz) - 1.0);
    m.launch_s = 9e-6;
    stencil_gpu_model_out r;
    if (stencil_model_gpu(&m, &r) != ST_OK) return 0.0;
    return r.gcells;
}

}  // namespace

namespace stn {
// the batch's (T, V) choice uses the same calibrated model; seg_rows: rows per queue item (each
// item streams 2T rows more than it stores)
double batch_model_gcells(int kind, int nx, int ny, int steps, int sms, int T, int V, int bps,
                          int seg_rows)
{
    stencil_desc d = {};
    d.kind = kind;
    d.ndim = 2;
    d.nx = nx;
    d.ny = ny;
    d.nz = 1;
    return model_gcells_2d(d, sms, Cand2D{T, V, 1}, bps, steps, std::min(seg_rows, ny));
}
}  // namespace stn

namespace {

// ---- resident tiles (res2d.cu) ---------------------------------------------------------------
// A 2D grid that fits the co-resident blocks is held on chip for the whole run; the chosen
// (T, cells per thread, block rows) minimises the same kind of restated run time as Eqs. 3-9:
//   t(steps) = steps * t_step + (epochs - 1) * t_x + t_launch + t_io,
//   t_step   = (cells held per SM) * ops / (issue rate of an SM) + t_bar,
// a cell held being one of a tile incl. its halos (Sec. 3.2's redundant compute), ops the issued
// thread instructions per cell and step (the Table 2 operations, the shuffles of the lane edges,
// the row exchange between warps, loop overhead), t_bar the per-step barrier of that exchange,
// t_x one exchange through L2 after every T steps (publish, neighbour wait, halo reload), t_io
// the single read and write of the grid.  Calibrated on GB300: first by least squares over 93
// measured configurations of 512^2 and 1024^2 grids (T = 1..16, 2 and 4 cells per lane, both
// kinds, exact and contracted); then, after the step loop was unrolled and the x-edge work split
// by edge, on the step loops' clock64 cycles and the run times of 1024^2 at T = 12..20 (both
// kinds, exact and contracted, within 0.9-1.05): issue efficiency 0.73, t_x = 7.8 us, and two
// more operations per cell for exact plans (Table 2 order, no fused multiply-adds).
struct ResGeom {
    int T = 0, vx = 0, nw = 0, nbx = 0, nby = 0, cw = 0, ch = 0, hx = 0;
    double t = 0.0;   // predicted seconds for 1000 steps
};

constexpr long long kMaxBlocksSM = 32, kMaxWarpsSM = 64;   // what one SM (compute capability 10.x) holds

double res_time(const stencil_desc &d, int sms, const ResGeom &g, int steps)
{
    const int VY = res2d_rows_per_thread();
    const double per_sm = std::ceil((double)g.nbx * g.nby / sms);
    const double cells = per_sm * g.nw * 32.0 * g.vx * VY;
    double fp = d.kind == ST_DIFFUSION ? 5.0 : 6.0;
    if (d.exact) fp = d.kind == ST_DIFFUSION ? 11.0 : 15.0;
    const double ops = fp + 2.0 / g.vx + 4.0 / (g.vx * VY) + 1.0;
    const double t_step = cells * ops / (128.0 * 0.73 * 2.07e9) + 0.1e-6;
    const double t_x = 7.8e-6;
    const int epochs = (steps + g.T - 1) / g.T;
    return steps * t_step + (epochs - 1) * t_x + 5e-6 + (double)d.nx * d.ny * 8.0 / 6.8e12;
}

// The fastest resident geometry with T steps per exchange and vx cells per thread along x;
// false when the grid does not fit the co-resident blocks of the device.
bool res_geometry(const stencil_desc &d, int sms, int T, int vx, ResGeom *out)
{
    const int kind = d.kind;
    if (T < 1 || !res2d_available(kind, d.exact, vx)) return false;
    const int VY = res2d_rows_per_thread(), maxw = res2d_max_warps(kind, d.exact, vx);
    const int hx = (T + vx - 1) / vx * vx, hy = T;   // x-halo a multiple of vx: x = 0 is a cell 0
    const int cw = 32 * vx - 2 * hx;
    if (cw < 1) return false;
    const int nbx = (d.nx + cw - 1) / cw;
    if (nbx > 1 && cw < hx) return false;   // a halo must not reach past the next block
    const int ch_max = maxw * VY - 2 * hy;   // rows a block can hold besides its halos
    if (ch_max < 1) return false;
    std::vector<int> bps(maxw + 1, 0);
    bool found = false;
    ResGeom best;
    for (int nby = (d.ny + ch_max - 1) / ch_max; nby <= d.ny; nby++) {
        const int ch = (d.ny + nby - 1) / nby;
        if (nby > 1 && ch < hy) break;
        if ((long long)nbx * nby > sms * kMaxBlocksSM) break;   // more than the device can hold
        if ((long long)(nby - 1) * ch >= d.ny) continue;   // the last block would be empty
        const int nw = (ch + 2 * hy + VY - 1) / VY;
        if ((long long)nbx * nby * nw > sms * kMaxWarpsSM) continue;
        if (!bps[nw]) {
            int b = 0;
            if (res2d_occupancy(kind, d.exact, vx, nw, &b) != cudaSuccess) {
                (void)cudaGetLastError();
                b = 0;
            }
            bps[nw] = b > 0 ? b : -1;
        }
        if (bps[nw] < 1 || (long long)nbx * nby > (long long)sms * bps[nw]) continue;
        ResGeom g;
        g.T = T;
        g.vx = vx;
        g.nw = nw;
        g.nbx = nbx;
        g.nby = nby;
        g.cw = cw;
        g.ch = ch;
        g.hx = hx;
        g.t = res_time(d, sms, g, 1000);
        if (!found || g.t < best.t) {
            best = g;
            found = true;
        }
    }
    if (found) *out = best;
    return found;
}

// the best resident geometry over the compiled cells per thread and the candidate T (forced
// values restrict the search)
bool res_choose(const stencil_desc &d, int sms, ResGeom *out)
{
    bool found = false;
    for (int vx : {2, 4}) {
        if (d.force_vec && d.force_vec != vx) continue;
        for (int t : {1, 2, 3, 4, 6, 8, 12, 16, 20, 24, 32}) {
            if (d.force_T && t != d.force_T) continue;
            ResGeom g;
            if (res_geometry(d, sms, t, vx, &g) && (!found || g.t < out->t)) {
                *out = g;
                found = true;
            }
        }
        if (d.force_T && !found) {   // a forced T outside the list above
            ResGeom g;
            if (res_geometry(d, sms, d.force_T, vx, &g) && (!found || g.t < out->t)) {
                *out = g;
                found = true;
            }
        }
    }
    return found;
}

// smallest compiled kernel T >= want for the plan's family (or the largest compiled one)
int kernel_T_for(const stencil_plan_s *p, int want)
{
    int best = 0;
    for (int t : kTcand) {
        if (!available(p, t)) continue;
        if (t >= want) return t;
        best = t;
    }
    return best;
}

// Dealt segments on the device, [first segment of each block | segments], and their block count.
int upload_segments(const std::vector<Segment> &segs, int *ctas, int *seg_off, void **dev, cudaStream_t st)
{
    int n = 1;
    for (const Segment &q : segs) n = std::max(n, q.block + 1);
    *ctas = n;
    *seg_off = (n + 1 + 3) / 4 * 4;   // (the segments start 16-byte aligned)
    std::vector<int> host(*seg_off + 4 * segs.size(), 0), at(n, 0);
    for (const Segment &q : segs) at[q.block]++;
    for (int b = 0; b < n; b++) {
        host[b + 1] = host[b] + at[b];
        at[b] = host[b];
    }
    for (const Segment &q : segs) {
        int *h = host.data() + *seg_off + 4 * (size_t)at[q.block]++;
        h[0] = q.col;
        h[1] = q.z0;
        h[2] = q.z1;
    }
    cudaError_t e = stn::dev_malloc(dev, host.size() * sizeof(int));
    if (e == cudaSuccess) e = stn::dev_upload(*dev, host.data(), host.size() * sizeof(int), st);
    if (e != cudaSuccess) {
        if (*dev) stn::dev_free(*dev);
        *dev = nullptr;
    }
    return map_cuda(e);
}

// Segments of a contracted 2D pass: rows of tile columns dealt like the planes of the 3D passes
// (SegmentDealer), so that neighbouring columns stream the same rows at the same time and share
// their halo cells, and the partial sectors of their rows, in L2.  A segment's fill is 2T rows of
// which the idle stages are skipped.  A row of a tile column whose edge lies on a lane boundary
// (x = 0 always, x = nx-1 when nx is a multiple of the cells per thread) costs kEdge2, one whose
// last column lies inside a lane kGhost2 (its warps run a clamp select per cell), and a segment
// that starts at the top or ends at the bottom kTop2 T rows more (special rows run a loop with
// boundary tests).  Measured on GB300 against contiguous ranges balanced the same way: 12000^2
// diffusion 4001 -> 4184 GCell/s, 16384^2 4114 -> 4247, Hotspot 3058 -> 3107, 8192^2 Hotspot 2645
// -> 2761 (T = 8, 8 cells per thread); DRAM reads of a 16384^2 diffusion pass 1.31 -> 1.10 GB.
// halo: rows per side a segment streams besides its own (R T); V: cells per thread.
int segments_2d(stencil_plan_s *p, int bps, int halo, int V, PassCfg2D *c)
{
    std::vector<double> w(c->ntx, 1.0);
    w.front() = kEdge2;
    w.back() = p->d.nx % V == 0 ? kEdge2 : kGhost2;
    std::vector<Segment> segs;
    // A scheduler issues from its oldest ready warp first, so of the one-warp blocks that share one
    // the first to arrive (blocks arrive in order, one per SM and round, four rounds per warp
    // rank) runs ahead of the others (equal shares, 12000^2 diffusion: the first half of the
    // blocks took 204 us, the second 265; ahead by 0 / 0.05 / 0.1 / 0.15, 16384^2 diffusion:
    // 4071 / 4160 / 3986 / 3814 GCell/s)
    const int slots = p->sms * bps, ranks = (bps + 3) / 4;
    std::vector<double> speed(slots, 1.0);
    for (int b = 0; b < slots && ranks > 1; b++)
        speed[b] = 1.0 + kAhead2 * (1.0 - 2.0 * (b / p->sms / 4) / (ranks - 1));
    SegmentDealer(p->d.ny, slots, kFill2 * halo, (V == 8 ? kTop2V8 : kTop2V4) * halo, w, speed).best(0.5, &segs);
    return upload_segments(segs, &c->ctas, &c->seg_off, &c->segs, p->stream);
}

// A remainder pass (fewer steps than the plan's T) gets its own shorter kernel, whose segments are
// dealt and uploaded on its first use, under stream capture too (the graph then holds that kernel).
// Where no memory is left for them, the plan's own kernel runs the fewer steps instead.
int prepare2(stencil_plan_s *p, int Tk, PassCfg2D **out)
{
    if ((int)p->cfg2.size() <= Tk) p->cfg2.resize(Tk + 1);
    PassCfg2D &c = p->cfg2[Tk];
    if (!c.ready) {
        c.shape = Shape2D{p->d.kind, p->d.exact ? 1 : 0, Tk, p->V, p->W, shape_stor(p)};
        if (!tb2d_available(c.shape)) return ST_ERR_UNSUPPORTED;
        const stn::RelaxedCapture relaxed;
        int bps = 0;
        cudaError_t e = tb2d_prepare(c.shape, &bps);
        if (e != cudaSuccess) return map_cuda(e);
        if (bps < 1) return ST_ERR_UNSUPPORTED;
        const int bx = tb2d_tile_width(c.shape), h = tb2d_halo(c.shape);
        const int cx = bx - 2 * h;
        c.ntx = (p->d.nx + cx - 1) / cx;
        c.total = (long long)c.ntx * p->d.ny;
        // each block streams at least ~8T rows so the y-halo (2T rows per segment) stays small
        const long long min_rows = 4;   // short segments keep small grids parallel
        long long ctas = std::min<long long>((long long)p->sms * bps,
                                             std::max<long long>(1, c.total / min_rows));
        c.rows_per_cta = (c.total + ctas - 1) / ctas;
        c.ctas = (int)((c.total + c.rows_per_cta - 1) / c.rows_per_cta);
        if (tb2d_segments(c.shape)) {
            const int rc = segments_2d(p, bps, c.shape.T, c.shape.V, &c);
            if (rc == ST_ERR_OOM && Tk < p->T) {
                (void)cudaGetLastError();
                return prepare2(p, p->T, out);
            }
            if (rc != ST_OK) return rc;
        }
        c.ready = true;
    }
    *out = &c;
    return ST_OK;
}

// Trajectory passes run the in-place T = 8, V = 8 contracted kernel that also writes every
// fused step; same launch geometry rules as the plan's own passes.
constexpr int kTrajT = 8;

int prepare_traj(stencil_plan_s *p, PassCfg2D **out)
{
    PassCfg2D &c = p->traj;
    if (!c.ready) {
        c.shape = Shape2D{p->d.kind, 0, kTrajT, 8, 0,
                          (p->d.kind == ST_THERMAL ? (int)STOR_SRC : 0) | (int)STOR_ALL};
        if (!tb2d_available(c.shape)) return ST_ERR_UNSUPPORTED;
        int bps = 0;
        cudaError_t e = tb2d_prepare(c.shape, &bps);
        if (e != cudaSuccess) return map_cuda(e);
        if (bps < 1) return ST_ERR_UNSUPPORTED;
        const int cx = tb2d_tile_width(c.shape) - 2 * tb2d_halo(c.shape);
        c.ntx = (p->d.nx + cx - 1) / cx;
        c.total = (long long)c.ntx * p->d.ny;
        // even shares: these passes wait for their writes (every fused step goes to memory), and
        // nothing is allocated on the first call
        const long long ctas = std::min<long long>((long long)p->sms * bps,
                                                   std::max<long long>(1, c.total / 4));
        c.rows_per_cta = (c.total + ctas - 1) / ctas;
        c.ctas = (int)((c.total + c.rows_per_cta - 1) / c.rows_per_cta);
        c.ready = true;
    }
    *out = &c;
    return ST_OK;
}

// The streamed radius-2 star: T = 1, 2 or 4 steps fused.
int prepare_star2f(stencil_plan_s *p, int Tk, PassCfg2D **out)
{
    if ((int)p->cfg2.size() <= Tk) p->cfg2.resize(Tk + 1);
    PassCfg2D &c = p->cfg2[Tk];
    if (!c.ready) {
        const stn::RelaxedCapture relaxed;
        int bps = 0;
        const cudaError_t e = star2f_prepare(Tk, &bps);
        if (e != cudaSuccess) return map_cuda(e);
        if (bps < 1) return ST_ERR_UNSUPPORTED;
        c.shape.T = Tk;
        c.ntx = (p->d.nx + star2f_compute_width() - 1) / star2f_compute_width();
        const int rc = segments_2d(p, bps, 2 * Tk, 8, &c);
        if (rc == ST_ERR_OOM && Tk < p->T) {
            (void)cudaGetLastError();
            return prepare_star2f(p, p->T, out);
        }
        if (rc != ST_OK) return rc;
        c.ready = true;
    }
    *out = &c;
    return ST_OK;
}

int prepare3(stencil_plan_s *p, int Tk, PassCfg3D **out)
{
    if ((int)p->cfg3.size() <= Tk) p->cfg3.resize(Tk + 1);
    PassCfg3D &c = p->cfg3[Tk];
    if (!c.ready) {
        c.shape = Shape3D{p->d.kind, p->d.exact ? 1 : 0, Tk, p->VY, p->NW, p->alg3, p->VX3};
        if (!tb3d_available(c.shape)) return ST_ERR_UNSUPPORTED;
        const stn::RelaxedCapture relaxed;
        int bps = 0;
        cudaError_t e = tb3d_prepare(c.shape, &bps);
        if (e != cudaSuccess) return map_cuda(e);
        if (bps < 1) return ST_ERR_UNSUPPORTED;
        const int hx = (Tk + 3) / 4 * 4, hy = Tk;
        const int cx = 32 * p->VX3 - 2 * hx, cy = p->VY * p->NW - 2 * hy;
        c.ntx = (p->d.nx + cx - 1) / cx;
        c.nty = (p->d.ny + cy - 1) / cy;
        c.cols = (long long)c.ntx * c.nty;
        const long long total = c.cols * p->d.nz;
        const long long min_planes = std::max(16, 8 * Tk);
        long long ctas = std::min<long long>((long long)p->sms * bps,
                                             std::max<long long>(1, total / min_planes));
        c.planes_per_cta = (total + ctas - 1) / ctas;
        c.ctas = (int)((total + c.planes_per_cta - 1) / c.planes_per_cta);
        if (p->alg3) {
            // segments dealt to the blocks (SegmentDealer): a plane of a tile column at the x
            // edge costs 1.4, at the y edge 1.2 (only they run instances with the clamp fix-ups,
            // and the barrier makes a block wait for its slowest warp; swept 1.0-1.4 on GB300,
            // T = 3: 512^3 diffusion 1188 GCell/s at 1.1 / 1.05, 1318 at 1.4 / 1.2).  Dealt
            // level by level against contiguous ranges balanced the same way: 512^2 x 256 Hotspot
            // 940 -> 1044 GCell/s at T = 3, 611 -> 912 at T = 2 (DRAM reads of a 512^2 x 256
            // diffusion pass 491 -> 302 MB); a plan of few columns is spread over more blocks
            // (187 x 141 x 93 diffusion x 30: 427 -> 242 us)
            std::vector<Segment> segs;
            SegmentDealer(p->d.nz, p->sms * bps, 3.0 * Tk - 1, 0.0, column_weights(c.ntx, c.nty)).best(0.25, &segs);
            const int rc = upload_segments(segs, &c.ctas, &c.seg_off, &c.segs, p->stream);
            if (rc == ST_ERR_OOM && Tk < p->T) {
                (void)cudaGetLastError();
                return prepare3(p, p->T, out);
            }
            if (rc != ST_OK) return rc;
        }
        c.ready = true;
    }
    *out = &c;
    return ST_OK;
}

bool ranges_overlap(const void *a, const void *b, size_t n)
{
    const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
    return x < y + n && y < x + n;
}

// [a, a + na) and [b, b + nb) share a byte
bool ranges_overlap2(const void *a, size_t na, const void *b, size_t nb)
{
    const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
    return x < y + nb && y < x + na;
}

bool stable(const stencil_desc &d, const float *k)
{
    const double eps = 1e-6;
    for (int i = 0; i < ncoef(d); i++)
        if (!std::isfinite(k[i])) return false;
    if (d.kind == ST_DIFFUSION) {
        double s = 0;
        for (int i = 0; i < ncoef(d); i++) {
            if (k[i] < 0) return false;
            s += k[i];
        }
        return s <= 1.0 + eps;
    }
    if (d.ndim == 2) {
        const double kdt = k[0], rx = k[1], ry = k[2], rz = k[3];
        if (kdt < 0 || rx < 0 || ry < 0 || rz < 0) return false;
        return kdt * (2 * rx + 2 * ry + rz) <= 1.0 + eps;
    }
    for (int i = 0; i < 8; i++)
        if (k[i] < 0) return false;
    return true;
}

cudaError_t record(stencil_plan_s *p, bool begin)
{
    if (!p->timing) return cudaSuccess;
    if (begin && p->ev_used + 2 > p->ev.size()) {
        for (int i = 0; i < 64; i++) {
            cudaEvent_t e;
            cudaError_t err = cudaEventCreate(&e);
            if (err != cudaSuccess) return err;
            p->ev.push_back(e);
        }
    }
    cudaError_t err = cudaEventRecord(p->ev[p->ev_used], p->stream);
    p->ev_used++;
    return err;
}

int flush_timing(stencil_plan_s *p)
{
    if (p->ev_used == 0) return ST_OK;
    cudaError_t e = cudaEventSynchronize(p->ev[p->ev_used - 1]);
    if (e != cudaSuccess) return map_cuda(e);
    for (size_t i = 0; i + 1 < p->ev_used; i += 2) {
        float ms = 0.f;
        e = cudaEventElapsedTime(&ms, p->ev[i], p->ev[i + 1]);
        if (e != cudaSuccess) return map_cuda(e);
        p->ms_acc += ms;
        p->launches++;
    }
    p->ev_used = 0;
    return ST_OK;
}

// traj (trajectory passes): its configuration, and where the pass's intermediate steps go
int run_pass2(stencil_plan_s *p, const float *src, long long lds, float *dst, long long ldd,
              const float *pw, const float *k, int tsteps, PassCfg2D *traj = nullptr,
              float *states = nullptr, long long stride = 0)
{
    PassCfg2D *c = traj;
    int rc = traj ? ST_OK : prepare2(p, kernel_T_for(p, tsteps), &c);
    if (rc != ST_OK) return rc;
    Pass2D a = {};
    a.states = states;
    a.state_stride = stride;
    a.in = src;
    a.out = dst;
    a.pw = pw;
    a.ld_in = lds;
    a.ld_out = ldd;
    a.ld_pw = (p->src && pw == p->src) ? p->ld_src : p->d.nx;
    a.pw_plane = (long long)p->d.nx * p->d.ny;   // per-cell coefficient planes, dense
    a.nx = p->d.nx;
    a.ny = p->d.ny;
    a.tsteps = tsteps;
    a.ntx = c->ntx;
    a.total_rows = c->total;
    a.rows_per_cta = c->rows_per_cta;
    a.seg_first = static_cast<const int *>(c->segs);
    a.segs = c->segs ? reinterpret_cast<const int4 *>(a.seg_first + c->seg_off) : nullptr;
    a.ctas = c->ctas;
    for (int i = 0; i < 5; i++) a.k[i] = a.kf[i] = k[i];
    a.kf[5] = k[0] * k[2];    // Hotspot: sdc * Ry, rounded once (float32)
    a.kf[6] = -2.0f * k[2];   // Hotspot: -2 Ry (exact)
    if (stor_src_bits(c->shape.stor)) hot_coeffs_src(k, a.kf);
    a.vec_in = ((uintptr_t)src % 16 == 0) && (lds % 4 == 0);
    a.vec_out = ((uintptr_t)dst % 16 == 0) && (ldd % 4 == 0) &&
                (!states || ((uintptr_t)states % 16 == 0 && stride % 4 == 0));
    a.vec_pw = pw ? (((uintptr_t)pw % 16 == 0) && (a.ld_pw % 4 == 0)) : 0;
    if (p->timing && p->ev_used + 2 > 2 * 1024) {
        rc = flush_timing(p);
        if (rc != ST_OK) return rc;
    }
    cudaError_t e = record(p, true);
    if (e == cudaSuccess) e = tb2d_launch(c->shape, a, p->stream);
    if (e == cudaSuccess) e = record(p, false);
    return map_cuda(e);
}

// a run of a resident-tile plan: one cooperative launch.  The blocks' epoch counters grow from run
// to run (each run starts at a base that no counter is above), so a run launched now needs no reset.
// A captured run does: every replay gets the arguments of the capture, so its graph zeroes the
// counters and counts from 0, and later plain runs start above what a replay may have left.
int run_resident(stencil_plan_s *p, const float *in, float *out, const float *pw, const float *k,
                 int steps)
{
    const stencil_desc &d = p->d;
    Res2D a = {};
    a.in = in;
    a.ld_in = d.nx;
    a.out = out;
    cudaError_t e = cudaSuccess;
    const int epochs = (steps + p->T - 1) / p->T;
    if (in == out && epochs == 1) {
        // in place with no exchange between the blocks' first read and last write: a block
        // could overwrite cells a neighbour has yet to read, so the run reads a copy (in the
        // exchange grids, unused by a single epoch)
        float *cp = p->res_xg;
        e = cudaMemcpy2DAsync(cp, (size_t)p->res_ld * sizeof(float), in, (size_t)d.nx * sizeof(float),
                              (size_t)d.nx * sizeof(float), d.ny, cudaMemcpyDeviceToDevice, p->stream);
        if (e != cudaSuccess) return map_cuda(e);
        a.in = cp;
        a.ld_in = p->res_ld;
    }
    a.aux = pw;
    a.ld_aux = d.nx;
    a.xg = p->res_xg;
    a.xplane = p->res_ld * d.ny;
    a.ld_x = p->res_ld;
    if (epochs > 1) {
        const bool cap = stn::stream_captured(p->stream);
        if (cap) p->res_captured = std::max(p->res_captured, epochs);
        if (cap || p->res_epoch > 0x7fffffff - epochs) {   // (or the counters would overflow)
            e = cudaMemsetAsync(p->res_flags, 0, (size_t)p->res_nbx * p->res_nby * sizeof(int), p->stream);
            if (e != cudaSuccess) return map_cuda(e);
            a.epoch0 = 0;
            p->res_epoch = std::max(cap ? p->res_epoch : epochs, p->res_captured);
        } else {
            a.epoch0 = p->res_epoch;
            p->res_epoch += epochs;
        }
    }
    a.flags = p->res_flags;
    a.status = p->err;
    a.wait_ns = p->res_wait_ns;
    a.hold_block = p->res_hold_block;
    a.hold_epoch = p->res_hold_epoch;
    a.nx = d.nx;
    a.ny = d.ny;
    a.steps = steps;
    a.T = p->T;
    a.nbx = p->res_nbx;
    a.nby = p->res_nby;
    a.cw = p->res_cw;
    a.ch = p->res_ch;
    a.hx = p->res_hx;
    a.hy = p->T;
    if (d.kind == ST_THERMAL && !d.exact) {
        // the expanded weights cc, cx, cy, cz of the contracted Hotspot kernels
        float kf[7];
        hot_coeffs_src(k, kf);
        for (int i = 0; i < 4; i++) a.k[i] = kf[i];
        a.src_sdc = k[0];
        a.src_a = k[4] * k[3];   // amb * Rz, rounded once
    } else {
        for (int i = 0; i < 5; i++) a.k[i] = k[i];
    }
    if (p->timing && p->ev_used + 2 > 2 * 1024) {
        const int rc = flush_timing(p);
        if (rc != ST_OK) return rc;
    }
    e = record(p, true);
    if (e == cudaSuccess)
        e = res2d_launch(d.kind, d.exact, p->res_vx, p->res_nw, a,
                         p->stream);
    if (e == cudaSuccess) e = record(p, false);
    return map_cuda(e);
}

// one pass of a 16-bit plan: coded grid q[src] -> q[dst], always the plan's T kernel (the
// trailing stages forward when tsteps < T), so the block codes keep the plan's tiling
int run_pass2q(stencil_plan_s *p, int src, int dst, const float *k, int tsteps)
{
    PassCfg2D *c = nullptr;
    int rc = prepare2(p, p->T, &c);
    if (rc != ST_OK) return rc;
    Pass2D a = {};
    a.nx = p->d.nx;
    a.ny = p->d.ny;
    a.tsteps = tsteps;
    a.ntx = c->ntx;
    a.total_rows = c->total;
    a.rows_per_cta = c->rows_per_cta;
    a.seg_first = static_cast<const int *>(c->segs);
    a.segs = c->segs ? reinterpret_cast<const int4 *>(a.seg_first + c->seg_off) : nullptr;
    a.ctas = c->ctas;
    for (int i = 0; i < 5; i++) a.k[i] = a.kf[i] = k[i];
    a.kf[5] = k[0] * k[2];
    a.kf[6] = -2.0f * k[2];
    if (stor_src_bits(c->shape.stor)) hot_coeffs_src(k, a.kf);
    a.vec_in = a.vec_out = a.vec_pw = 1;
    a.stor = p->stor;
    a.qin = p->q[src];
    a.qout = p->q[dst];
    a.min_ = p->qm[src];
    a.mout = p->qm[dst];
    a.qpw = p->qp;
    a.mpw = p->qpm;
    a.ld_q = p->ld_q;
    cudaError_t e = record(p, true);
    if (e == cudaSuccess) e = tb2d_launch(c->shape, a, p->stream);
    if (e == cudaSuccess) e = record(p, false);
    return map_cuda(e);
}

int run_pass_star3(stencil_plan_s *p, const float *src, float *dst, const float *k, int tsteps)
{
    PassStar3D a = {};
    a.in = src;
    a.out = dst;
    a.nx = p->d.nx;
    a.ny = p->d.ny;
    a.nz = p->d.nz;
    a.tsteps = tsteps;
    a.ntx = p->ntx_star;
    a.nty = p->nty_star;
    a.nseg = p->nseg_star;
    a.zseg = p->zseg_star;
    for (int i = 0; i < ncoef(p->d) && i < 25; i++) a.k[i] = k[i];
    a.vec_out = ((uintptr_t)dst % 16 == 0) && (p->d.nx % 4 == 0);
    a.err = p->err;
    CUtensorMap tm;
    std::memset(&tm, 0, sizeof(tm));
    a.use_tma = tma3d_encode(&tm, src, p->d.nx, p->d.ny, p->d.nz, p->d.nx, 64, 64) ? 1 : 0;
    if (p->timing && p->ev_used + 2 > 2 * 1024) {
        const int rc = flush_timing(p);
        if (rc != ST_OK) return rc;
    }
    cudaError_t e = record(p, true);
    if (e == cudaSuccess) e = star3d_launch(p->d.rad, p->d.exact, p->T, a, tm, p->stream);
    if (e == cudaSuccess) e = record(p, false);
    return map_cuda(e);
}

int run_pass_star2f(stencil_plan_s *p, const float *src, long long lds, float *dst, long long ldd,
                    const float *k, int tsteps)
{
    PassCfg2D *c = nullptr;
    int rc = prepare_star2f(p, tsteps <= 1 ? 1 : tsteps <= 2 ? 2 : 4, &c);
    if (rc != ST_OK) return rc;
    Pass2D a = {};
    a.in = src;
    a.out = dst;
    a.ld_in = lds;
    a.ld_out = ldd;
    a.nx = p->d.nx;
    a.ny = p->d.ny;
    a.tsteps = tsteps;
    a.ntx = c->ntx;
    a.seg_first = static_cast<const int *>(c->segs);
    a.segs = reinterpret_cast<const int4 *>(a.seg_first + c->seg_off);
    a.ctas = c->ctas;
    a.vec_in = ((uintptr_t)src % 16 == 0) && (lds % 4 == 0);
    a.vec_out = ((uintptr_t)dst % 16 == 0) && (ldd % 4 == 0);
    StarCoef2 ks;
    for (int i = 0; i < 9; i++) ks.k[i] = k[i];
    if (p->timing && p->ev_used + 2 > 2 * 1024) {
        rc = flush_timing(p);
        if (rc != ST_OK) return rc;
    }
    cudaError_t e = record(p, true);
    if (e == cudaSuccess) e = star2f_launch(c->shape.T, a, ks, p->stream);
    if (e == cudaSuccess) e = record(p, false);
    return map_cuda(e);
}

int run_pass_star(stencil_plan_s *p, const float *src, long long lds, float *dst, long long ldd,
                  const float *k, int tsteps)
{
    if (p->star_rows) return run_pass_star2f(p, src, lds, dst, ldd, k, tsteps);
    if (p->d.ndim == 3) return run_pass_star3(p, src, dst, k, tsteps);
    PassStar2D a = {};
    a.in = src;
    a.out = dst;
    a.ld_in = p->d.nx;
    a.ld_out = p->d.nx;
    a.nx = p->d.nx;
    a.ny = p->d.ny;
    a.tsteps = tsteps;
    a.ntx = p->ntx_star;
    a.nty = p->nty_star;
    for (int i = 0; i < ncoef(p->d) && i < 17; i++) a.k[i] = k[i];
    a.vec_out = ((uintptr_t)dst % 16 == 0) && (p->d.nx % 4 == 0);
    a.err = p->err;
    CUtensorMap tm;
    std::memset(&tm, 0, sizeof(tm));
    a.use_tma = tma3d_encode(&tm, src, p->d.nx, p->d.ny, 1, p->d.nx, 128, 128) ? 1 : 0;
    if (p->timing && p->ev_used + 2 > 2 * 1024) {
        const int rc = flush_timing(p);
        if (rc != ST_OK) return rc;
    }
    cudaError_t e = record(p, true);
    if (e == cudaSuccess) e = star2d_launch(p->d.rad, p->d.exact, p->T, a, tm, p->stream);
    if (e == cudaSuccess) e = record(p, false);
    return map_cuda(e);
}

// row pitches lds, ldd, ldp of the input, the output and the power map, in floats
int run_pass3(stencil_plan_s *p, const float *src, long long lds, float *dst, long long ldd,
              const float *pw, long long ldp, const float *k, int tsteps)
{
    PassCfg3D *c = nullptr;
    int rc = prepare3(p, kernel_T_for(p, tsteps), &c);
    if (rc != ST_OK) return rc;
    Pass3D a;
    a.in = src;
    a.out = dst;
    a.pw = pw;
    a.nx = p->d.nx;
    a.ny = p->d.ny;
    a.nz = p->d.nz;
    a.tsteps = tsteps;
    a.ntx = c->ntx;
    a.nty = c->nty;
    a.total_cols = c->cols;
    a.planes_per_cta = c->planes_per_cta;
    a.ctas = c->ctas;
    a.seg_first = static_cast<const int *>(c->segs);
    a.segs = c->segs ? reinterpret_cast<const int4 *>(a.seg_first + c->seg_off) : nullptr;
    for (int i = 0; i < 9; i++) a.k[i] = i < ncoef(p->d) ? k[i] : 0.f;
    a.ld_in = lds;
    a.ld_out = ldd;
    a.ld_pw = ldp;
    a.vec = ((uintptr_t)src % 16 == 0) && (lds % 4 == 0);
    a.vec_out = ((uintptr_t)dst % 16 == 0) && (ldd % 4 == 0);
    if (!p->alg3) a.vec = a.vec && a.vec_out;
    a.vec_pw = pw && ((uintptr_t)pw % 16 == 0) && (ldp % 4 == 0);
    a.err = p->err;
    a.use_tma = 0;
    Tma3D tm;
    std::memset(&tm, 0, sizeof(tm));
    if (p->alg3 && a.vec) {
        const int bx = 32 * p->VX3, by = p->VY * p->NW;
        bool ok = tma3d_encode(&tm.in, src, p->d.nx, p->d.ny, p->d.nz, lds, bx, by);
        if (ok && pw) ok = a.vec_pw && tma3d_encode(&tm.pw, pw, p->d.nx, p->d.ny, p->d.nz, ldp, bx, by);
        a.use_tma = ok ? 1 : 0;
    }
    if (p->timing && p->ev_used + 2 > 2 * 1024) {
        rc = flush_timing(p);
        if (rc != ST_OK) return rc;
    }
    cudaError_t e = record(p, true);
    if (e == cudaSuccess) e = tb3d_launch(c->shape, a, tm, p->stream);
    if (e == cudaSuccess) e = record(p, false);
    return map_cuda(e);
}

// Contracted first-order plans on rows that are no whole 16-byte chunks (nx not a multiple of 4):
// the passes between the first and the last run between two padded scratch grids, so that only
// those two touch the caller's rows (staged and stored cell by cell).  The second grid (and the
// padded power map of 3D Hotspot) is taken where memory is no concern: up to 16 GiB a grid and a
// quarter of what is free once the plan has all it needs.  Otherwise, and if the allocation fails,
// the passes alternate between one scratch grid and the output.
int extra_grids(stencil_plan_s *p)
{
    const stencil_desc &d = p->d;
    if (d.nx % 4 == 0 || d.exact || p->res || p->stor || (d.rad > 1 && !p->star_rows) ||
        (d.ndim == 3 && !p->alg3) || p->scratch_bytes > (size_t)16 << 30)
        return ST_OK;
    const bool pad_pw = d.ndim == 3 && d.kind == ST_THERMAL;
    size_t free_b = 0, total_b = 0;
    cudaError_t e = cudaMemGetInfo(&free_b, &total_b);
    if (e != cudaSuccess) return map_cuda(e);
    if (p->scratch_bytes * (pad_pw ? 2 : 1) > free_b / 4) return ST_OK;
    float *grid = nullptr, *pw = nullptr;
    e = stn::dev_malloc(&grid, p->scratch_bytes);
    if (e == cudaSuccess && pad_pw) e = stn::dev_malloc(&pw, p->scratch_bytes);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        if (grid) stn::dev_free(grid);
        return e == cudaErrorMemoryAllocation ? ST_OK : map_cuda(e);
    }
    p->scratch2 = grid;
    p->scratch_bytes *= 2;
    if (pad_pw) {
        p->src = pw;
        p->ld_src = p->ld_scratch;
    }
    return ST_OK;
}

}  // namespace

extern "C" {

int stencil_abi_version(void) { return ST_ABI_VERSION; }

const char *stencil_strerror(int code)
{
    switch (code) {
    case ST_OK: return "ok";
    case ST_ERR_INVALID_ARG: return "invalid argument";
    case ST_ERR_DIMS_MISMATCH: return "grid dimensions differ from the plan's";
    case ST_ERR_UNSTABLE_COEFFS: return "coefficients violate the explicit stability bound";
    case ST_ERR_CUDA: return "CUDA runtime error";
    case ST_ERR_OOM: return "device memory allocation failed";
    case ST_ERR_TIMEOUT: return "bounded device wait timed out";
    case ST_ERR_UNSUPPORTED: return "unsupported parameter combination";
    case ST_ERR_TOO_LARGE: return "grid larger than the allocation-free entry point's fixed buffer";
    default: return "unknown status";
    }
}

int stencil_plan_destroy(stencil_plan p);

static int plan_create(stencil_plan *out, const stencil_desc *desc);

int stencil_plan_create(stencil_plan *out, const stencil_desc *desc)
{
    // nothing forced and a measured choice cached for this problem: take it (an entry this
    // build cannot make falls back to the model's choice)
    if (out && desc && !desc->force_T && !desc->force_bx && !desc->force_by && !desc->force_vec &&
        !desc->partial_rows && !desc->resident) {
        stencil_desc t = *desc;
        int f[6];
        if (tune_cache_lookup(t, f)) {
            t.force_T = f[0];
            t.force_bx = f[1];
            t.force_by = f[2];
            t.force_vec = f[3];
            t.partial_rows = f[4];
            t.resident = f[5];
            const int rc = plan_create(out, &t);
            if (rc == ST_OK) {
                (*out)->tuned = 1;
                return rc;
            }
            if (rc != ST_ERR_UNSUPPORTED) return rc;
        }
    }
    return plan_create(out, desc);
}

int stencil_plan_tuned(stencil_plan p) { return p ? p->tuned : 0; }

static int plan_create(stencil_plan *out, const stencil_desc *desc)
{
    if (!out) return ST_ERR_INVALID_ARG;
    *out = nullptr;
    if (!desc) return ST_ERR_INVALID_ARG;
    stencil_desc d = *desc;
    if (d.kind != ST_DIFFUSION && d.kind != ST_THERMAL && d.kind != ST_DIFFUSION_VAR)
        return ST_ERR_INVALID_ARG;
    if (d.ndim != 2 && d.ndim != 3) return ST_ERR_INVALID_ARG;
    if (d.ndim == 2) d.nz = 1;
    if (d.nx < 1 || d.ny < 1 || d.nz < 1) return ST_ERR_INVALID_ARG;
    if (d.storage != ST_F32 && d.storage != ST_BF16 && d.storage != ST_F16)
        return ST_ERR_INVALID_ARG;
    // 16-bit storage: 2D contracted plans only
    if (d.storage != ST_F32 && (d.ndim != 2 || d.exact)) return ST_ERR_UNSUPPORTED;
    if (d.force_T < 0 || d.force_bx < 0 || d.force_by < 0 || d.force_vec < 0)
        return ST_ERR_INVALID_ARG;
    if (d.rad < 0) return ST_ERR_INVALID_ARG;
    if (d.partial_rows < 0 || d.partial_rows > 2 || d.resident < -1 || d.resident > 1)
        return ST_ERR_INVALID_ARG;
    if (d.ndim == 2 && d.rad <= 1 && d.force_by) return ST_ERR_INVALID_ARG;   // no 2D tile height
    if (d.partial_rows && (d.ndim != 2 || d.exact || d.kind == ST_DIFFUSION_VAR || d.rad > 1))
        return ST_ERR_UNSUPPORTED;
    if (d.resident == 1 && (d.ndim != 2 || d.rad > 1 || d.kind == ST_DIFFUSION_VAR ||
                            d.storage != ST_F32 || d.force_bx || d.partial_rows))
        return ST_ERR_UNSUPPORTED;
    // per-cell coefficients: 2D float32 plans of the windowed kernel (V = 4, 128 or 512 cells
    // wide); the stability check of strict plans needs host coefficients
    if (d.kind == ST_DIFFUSION_VAR &&
        (d.ndim != 2 || d.storage != ST_F32 || d.rad > 1 || d.strict || d.force_by ||
         (d.force_vec && d.force_vec != 4) || (d.force_bx && d.force_bx != 128 && d.force_bx != 512)))
        return ST_ERR_UNSUPPORTED;
    if (d.rad > 1) {
        const int tile = d.ndim == 2 ? 128 : 64;   // star tiles: 128 x 128 in 2D, 64 x 64 in 3D
        if (d.kind != ST_DIFFUSION || d.storage != ST_F32 || d.rad > 4 ||
            (d.force_bx && d.force_bx != tile) || (d.force_by && d.force_by != tile) ||
            (d.force_vec && d.force_vec != (d.ndim == 2 ? 4 : 16)))
            return ST_ERR_UNSUPPORTED;
    }

    stencil_plan_s *p = new (std::nothrow) stencil_plan_s();
    if (!p) return ST_ERR_OOM;
    p->d = d;
    p->stream = static_cast<cudaStream_t>(d.stream);
    int rc = ST_OK;
    cudaError_t e = cudaGetDevice(&p->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&p->sms, cudaDevAttrMultiProcessorCount, p->device);
    if (e != cudaSuccess) {
        delete p;
        return map_cuda(e);
    }

    p->stor = d.storage == ST_BF16 ? 1 : (d.storage == ST_F16 ? 2 : 0);
    if (d.rad > 1 && d.ndim == 3) {
        // 3D star diffusion: 64 x 64 tiles streamed along z, T = 1 unless forced: measured on
        // 512^3, R = 2 (GB300), T = 1 runs at 382 GCell/s and T = 2 at 271 -- the second ring
        // of planes leaves one 8-warp block per SM and adds a barrier per plane
        const int T = d.force_T ? d.force_T : 1;
        int bps = 0;
        if (!star3d_available(d.rad, d.exact, T)) rc = ST_ERR_UNSUPPORTED;
        if (rc == ST_OK) {
            e = star3d_prepare(d.rad, d.exact, T, &bps);
            if (e != cudaSuccess) rc = map_cuda(e);
            else if (bps < 1) rc = ST_ERR_UNSUPPORTED;
        }
        if (rc == ST_OK) {
            p->T = T;
            int cx = 0, cy = 0;
            star3d_tile(d.rad, T, &cx, &cy);
            p->ntx_star = (d.nx + cx - 1) / cx;
            p->nty_star = (d.ny + cy - 1) / cy;
            // z-segments: the count that keeps the most block slots busy, discounted by the
            // planes a segment re-reads (R T at either end); segments at least 8 R T long
            const long long cols = (long long)p->ntx_star * p->nty_star;
            const long long slots = (long long)p->sms * bps;
            const int max_seg = std::max(1, d.nz / (8 * d.rad * T));
            double best = -1.0;
            long long nseg = 1;
            for (int n = 1; n <= max_seg; n++) {
                const long long blocks = cols * n, waves = (blocks + slots - 1) / slots;
                const double zs = (double)((d.nz + n - 1) / n);
                const double eff = (double)blocks / (double)(waves * slots) * zs / (zs + 2.0 * d.rad * T);
                if (eff > best + 1e-9) {
                    best = eff;
                    nseg = n;
                }
            }
            p->zseg_star = (int)((d.nz + nseg - 1) / nseg);
            p->nseg_star = (d.nz + p->zseg_star - 1) / p->zseg_star;
            p->ld_scratch = d.nx;
            p->scratch_bytes = (size_t)cells_of(d) * sizeof(float);
        }
    } else if (d.rad > 1) {
        // star diffusion: 128 x 128 tiles, T from {1, 2, 4} (default: the largest whose halos
        // leave at least 70 % of the tile's cells in its compute block)
        int T = d.force_T;
        if (!T) {
            T = 1;
            for (int t : {2, 4}) {
                const double cx = 128 - 2 * ((d.rad * t + 3) / 4 * 4), cy = 128 - 2 * d.rad * t;
                if (cx > 0 && cy > 0 && cx * cy >= 0.7 * 128 * 128) T = t;
            }
        }
        // contracted, radius 2, no tile asked for: streamed by one-warp blocks, T = 4 unless forced
        // (8192^2 x 64: 2327 us; T = 2 3227 us, tiles 4026 us)
        if (d.rad == 2 && !d.exact && !d.force_bx && !d.force_by && !d.force_vec &&
            (T == 1 || T == 2 || T == 4)) {
            PassCfg2D *c = nullptr;
            p->T = T;
            rc = prepare_star2f(p, T, &c);
            if (rc == ST_OK) {
                p->star_rows = 1;
                p->ld_scratch = ((long long)d.nx + 31) / 32 * 32;
                p->scratch_bytes = (size_t)p->ld_scratch * d.ny * sizeof(float);
            }
        } else if (!star2d_available(d.rad, d.exact, T)) {
            rc = ST_ERR_UNSUPPORTED;
        }
        if (rc == ST_OK && !p->star_rows) {
            e = star2d_prepare(d.rad, d.exact, T);
            if (e != cudaSuccess) rc = map_cuda(e);
        }
        if (rc == ST_OK && !p->star_rows) {
            p->T = T;
            const int cx = 128 - 2 * star2d_halo_x(d.rad, T), cy = 128 - 2 * star2d_halo_y(d.rad, T);
            p->ntx_star = (d.nx + cx - 1) / cx;
            p->nty_star = (d.ny + cy - 1) / cy;
            p->ld_scratch = d.nx;   // dense rows: the tensor map of a grid uses the grid's pitch
            p->scratch_bytes = (size_t)d.nx * d.ny * sizeof(float);
        }
    } else if (d.ndim == 2) {
        // resident tiles: when asked for, or compared below with the passes when nothing else
        // is forced
        ResGeom rg;
        bool res = false;
        if (d.resident == 1) {
            res = res_choose(d, p->sms, &rg);
            if (!res) rc = ST_ERR_UNSUPPORTED;
        } else if (d.resident == 0 && !d.force_T && !d.force_vec && !d.force_bx && !d.partial_rows &&
                   d.kind != ST_DIFFUSION_VAR && !p->stor) {
            res = res_choose(d, p->sms, &rg);
        }
        const double res_g = res ? 1000.0 * d.nx * d.ny / rg.t / 1e9 : 0.0;
        if (d.resident != 1) {
            // Contracted plans run one-warp tiles of V = 8 cells per thread (bsize_x = 256) with
            // partial-sum stages; exact plans run the rotating-window kernel, V = 4, with W warps
            // per tile (bsize_x = 128 W).
            // Where only T is forced, Hotspot takes V = 4: T = 8 against V = 8 (the better of its two
            // variants) 601 / 677 us on 3000 x 2000 x 160, 1467 / 1570 on 4096^2 x 200, 3985 / 3700 on
            // 8192^2 x 160, 7517 / 6951 on 16384^2 x 80.  With nothing forced the model chooses below.
            const bool var = d.kind == ST_DIFFUSION_VAR;   // windowed kernel, exact or contracted
            p->V = d.force_vec ? d.force_vec : ((d.exact || d.kind != ST_DIFFUSION) ? 4 : 8);
            if (d.force_bx) {
                if (d.force_bx % (32 * p->V)) rc = ST_ERR_UNSUPPORTED;
                p->W = d.force_bx / (32 * p->V);
            } else {
                p->W = 1;
                if (d.exact && d.nx >= 512) p->W = 4;
            }
            if (!d.exact && d.partial_rows == 1) p->W = 0;   // partial rows updated in place
            if (!d.exact && d.partial_rows == 2) p->W = 1;   // two alternating sets of partial rows
            if (p->stor && !d.force_T && !d.force_vec && !d.force_bx && !d.partial_rows) {
                // 16-bit storage, nothing forced: T = 8 with 8 cells per lane, rows in place, or,
                // where a block has few rows, 4 cells per lane (three warps per scheduler).  The
                // line is the float32 kernels' (their model).  Measured on GB300, 8 against 4 cells,
                // bf16 Hotspot: 8192^2 x 200 5222 / 6396 us, 16384^2 x 80 8993 / 11093; on the other
                // side of the line 3000 x 2000 x 150 703 / 713, 1100 x 6000 x 100 578 / 541
                int b8 = 0, b4 = 0;
                const Shape2D s8{d.kind, 0, 8, 8, 0, shape_stor(p)}, s4{d.kind, 0, 8, 4, 1, shape_stor(p)};
                p->V = 8;
                p->W = 0;
                if (tb2d_available(s4) && tb2d_prepare(s8, &b8) == cudaSuccess &&
                    tb2d_prepare(s4, &b4) == cudaSuccess && b8 > 0 && b4 > 0 &&
                    model_gcells_2d(d, p->sms, Cand2D{8, 4, 1}, b4, 1000) >
                        1.08 * model_gcells_2d(d, p->sms, Cand2D{8, 8, 0}, b8, 1000)) {
                    p->V = 4;
                    p->W = 1;
                }
                (void)cudaGetLastError();
            }
            if (!d.exact && !var && !p->stor && !d.force_T && !d.force_vec && !d.force_bx && !d.partial_rows) {
                // contracted, nothing forced: the compiled (T, V, variant) the model rates best
                const Cand2D cands[] = {{4, 4, 1}, {8, 4, 1}, {12, 4, 1}, {4, 8, 1}, {6, 8, 1},
                                        {8, 8, 1}, {8, 8, 0}, {12, 4, 0}};
                double best = -1.0;
                for (const Cand2D &k : cands) {
                    const Shape2D sh{d.kind, 0, k.T, k.V, k.W, d.kind == ST_THERMAL ? STOR_SRC : 0};
                    if (!tb2d_available(sh)) continue;
                    int bps = 0;
                    if (tb2d_prepare(sh, &bps) != cudaSuccess || bps < 1) continue;
                    const double g = model_gcells_2d(d, p->sms, k, bps, 1000);
                    if (g > best) {
                        best = g;
                        p->V = k.V;
                        p->W = k.W;
                    }
                }
                (void)cudaGetLastError();
            }
            // per-cell coefficients: every fused step keeps five more weight rows per tile column in
            // shared memory, so deeper fusion costs resident warps; measured on 8192^2 (GB300):
            // T = 4 with one-warp tiles 608 GCell/s, T = 8 545, four-warp tiles 532 / 451
            const int want = d.force_T ? d.force_T : (var ? 4 : 8);
            p->T = kernel_T_for(p, want);
            if (!d.exact && !var && !p->stor && !d.force_T && !d.force_vec && !d.force_bx && !d.partial_rows) {
                // and the T the model rates best within that family
                double best = -1.0;
                for (int t : kTcand) {
                    const Shape2D sh{d.kind, 0, t, p->V, p->W, d.kind == ST_THERMAL ? STOR_SRC : 0};
                    if (!tb2d_available(sh)) continue;
                    int bps = 0;
                    if (tb2d_prepare(sh, &bps) != cudaSuccess || bps < 1) continue;
                    const double g = model_gcells_2d(d, p->sms, Cand2D{t, p->V, p->W}, bps, 1000);
                    if (g > best) {
                        best = g;
                        p->T = t;
                    }
                }
                (void)cudaGetLastError();
            }
            if (p->T == 0 || (d.force_T && p->T != d.force_T)) rc = ST_ERR_UNSUPPORTED;
            if (res && d.resident == 0 && rc == ST_OK && !d.exact) {
                // contracted: resident tiles only where the model rates them above the passes
                // (exact plans: always when the grid fits; the exact passes have no calibration)
                int bps = 0;
                const Shape2D sh{d.kind, 0, p->T, p->V, p->W, d.kind == ST_THERMAL ? STOR_SRC : 0};
                if (tb2d_prepare(sh, &bps) == cudaSuccess && bps > 0 &&
                    model_gcells_2d(d, p->sms, Cand2D{p->T, p->V, p->W}, bps, 1000) >= res_g)
                    res = false;
                (void)cudaGetLastError();
            }
            PassCfg2D *c = nullptr;
            if (rc == ST_OK && !res) rc = prepare2(p, p->T, &c);
            if (rc == ST_OK && p->stor) {
                // coded grids: rows padded to 8 cells (16 bytes), codes per (row, tile column)
                p->cx = tb2d_tile_width(c->shape) - 2 * tb2d_halo(c->shape);
                p->ntx = (d.nx + p->cx - 1) / p->cx;
                p->ld_q = ((long long)d.nx + 7) / 8 * 8;
                const size_t qb = (size_t)p->ld_q * d.ny * 2, mb = (size_t)p->ntx * d.ny * sizeof(float2);
                for (int b = 0; b < 2 && rc == ST_OK; b++) {
                    e = stn::dev_malloc(&p->q[b], qb);
                    if (e == cudaSuccess) e = stn::dev_malloc(&p->qm[b], mb);
                    if (e != cudaSuccess) rc = map_cuda(e);
                }
                if (rc == ST_OK && d.kind == ST_THERMAL) {
                    e = stn::dev_malloc(&p->qp, qb);
                    if (e == cudaSuccess) e = stn::dev_malloc(&p->qpm, mb);
                    if (e != cudaSuccess) rc = map_cuda(e);
                }
                p->scratch_bytes = 0;   // no float32 scratch: the coded grids take its place
            } else if (rc == ST_OK && !res) {
                p->ld_scratch = ((long long)d.nx + 31) / 32 * 32;
                p->scratch_bytes = (size_t)p->ld_scratch * d.ny * sizeof(float);
            }
        }
        if (res && rc == ST_OK) {
            p->res = 1;
            p->T = rg.T;
            p->res_vx = rg.vx;
            p->res_nw = rg.nw;
            p->res_nbx = rg.nbx;
            p->res_nby = rg.nby;
            p->res_cw = rg.cw;
            p->res_ch = rg.ch;
            p->res_hx = rg.hx;
            p->res_ld = ((long long)d.nx + 3) / 4 * 4;
            p->scratch_bytes = 0;   // the two exchange grids take the scratch grid's place
            p->model = res_g;
        }
    } else {
        // tile width 64 (2 cells per lane) or 128 (4 cells per lane), tile height, cells per
        // thread; 64 x 64 with 16 cells per thread is the three-plane-window kernel (exact or
        // contracted), every other shape the partial-sum kernel (contracted)
        const bool free_tile = !d.exact && !d.force_bx && !d.force_by && !d.force_vec;
        int bx = d.force_bx ? d.force_bx : 64;
        int by = d.force_by ? d.force_by : (bx == 128 || free_tile ? 32 : 64);
        int cells = d.force_vec ? d.force_vec : (d.exact ? 16 : 8);
        int model_T = 0;
        if (free_tile && !d.force_T && d.rad <= 1) {
            // nothing forced, contracted: the compiled partial-sum (tile, T) the calibrated
            // model rates best
            const int shapes[][3] = {{64, 64, 8}, {64, 32, 8}, {128, 32, 8}, {64, 64, 4}};
            // (the rating of one deals its segments, so the most promising come first and the search
            // ends where the upper bound of the next is no better)
            struct Cand3 { double bound; int bx, by, cells, t; };
            std::vector<Cand3> cands;
            for (const auto &sh : shapes)
                for (int t : {3, 2, 4, 1}) {
                    const int vx = sh[0] / 32, vy = sh[2] / vx, nw = sh[1] / vy;
                    if (tb3d_available(Shape3D{d.kind, 0, t, vy, nw, 1, vx}))
                        cands.push_back({model_gcells_3d(d, p->sms, t, vx, vy, nw, true), sh[0], sh[1], sh[2], t});
                }
            std::stable_sort(cands.begin(), cands.end(), [](const Cand3 &a, const Cand3 &b) { return a.bound > b.bound; });
            double best = -1.0;
            for (const Cand3 &k : cands) {
                if (k.bound <= best) break;
                const int vx = k.bx / 32, vy = k.cells / vx;
                const double g = model_gcells_3d(d, p->sms, k.t, vx, vy, k.by / vy);
                if (g > best) {
                    best = g;
                    bx = k.bx;
                    by = k.by;
                    cells = k.cells;
                    model_T = k.t;
                }
            }
            p->model = std::max(best, 0.0);
        }
        if (bx != 64 && bx != 128) rc = ST_ERR_UNSUPPORTED;
        p->VX3 = bx / 32;
        if (rc == ST_OK && (cells % p->VX3 != 0 || by % (cells / p->VX3) != 0))
            rc = ST_ERR_UNSUPPORTED;
        if (rc == ST_OK) {
            p->VY = cells / p->VX3;
            p->NW = by / p->VY;
            p->alg3 = (p->VX3 == 2 && p->VY == 8 && p->NW == 8) ? 0 : 1;
            if (p->alg3 && d.exact) rc = ST_ERR_UNSUPPORTED;
        }
        const int want = d.force_T ? d.force_T : (model_T ? model_T : 4);
        p->T = kernel_T_for(p, want);
        if (p->T == 0 || (d.force_T && p->T != d.force_T)) rc = ST_ERR_UNSUPPORTED;
        PassCfg3D *c = nullptr;
        if (rc == ST_OK) rc = prepare3(p, p->T, &c);
        // the partial-sum kernel's scratch rows are padded to whole 16-byte chunks
        p->ld_scratch = p->alg3 ? ((long long)d.nx + 3) / 4 * 4 : d.nx;
        p->scratch_bytes = (size_t)p->ld_scratch * d.ny * d.nz * sizeof(float);
    }
    if (rc == ST_OK && p->scratch_bytes) {
        e = stn::dev_malloc(&p->scratch, p->scratch_bytes);
        if (e != cudaSuccess) rc = map_cuda(e);
    }
    if (rc == ST_OK && d.ndim == 2 && d.kind == ST_THERMAL && !d.exact && !p->stor) {
        // rows padded to 32 cells like the scratch grid: 16-byte aligned rows for any nx
        p->ld_src = ((long long)d.nx + 31) / 32 * 32;
        e = stn::dev_malloc(&p->src, (size_t)p->ld_src * d.ny * sizeof(float));
        if (e != cudaSuccess) rc = map_cuda(e);
    }
    if (rc == ST_OK && p->res) {
        const size_t fb = (size_t)p->res_nbx * p->res_nby * sizeof(int);
        e = stn::dev_malloc(&p->res_xg, (size_t)2 * p->res_ld * d.ny * sizeof(float));
        if (e == cudaSuccess) e = stn::dev_malloc(&p->res_flags, fb);
        if (e == cudaSuccess) e = stn::dev_zero(p->res_flags, fb, p->stream);
        if (e != cudaSuccess) rc = map_cuda(e);
    }
    if (rc == ST_OK && !p->res && !d.exact && !p->stor && d.rad <= 1 && d.kind != ST_DIFFUSION_VAR) {
        if (d.ndim == 2) {
            int bps = 0;
            const Shape2D sh{d.kind, 0, p->T, p->V, p->W, d.kind == ST_THERMAL ? STOR_SRC : 0};
            if (tb2d_prepare(sh, &bps) == cudaSuccess && bps > 0)
                p->model = model_gcells_2d(d, p->sms, Cand2D{p->T, p->V, p->W}, bps, 1000);
            (void)cudaGetLastError();
        } else if (p->alg3 && p->model <= 0.0) {   // forced
            p->model = model_gcells_3d(d, p->sms, p->T, p->VX3, p->VY, p->NW);
        }
    }
    if (rc == ST_OK) {
        e = stn::dev_malloc(&p->err, sizeof(int));
        if (e == cudaSuccess) e = stn::dev_zero(p->err, sizeof(int), p->stream);
        if (e != cudaSuccess) rc = map_cuda(e);
    }
    if (rc == ST_OK) rc = extra_grids(p);   // last: nothing the plan needs comes after it
    if (rc != ST_OK) {
        stencil_plan_destroy(p);
        return rc;
    }
    *out = p;
    return ST_OK;
}

int stencil_run(stencil_plan p, const void *grid_in, void *grid_out, const void *power,
                const float *coeffs, int nx, int ny, int nz, int steps)
{
    if (!p || !grid_in || !grid_out || steps < 0) return ST_ERR_INVALID_ARG;
    const stencil_desc &d = p->d;
    // per-cell coefficients come as device planes in `power`; host coefficients are unused
    static const float no_coeffs[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    if (!coeffs) {
        if (d.kind != ST_DIFFUSION_VAR) return ST_ERR_INVALID_ARG;
        coeffs = no_coeffs;
    }
    if (d.ndim == 2 && nz != 1) return ST_ERR_DIMS_MISMATCH;
    if (nx != d.nx || ny != d.ny || nz != d.nz) return ST_ERR_DIMS_MISMATCH;
    if ((d.kind != ST_DIFFUSION) != (power != nullptr)) return ST_ERR_INVALID_ARG;
    const size_t bytes = (size_t)cells_of(d) * sizeof(float);
    const size_t pw_bytes = d.kind == ST_DIFFUSION_VAR ? 5 * bytes : bytes;
    if (grid_in != grid_out && ranges_overlap(grid_in, grid_out, bytes)) return ST_ERR_INVALID_ARG;
    if (power && ranges_overlap2(power, pw_bytes, grid_out, bytes)) return ST_ERR_INVALID_ARG;
    if (d.strict && !stable(d, coeffs)) return ST_ERR_UNSTABLE_COEFFS;
    if (p->sticky != ST_OK) return p->sticky;
    const stn::NvtxRange r_run("stencil_run");

    const float *in = static_cast<const float *>(grid_in);
    float *out = static_cast<float *>(grid_out);
    const float *pw = static_cast<const float *>(power);
    cudaError_t e;
    if (steps == 0) {
        if (in == out) return ST_OK;
        e = cudaMemcpyAsync(out, in, bytes, cudaMemcpyDeviceToDevice, p->stream);
        return map_cuda(e);
    }
    if (p->res) {
        const int rc = run_resident(p, in, out, pw, coeffs, steps);
        if (rc != ST_OK) p->sticky = rc;
        return rc;
    }
    const int T = p->T;
    const int passes = (steps + T - 1) / T;
    const int last = steps - T * (passes - 1);
    if (p->stor) {
        // 16-bit storage: code the field (and the power map), run every pass on the coded
        // grids, decode into the output
        e = lp_encode(p->stor, in, d.nx, p->q[0], p->ld_q, p->qm[0], d.nx, d.ny, p->cx, p->stream);
        // the power map is coded as the Hotspot source map sdc*(p + amb*Rz) the kernels read
        if (e == cudaSuccess && pw)
            e = lp_encode(p->stor, pw, d.nx, p->qp, p->ld_q, p->qpm, d.nx, d.ny, p->cx, p->stream,
                          coeffs[4] * coeffs[3], coeffs[0]);
        if (e != cudaSuccess) return map_cuda(e);
        int cur = 0;
        for (int i = 0; i < passes; i++) {
            const stn::NvtxRange r_pass("pass");
            const int rc = run_pass2q(p, cur, 1 - cur, coeffs, (i == passes - 1) ? last : T);
            if (rc != ST_OK) {
                p->sticky = rc;
                return rc;
            }
            cur = 1 - cur;
        }
        e = lp_decode(p->stor, p->q[cur], p->ld_q, p->qm[cur], out, d.nx, d.nx, d.ny, p->cx,
                      p->stream);
        return map_cuda(e);
    }
    // buffer of pass i: the caller's output when (passes-1-i) is even, else the scratch grid;
    // in place with an odd pass count, pass 0 cannot write the input it reads, so every pass
    // shifts by one and a final copy brings the scratch result to the output.
    // With two scratch grids the passes between the first and the last use only those.
    const bool two = p->scratch2 != nullptr;
    const bool shift = (in == out) && (two ? passes == 1 : passes % 2 == 1);
    const long long ldo = d.nx, ldsc = p->ld_scratch;
    long long ldp = d.nx;
    if (p->src && d.ndim == 3) {
        if (passes > 1) {   // padded rows: one copy instead of unaligned reads in every pass
            e = cudaMemcpy2DAsync(p->src, (size_t)p->ld_src * sizeof(float), pw,
                                  (size_t)d.nx * sizeof(float), (size_t)d.nx * sizeof(float),
                                  (size_t)d.ny * d.nz, cudaMemcpyDeviceToDevice, p->stream);
            if (e != cudaSuccess) return map_cuda(e);
            pw = p->src;
            ldp = p->ld_src;
        }
    } else if (p->src) {
        // contracted Hotspot 2D kernels stage sdc*(p + amb*Rz) (Table 2's source and ambient
        // terms folded into one map)
        e = hot_source(pw, d.nx, p->src, p->ld_src, d.nx, d.ny, coeffs[4], coeffs[3], coeffs[0],
                       p->V, p->stream);
        if (e != cudaSuccess) return map_cuda(e);
        pw = p->src;
    }
    const float *src = in;
    long long lds = d.nx;
    for (int i = 0; i < passes; i++) {
        const stn::NvtxRange r_pass("pass");
        const int ts = (i == passes - 1) ? last : T;
        const bool to_out = two ? !shift && i == passes - 1
                            : shift ? ((passes - i) % 2 == 0) : ((passes - 1 - i) % 2 == 0);
        float *dst = to_out ? out : (two && i % 2) ? p->scratch2 : p->scratch;
        const long long ldd = to_out ? ldo : ldsc;
        int rc = d.rad > 1     ? run_pass_star(p, src, lds, dst, ldd, coeffs, ts)
                 : d.ndim == 2 ? run_pass2(p, src, lds, dst, ldd, pw, coeffs, ts)
                               : run_pass3(p, src, lds, dst, ldd, pw, ldp, coeffs, ts);
        if (rc != ST_OK) {
            p->sticky = rc;
            return rc;
        }
        src = dst;
        lds = ldd;
    }
    if (shift) {
        if (ldsc != d.nx)
            e = cudaMemcpy2DAsync(out, (size_t)d.nx * sizeof(float), p->scratch,
                                  (size_t)ldsc * sizeof(float), (size_t)d.nx * sizeof(float),
                                  (size_t)d.ny * d.nz, cudaMemcpyDeviceToDevice, p->stream);
        else
            e = cudaMemcpyAsync(out, p->scratch, bytes, cudaMemcpyDeviceToDevice, p->stream);
        if (e != cudaSuccess) return map_cuda(e);
    }
    return ST_OK;
}

int stencil_run_trajectory(stencil_plan p, const void *grid_in, void *states, long long stride,
                           const void *power, const float *coeffs, int steps)
{
    if (!p || !grid_in || !states || !coeffs || steps < 1) return ST_ERR_INVALID_ARG;
    const stencil_desc &d = p->d;
    if (d.ndim != 2 || d.exact || p->stor || d.rad > 1 || d.kind == ST_DIFFUSION_VAR)
        return ST_ERR_UNSUPPORTED;
    const long long n = (long long)d.nx * d.ny;
    if (stride < n) return ST_ERR_INVALID_ARG;
    if ((d.kind == ST_THERMAL) != (power != nullptr)) return ST_ERR_INVALID_ARG;
    const size_t bytes = (size_t)n * sizeof(float);
    const size_t span = ((size_t)(steps - 1) * stride + n) * sizeof(float);
    if (ranges_overlap2(grid_in, bytes, states, span)) return ST_ERR_INVALID_ARG;
    if (power && ranges_overlap2(power, bytes, states, span)) return ST_ERR_INVALID_ARG;
    if (d.strict && !stable(d, coeffs)) return ST_ERR_UNSTABLE_COEFFS;
    if (p->sticky != ST_OK) return p->sticky;
    PassCfg2D *c = nullptr;
    int rc = prepare_traj(p, &c);
    if (rc != ST_OK) return rc;
    const float *pw = static_cast<const float *>(power);
    if (p->src) {
        // contracted Hotspot kernels stage sdc*(p + amb*Rz) (Table 2's source and ambient terms
        // folded into one map)
        const cudaError_t e = hot_source(pw, d.nx, p->src, p->ld_src, d.nx, d.ny, coeffs[4],
                                         coeffs[3], coeffs[0], c->shape.V, p->stream);
        if (e != cudaSuccess) return map_cuda(e);
        pw = p->src;
    }
    float *st = static_cast<float *>(states);
    const int passes = (steps + kTrajT - 1) / kTrajT;
    for (int i = 0; i < passes; i++) {
        const int ts = std::min(kTrajT, steps - i * kTrajT);
        const float *src = i == 0 ? static_cast<const float *>(grid_in)
                                  : st + ((long long)i * kTrajT - 1) * stride;
        float *dst = st + ((long long)i * kTrajT + ts - 1) * stride;
        rc = run_pass2(p, src, d.nx, dst, d.nx, pw, coeffs, ts, c,
                       st + (long long)i * kTrajT * stride, stride);
        if (rc != ST_OK) {
            p->sticky = rc;
            return rc;
        }
    }
    return ST_OK;
}

int stencil_plan_sync(stencil_plan p)
{
    if (!p) return ST_ERR_INVALID_ARG;
    cudaError_t e = cudaStreamSynchronize(p->stream);
    if (e != cudaSuccess) return map_cuda(e);
    if (p->err) {
        int flag = 0;
        e = cudaMemcpy(&flag, p->err, sizeof(int), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return map_cuda(e);
        if (flag) {
            (void)stn::dev_zero(p->err, sizeof(int), p->stream);
            return ST_ERR_TIMEOUT;
        }
    }
    return p->sticky;
}

int stencil_plan_set_wait(stencil_plan p, long long wait_ns, int hold_block, int hold_epoch)
{
    if (!p || wait_ns <= 0 || hold_block < -1) return ST_ERR_INVALID_ARG;
    if (!p->res) return ST_ERR_UNSUPPORTED;
    p->res_wait_ns = wait_ns;
    p->res_hold_block = hold_block;
    p->res_hold_epoch = hold_block >= 0 ? hold_epoch : -1;
    return ST_OK;
}

int stencil_plan_get_info(stencil_plan p, stencil_plan_info *info)
{
    if (!p || !info) return ST_ERR_INVALID_ARG;
    std::memset(info, 0, sizeof(*info));
    info->T = p->T;
    info->model_gcells = p->model;
    info->sms = p->sms;
    info->scratch_bytes = (long long)p->scratch_bytes;
    info->exact = p->d.exact;
    info->partial_rows = (p->d.ndim == 2 && !p->d.exact && p->d.rad <= 1 && !p->res &&
                          p->d.kind != ST_DIFFUSION_VAR) ? (p->W == 0 ? 1 : 2) : 0;
    if (p->res) {
        info->resident = 1;
        info->bx = 32 * p->res_vx;
        info->by = p->res_nw * res2d_rows_per_thread();
        info->halo = p->res_hx;
        info->vec = p->res_vx;
        info->warps = p->res_nw;
        info->ctas = p->res_nbx * p->res_nby;
        info->scratch_bytes = (long long)2 * p->res_ld * p->d.ny * sizeof(float);
        info->kernel_id = 7;
        return ST_OK;
    }
    if (p->d.rad > 1 && p->d.ndim == 3) {
        int cx = 0, cy = 0;
        star3d_tile(p->d.rad, p->T, &cx, &cy);
        info->bx = 64;
        info->by = 64;
        info->halo = (64 - cx) / 2;
        info->vec = 16;
        info->warps = 8;
        info->ctas = p->ntx_star * p->nty_star * p->nseg_star;
        info->kernel_id = 6;
    } else if (p->star_rows) {
        PassCfg2D *c = nullptr;
        const int rc = prepare_star2f(p, p->T, &c);
        if (rc != ST_OK) return rc;
        info->bx = star2f_tile_width();
        info->by = 0;
        info->halo = (star2f_tile_width() - star2f_compute_width()) / 2;
        info->vec = 8;
        info->warps = 1;
        info->ctas = c->ctas;
        info->kernel_id = 8;
    } else if (p->d.rad > 1) {
        info->bx = 128;
        info->by = 128;
        info->halo = star2d_halo_x(p->d.rad, p->T);
        info->vec = 4;
        info->warps = 16;
        info->ctas = std::min(p->ntx_star * p->nty_star, p->sms);   // persistent, one per SM
        info->kernel_id = 5;
    } else if (p->d.ndim == 2) {
        PassCfg2D *c = nullptr;
        int rc = prepare2(p, p->T, &c);
        if (rc != ST_OK) return rc;
        const int warps = std::max(p->W, 1);   // W = 0 marks the one-warp in-place variant
        info->bx = 32 * p->V * warps;
        info->by = 0;
        info->halo = tb2d_halo(c->shape);
        info->vec = p->V;
        info->warps = warps;
        info->ctas = c->ctas;
        info->kernel_id = 2;
    } else {
        PassCfg3D *c = nullptr;
        int rc = prepare3(p, p->T, &c);
        if (rc != ST_OK) return rc;
        info->bx = 32 * p->VX3;
        info->by = p->VY * p->NW;
        info->halo = p->T;
        info->vec = p->VX3 * p->VY;
        info->warps = p->NW;
        info->ctas = c->ctas;
        info->kernel_id = p->alg3 ? 4 : 3;
    }
    return ST_OK;
}

int stencil_plan_set_timing(stencil_plan p, int enable)
{
    if (!p) return ST_ERR_INVALID_ARG;
    p->timing = enable != 0;
    return ST_OK;
}

int stencil_plan_kernel_time(stencil_plan p, double *ms, long long *launches, int reset)
{
    if (!p || !ms || !launches) return ST_ERR_INVALID_ARG;
    int rc = flush_timing(p);
    if (rc != ST_OK) return rc;
    *ms = p->ms_acc;
    *launches = p->launches;
    if (reset) {
        p->ms_acc = 0.0;
        p->launches = 0;
    }
    return ST_OK;
}

int stencil_plan_destroy(stencil_plan p)
{
    if (!p) return ST_OK;
    if (p->ev_used) cudaStreamSynchronize(p->stream);
    for (cudaEvent_t e : p->ev) cudaEventDestroy(e);
    if (p->scratch) stn::dev_free(p->scratch);
    if (p->scratch2) stn::dev_free(p->scratch2);
    for (int b = 0; b < 2; b++) {
        if (p->q[b]) stn::dev_free(p->q[b]);
        if (p->qm[b]) stn::dev_free(p->qm[b]);
    }
    if (p->qp) stn::dev_free(p->qp);
    if (p->qpm) stn::dev_free(p->qpm);
    if (p->err) stn::dev_free(p->err);
    if (p->src) stn::dev_free(p->src);
    if (p->res_xg) stn::dev_free(p->res_xg);
    if (p->res_flags) stn::dev_free(p->res_flags);
    for (PassCfg2D &c : p->cfg2)
        if (c.segs) stn::dev_free(c.segs);
    for (PassCfg3D &c : p->cfg3)
        if (c.segs) stn::dev_free(c.segs);
    delete p;
    return ST_OK;
}

}  // extern "C"
