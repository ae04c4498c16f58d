// tb2.cu -- launch of the two-step temporally blocked kernel yee_tb2 (tile
// variant 7): windows, the flattened (window, plane) work split into ranges
// of equal estimated cost over one wave of resident CTAs, and the source time
// factors of both steps.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "grid_impl.h"
#include "tma_host.h"
#include "yee_tb2.cuh"

namespace fdtd {

// Window rows of the kernel that serves tile height ty on a box: ty 16 takes
// the small windows too where the large ones hold so few planes per SM that a
// launch is the latency of a handful of planes, which a plane of six warps has
// less of than one of twelve.  The small windows' kernel has the fluence terms
// always, so that without a fluence the line lies lower.  us per step, 24 rows /
// 12 rows, and (window, plane) items per SM: 48 x 40 x 16 8.2 / 6.3 (0.4), 64 x 48 x
// 12 8.2 / 7.2 (0.7), 40 x 40 x 32 8.2 / 7.2 (0.8), 64 x 64 x 32 9.8 / 9.3 (2.5), 80 x 80 x
// 40 11.3 / 13.3 (4.2), 40 x 40 x 160 11.9 / 13.1 (4.2); without a fluence 48 x 40 x 16 7.2 /
// 6.4, 64 x 48 x 12 7.2 / 7.2, 80 x 80 x 16 8.2 / 9.3 (1.7), 64 x 64 x 32 8.2 / 9.3.
constexpr double kFewItems = 2.6, kFewItemsNoFlu = 0.7;
static int tb2_rows(const fdtd_grid* g, int ty)
{
    if (ty == 8) return kTb2RowsSmall;
    int t, u;
    tb2_windows(g->desc, kTb2Rows, &t, &u);
    const double items = double(t) * u * g->desc.nz / (g->sm_count > 0 ? g->sm_count : 152);
    return items <= (g->desc.fluence ? kFewItems : kFewItemsNoFlu) ? kTb2RowsSmall : kTb2Rows;
}

void tb2_windows(const fdtd_grid_desc& d, int ry, int* t, int* u)
{
    *t = (d.nx + kTb2Sx - 1) / kTb2Sx;
    *u = (d.ny + ry - 5) / (ry - 4);
}

// True if the windows of column wx of T (of row wy of U) run the x (y) shell
// and wall code.
static bool shell_x(const fdtd_grid_desc& d, int wx, int T)
{
    const int L0 = kTb2Sx * wx - kTb2Ox;
    return wx == 0 || wx == T - 1 || (d.npml > 0 && (L0 < d.npml || L0 + kTb2Wx > d.nx - d.npml));
}
static bool shell_y(const fdtd_grid_desc& d, int ry, int wy, int U)
{
    const int M0 = (ry - 4) * wy - kTb2Oy;
    return wy == 0 || wy == U - 1 || (d.npml > 0 && (M0 < d.npml || M0 + ry > d.ny - d.npml));
}

std::vector<long long> tb2_refined_ranges(const std::vector<long long>& s, const unsigned long long* cycles,
                                          double step)
{
    const int slots = int(s.size()) - 1;
    double total = 0.0;
    for (int c = 0; c < slots; ++c)
        if (s[size_t(c) + 1] > s[size_t(c)]) total += double(cycles[c]);
    if (!(total > 0.0)) return s;
    // cost of the items [0, x): piecewise linear, CTA c's items at cycles_c / (its item count) each
    std::vector<long long> ns(size_t(slots) + 1, s.back());
    ns[0] = 0;
    int c = 0;
    double cum = 0.0;
    for (int k = 1; k < slots; ++k) {
        const double target = total * k / slots;
        while (c < slots && (s[size_t(c) + 1] == s[size_t(c)] || cum + double(cycles[c]) < target)) {
            if (s[size_t(c) + 1] > s[size_t(c)]) cum += double(cycles[c]);
            ++c;
        }
        double x = double(s.back());
        if (c < slots) {
            const double frac = (target - cum) / double(cycles[c]);
            x = double(s[size_t(c)]) + frac * double(s[size_t(c) + 1] - s[size_t(c)]);
        }
        // move the boundary `step` of the way (damping against oscillation)
        const long long y = std::llround(double(s[size_t(k)]) + step * (x - double(s[size_t(k)])));
        ns[size_t(k)] = std::max(ns[size_t(k) - 1], std::min(y, s.back()));
    }
    return ns;
}

void tb2_refine(fdtd_grid* g, int ty, int slots, const unsigned long long* cycles, double step)
{
    const int ry = tb2_rows(g, ty);
    // the ranges the measured launches ran: the cached plan of this shape
    if (g->tb2_key.ry != ry || g->tb2_key.slots != slots || g->tb2_start.size() != size_t(slots) + 1) return;
    g->tb2_refined = tb2_refined_ranges(g->tb2_start, cycles, step);
    g->tb2_ref_order = g->tb2_key.order;
    g->tb2_ref_ry = ry;
    g->tb2_ref_slots = slots;
    g->tb2_ref_src = g->src_gen;
    g->tb2_ref_gen += 1;
}

// Rows interleaved by D (see Tb2Plan) for window order `mode` 2, row by row
// (D = 1) otherwise: D in [1, 16] such that D windows of planes come closest
// to a whole number of CTA shares.
static int tb2_order_d(int T, int U, int nz, int slots, int mode)
{
    if (mode != 2) return 1;
    const double share = double(T) * U * nz / slots;
    int best = 1;
    double bd = 1e30;
    for (int D = 1; D <= 16 && D <= U; ++D) {
        const double r = std::fmod(double(nz) * D, share), dist = std::min(r, share - r);
        if (dist < bd - 1e-9) { bd = dist; best = D; }
    }
    return best;
}

// Window at flattened position pos (the host copy of tb2_window_at).
static int tb2_window_host(int T, int U, int D, int pos)
{
    if (D <= 1) return pos;
    const int grp = pos / (T * D);
    const int rows = std::min(D, U - grp * D);
    const int r = pos - grp * T * D;
    const int wx = r / rows, l = r - wx * rows;
    return (grp * D + l) * T + wx;
}

// CTA work ranges of variant 7 on grid g: windows of 32 x RY columns, `slots`
// resident CTAs.  Each CTA gets a contiguous range of (window, plane) items,
// on the default tile and with lz 3 after as many whole windows as every CTA can
// have (kWholeMost): CTA c takes the windows c, c + slots, ..., so that `slots` consecutive windows
// march up z together and find each other's halo planes in L2 (a range starts
// at any plane, and its neighbours' halos come from HBM: 105 bytes read per
// cell and launch, 32 needed).  us per step, ranges only / whole windows
// first: 512 x 512 x 64 199 / 182, 400 x 330 x 48 88.6 / 78.0, 411 x 411 x 738 with z
// walls 2184 / 1610; without fluence 384 x 384 x 96 159 / 134, 332 x 332 x 46 52.4 / 47.7.
// The ranges either have equal estimated cost -- a window-plane costs 1,
// plus w_shell for each of the x and y shell or wall codes the window runs and
// kCorner w_shell more for both, plus w_ant if it holds antenna columns,
// kZPlane times that in the z shells, and a window costs kRestart more planes
// at its start (the wavefront refills: four planes and the first loads'
// latency) -- or (tc.measured) are the ones tb2_refine moved until
// the CTAs' measured times were equal.  Cached on the grid until the antenna,
// the weights or the launch shape change.
// Measured on GB300 (cycles per plane, 256 x 256 x 128 cells): inner windows
// 2400, with antenna columns 2750, x shell 3340, y shell 3380, both 4720; the
// default weights 0.4 and 0.2 follow (0.15 is slower by up to 2 %).  A z-shell
// plane takes about 2.3 inner ones (411 x 411 x 192: 448 us per step with 4 cells of
// z CPML, 508 with 16), and a launch 15 to 55 us more for having any, whatever
// their number.  The split does best with less weight than that: us per step at
// kZPlane 1.6 / 2.2 / 3 / 4, 411 x 411 x 192 with 16 cells 508 / 519 / 520 / 521, 340 x
// 340 x 192 417 / 423 / 426 / 431, 205 x 205 x 400 with 8 417 / 429 / 438 / 456, 332 x 332 x 40
// with 1 91 / 82 / 82 / 81.
constexpr double kRestart = 5.3;
constexpr double kCorner = 0.4;
constexpr double kZPlane = 1.6;
// Whole windows first only as far as no CTA's whole windows cost more than this
// times a CTA's mean share: few windows per CTA and the dear ones on the shell
// would leave the others waiting (288 x 252 x 128, 156 windows on 152 SMs: 151 us
// per step with one round of whole windows, 113 with ranges only).  us per
// step at limits 1.0 / 1.12 / 1.18 / 1.25: 332 x 332 x 46 52.4 / 47.7 / 47.7 / 47.6,
// 360 x 300 x 64 82.3 / 82.4 / 76.9 / 76.9, 430 x 350 x 64 87.1 / 87.1 / 86.3 / 91.9, 600 x
// 500 x 24 87.4 / 87.4 / 87.0 / 94.5.
constexpr double kWholeMost = 1.18;
static void tb2_plan(fdtd_grid* g, int RY, int slots, const TileConfig& tc, Tb2Plan& P)
{
    const fdtd_grid_desc& d = g->desc;
    tb2_windows(d, RY, &P.T, &P.U);
    P.prof = nullptr;
    P.dt16 = float(g->dt * 0.0625);
    P.err = reinterpret_cast<int*>(static_cast<char*>(g->arena) + g->L.err);
    // whole windows first (0), rows interleaved (2) or row by row (1); measured
    // ranges, and the launches that measure them, hold every window
    const bool measure = tc.measured || g->tb2_profile;
    const int order = tc.automatic || (tc.lz == 3 && !measure) ? 0 : (tc.lz == 2 ? 2 : 1);
    P.D = tb2_order_d(P.T, P.U, d.nz, slots, order);
    const bool meas = tc.measured && g->tb2_ref_ry == RY && g->tb2_ref_slots == slots &&
                      g->tb2_ref_src == g->src_gen && g->tb2_refined.size() == size_t(slots) + 1 &&
                      g->tb2_ref_order == order;
    auto& key = g->tb2_key;
    if (key.ry != RY || key.slots != slots || key.src_gen != g->src_gen || key.measured != meas ||
        key.order != order ||
        (meas ? key.cost_gen != g->tb2_ref_gen : (key.w_shell != tc.w_shell || key.w_ant != tc.w_ant))) {
        if (meas) {
            g->tb2_start = g->tb2_refined;
            g->tb2_whole = 0;
        } else {
            const int nx = d.nx, ny = d.ny, nz = d.nz;
            const int nw = P.T * P.U;
            std::vector<double> cost(size_t(nw), 1.0);
            for (int wy = 0; wy < P.U; ++wy)
                for (int wx = 0; wx < P.T; ++wx) {
                    const int L0 = kTb2Sx * wx - kTb2Ox, M0 = (RY - 4) * wy - kTb2Oy;
                    const int i0 = std::max(L0, 0), i1 = std::min(L0 + kTb2Wx, nx);
                    const int j0 = std::max(M0, 0), j1 = std::min(M0 + RY, ny);
                    const int sx = shell_x(d, wx, P.T), sy = shell_y(d, RY, wy, P.U);
                    bool ant = false;
                    if (!g->hmask.empty())
                        for (int j = j0; j < j1 && !ant; ++j)
                            for (int i = i0; i < i1 && !ant; ++i) ant = g->hmask[size_t(j) * nx + i] != 0;
                    cost[size_t(wy) * P.T + wx] = 1.0 + (sx + sy + kCorner * sx * sy) * tc.w_shell + (ant ? tc.w_ant : 0.0);
                }
            // planes of the z shells cost kZPlane times a plain one
            std::vector<double> zc(size_t(nz) + 1, 0.0);   // cost of the planes [0, k)
            const bool zw = d.z_boundary == FDTD_Z_WALLS;
            const int pz = zw ? d.npml_z : 0;
            for (int k = 0; k < nz; ++k) zc[size_t(k) + 1] = zc[size_t(k)] + (k < pz || k >= nz - pz ? kZPlane : 1.0);
            const double zsum = zc[size_t(nz)];
            if (P.D > 1) {   // costs by position
                std::vector<double> byp(cost.size());
                for (int m = 0; m < nw; ++m) byp[size_t(m)] = cost[size_t(tb2_window_host(P.T, P.U, P.D, m))];
                cost.swap(byp);
            }
            // the whole windows, then ranges of the others (from first on) that
            // bring every CTA to the same cost: CTA c's share of them is what its
            // whole windows leave below the level
            double rest = 0.0;
            for (int w = 0; w < nw; ++w) rest += cost[size_t(w)] * (zsum + kRestart);
            const double most = kWholeMost * rest / slots;
            std::vector<double> own(size_t(slots), 0.0), reach(size_t(slots) + 1, 0.0);
            int first = order == 0 ? nw / slots * slots : 0;
            for (;; first -= slots) {
                std::fill(own.begin(), own.end(), 0.0);
                for (int w = 0; w < first; ++w) own[size_t(w % slots)] += cost[size_t(w)] * (zsum + kRestart);
                if (first == 0 || *std::max_element(own.begin(), own.end()) <= most) break;
            }
            g->tb2_whole = first;
            rest = 0.0;
            for (int w = first; w < nw; ++w) rest += cost[size_t(w)] * (zsum + kRestart);
            std::vector<double> level(own);
            std::sort(level.begin(), level.end());
            double top = 0.0, below = 0.0;
            for (int n = 1; n <= slots; ++n) {   // the n CTAs with the least share the rest
                below += level[size_t(n) - 1];
                top = (rest + below) / n;
                if (n == slots || top <= level[size_t(n)]) break;
            }
            for (int c = 0; c < slots; ++c) reach[size_t(c) + 1] = reach[size_t(c)] + std::max(0.0, top - own[size_t(c)]);
            std::vector<long long> start(size_t(slots) + 1, (long long)(nw - first) * nz);
            start[0] = 0;
            int c = 1;
            double cum = 0.0;
            for (int w = 0; w < nw - first && c < slots; ++w) {
                const double cw = cost[size_t(first + w)];
                const double span = cw * (zsum + kRestart), base = cum + cw * kRestart;
                while (c < slots && reach[size_t(c)] < cum + span) {
                    // the first plane whose cost from the window's start reaches the share
                    long long k = std::lower_bound(zc.begin(), zc.end(), (reach[size_t(c)] - base) / cw) - zc.begin();
                    k = std::max(0LL, std::min((long long)nz, k));
                    start[size_t(c)] = std::max(start[size_t(c) - 1], (long long)w * nz + k);
                    ++c;
                }
                cum += span;
            }
            g->tb2_start = start;
        }
        key.ry = RY; key.slots = slots; key.src_gen = g->src_gen;
        key.w_shell = tc.w_shell; key.w_ant = tc.w_ant;
        key.measured = meas; key.cost_gen = g->tb2_ref_gen; key.order = order;
    }
    P.whole = g->tb2_whole;
    for (int c = 0; c <= slots; ++c) P.start[c] = g->tb2_start[size_t(c)];
}

// Resident CTAs per SM of the kernels of one RY on the device `device`, the
// current one (dynamic shared memory set on the device's first use).
template <int RY>
static cudaError_t tb2_blocks_per_sm(int device, int* out)
{
    using S = Tb2Smem<RY>;
    static_assert(S::bytes() <= 232448, "the window's shared memory exceeds the 227 KB a CTA can hold");
    static PerDevice blocks_per_sm;
    return blocks_per_sm.get(device, out, [](int* n) {
        const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
        const int bytes = int(S::bytes());
        cudaError_t e = cudaFuncSetAttribute(yee_tb2<RY, false, false, true>, at, bytes);
        if constexpr (RY == kTb2Rows) {
            if (e == cudaSuccess) e = cudaFuncSetAttribute(yee_tb2<RY, false, false, false>, at, bytes);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(yee_tb2<RY, false, true, true>, at, bytes);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(yee_tb2<RY, false, true, false>, at, bytes);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(yee_tb2<RY, true, true, true>, at, bytes);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(yee_tb2_t<RY, false, false, true>, at, bytes);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(yee_tb2_t<RY, false, true, true>, at, bytes);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(yee_tb2_t<RY, true, true, true>, at, bytes);
        }
        if (e != cudaSuccess) return e;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, yee_tb2<RY, false, false, true>, S::NT, S::bytes());
        return e == cudaSuccess && *n < 1 ? cudaErrorInvalidConfiguration : e;
    });
}

// ---- the route of the default tile
// Estimated us per step of the two kernels that a pair of steps can take.  The
// bits are the same, so the default tile takes the one estimated to be faster.
// The constants were fitted to 1123 boxes measured both ways on GB300 (2 x 2 x 1
// to 2048 x 2048 x 12 and 8 x 8 x 16384 cells, with and without fluence, CPML, z
// walls, z CPML and sheet): the faster kernel is taken, or one within 3 % of it,
// for 1044 of them, and the others cost 11 % on average.  us per step, two-step /
// cell passes: 2048 x 2048 x 1 224 / 79, x 3 295 / 273, x 12 603 / 1075; 560 x 560 x
// 2 24.6 / 16.5, x 12 56 / 75; 32 x 32 x 1024 36 / 25, 20 x 20 x 4096 38 / 69; 332 x
// 332 x 46 62 / 109; 16 x 16 x 64 7.2 / 8.2; z walls, 360 x 360 x 6 34 / 21, 411 x 411
// x 192 with 16 z-CPML cells 508 / 684, 205 x 205 x 400 with 8 417 / 402.
//
// Two-step kernel on `ctas` CTAs: the planes of a CTA's share, and kRefill for
// each window it starts and for the range in which it goes on inside one,
// times the time of a plane.
constexpr double kRefill = 5.6;                       // planes
constexpr double kPlane = 1.24, kPlaneNoFlu = 1.0;    // us, an inner window's, with and without the fluence terms
constexpr double kPlaneWall = 1.43, kPlaneWallNoFlu = 1.6;   // the wall kernel's, which has the terms always
constexpr double kShellWall = 0.3;                    // as w_shell, for the wall kernel
constexpr double kOddShell = 0.32;                    // more for an x shell off even columns (4-byte psi accesses)
constexpr double kZShell = 2.1;                       // a z-shell plane, in planes
constexpr double kZCode = 1.27, kZCodeFew = 1.6;      // all of it with a z CPML: many and few windows per CTA
constexpr double kManyWindows = 1.5;
constexpr double kWallFloor = 8.5;
double two_step_us(const fdtd_grid_desc& d, bool sheet, int ctas, bool terms)
{
    int T, U;
    tb2_windows(d, kTb2Rows, &T, &U);
    const bool zw = d.z_boundary == FDTD_Z_WALLS, wall = zw || sheet;
    double fx = 0.0, fy = 0.0;   // shares of the windows with x and with y shell code
    for (int wx = 0; wx < T; ++wx) fx += shell_x(d, wx, T) ? 1.0 / T : 0.0;
    for (int wy = 0; wy < U; ++wy) fy += shell_y(d, kTb2Rows, wy, U) ? 1.0 / U : 0.0;
    const double odd = d.npml > 0 && ((d.nx | d.npml) & 1) ? kOddShell : 0.0;
    const double cost = 1.0 + (wall ? kShellWall : TileConfig().w_shell) * (fx * (1.0 + odd) + fy + kCorner * fx * fy);
    const double windows = double(T) * U / ctas;   // per CTA
    const int npz = zw ? d.npml_z : 0;
    const double nz = d.nz, z = nz + 2.0 * npz * (kZShell - 1.0);
    const double planes = std::max(windows * z, z / nz) + (kRefill + (zw ? 1.0 : 0.0)) * (windows + 1.0);
    const double plane = wall ? (d.fluence ? kPlaneWall : kPlaneWallNoFlu) : (terms ? kPlane : kPlaneNoFlu);
    const double us = 0.5 * cost * planes * plane * (npz == 0 ? 1.0 : (windows < kManyWindows ? kZCodeFew : kZCode));
    return wall ? std::max(us, kWallFloor) : us;
}

// Cell passes: two launches, and from some 10^5 cells on the cells (in whole
// 32 x 4 blocks) at the rate of the passes, the shells' with half a cell's
// work more.
constexpr double kCellRate = 52.0e3, kCellRateNoFlu = 70.0e3;   // cells per us
constexpr double kCellShell = 0.55;
static double cell_blocks(const fdtd_grid_desc& d)   // cells in whole blocks
{
    return double((d.nx + 31) / 32 * 32) * ((d.ny + 3) / 4 * 4) * d.nz;
}

double cell_work_us(const fdtd_grid_desc& d)
{
    const double inner = std::max(0.0, 1.0 - 2.0 * d.npml / d.nx) * std::max(0.0, 1.0 - 2.0 * d.npml / d.ny);
    const int npz = d.z_boundary == FDTD_Z_WALLS ? d.npml_z : 0;
    const double shell = 1.0 - (d.npml > 0 ? inner : 1.0) * (1.0 - 2.0 * npz / d.nz);
    return cell_blocks(d) * (1.0 + kCellShell * shell) / (d.fluence ? kCellRate : kCellRateNoFlu);
}

double cell_step_us(const fdtd_grid_desc& d)
{
    const double cells = cell_blocks(d);
    const double launches = d.fluence ? std::max(8.9, 8.2 + std::min(cells / 65e3, 4.1))
                                      : 8.2 + std::min(std::max(0.0, cells - 190e3) / 20e3, 4.1);
    return std::max(launches, 2.9 + cell_work_us(d));
}

bool default_two_step(const fdtd_grid* g)
{
    if (g->desc.precision != FDTD_F32) return false;
    if (g->route != 0) return g->route == 1;
    return two_step_us(g->desc, g->has_wall, g->sm_count > 0 ? g->sm_count : 152, g->desc.fluence != 0) <
           cell_step_us(g->desc);
}

int tb2_slots(const fdtd_grid* g, int ty)
{
    int per_sm = 0;
    const cudaError_t e = tb2_rows(g, ty) == kTb2RowsSmall
                              ? tb2_blocks_per_sm<kTb2RowsSmall>(g->device, &per_sm)
                              : tb2_blocks_per_sm<kTb2Rows>(g->device, &per_sm);
    if (e != cudaSuccess) return -1;
    return std::min(kTb2MaxCtas, (g->sm_count > 0 ? g->sm_count : 152) * per_sm);
}

// Tensor maps of the fields of copy `cur` and of the fluence accumulator, in
// boxes of one window (32 x RY columns of one plane).
template <int RY>
static bool tb2_maps(fdtd_grid* g, int cur, TmaMaps** out)
{
    const int sl = RY == kTb2RowsSmall ? 0 : 1;
    TmaMaps& m = g->tb2maps[cur][sl];
    if (!g->tb2maps_ok[cur][sl]) {
        char* A = static_cast<char*>(g->arena);
        bool ok = true;
        for (int c = 0; c < 3; ++c) {
            ok = ok && encode_map(&m.e[c], A + g->L.field[cur][c], 4, g->desc, g->L.pitch, kTb2Wx, RY, CU_TENSOR_MAP_L2_PROMOTION_L2_64B);
            ok = ok && encode_map(&m.h[c], A + g->L.field[cur][3 + c], 4, g->desc, g->L.pitch, kTb2Wx, RY, CU_TENSOR_MAP_L2_PROMOTION_L2_64B);
        }
        void* f = g->desc.fluence ? A + g->L.fluence : A + g->L.field[cur][0];   // unused without a fluence
        if (g->desc.fluence) ok = ok && encode_map(&m.f, f, 8, g->desc, g->L.pitch, kTb2Wx, RY, CU_TENSOR_MAP_L2_PROMOTION_L2_64B);
        else m.f = m.e[0];
        if (!ok) return false;
        g->tb2maps_ok[cur][sl] = true;
    }
    *out = &m;
    return true;
}

template <int RY>
static cudaError_t launch_tb2_t(const fdtd_grid* cg, int cur, long long n, const TileConfig& tc, cudaStream_t s)
{
    fdtd_grid* g = const_cast<fdtd_grid*>(cg);
    using S = Tb2Smem<RY>;
    int per_sm = 0;
    cudaError_t e = tb2_blocks_per_sm<RY>(g->device, &per_sm);
    if (e != cudaSuccess) return e;
    const int slots = std::min(kTb2MaxCtas, (g->sm_count > 0 ? g->sm_count : 152) * per_sm);
    Tb2Plan plan;
    tb2_plan(g, RY, slots, tc, plan);
    if (g->tb2_profile)
        plan.prof = reinterpret_cast<unsigned long long*>(static_cast<char*>(g->arena) + g->L.tb2prof);
    const SrcTime* wall = g->has_wall ? &g->wallt : nullptr;
    const StepTime<float> t0 = step_time<float>(g->srct, wall, g->dt, n);
    const StepTime<float> t1 = step_time<float>(g->srct, wall, g->dt, n + 1);
    Tb2Times tt;
    tt.th0 = t0.th; tt.te0 = t0.te; tt.tw0 = t0.tw;
    tt.th1 = t1.th; tt.te1 = t1.te; tt.tw1 = t1.tw;
    TmaMaps* m = nullptr;
    if (!tb2_maps<RY>(g, cur, &m)) return cudaErrorInvalidValue;
    mark_waits(g, s);
    const StepArgs<float> a = make_args<float>(g, cur);
    const unsigned ctas = unsigned(slots);
    if constexpr (RY == kTb2Rows) {
        const bool flu = g->desc.fluence != 0;
        if (tc.automatic) {   // runs on the default tile: the cell passes' roundings
            if (has_walls(g)) yee_tb2<RY, true, true, true><<<ctas, S::NT, S::bytes(), s>>>(a, tt, *m, plan);
            else if (flu) yee_tb2<RY, false, true, true><<<ctas, S::NT, S::bytes(), s>>>(a, tt, *m, plan);
            else yee_tb2<RY, false, true, false><<<ctas, S::NT, S::bytes(), s>>>(a, tt, *m, plan);
            return cudaGetLastError();
        }
        if (!flu) {
            yee_tb2<RY, false, false, false><<<ctas, S::NT, S::bytes(), s>>>(a, tt, *m, plan);
            return cudaGetLastError();
        }
    }
    yee_tb2<RY, false, false, true><<<ctas, S::NT, S::bytes(), s>>>(a, tt, *m, plan);
    return cudaGetLastError();
}

cudaError_t launch_tb2(const fdtd_grid* g, int cur, long long n, const TileConfig& tc, cudaStream_t s)
{
    if (g->desc.precision != FDTD_F32 || (has_walls(g) && !tc.automatic)) return cudaErrorInvalidValue;
    if (!tc.automatic && tb2_rows(g, tc.ty) == kTb2RowsSmall) return launch_tb2_t<kTb2RowsSmall>(g, cur, n, tc, s);
    return launch_tb2_t<kTb2Rows>(g, cur, n, tc, s);
}

cudaError_t launch_tb2_table(const fdtd_grid* cg, int cur, const StepTime<float>* times, int i0, int i1,
                             int max_ctas, bool automatic, cudaStream_t s)
{
    fdtd_grid* g = const_cast<fdtd_grid*>(cg);
    if (g->desc.precision != FDTD_F32 || (has_walls(g) && !automatic)) return cudaErrorInvalidValue;
    constexpr int RY = kTb2Rows;
    using S = Tb2Smem<RY>;
    int per_sm = 0;
    cudaError_t e = tb2_blocks_per_sm<RY>(g->device, &per_sm);
    if (e != cudaSuccess) return e;
    const int all = std::min(kTb2MaxCtas, (g->sm_count > 0 ? g->sm_count : 152) * per_sm);
    const int slots = std::max(1, std::min(all, max_ctas));
    // an automatic launch has the default tile's work split, whatever tile the
    // grid's own steps take
    const TileConfig tc = automatic ? default_tile(g->desc, g->sm_count) : g->tile;
    Tb2Plan plan;
    tb2_plan(g, RY, slots, tc, plan);
    TmaMaps* m = nullptr;
    if (!tb2_maps<RY>(g, cur, &m)) return cudaErrorInvalidValue;
    const StepArgs<float> a = make_args<float>(g, cur);
    const unsigned ctas = unsigned(slots);
    if (!automatic) yee_tb2_t<RY, false, false, true><<<ctas, S::NT, S::bytes(), s>>>(a, times, i0, i1, *m, plan);
    else if (has_walls(g)) yee_tb2_t<RY, true, true, true><<<ctas, S::NT, S::bytes(), s>>>(a, times, i0, i1, *m, plan);
    else yee_tb2_t<RY, false, true, true><<<ctas, S::NT, S::bytes(), s>>>(a, times, i0, i1, *m, plan);
    return cudaGetLastError();
}

}  // namespace fdtd

using namespace fdtd;

extern "C" {

int fdtd_debug_tb2_order(int t, int u, int nz, int slots, int order, int* out)
{
    if (t < 1 || u < 1 || nz < 1 || slots < 1 || !out) return -1;
    const int D = tb2_order_d(t, u, nz, slots, order == 2 ? 2 : 1);
    for (int m = 0; m < t * u; ++m) out[m] = tb2_window_host(t, u, D, m);
    return D;
}

fdtd_status fdtd_debug_route_us(const fdtd_grid_desc* d, int sheet, int ctas, double* two_step, double* cells)
{
    const fdtd_status st = validate(d);
    if (st != FDTD_OK) return st;
    if (ctas < 1 || !two_step || !cells) return fail(FDTD_EINVAL, "invalid argument");
    *two_step = two_step_us(*d, sheet != 0, ctas, d->fluence != 0);
    *cells = cell_step_us(*d);
    return FDTD_OK;
}

fdtd_status fdtd_debug_set_route(fdtd_grid* g, int route)
{
    if (!g || route < 0 || route > 2 || (route == 1 && g->desc.precision != FDTD_F32))
        return fail(FDTD_EINVAL, "invalid argument");
    if (g->batch_refs > 0) return fail(FDTD_ESTATE, "fdtd_debug_set_route: the grid belongs to a batch");
    g->route = route;
    return FDTD_OK;
}

int fdtd_debug_get_route(const fdtd_grid* g)
{
    if (!g) return -1;
    return g->tile.variant == 7 || (g->tile.automatic && default_two_step(g)) ? 1 : 2;
}

fdtd_status fdtd_debug_per_device(const int* devices, const int* results, int n, int* values)
{
    if (!devices || !results || !values || n < 1) return fail(FDTD_EINVAL, "invalid argument");
    PerDevice p;
    for (int q = 0; q < n; ++q) {
        values[q] = 0;
        const cudaError_t e = p.get(devices[q], &values[q], [&](int* v) {
            *v = results[q];
            return results[q] > 0 ? cudaSuccess : cudaErrorInvalidValue;
        });
        if (e != cudaSuccess) values[q] = -1;
    }
    return FDTD_OK;
}

fdtd_status fdtd_debug_tb2_refine(int slots, const long long* starts, const unsigned long long* cycles, double step,
                                  long long* out)
{
    if (slots < 1 || !starts || !cycles || !out || !(step > 0.0 && step <= 1.0))
        return fail(FDTD_EINVAL, "invalid argument");
    std::vector<long long> s(starts, starts + slots + 1);
    if (s[0] != 0) return fail(FDTD_EINVAL, "starts[0] must be 0");
    for (int c = 0; c < slots; ++c)
        if (s[size_t(c) + 1] < s[size_t(c)]) return fail(FDTD_EINVAL, "starts must not decrease");
    const std::vector<long long> ns = tb2_refined_ranges(s, cycles, step);
    for (int c = 0; c <= slots; ++c) out[c] = ns[size_t(c)];
    return FDTD_OK;
}

}  // extern "C"
