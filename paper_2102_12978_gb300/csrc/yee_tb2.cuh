// yee_tb2.cuh -- two Yee steps per launch (temporal blocking), FP32 (sm_103a).
//
// One launch advances the grid from (E^n, H^{n-1/2}) to (E^{n+2}, H^{n+3/2})
// and adds the fluence terms of steps n and n+1, so that the fields, the
// fluence accumulator and the CPML psi cross HBM once per two steps: half the
// bytes per cell-update of any one-step pass.  Every arithmetic step is the
// one of the cell passes (Section 4 Yee update with the Roden-Gedney CPML,
// the soft source of Eq. 13, the fluence of Section 2), in the same order; with
// CR (see tb2_flux) the two agree bit for bit.
//
// Work decomposition.
//   * A CTA owns a window of 32 x RY (i, j) columns and marches along z; each
//     thread owns two x-adjacent columns (16 RY threads, a half warp per
//     row).  A window writes E^{n+2} and H^{n+3/2} only on its own 24 x
//     (RY - 4) columns, which start 4 columns and 2 rows in, and recomputes
//     what they need around them itself (E^{n+2} can be had from 2 columns and
//     rows in).  Columns past the box hold exact zeros at every stage
//     (zero-filled loads, zero coefficients): the wall values the stencil
//     reads there.
//   * Own columns start at multiples of 8, so that every store fills whole
//     32-byte sectors.  Stores of partial sectors were what held the kernel:
//     with own columns 28 wide (of the same 32), whose rows begin and end
//     inside a sector, a plane of an inner window took 3900 cycles, against
//     2380 with full sectors and 2050 without any loads and stores
//     (256 x 256 x 128 cells, one GB300); the 24-wide windows are a fifth more
//     and still faster by a third.
//   * Two columns per thread, because the kernel is bound by instruction
//     issue and latency before HBM and the FP32 pipe: the FP32 arithmetic of
//     the two columns is one packed instruction (fma.rn.f32x2 and its kin run
//     at half the rate of the scalar ones, so the pipe is as busy and the
//     issue slots are halved), shared-memory accesses and stores move both
//     columns at once, the x neighbours of the pair take one shuffle, and a
//     window of 32 x 24 columns fits the register file with 12 warps.  430
//     instructions per warp and plane of 64 columns, against 385 per 32
//     columns with one column per thread.
//   * z-march with a wavefront of four stages per plane p: A, H^{n+1/2} of
//     plane p-1; B, E^{n+1} of plane p-1; C, H^{n+3/2} of plane p-2; D,
//     E^{n+2} of plane p-2.  The y neighbours come from per-plane shared
//     exchange buffers (E^n straight from the ring of loaded planes), the
//     z neighbours from registers carried from plane to plane; two CTA
//     barriers per plane.
//   * Planes are loaded by TMA, one box per array (32 x RY columns of E^n and
//     H^{n-1/2} of plane p + 3 and of the fluence of plane p), zero-filled
//     past the box, into a ring of four slots; a slot completes on its own
//     mbarrier.  A thread copies the CPML psi of its own shell columns by
//     cp.async into two slots of its own.
//   * The antenna coefficients of a window's columns are staged in shared
//     memory when the window starts; the per-plane phase e^{i beta z_k} is
//     loaded one plane ahead.
//   * The fluence of cell (i, j, k) needs E and H at i+1, j+1, k+1; a
//     window's fluence cells are its own columns, their rows and planes
//     shifted by -1 (plus the last row before the far wall; on z-walled grids
//     the last plane too), so that the H^{n+3/2} they need lie inside the
//     window.  Both terms of a cell (steps n and n+1) are
//     added, Kahan-compensated, in one read-modify-write.
//   * Reading step n from one copy of the fields and psi and writing step
//     n+2 into the other (ping-pong, E-side psi included) makes the halo
//     recompute race-free.
//   * Every row of a window runs every stage, whether or not a column the
//     window writes depends on it, so that the stage code has no branches
//     on the row; a warp with antenna points adds the source terms on all its
//     lanes (zero terms where a column has none), and the x-shell windows
//     update the x psi on all lanes (zero coefficients off the shell).
//     Windows off the x (y) faces and shells run code without the checks of
//     the x (y) walls, psi and columns past the box (template flags GX, GY).
//     A plane of an inner window takes 2400 cycles, of an x- or y-shell window
//     3400, of a corner 4700.
//   * On the default tile (and with lz 3) a CTA takes whole windows first, so
//     that neighbouring windows march together and share halo planes in L2,
//     then a range of what is left (tb2_plan).  On other tiles it takes
//     a contiguous range of the flattened (window, plane) work:
//     ranges of equal estimated cost (windows with CPML shell or antenna
//     columns weigh more, with weights the autotuner picks by timing), or
//     ranges the host refined until the CTAs' measured times were equal
//     (the kernel records each CTA's SM cycles when asked).  The window rows
//     may be interleaved in the flattened order, so that x-neighbouring
//     windows march side by side (tb2_window_at).  Where a range starts or
//     crosses into the next window the wavefront restarts, which costs four
//     planes of recompute and the latency of the first loads.
//   * Outputs are stored with the L2 evict-last policy; every sum of two
//     products is rounded explicitly (see below).
//   * Grids with z walls or a wall sheet run an instantiation of their own
//     (W), whose planes off the z shells run the loop above with the walls'
//     few extra tests; z-shell planes run apart.
// FP32 fields with the Kahan FP32 fluence.  256 x 256 x 128 cells with a
// 16-cell CPML, antenna and fluence: 104 us per step (one column per thread,
// windows of 32 x 16 with 28 x 12 own columns: 122-130 us); 512 x 512 x 64: 182 us.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "yee_cell.cuh"

namespace fdtd {

// Source time factors f e^{-i Phi} of the two steps: H at (n+1/2) dt and
// (n+3/2) dt, E (and the wall sheet) at (n+1) dt and (n+2) dt.
struct Tb2Times {
    Cpx<float> th0, te0, th1, te1, tw0, tw1;
};

// Flattened work: windows T (along x) by U (along y), nz planes each, items
// (window, plane) numbered window * nz + plane.  CTA c takes the items
// [start[c], start[c + 1]): ranges of equal estimated cost (a window's planes
// cost more where the window holds CPML shell or antenna columns), chosen on
// the host.
// prof, if not null, receives per CTA c the SM cycles it ran (prof[c] is
// added to): the host moves the ranges' boundaries so that every CTA takes
// the same time.
constexpr int kTb2MaxCtas = 512;
// D > 1: the windows of D window rows are interleaved in the flattened
// order (position item / nz): group g of rows gD .. gD + D - 1 (fewer in the
// last group) takes the positions from g T D on, window (wx, gD + l) at
// position g T D + wx * (rows in the group) + l, so that x-neighbours lie D
// positions apart.  The host picks D so that D windows of planes are close to
// a whole number of CTA shares: x-neighbours then start at nearly the same
// plane and march side by side.  D = 1: row by row.
// whole > 0: CTA c first takes the windows c, c + CTAs, ... below whole, from
// plane 0 to nz; the items then are those of the windows from whole on.
struct Tb2Plan {
    int T, U, D, whole;
    unsigned long long* prof;
    int* err;                    // the grid's error word (an expired wait raises it)
    float dt16;                  // dt / 16
    long long start[kTb2MaxCtas + 1];
};

__device__ __forceinline__ int tb2_window_at(const Tb2Plan& tw, int pos)
{
    if (tw.D <= 1) return pos;
    const int grp = pos / (tw.T * tw.D);
    const int rows = tw.U - grp * tw.D < tw.D ? tw.U - grp * tw.D : tw.D;
    const int r = pos - grp * tw.T * tw.D;
    const int wx = r / rows, l = r - wx * rows;
    return (grp * tw.D + l) * tw.T + wx;
}

// Columns per window along x, and the stride between windows.
constexpr int kTb2Wx = 32;
constexpr int kTb2Sx = 24;
constexpr int kTb2Ox = 4;   // first own column of a window
constexpr int kTb2Oy = 2;   // first own row
// Window rows: tile heights (ty) 16 and 8.
constexpr int kTb2Rows = 24;
constexpr int kTb2RowsSmall = 12;

template <int RY>
struct Tb2Smem {
    static constexpr int NT = 16 * RY;   // threads: two columns each
    static constexpr int NC = 32 * RY;   // columns per window
    static constexpr int R = 4;          // ring slots (see tb2_issue)
    static constexpr int SLOT = 8 * NC;  // floats per slot: E^n 3, H^{n-1/2} 3, fluence (float2)
    static constexpr int NP = 8;         // psi values per column and slot (two slots)
    // exchange arrays, and a row's room before the first and after the last
    // (a y neighbour past the window's rows reads there, for halo rows only)
    static constexpr int XS = NC, XO = 32;
    static constexpr int NX = 10;        // 3 H^{n+1/2}, 2x2 E^{n+1}, 3 H^{n+3/2}
    static constexpr size_t bytes()
    {
        return size_t(R) * SLOT * 4 + size_t(2) * NP * NC * 4    // planes, psi
               + (size_t(NX) * XS + 64) * 4                      // exchange arrays
               + size_t(12) * NC * 4                             // antenna coefficients of the columns (6 complex)
               + R * 8 + 128;                                    // mbarriers, alignment
    }
};

// ---- pairs of columns: packed FP32, rounded as the scalar operations.  The
// compiler may contract a packed multiply whose result feeds a packed add or
// subtract (it does so across one side of an unrolled loop and not the
// other, which would make results depend on the work split): no mul2 below
// feeds an add2 or sub2, only the addend of an fma2.
__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

__device__ __forceinline__ void cpa4(float* dst, const float* src, bool valid)
{
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(valid ? 4 : 0)
                 : "memory");
}
// bytes: 8, or 4 (the second element zero-filled), or 0
__device__ __forceinline__ void cpa8(float* dst, const float* src, int bytes)
{
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cpa_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ void cpa_wait0() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// |E x Hbar| of a cell from its centre sums, times dt16 unless CR (the 1/16 of
// the four-edge E means and the two-face, two-time H means is folded into
// dt16).  CR: the roundings of the cell passes, which fuse the product with
// dt16 into the accumulator's add and take the CPML products in the other order
// (runs on the default tile, which mix both kernels); otherwise those of tile
// variant 7.
template <bool CR>
__device__ __forceinline__ float2 tb2_flux(float2 cx, float2 cy, float2 cc, float2 hbx, float2 hby, float2 hbz,
                                           float dt16)
{
    const float2 sx = fma2(cy, hbz, neg2(mul2(cc, hby)));
    const float2 sy = fma2(cc, hbx, neg2(mul2(cx, hbz)));
    const float2 sz = fma2(cx, hby, neg2(mul2(cy, hbx)));
    const float2 s = fma2(sz, sz, fma2(sy, sy, mul2(sx, sx)));
    if (CR) return make_float2(vec_norm(s.x), vec_norm(s.y));
    return make_float2(mul_rn(vec_norm(s.x), dt16), mul_rn(vec_norm(s.y), dt16));
}

__device__ __forceinline__ Cpx<float> cmul(Cpx<float> z, Cpx<float> t)
{
    return Cpx<float>{fma_rn(z.x, t.x, -mul_rn(z.y, t.y)), fma_rn(z.x, t.y, mul_rn(z.y, t.x))};
}

// Stores of the window's outputs with the L2 evict-last priority: a window
// writes 96 bytes of a row, so its first or last 128-byte line is shared with a
// neighbouring window, which writes its part at another time.
__device__ __forceinline__ uint64_t tb2_store_policy()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void st_keep(float* q, float v, uint64_t pol)
{
    asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(q), "f"(v), "l"(pol) : "memory");
}
__device__ __forceinline__ void st_keep(float2* q, float2 v, uint64_t pol)
{
    asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(q), "f"(v.x), "f"(v.y), "l"(pol)
                 : "memory");
}
__device__ __forceinline__ void st_keep(float4* q, float4 v, uint64_t pol)
{
    asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(q), "f"(v.x), "f"(v.y),
                 "f"(v.z), "f"(v.w), "l"(pol)
                 : "memory");
}

// CPML psi update b psi + a d (CR: rounded as the cell passes' psi_next).
template <bool CR>
__device__ __forceinline__ float2 psi2(float2 b, float2 psi, float2 aa, float2 d)
{
    return CR ? fma2(aa, d, mul2(b, psi)) : fma2(b, psi, mul2(aa, d));
}

// Per-window constants of a thread's two columns (i, j), (i + 1, j).
struct Tb2Col {
    int i, j, l, row, at;                 // l: half-warp lane; at: the pair's offset in a window array
    bool own0, own1, f0, f1;              // columns whose fields / fluence the window writes
    bool sx0, sx1, sy;                    // columns in an x shell, row in a y shell
    bool in0, in1;                        // columns inside the box
    bool xpair;                           // nx and npml even: an x shell holds whole pairs at even offsets
    bool ant, anth, ante;                 // the window holds antenna columns; the warp holds H / E points
    int col, colx, coly;
    float2 chx, chy, cex, cey, bhx, ahx, bex, aex, bhy, ahy, bey, aey;
};

// Values carried from plane to plane (planes relative to the current p).
struct Tb2Carry {
    float2 e0[3];                  // E^n(p-1)
    float2 h1p[3];                 // H^{n+1/2}(p-2)
    float2 e1p[3];                 // E^{n+1}(p-2)
    float2 h2px, h2py;             // H^{n+3/2}(p-3), x and y
    // fluence centre sums: step n of plane p-2 (f), step n+1 of plane p-3 (g)
    float2 fPEx, fPEy, fcz, fhbx, fhby, fHsz;
    float2 gPEx, gPEy, gcz, ghbx, ghby, gHsz;
    float2 tn;                     // fluence term of step n, plane p-3
    float2 px[4], py[4];           // psi of plane p-2 after step n: Hyx Hzx Eyx Ezx, Hxy Hzy Exy Ezy
    int kp, kq, kr, k3, ki;        // planes of p, p-1, p-2, p-3 and p+3 (modulo nz; as they are on z-walled grids)
    Cpx<float> zq, zr;             // e^{i beta z} of planes p-1 and p-2
};

template <int RY>
struct Tb2Bufs {
    float* ring;     // [R][SLOT]: E^n, H^{n-1/2} [6][RY][32], fluence [RY][32] (float2)
    float* psi;      // [2][NP][NC]: Hyx Hzx Hxy Hzy Eyx Ezx Exy Ezy
    float* HB;       // [Hx, Hz, Hy^{n-1/2} + Hy^{n+1/2}][XS]
    float* E1B;      // [2][Ez, Ex][XS]: E^{n+1}
    float* H1B;      // [Hx, Hz, Hy^{n+1/2} + Hy^{n+3/2}][XS]
    float* SC;       // [6][re, im][NC]: antenna coefficients (zero where a column has no point of the component)
    uint64_t* bars;  // [R]
    int* err;        // the grid's error word
    uint64_t pol;    // L2 evict-last policy of the stores
};

__device__ __forceinline__ int next_plane(int k, int nz) { return k + 1 == nz ? 0 : k + 1; }
// The plane after k; W: planes past the walls of a z-walled grid are real
// indices (their boxes read as zeros, the wall's values).
template <bool W>
__device__ __forceinline__ int tb2_next(const StepArgs<float>& a, int k)
{
    return W && a.zw ? k + 1 : next_plane(k, a.nz);
}

__device__ __forceinline__ float2 ld2(const float* q) { return *reinterpret_cast<const float2*>(q); }
__device__ __forceinline__ void st2(float* q, float2 v) { *reinterpret_cast<float2*>(q) = v; }

// Box loads of one iteration into ring slot s: E^n and H^{n-1/2} of plane k,
// the fluence of plane kf, at window corner (x, y).  Called by every thread;
// lane 0 of each of the first seven warps issues one box (warps loop where
// there are fewer), lane 0 of warp 0 arms the slot's mbarrier (bytes landing
// before it does keep the phase open: its arrival is the one the phase waits
// for).
template <int RY>
__device__ __forceinline__ void tb2_issue(const StepArgs<float>& a, const TmaMaps& m, const Tb2Bufs<RY>& b, int s,
                                          int k, int kf, int x, int y)
{
    using S = Tb2Smem<RY>;
    if ((threadIdx.x & 31) != 0) return;
    float* dst = b.ring + s * S::SLOT;
    uint64_t* bar = b.bars + s;
    const int nbox = a.fluence ? 7 : 6;
    #pragma unroll 1
    for (int q = threadIdx.x >> 5; q < nbox; q += S::NT / 32) {
        if (q == 0) mbar_expect_tx(bar, uint32_t((a.fluence ? 8 : 6) * S::NC * 4));
        tma_load_3d(dst + q * S::NC, &m.e[0] + q, bar, x, y, q < 6 ? k : kf);
    }
}

// The CPML psi of this thread's shell columns in plane k into psi slot s, one
// cp.async group.
template <int RY, int G, bool W>
__device__ __forceinline__ void tb2_issue_psi(const StepArgs<float>& a, const Tb2Col& c, const Tb2Bufs<RY>& b, int s,
                                              int k)
{
    using S = Tb2Smem<RY>;
    constexpr int NC = S::NC;
    constexpr bool GX = G & 1, GY = G & 2;
    if (!GX && !GY) return;
    const bool in = !(W && a.zw) || (k >= 0 && k < a.nz);   // zeros past a z wall
    if (W && !in) k = 0;
    float* r = b.psi + s * S::NP * NC + c.at;
    if (GX) {   // every lane: zeros where the column is not in an x shell
        const int q = k * a.ny * (2 * a.npml) + c.colx;
        const float* src[4] = {a.phx_in[0], a.phx_in[1], a.pex[0], a.pex[1]};
        constexpr int slot[4] = {0, 1, 4, 5};
        if (c.xpair) {
            #pragma unroll
            for (int v = 0; v < 4; ++v) cpa8(r + slot[v] * NC, src[v] + q, in && c.sx0 ? 8 : 0);
        } else
        #pragma unroll
        for (int v = 0; v < 4; ++v) {
            cpa4(r + slot[v] * NC, src[v] + q, in && c.sx0);
            cpa4(r + slot[v] * NC + 1, src[v] + q + (c.sx1 ? 1 : 0), in && c.sx1);
        }
    }
    if (GY) {
        const int q = k * (2 * a.npml) * a.pitch + c.coly;
        const int bytes = in && c.sy ? (c.in1 ? 8 : (c.in0 ? 4 : 0)) : 0;
        cpa8(r + 2 * NC, a.phy_in[0] + q, bytes);
        cpa8(r + 3 * NC, a.phy_in[1] + q, bytes);
        cpa8(r + 6 * NC, a.pey[0] + q, bytes);
        cpa8(r + 7 * NC, a.pey[1] + q, bytes);
    }
    cpa_commit();
}

// Soft-source increment Re{coef_c u} of component comp (coefficients staged in
// SC; zero, and the increment a signed zero, where the column has no point of
// the component).
template <int RY>
__device__ __forceinline__ float2 tb2_src(const Tb2Bufs<RY>& b, const Tb2Col& c, int comp, Cpx<float> u)
{
    constexpr int NC = Tb2Smem<RY>::NC;
    const float2 re = ld2(b.SC + (2 * comp) * NC + c.at), im = ld2(b.SC + (2 * comp + 1) * NC + c.at);
    return fma2(re, dup2(u.x), neg2(mul2(im, dup2(u.y))));
}

// x-shell psi of the pair stored from values v (offset q of the first column;
// xpair: the pair lies in the shell as a whole, at an even offset).
__device__ __forceinline__ void st_psix(float* p, int q, float2 v, bool w0, bool w1, bool xpair, uint64_t pol)
{
    if (xpair) {
        if (w0) st_keep(reinterpret_cast<float2*>(p + q), v, pol);
        return;
    }
    if (w0) st_keep(p + q, v.x, pol);
    if (w1) st_keep(p + q + 1, v.y, pol);
}

// A pair of row-contiguous values at element q of p (q even).
__device__ __forceinline__ void st_pair(float* p, int q, float2 v, bool w0, bool w1, uint64_t pol)
{
    if (w1) st_keep(reinterpret_cast<float2*>(p + q), v, pol);
    else if (w0) st_keep(p + q, v.x, pol);
}

// z-shell index of plane k, or -1.
__device__ __forceinline__ int tb2_zshell(const StepArgs<float>& a, int k)
{
    if (k < 0 || k >= a.nz) return -1;
    return k < a.npz ? k : (k >= a.nz - a.npz ? k - a.nz + 2 * a.npz : -1);
}

// z-shell psi update of a pair of columns: the value read from array t.
__device__ __forceinline__ float2 tb2_ldz(const float* t, const StepArgs<float>& a, const Tb2Col& c, int kk)
{
    const float* q = t + (long long)kk * (a.pitch * a.ny) + c.col;
    return make_float2(c.in0 ? q[0] : 0.0f, c.in1 ? q[1] : 0.0f);
}

// The wall sheet's E_x increment at the pair's columns.
__device__ __forceinline__ float2 tb2_sheet(const StepArgs<float>& a, const Tb2Col& c, Cpx<float> tw)
{
    const Cpx<float>* t = static_cast<const Cpx<float>*>(a.wcoefr) + c.j * a.nx + c.i;
    const Cpx<float> zero{0.0f, 0.0f}, w0 = c.in0 ? t[0] : zero, w1 = c.in1 ? t[1] : zero;
    return make_float2(fma_rn(w0.x, tw.x, -mul_rn(w0.y, tw.y)), fma_rn(w1.x, tw.x, -mul_rn(w1.y, tw.y)));
}

// One plane p of the wavefront: u = ring slot of plane p, U = (p - P0) mod 2
// gives the exchange-buffer parities at compile time.  Every row runs every
// stage: a row whose results no written column needs computes values that
// reach no output (rows beyond the window read the zero rows of the exchange
// arrays), and the stage code stays free of branches.
// W: 1, the z walls and the wall sheet compiled in; 2, the z CPML too (planes
// of the z shells).  valid: plane p-2's fields are the range's to store; okF:
// plane p-3's fluence.
//
// The walls: E_x and E_y are zero on the planes 0 and nz (plane nz reads as
// zeros; its E^{n+1} is set to zero here), and with that no value of a plane
// below 0 or above nz reaches a stored one.
template <int RY, int U, int G, int W, bool CR, bool FL>
__device__ __forceinline__ void tb2_plane(const StepArgs<float>& a, const TmaMaps& m, const Tb2Times& tt,
                                          const Tb2Col& c, const Tb2Bufs<RY>& b, Tb2Carry& s, bool valid, bool okF,
                                          bool issue_next, bool issue_psi, float dt16, uint32_t gq, int wx0, int wy0, bool& dead)
{
    using S = Tb2Smem<RY>;
    constexpr int NC = S::NC, XS = S::XS;
    constexpr bool GX = G & 1, GY = G & 2;
    const uint32_t SP = gq & 3, SQ = (gq + 3) & 3;                 // ring slots of planes p, p-1
    constexpr int PP = U & 1, PQ = PP ^ 1;                         // exchange parities of planes p, p-1
    // (past the window's edge: the edge column's own value; a column so
    // computed is halo and reaches no column the window writes)
    auto xp = [&](float2 v) {   // value of the +x neighbours
        float w = __shfl_down_sync(0xffffffffu, v.x, 1, 16);
        return make_float2(v.y, w);
    };
    auto xm = [&](float2 v) {   // value of the -x neighbours
        float w = __shfl_up_sync(0xffffffffu, v.y, 1, 16);
        return make_float2(w, v.x);
    };
    // y neighbours from the exchange arrays (past the window's rows: another
    // array's row, for halo rows only)
    auto yp = [&](const float* q) { return ld2(q + S::XO + c.at + 32); };
    auto ym = [&](const float* q) { return ld2(q + S::XO + c.at - 32); };
    auto put = [&](float* q, float2 v) { st2(q + S::XO + c.at, v); };
    // +y neighbour of E^n from the ring
    auto ype = [&](const float* q) { return ld2(q + c.at + 32); };
    const float2 cz = dup2(a.cz);
    // dt / (kappa dz) at the H and E positions of planes p-1 and p-2
    auto czat = [&](const float* t, int k) { return W == 2 ? dup2(t[min(max(k, 0), a.nz - 1)]) : cz; };
    const float2 czh = czat(a.chz, s.kq), cze = czat(a.cez, s.kq), czh1 = czat(a.chz, s.kr), cze1 = czat(a.cez, s.kr);
    const float2 zero2 = make_float2(0.0f, 0.0f);
    const int zsq = W == 2 ? tb2_zshell(a, s.kq) : -1, zsr = W == 2 ? tb2_zshell(a, s.kr) : -1;
    // the z-shell psi: of plane p-1 read ahead of the wait below, updated by
    // step n into this thread's place in shared memory (the antenna's, which
    // z-walled grids do not have), from there by step n+1 one plane later
    float2 ipz[4] = {zero2, zero2, zero2, zero2};
    if (W == 2 && zsq >= 0) {
        ipz[0] = tb2_ldz(a.phz_in[0], a, c, zsq); ipz[1] = tb2_ldz(a.phz_in[1], a, c, zsq);
        ipz[2] = tb2_ldz(a.pez[0], a, c, zsq); ipz[3] = tb2_ldz(a.pez[1], a, c, zsq);
    }
    float* zw = b.SC + PP * 4 * NC + c.at;         // psi of plane p-1 after step n: Hxz Hyz Exz Eyz
    const float* zr = b.SC + PQ * 4 * NC + c.at;   // of plane p-2

    if (!dead && !mbar_wait_bounded(b.bars + SP, (gq >> 2) & 1)) {
        dead = true;
        atomicOr(b.err, 1);
    }
    if (GX || GY) cpa_wait1();                                       // and the last plane's psi
    const float* rp = b.ring + SP * S::SLOT + c.at;
    const float* rq = b.ring + SQ * S::SLOT;
    float* ps = b.psi + PQ * S::NP * NC + c.at;                      // psi of plane p-1
    // e^{i beta z} of plane p, used from the next plane on
    Cpx<float> zn{0.0f, 0.0f};
    if (c.ant) zn = static_cast<const Cpx<float>*>(a.zphr)[s.kp];

    // ---- stage A: H^{n+1/2} of plane q = p-1
    const float2 en0 = ld2(rp), en1 = ld2(rp + NC), en2 = ld2(rp + 2 * NC);   // E^n(p)
    const float2 ex = s.e0[0], ey = s.e0[1], ez = s.e0[2];
    float2 hx, hy, hz, hsy, npx[4], npy[4];
    float2 nPEx, nPEy, ncz, nHsz, nhbx;
    {
        const float2 ox = ld2(rq + 3 * NC + c.at), oy = ld2(rq + 4 * NC + c.at), oz = ld2(rq + 5 * NC + c.at);
        const float2 ezj = ype(rq + 2 * NC), exj = ype(rq);
        const float2 ezi = xp(ez), eyi = xp(ey);
        const float2 dEz_y = sub2(ezj, ez), dEy_z = sub2(en1, ey), dEx_z = sub2(en0, ex);
        const float2 dEz_x = sub2(ezi, ez), dEy_x = sub2(eyi, ey), dEx_y = sub2(exj, ex);
        hx = fma2(czh, dEy_z, fma2(neg2(c.chy), dEz_y, ox));
        hy = fma2(c.chx, dEz_x, fma2(neg2(czh), dEx_z, oy));
        hz = fma2(c.chy, dEx_y, fma2(neg2(c.chx), dEy_x, oz));
        if (GX) {   // every lane (zero coefficients and psi off the x shells)
            npx[0] = psi2<CR>(c.bhx, ld2(ps + 0 * NC), c.ahx, dEz_x);   // Hyx
            npx[1] = psi2<CR>(c.bhx, ld2(ps + 1 * NC), c.ahx, dEy_x);   // Hzx
            hy = add2(hy, npx[0]);
            hz = sub2(hz, npx[1]);
        }
        if (GY) {
            npy[0] = psi2<CR>(c.bhy, ld2(ps + 2 * NC), c.ahy, dEz_y);   // Hxy
            npy[1] = psi2<CR>(c.bhy, ld2(ps + 3 * NC), c.ahy, dEx_y);   // Hzy
            hx = sub2(hx, npy[0]);
            hz = add2(hz, npy[1]);
        }
        if (W == 2 && zsq >= 0) {
            const float2 bz = dup2(a.bhz[zsq]), az = dup2(a.ahz[zsq]);
            const float2 p0 = psi2<CR>(bz, ipz[0], az, dEy_z);   // Hxz
            const float2 p1 = psi2<CR>(bz, ipz[1], az, dEx_z);   // Hyz
            hx = add2(hx, p0);
            hy = sub2(hy, p1);
            st2(zw, p0);
            st2(zw + NC, p1);
        }
        if (c.anth) {   // the whole warp: zero terms where a column has no point
            const Cpx<float> u = cmul(s.zq, tt.th0);
            hx = add2(hx, tb2_src(b, c, 3, u));
            hy = add2(hy, tb2_src(b, c, 4, u));
            hz = add2(hz, tb2_src(b, c, 5, u));
        }
        if constexpr (FL) {   // centre sums of step n for plane q
            nPEx = add2(ex, exj);
            nPEy = add2(ey, eyi);
            ncz = add2(add2(ez, ezi), add2(ezj, xp(ezj)));
            const float2 hsx = add2(ox, hx);
            hsy = add2(oy, hy);
            nHsz = add2(oz, hz);
            nhbx = add2(hsx, xp(hsx));
        }
    }
    put(b.HB, hx);
    put(b.HB + XS, hz);
    if constexpr (FL) put(b.HB + 2 * XS, hsy);
    __syncthreads();   // H^{n+1/2} of plane q is there, and every read of ring slot SQ is done
    // refill: the boxes of the iteration of plane p + 3 into the slot of p - 1
    if (issue_next) tb2_issue<RY>(a, m, b, SQ, s.ki, s.kp, wx0, wy0);

    // ---- stage B: E^{n+1} of plane q
    float2 nex, ney, nez;
    {
        const float2 hyi = xm(hy), hzi = xm(hz);
        const float2 hxj = ym(b.HB), hzj = ym(b.HB + XS);
        const float2 dHz_y = sub2(hz, hzj), dHy_z = sub2(hy, s.h1p[1]), dHx_z = sub2(hx, s.h1p[0]);
        const float2 dHz_x = sub2(hz, hzi), dHy_x = sub2(hy, hyi), dHx_y = sub2(hx, hxj);
        nex = fma2(neg2(cze), dHy_z, fma2(c.cey, dHz_y, ex));
        ney = fma2(neg2(c.cex), dHz_x, fma2(cze, dHx_z, ey));
        nez = fma2(neg2(c.cey), dHx_y, fma2(c.cex, dHy_x, ez));
        if (GX) {   // every lane (zero coefficients and psi off the x shells)
            npx[2] = psi2<CR>(c.bex, ld2(ps + 4 * NC), c.aex, dHz_x);   // Eyx
            npx[3] = psi2<CR>(c.bex, ld2(ps + 5 * NC), c.aex, dHy_x);   // Ezx
            ney = sub2(ney, npx[2]);
            nez = add2(nez, npx[3]);
        }
        if (GY) {
            npy[2] = psi2<CR>(c.bey, ld2(ps + 6 * NC), c.aey, dHz_y);   // Exy
            npy[3] = psi2<CR>(c.bey, ld2(ps + 7 * NC), c.aey, dHx_y);   // Ezy
            nex = add2(nex, npy[2]);
            nez = sub2(nez, npy[3]);
        }
        if (W == 2 && zsq >= 0) {
            const float2 bz = dup2(a.bez[zsq]), az = dup2(a.aez[zsq]);
            const float2 p0 = psi2<CR>(bz, ipz[2], az, dHy_z);   // Exz
            const float2 p1 = psi2<CR>(bz, ipz[3], az, dHx_z);   // Eyz
            nex = sub2(nex, p0);
            ney = add2(ney, p1);
            st2(zw + 2 * NC, p0);
            st2(zw + 3 * NC, p1);
        }
        if (c.ante) {   // the whole warp: zero terms where a column has no point
            const Cpx<float> u = cmul(s.zq, tt.te0);
            nex = add2(nex, tb2_src(b, c, 0, u));
            ney = add2(ney, tb2_src(b, c, 1, u));
            nez = add2(nez, tb2_src(b, c, 2, u));
        }
        if (W && a.wcoefr && s.kq == a.wplane) nex = add2(nex, tb2_sheet(a, c, tt.tw0));
        if (GY && c.j == 0) { nex = zero2; nez = zero2; }   // PEC: tangential E
        if (GX && c.i == 0) { ney.x = 0.0f; nez.x = 0.0f; }
        if (W && a.zw && (s.kq == 0 || s.kq == a.nz)) nex = ney = zero2;
    }
    // the psi of plane p + 1 into the slot of p - 1 (read above)
    if (GX || GY) {
        if (issue_psi) tb2_issue_psi<RY, G, W != 0>(a, c, b, PQ, tb2_next<W != 0>(a, s.kp));
        else cpa_commit();
    }
    // fluence term of step n for plane r = p-2 (sums of planes r and q)
    float2 nhby, tn_new;
    if constexpr (FL) {
        nhby = add2(hsy, yp(b.HB + 2 * XS));
        tn_new = tb2_flux<CR>(add2(s.fPEx, nPEx), add2(s.fPEy, nPEy), s.fcz, s.fhbx, s.fhby, add2(s.fHsz, nHsz), dt16);
    }

    // ---- stage C: H^{n+3/2} of plane r
    float2 h2x, h2y, h2z, gsy;
    float2 mPEx, mPEy, mcz, mHsz, mhbx;
    {
        const float* E1Br = b.E1B + PP * 2 * XS;   // written one plane ago (parity of r = parity of p)
        const float2 fezj = yp(E1Br), fexj = yp(E1Br + XS);
        const float2 fezi = xp(s.e1p[2]), feyi = xp(s.e1p[1]);
        const float2 dEz_y = sub2(fezj, s.e1p[2]), dEy_z = sub2(ney, s.e1p[1]), dEx_z = sub2(nex, s.e1p[0]);
        const float2 dEz_x = sub2(fezi, s.e1p[2]), dEy_x = sub2(feyi, s.e1p[1]), dEx_y = sub2(fexj, s.e1p[0]);
        h2x = fma2(czh1, dEy_z, fma2(neg2(c.chy), dEz_y, s.h1p[0]));
        h2y = fma2(c.chx, dEz_x, fma2(neg2(czh1), dEx_z, s.h1p[1]));
        h2z = fma2(c.chy, dEx_y, fma2(neg2(c.chx), dEy_x, s.h1p[2]));
        if (GX) {   // every lane (zero coefficients and psi off the x shells)
            const float2 p0 = psi2<CR>(c.bhx, s.px[0], c.ahx, dEz_x);
            const float2 p1 = psi2<CR>(c.bhx, s.px[1], c.ahx, dEy_x);
            h2y = add2(h2y, p0);
            h2z = sub2(h2z, p1);
            if (valid && (c.sx0 || c.sx1)) {
                const int qo = s.kr * a.ny * (2 * a.npml) + c.colx;
                const uint64_t pol = b.pol;
                st_psix(a.phx_out[0], qo, p0, c.own0 && c.sx0, c.own1 && c.sx1, c.xpair, pol);
                st_psix(a.phx_out[1], qo, p1, c.own0 && c.sx0, c.own1 && c.sx1, c.xpair, pol);
            }
        }
        if (GY) {
            const float2 p0 = psi2<CR>(c.bhy, s.py[0], c.ahy, dEz_y);
            const float2 p1 = psi2<CR>(c.bhy, s.py[1], c.ahy, dEx_y);
            h2x = sub2(h2x, p0);
            h2z = add2(h2z, p1);
            if (valid && c.sy) {
                const int qo = s.kr * (2 * a.npml) * a.pitch + c.coly;
                const uint64_t pol = b.pol;
                st_pair(a.phy_out[0], qo, p0, c.own0, c.own1, pol);
                st_pair(a.phy_out[1], qo, p1, c.own0, c.own1, pol);
            }
        }
        if (W == 2 && zsr >= 0) {
            const float2 bz = dup2(a.bhz[zsr]), az = dup2(a.ahz[zsr]);
            const float2 p0 = psi2<CR>(bz, ld2(zr), az, dEy_z), p1 = psi2<CR>(bz, ld2(zr + NC), az, dEx_z);
            h2x = add2(h2x, p0);
            h2y = sub2(h2y, p1);
            if (valid) {
                const int qo = zsr * (a.pitch * a.ny) + c.col;
                st_pair(a.phz_out[0], qo, p0, c.own0, c.own1, b.pol);
                st_pair(a.phz_out[1], qo, p1, c.own0, c.own1, b.pol);
            }
        }
        if (c.anth) {   // the whole warp: zero terms where a column has no point
            const Cpx<float> u = cmul(s.zr, tt.th1);
            h2x = add2(h2x, tb2_src(b, c, 3, u));
            h2y = add2(h2y, tb2_src(b, c, 4, u));
            h2z = add2(h2z, tb2_src(b, c, 5, u));
        }
        if constexpr (FL) {   // centre sums of step n+1 for plane r
            mPEx = add2(s.e1p[0], fexj);
            mPEy = add2(s.e1p[1], feyi);
            mcz = add2(add2(s.e1p[2], fezi), add2(fezj, xp(fezj)));
            const float2 gsx = add2(s.h1p[0], h2x);
            gsy = add2(s.h1p[1], h2y);
            mHsz = add2(s.h1p[2], h2z);
            mhbx = add2(gsx, xp(gsx));
        }
    }
    {
        float* E1Bq = b.E1B + PQ * 2 * XS;
        put(E1Bq, nez);
        put(E1Bq + XS, nex);
        put(b.H1B, h2x);
        put(b.H1B + XS, h2z);
        if constexpr (FL) put(b.H1B + 2 * XS, gsy);
    }
    __syncthreads();

    // ---- stage D: E^{n+2} of plane r
    {
        const float2 hyi = xm(h2y), hzi = xm(h2z);
        const float2 hxj = ym(b.H1B), hzj = ym(b.H1B + XS);
        const float2 dHz_y = sub2(h2z, hzj), dHy_z = sub2(h2y, s.h2py), dHx_z = sub2(h2x, s.h2px);
        const float2 dHz_x = sub2(h2z, hzi), dHy_x = sub2(h2y, hyi), dHx_y = sub2(h2x, hxj);
        float2 fx = fma2(neg2(cze1), dHy_z, fma2(c.cey, dHz_y, s.e1p[0]));
        float2 fy = fma2(neg2(c.cex), dHz_x, fma2(cze1, dHx_z, s.e1p[1]));
        float2 fz = fma2(neg2(c.cey), dHx_y, fma2(c.cex, dHy_x, s.e1p[2]));
        if (GX) {   // every lane (zero coefficients and psi off the x shells)
            const float2 p0 = psi2<CR>(c.bex, s.px[2], c.aex, dHz_x);
            const float2 p1 = psi2<CR>(c.bex, s.px[3], c.aex, dHy_x);
            fy = sub2(fy, p0);
            fz = add2(fz, p1);
            if (valid && (c.sx0 || c.sx1)) {
                const int qo = s.kr * a.ny * (2 * a.npml) + c.colx;
                const uint64_t pol = b.pol;
                st_psix(a.pex_out[0], qo, p0, c.own0 && c.sx0, c.own1 && c.sx1, c.xpair, pol);
                st_psix(a.pex_out[1], qo, p1, c.own0 && c.sx0, c.own1 && c.sx1, c.xpair, pol);
            }
        }
        if (GY) {
            const float2 p0 = psi2<CR>(c.bey, s.py[2], c.aey, dHz_y);
            const float2 p1 = psi2<CR>(c.bey, s.py[3], c.aey, dHx_y);
            fx = add2(fx, p0);
            fz = sub2(fz, p1);
            if (valid && c.sy) {
                const int qo = s.kr * (2 * a.npml) * a.pitch + c.coly;
                const uint64_t pol = b.pol;
                st_pair(a.pey_out[0], qo, p0, c.own0, c.own1, pol);
                st_pair(a.pey_out[1], qo, p1, c.own0, c.own1, pol);
            }
        }
        if (W == 2 && zsr >= 0) {
            const float2 bz = dup2(a.bez[zsr]), az = dup2(a.aez[zsr]);
            const float2 p0 = psi2<CR>(bz, ld2(zr + 2 * NC), az, dHy_z), p1 = psi2<CR>(bz, ld2(zr + 3 * NC), az, dHx_z);
            fx = sub2(fx, p0);
            fy = add2(fy, p1);
            if (valid) {
                const int qo = zsr * (a.pitch * a.ny) + c.col;
                st_pair(a.pez_out[0], qo, p0, c.own0, c.own1, b.pol);
                st_pair(a.pez_out[1], qo, p1, c.own0, c.own1, b.pol);
            }
        }
        if (c.ante) {   // the whole warp: zero terms where a column has no point
            const Cpx<float> u = cmul(s.zr, tt.te1);
            fx = add2(fx, tb2_src(b, c, 0, u));
            fy = add2(fy, tb2_src(b, c, 1, u));
            fz = add2(fz, tb2_src(b, c, 2, u));
        }
        if (W && a.wcoefr && s.kr == a.wplane) fx = add2(fx, tb2_sheet(a, c, tt.tw1));
        if (GY && c.j == 0) { fx = zero2; fz = zero2; }
        if (GX && c.i == 0) { fy.x = 0.0f; fz.x = 0.0f; }
        if (W && a.zw && s.kr == 0) fx = fy = zero2;
        if (valid && c.own0) {
            const int g = s.kr * (a.pitch * a.ny) + c.col;
            const uint64_t pol = b.pol;
            const bool w1 = !GX || c.own1;   // off the x faces the window writes whole pairs
            st_pair(a.eout[0], g, fx, true, w1, pol);
            st_pair(a.eout[1], g, fy, true, w1, pol);
            st_pair(a.eout[2], g, fz, true, w1, pol);
            st_pair(a.hout[0], g, h2x, true, w1, pol);
            st_pair(a.hout[1], g, h2y, true, w1, pol);
            st_pair(a.hout[2], g, h2z, true, w1, pol);
        }
    }
    // fluence of plane p-3: the step-n term from the last plane, then step n+1
    float2 mhby;
    if constexpr (FL) {   // every lane computes it (no divergent branch); the fluence cells store it
        mhby = add2(gsy, yp(b.H1B + 2 * XS));
        const float2 t1 = tb2_flux<CR>(add2(s.gPEx, mPEx), add2(s.gPEy, mPEy), s.gcz, s.ghbx, s.ghby, add2(s.gHsz, mHsz),
                                   dt16);
        const float4 f = *reinterpret_cast<const float4*>(b.ring + SP * S::SLOT + 6 * NC + 2 * c.at);
        // FluAcc<float>::add (CR: add_fma), twice
        float2 sum = make_float2(f.x, f.z), comp = make_float2(f.y, f.w);
        #pragma unroll
        for (int n = 0; n < 2; ++n) {
            const float2 v = n == 0 ? s.tn : t1;
            const float2 y = CR ? fma2(v, dup2(dt16), neg2(comp)) : sub2(v, comp);
            const float2 t = add2(sum, y);
            comp = sub2(sub2(t, sum), y);
            sum = t;
        }
        if (okF) {
            float2* F = static_cast<float2*>(a.fluence) + (s.k3 * (a.pitch * a.ny) + c.col);
            const uint64_t pol = b.pol;
            if (GX ? c.f1 : c.f0)
                st_keep(reinterpret_cast<float4*>(F), make_float4(sum.x, comp.x, sum.y, comp.y), pol);
            else if (GX && c.f0) st_keep(F, make_float2(sum.x, comp.x), pol);
        }
    }

    // ---- carry to the next plane
    s.e0[0] = en0; s.e0[1] = en1; s.e0[2] = en2;
    s.h1p[0] = hx; s.h1p[1] = hy; s.h1p[2] = hz;
    s.e1p[0] = nex; s.e1p[1] = ney; s.e1p[2] = nez;
    s.h2px = h2x; s.h2py = h2y;
    if constexpr (FL) {
        s.fPEx = nPEx; s.fPEy = nPEy; s.fcz = ncz; s.fhbx = nhbx; s.fhby = nhby; s.fHsz = nHsz;
        s.gPEx = mPEx; s.gPEy = mPEy; s.gcz = mcz; s.ghbx = mhbx; s.ghby = mhby; s.gHsz = mHsz;
        s.tn = tn_new;
    }
    #pragma unroll
    for (int v = 0; v < 4; ++v) {
        if (GX) s.px[v] = npx[v];
        if (GY) s.py[v] = npy[v];
    }
    s.zr = s.zq; s.zq = zn;
    s.k3 = s.kr; s.kr = s.kq; s.kq = s.kp;
    s.kp = tb2_next<W != 0>(a, s.kp);
    s.ki = tb2_next<W != 0>(a, s.ki);
}

// A plane p whose planes p-1 and p-2 lie off the z shells.
__device__ __forceinline__ bool tb2_plain(const StepArgs<float>& a, const Tb2Carry& s)
{
    return a.npz == 0 || (s.kr >= a.npz && s.kq < a.nz - a.npz);
}

// One window, planes [kb, ke) of its E^{n+2} / H^{n+3/2} output (fluence
// planes [kb-1, ke-1), modulo nz).  gq counts the CTA's iterations: ring slot
// gq mod 4, mbarrier parity (gq / 4) mod 2.
template <int RY, int G, bool W, bool CR, bool FL>
__device__ __forceinline__ void tb2_window(const StepArgs<float>& a, const TmaMaps& m, const Tb2Times& tt,
                                           const Tb2Plan& tw, int window, int kb, int ke, const Tb2Bufs<RY>& b,
                                           uint32_t& gq, bool& dead)
{
    using S = Tb2Smem<RY>;
    constexpr int NC = S::NC;
    constexpr bool GX = G & 1, GY = G & 2;
    Tb2Col c;
    c.l = threadIdx.x & 15; c.row = threadIdx.x >> 4; c.at = c.row * 32 + 2 * c.l;
    const int nx = a.nx, ny = a.ny, nz = a.nz, npml = a.npml, w2 = 2 * npml;
    const int wx = window % tw.T, wy = window / tw.T;
    const int L0 = kTb2Sx * wx - kTb2Ox, M0 = (RY - 4) * wy - kTb2Oy;
    c.i = L0 + 2 * c.l; c.j = M0 + c.row;
    const bool inj = c.j >= 0 && c.j < ny;
    c.in0 = inj && c.i >= 0 && c.i < nx;
    c.in1 = inj && c.i >= 0 && c.i + 1 < nx;
    // E^{n+2} / H^{n+3/2} columns this window writes, and its fluence cells
    // (the same columns, the rows shifted by -1)
    const int xa = kTb2Sx * wx, xb = xa + kTb2Sx < nx ? xa + kTb2Sx : nx;
    const int ya = (RY - 4) * wy, yb = wy == tw.U - 1 ? ny : ya + RY - 4;
    const int fya = wy == 0 ? 0 : ya - 1, fyb = wy == tw.U - 1 ? ny : yb - 1;
    const bool x0 = c.i >= xa && c.i < xb, x1 = c.i >= xa && c.i + 1 < xb;   // xa is even: x1 implies x0
    const bool oy = c.j >= ya && c.j < yb;
    c.own0 = oy && x0;
    c.own1 = oy && x1;
    const bool fy = a.fluence != nullptr && c.j >= fya && c.j < fyb;
    c.f0 = fy && x0;
    c.f1 = fy && x1;
    auto shell = [&](int i) { return npml > 0 && (i < npml || i >= nx - npml); };
    c.xpair = ((nx | npml) & 1) == 0;
    c.sx0 = c.in0 && shell(c.i);
    c.sx1 = c.in1 && shell(c.i + 1);
    c.sy = c.in0 && npml > 0 && (c.j < npml || c.j >= ny - npml);
    auto shx = [&](int i) { return i < npml ? i : i - nx + w2; };
    const int i0 = c.sx0 ? shx(c.i) : 0, i1 = c.sx1 ? shx(c.i + 1) : 0;
    const int jj = c.sy ? (c.j < npml ? c.j : c.j - ny + w2) : 0;
    c.col = c.in0 ? c.j * a.pitch + c.i : 0;
    // x-shell offset of the first column of the pair, such that the second is
    // one on wherever it is in a shell
    c.colx = c.sx0 ? c.j * w2 + i0 : (c.sx1 ? c.j * w2 + i1 - 1 : 0);
    c.coly = c.sy ? jj * a.pitch + c.i : 0;
    // coefficients of a column past the box are zero: its values stay zero
    auto pair = [&](const float* t, bool v0, int q0, bool v1, int q1) {
        return make_float2(v0 ? t[q0] : 0.0f, v1 ? t[q1] : 0.0f);
    };
    c.chx = pair(a.chx, c.in0, c.i, c.in1, c.i + 1);
    c.cex = pair(a.cex, c.in0, c.i, c.in1, c.i + 1);
    c.chy = dup2(c.in0 ? a.chy[c.j] : 0.0f);
    c.cey = dup2(c.in0 ? a.cey[c.j] : 0.0f);
    if (GX) {
        c.bhx = pair(a.bhx, c.sx0, i0, c.sx1, i1); c.ahx = pair(a.ahx, c.sx0, i0, c.sx1, i1);
        c.bex = pair(a.bex, c.sx0, i0, c.sx1, i1); c.aex = pair(a.aex, c.sx0, i0, c.sx1, i1);
    }
    if (GY) {
        c.bhy = dup2(c.sy ? a.bhy[jj] : 0.0f); c.ahy = dup2(c.sy ? a.ahy[jj] : 0.0f);
        c.bey = dup2(c.sy ? a.bey[jj] : 0.0f); c.aey = dup2(c.sy ? a.aey[jj] : 0.0f);
    }
    const uint8_t m0 = (c.in0 && a.smask) ? (a.smask[c.j * nx + c.i] & 0x3f) : uint8_t(0);
    const uint8_t m1 = (c.in1 && a.smask) ? (a.smask[c.j * nx + c.i + 1] & 0x3f) : uint8_t(0);
    c.ant = __syncthreads_or((m0 | m1) != 0) != 0;
    c.anth = __any_sync(0xffffffffu, ((m0 | m1) & 0x38) != 0);
    c.ante = __any_sync(0xffffffffu, ((m0 | m1) & 0x07) != 0);
    if (c.ant) {   // every column of the window, zeros where it has no point of a component
        const Cpx<float>* coef = static_cast<const Cpx<float>*>(a.scoefr);
        const Cpx<float> zero{0.0f, 0.0f};
        for (int q = 0; q < 6; ++q) {
            const Cpx<float>* t = coef + q * nx * ny + c.j * nx + c.i;
            const Cpx<float> v0 = (m0 >> q) & 1 ? t[0] : zero, v1 = (m1 >> q) & 1 ? t[1] : zero;
            st2(b.SC + (2 * q) * NC + c.at, make_float2(v0.x, v1.x));
            st2(b.SC + (2 * q + 1) * NC + c.at, make_float2(v0.y, v1.y));
        }
    }

    const float dt16 = tw.dt16;
    // planes streamed: kb-2 .. ke+1, and one more before the upper z wall,
    // where the range holds the fluence of the last plane too
    const int P0 = kb - 2, P1 = ke + 1 + (W && a.zw && ke == nz ? 1 : 0);
    Tb2Carry s;
    const float2 z2 = dup2(0.0f);
    for (int q = 0; q < 3; ++q) { s.e0[q] = z2; s.h1p[q] = z2; s.e1p[q] = z2; }
    s.h2px = s.h2py = z2;
    s.fPEx = s.fPEy = s.fcz = s.fhbx = s.fhby = s.fHsz = z2;
    s.gPEx = s.gPEy = s.gcz = s.ghbx = s.ghby = s.gHsz = z2;
    s.tn = z2;
    for (int q = 0; q < 4; ++q) { s.px[q] = z2; s.py[q] = z2; }
    s.zq = s.zr = Cpx<float>{0.0f, 0.0f};
    const bool raw = W && a.zw;   // z walls: planes as they are
    s.kp = raw ? P0 : (P0 % nz + nz) % nz;
    s.kq = raw ? P0 - 1 : (s.kp == 0 ? nz - 1 : s.kp - 1);
    s.kr = raw ? P0 - 2 : (s.kq == 0 ? nz - 1 : s.kq - 1);
    s.k3 = raw ? P0 - 3 : (s.kr == 0 ? nz - 1 : s.kr - 1);
    // prologue: the boxes of the iterations of planes P0, P0 + 1, P0 + 2 (their
    // fluence planes P0 - 3, P0 - 2, P0 - 1), the psi of planes P0 - 1 and P0.
    // The first iteration reads E^n and H^{n-1/2} of plane P0 - 1 from the slot
    // before the first: stale values, that (like the zero carry) only reach
    // the recomputed planes below kb.
    const int k1 = tb2_next<W>(a, s.kp), k2 = tb2_next<W>(a, k1);
    tb2_issue<RY>(a, m, b, gq & 3, s.kp, s.k3, L0, M0);
    tb2_issue<RY>(a, m, b, (gq + 1) & 3, k1, s.kr, L0, M0);
    tb2_issue<RY>(a, m, b, (gq + 2) & 3, k2, s.kq, L0, M0);
    if (GX || GY) {
        tb2_issue_psi<RY, G, W>(a, c, b, 1, s.kq);
        tb2_issue_psi<RY, G, W>(a, c, b, 0, s.kp);
    }
    s.ki = tb2_next<W>(a, k2);
    // stores: fields of plane p-2 in [kb, ke), fluence of plane p-3 in
    // [kb-1, ke-1) (modulo nz; on z-walled grids [max(kb-1, 0), ke-1), to nz
    // where ke = nz)
    int p = P0;
    auto valid = [&]() { return p >= kb + 2 && (!W || p < ke + 2); };
    auto okF = [&]() { return p >= kb + 2 && (!raw || p >= 3); };
    // W: planes of the z shells run their code one by one, the others in a loop
    // as lean as the z-periodic kernel's (with a choice per plane inside the
    // loop the body left the instruction cache)
    int u = 0;   // (p - P0) mod 2
    bool more = true;
    while (more) {
        if constexpr (W) {
            if (u == 1 || !tb2_plain(a, s)) {
                if (u == 0)
                    tb2_plane<RY, 0, G, 2, CR, FL>(a, m, tt, c, b, s, valid(), okF(), p + 3 <= P1, p + 2 <= P1, dt16, gq,
                                                  L0, M0, dead);
                else
                    tb2_plane<RY, 1, G, 2, CR, FL>(a, m, tt, c, b, s, valid(), okF(), p + 3 <= P1, p + 2 <= P1, dt16, gq,
                                                  L0, M0, dead);
                u ^= 1;
                ++gq;
                more = ++p <= P1;
                continue;
            }
        }
        #pragma unroll 1
        for (;;) {
            tb2_plane<RY, 0, G, W ? 1 : 0, CR, FL>(a, m, tt, c, b, s, valid(), okF(), p + 3 <= P1, p + 2 <= P1, dt16, gq, L0,
                                           M0, dead);
            ++gq;
            u = 1;
            if (!(more = ++p <= P1)) break;
            if (W && !tb2_plain(a, s)) break;
            tb2_plane<RY, 1, G, W ? 1 : 0, CR, FL>(a, m, tt, c, b, s, valid(), okF(), p + 3 <= P1, p + 2 <= P1, dt16, gq, L0,
                                           M0, dead);
            ++gq;
            u = 0;
            if (!(more = ++p <= P1)) break;
            if (W && !tb2_plain(a, s)) break;
        }
    }
    cpa_wait0();
}

template <int RY, bool W, bool CR, bool FL>
__device__ __forceinline__ void tb2_run(const StepArgs<float>& a, const TmaMaps& m, const Tb2Times& tt,
                                        const Tb2Plan& tw)
{
    using S = Tb2Smem<RY>;
    constexpr int NT = S::NT, NC = S::NC, R = S::R, XS = S::XS;
    extern __shared__ unsigned char tb2_smem_raw[];
    Tb2Bufs<RY> b;
    b.ring = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(tb2_smem_raw) + 127) & ~uintptr_t(127));
    b.psi = b.ring + R * S::SLOT;
    b.HB = b.psi + 2 * S::NP * NC;
    b.E1B = b.HB + 3 * XS;
    b.H1B = b.E1B + 4 * XS;
    b.SC = b.H1B + 3 * XS + 64;
    b.bars = reinterpret_cast<uint64_t*>(b.SC + 12 * NC);
    b.err = tw.err;
    b.pol = tb2_store_policy();
    if (threadIdx.x == 0) {
        for (int q = 0; q < R; ++q) mbar_init(b.bars + q, 1);
        mbar_fence_init();
    }
    __syncthreads();
    uint32_t gq = 0;
    bool dead = false;   // a wait expired: run on without waiting, the error word is raised
    const long long t0 = tw.prof ? clock64() : 0;
    // this CTA's work: its whole windows, then its range of items.  The first
    // thread keeps the place in shared memory: held in registers over the z
    // march it spills there (FL: 145 us per step at 256 x 256 x 128, 104 so).
    __shared__ long long at;     // the next item
    __shared__ int pos, work[3]; // the next whole window; window, kb, ke of this turn
    if (threadIdx.x == 0) {
        pos = blockIdx.x;
        at = tw.start[blockIdx.x];
    }
    for (;;) {
        if (threadIdx.x == 0) {
            if (pos < tw.whole) {
                work[0] = tb2_window_at(tw, pos);
                work[1] = 0;
                work[2] = a.nz;
                pos += gridDim.x;
            } else {
                const long long left = tw.start[blockIdx.x + 1] - at;
                const int kb = int(at % a.nz), n = left < (long long)(a.nz - kb) ? int(left) : a.nz - kb;
                work[0] = n > 0 ? tb2_window_at(tw, tw.whole + int(at / a.nz)) : -1;
                work[1] = kb;
                work[2] = kb + n;
                at += n;
            }
        }
        __syncthreads();
        const int window = work[0], kb = work[1], ke = work[2];
        if (window < 0) break;
        // a window off the x (y) faces and shells runs without the checks of
        // the x (y) walls, psi and columns past the box
        const int wx = window % tw.T, wy = window / tw.T;
        const int L0 = kTb2Sx * wx - kTb2Ox, M0 = (RY - 4) * wy - kTb2Oy;
        const bool gx = wx == 0 || wx == tw.T - 1 || (a.npml > 0 && (L0 < a.npml || L0 + kTb2Wx > a.nx - a.npml));
        const bool gy = wy == 0 || wy == tw.U - 1 || (a.npml > 0 && (M0 < a.npml || M0 + RY > a.ny - a.npml));
        if (!gx && !gy) tb2_window<RY, 0, W, CR, FL>(a, m, tt, tw, window, kb, ke, b, gq, dead);
        else if (!gy) tb2_window<RY, 1, W, CR, FL>(a, m, tt, tw, window, kb, ke, b, gq, dead);
        else if (!gx) tb2_window<RY, 2, W, CR, FL>(a, m, tt, tw, window, kb, ke, b, gq, dead);
        else tb2_window<RY, 3, W, CR, FL>(a, m, tt, tw, window, kb, ke, b, gq, dead);
        __syncthreads();   // the ring and the exchange buffers are reused by the next window
    }
    if (dead) {   // copies may still be in flight: give each slot's last phase one more bounded wait
        for (int q = 0; q < R && q < int(gq); ++q) {
            const uint32_t last = gq - 1 - ((gq - 1 - q) & 3);   // last iteration that used slot q
            mbar_wait_bounded(b.bars + q, (last >> 2) & 1);
        }
    }
    if (tw.prof && threadIdx.x == 0) tw.prof[blockIdx.x] += static_cast<unsigned long long>(clock64() - t0);
}

// Steps n and n+1 with their source time factors as a parameter.  W: grids
// with z walls or a wall sheet (kept apart, so that the z-periodic kernel
// carries none of it).  CR: see tb2_flux.  FL: the fluence terms compiled in;
// z-periodic grids without a fluence accumulator take the kernels without (332
// x 332 x 46 cells 66 us per step with the terms compiled in, 54 without).
template <int RY, bool W, bool CR, bool FL>
__global__ void __launch_bounds__(16 * RY, 1)
yee_tb2(const StepArgs<float> a, const Tb2Times tt, const __grid_constant__ TmaMaps m,
        const __grid_constant__ Tb2Plan tw)
{
    tb2_run<RY, W, CR, FL>(a, m, tt, tw);
}

// The same with the time factors of the two steps read from a device table
// (times[i0] for step n, times[i1] for step n+1): the batched graph replays
// these launches with the table refreshed before each replay.
template <int RY, bool W, bool CR, bool FL>
__global__ void __launch_bounds__(16 * RY, 1)
yee_tb2_t(const StepArgs<float> a, const StepTime<float>* __restrict__ times, int i0, int i1,
          const __grid_constant__ TmaMaps m, const __grid_constant__ Tb2Plan tw)
{
    Tb2Times tt;
    tt.th0 = times[i0].th; tt.te0 = times[i0].te; tt.tw0 = times[i0].tw;
    tt.th1 = times[i1].th; tt.te1 = times[i1].te; tt.tw1 = times[i1].tw;
    tb2_run<RY, W, CR, FL>(a, m, tt, tw);
}

}  // namespace fdtd
