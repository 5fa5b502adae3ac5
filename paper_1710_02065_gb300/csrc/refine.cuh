// refine.cuh -- 2:1 grid coupling kernels of a parent / child level pair (Sec. II.B, Eq. couplingCF,
// Eq. couplingFC), D2Q9, and D3Q19 / D3Q27 (the 3D kernels, templated on the
// lattice, are at the end of the file).
// Below, "coarse" is the parent level of a pair and "fine" its child; nested
// levels apply these kernels pair by pair.
//
// Layout (vertex based, dx_f = dx_c / 2, dt_f = dt_c / 2): the fine patch
// covers the coarse nodes X0..X0+Wc, Y0..Y0+Hc; fine node (i, j) sits at
// (X0 + i/2, Y0 + j/2).  The fine boundary ring is a fixed set of nodes
// rebuilt from coarse data after every fine substep; the first ring of
// covered coarse nodes is rebuilt from fine data after every coarse step;
// deeper covered coarse nodes are fixed and never read.
//
// Exchanged data are pre-collision moments (rho - 1, u, Pi^neq); a receiving
// node is rebuilt in post-collision form feqH(rho, u) + (1 - 1/tau) fneqH(u,
// alpha Pi^neq) with alpha = tau_f / (2 tau_c) coarse -> fine and
// 2 tau_c / tau_f fine -> coarse (leading-order Chapman-Enskog f^neq ~ tau
// dt grad u with dt_f = dt_c / 2).
//
//   k_line_moments  : coarse moments at t = 0 on the four interface lines, extended
//                     by one node past each end (cubic stencils near corners)
//   k_level_step_2d : a substep of the fine level with its coupling: line moments
//                     at t + 1; fine ring from line moments mixed in time
//                     ((1-a) M0 + a M1, a = 1/2 at the fine half step) and
//                     interpolated in space (copy at coincident nodes,
//                     (-1, 9, 9, -1)/16 at mid nodes); covered coarse ring from
//                     the coincident fine node's rho, u and its 3 x 3
//                     full-weighted Pi^neq
#pragma once

#include "rr.cuh"
#include "step.cuh"

namespace rr {

struct RefineGeom {
    int X0, Y0, Wc, Hc;
    int nxc, nyc, nfx, nfy;
    // third axis of a 3D patch (zero / one for D2Q9)
    int Z0, Dc, nzc, nfz;
};

// number of line entries: two horizontal lines of Wc + 3, two vertical of Hc + 3
__host__ __device__ inline int line_count(const RefineGeom &g) { return 2 * (g.Wc + 3) + 2 * (g.Hc + 3); }

__device__ inline void line_coord(const RefineGeom &g, int e, int &x, int &y)
{
    const int nh = g.Wc + 3, nv = g.Hc + 3;
    if (e < nh) { x = g.X0 - 1 + e; y = g.Y0; }
    else if (e < 2 * nh) { x = g.X0 - 1 + (e - nh); y = g.Y0 + g.Hc; }
    else if (e < 2 * nh + nv) { x = g.X0; y = g.Y0 - 1 + (e - 2 * nh); }
    else { x = g.X0 + g.Wc; y = g.Y0 - 1 + (e - 2 * nh - nv); }
}

// entry of a coarse node on a horizontal line (top = 0/1) or vertical line (right = 0/1)
__device__ inline int entry_h(const RefineGeom &g, int x, int top) { return top * (g.Wc + 3) + (x - (g.X0 - 1)); }
__device__ inline int entry_v(const RefineGeom &g, int y, int right)
{
    return 2 * (g.Wc + 3) + right * (g.Hc + 3) + (y - (g.Y0 - 1));
}

// Arithmetic of the coupling runs in the storage format's compute type
// (FP32 for FP32/FP16/BF16 storage, FP64 for FP64); the interface moments
// are kept in FP64 arrays.
template <class S>
using CT = typename StoreC<S>::C;

// Pre-collision moments at node (x, y) of a 2D lattice: pull with periodic
// wrap and halfway bounce-back on mask == 1.  m = (rho - 1, ux, uy, Pxx, Pxy, Pyy).
template <class S>
__device__ void streamed_moments_2d(const S *__restrict__ f, const uint8_t *__restrict__ mask, int nx, int ny,
                                    int x, int y, CT<S> m[6])
{
    using C = CT<S>;
    const int64_t N = (int64_t)nx * ny;
    const int64_t cell = x + (int64_t)nx * y;
    C g[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        int sx = x - D2Q9::cx(i), sy = y - D2Q9::cy(i);
        sx = sx < 0 ? sx + nx : (sx >= nx ? sx - nx : sx);
        sy = sy < 0 ? sy + ny : (sy >= ny ? sy - ny : sy);
        const int64_t src = sx + (int64_t)nx * sy;
        if (mask && i != 0 && (mask[src] & MASK_TYPE) == MASK_SOLID)
            g[i] = Store<S>::ld(f + (int64_t)opp<D2Q9>(i) * N + cell);
        else
            g[i] = Store<S>::ld(f + (int64_t)i * N + src);
    }
    const Mom<C> mo = moments_pairs<D2Q9, C>(g);
    const C rho = C(1) + mo.dr;
    const C ux = mo.jx / rho, uy = mo.jy / rho;
    const Sym2<C> p = pi_neq<C>(mo, mo.dr, rho, ux, uy, C(0), 2);
    m[0] = mo.dr; m[1] = ux; m[2] = uy; m[3] = p.xx; m[4] = p.xy; m[5] = p.yy;
}

// Local (not streamed) moments of the stored populations at (x, y)
template <class S>
__device__ void local_moments_2d(const S *__restrict__ f, int nx, int ny, int x, int y, CT<S> m[6])
{
    using C = CT<S>;
    const int64_t N = (int64_t)nx * ny;
    const int64_t cell = x + (int64_t)nx * y;
    C g[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = Store<S>::ld(f + (int64_t)i * N + cell);
    const Mom<C> mo = moments_pairs<D2Q9, C>(g);
    const C rho = C(1) + mo.dr;
    const C ux = mo.jx / rho, uy = mo.jy / rho;
    const Sym2<C> p = pi_neq<C>(mo, mo.dr, rho, ux, uy, C(0), 2);
    m[0] = mo.dr; m[1] = ux; m[2] = uy; m[3] = p.xx; m[4] = p.xy; m[5] = p.yy;
}

// Store feqH(rho, u) + omega fneqH(u, alpha Pi^neq) at a cell, omega = 1 - 1/tau
// (alpha and omega come from the host in the compute type)
template <class S>
__device__ void store_rebuilt_2d(S *__restrict__ f, int64_t N, int64_t cell, const CT<S> m[6], CT<S> alpha,
                                 CT<S> omega)
{
    using C = CT<S>;
    Coef<C> k{};
    const C rho = C(1) + m[0];
    add_eq<C, 2>(k, C(1), m[0], rho, m[1], m[2], C(0));
    Sym2<C> p;
    p.xx = alpha * m[3]; p.xy = alpha * m[4]; p.yy = alpha * m[5];
    p.zz = p.xz = p.yz = C(0);
    add_neq<C, 2>(k, omega, m[1], m[2], C(0), p);
    const RebuildPre<C> r = rebuild_prep<D2Q9, C>(k);
    Store<S>::st(f + cell, rebuild_rest<D2Q9, C>(k, r));
#pragma unroll
    for (int i = 1; i <= D2Q9::HALF; ++i) {
        C gp, gm;
        rebuild_pair<D2Q9, C>(k, r, i, gp, gm);
        Store<S>::st(f + (int64_t)i * N + cell, gp);
        Store<S>::st(f + (int64_t)(i + D2Q9::HALF) * N + cell, gm);
    }
}

// Local moments of the stored coarse field on the interface lines (t = 0)
template <class S>
__global__ void k_line_moments(RefineGeom g, const S *__restrict__ fc, CT<S> *__restrict__ M)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= line_count(g)) return;
    int x, y;
    line_coord(g, e, x, y);
    CT<S> m[6];
    local_moments_2d<S>(fc, g.nxc, g.nyc, x, y, m);
#pragma unroll
    for (int k = 0; k < 6; ++k) M[6 * e + k] = m[k];
}

// One substep of a refined 2D level in one launch: the level's own update and,
// beside it, the coupling with its parent that the substep needs.  Blocks take
// one of four roles by index (the coupling roles first: their chains of loads
// are the longest of the launch):
//   line     (first substep) the parent-side interface moments at t + 1, kept
//            as the next step's moments at t
//   ring     the level's ring in the field written, at t + a (a = 1/2, then 1):
//            line moments mixed in time and interpolated in space.  The first
//            substep pulls the moments at t + 1 from the parent's pre-step
//            field itself (the line role stores them in the same launch); the
//            second reads the stored ones.  Four lanes per ring node, one per
//            stencil point.
//   restrict (second substep) the parent's covered ring from the level's
//            field at t + 1/2, the field this substep's update reads: 16 lanes
//            per node, one per point of the 3 x 3 filter
//   update   one thread per cell of the level (update_cell), ring cells fixed
// None of the roles reads what another writes: ring and restrict write cells
// that the updates of the two levels leave alone.
// The coupling is latency-bound (a few thousand nodes).  As launches of its
// own (line 2.2, ring 2 x 2.9, restrict 15.3 us with one thread per node and
// its 81 loads in a chain, between two updates of 4.4 us), a coarse step of the
// 800 x 400 + 641 x 321 cylinder took 35 us; with these two launches of 4.7 us
// beside the level-0 update it takes 13 us (GB300, FP32).
struct LevelStep2D {
    RefineGeom g;
    int nline, nring, nrestrict;  // blocks of each role
    const void *parent_old;       // parent field at t (pre-step)
    void *parent_new;             // parent field at t + 1 (covered ring written)
    const uint8_t *parent_links, *level_links;  // masks with solids, or null
    const void *M0;
    void *M1;
    double a;                     // time of the ring in the parent step
    int first;                    // first substep: moments at t + 1 are pulled, and stored by the line role
    double alpha_down, omega_down, alpha_up, omega_up;
};

// Ring node t of an nfx x nfy level
__device__ inline void ring_coord(int nfx, int nfy, int t, int &i, int &j)
{
    if (t < nfx) { i = t; j = 0; }
    else if (t < 2 * nfx) { i = t - nfx; j = nfy - 1; }
    else if (t < 2 * nfx + nfy - 2) { i = 0; j = 1 + t - 2 * nfx; }
    else { i = nfx - 1; j = 1 + t - 2 * nfx - (nfy - 2); }
}
__host__ __device__ inline int ring_count(int nfx, int nfy) { return 2 * nfx + 2 * (nfy - 2); }

constexpr int kLevelBlock = 128;  // default threads per block (lbm_set_launch)

template <class S>
__device__ __forceinline__ void level_line(const LevelStep2D &q, int e)
{
    using C = CT<S>;
    if (e >= line_count(q.g)) return;
    int x, y;
    line_coord(q.g, e, x, y);
    C m[6];
    streamed_moments_2d<S>((const S *)q.parent_old, q.parent_links, q.g.nxc, q.g.nyc, x, y, m);
#pragma unroll
    for (int k = 0; k < 6; ++k) ((C *)q.M1)[6 * e + k] = m[k];
}

template <class S>
__device__ __forceinline__ void level_ring(const LevelStep2D &q, int lane_id, S *ff)
{
    using C = CT<S>;
    const RefineGeom &g = q.g;
    const int t = lane_id >> 2, r = lane_id & 3;
    const bool node = t < ring_count(g.nfx, g.nfy);  // other lanes still join the shuffles
    int i = 0, j = 0;
    if (node) ring_coord(g.nfx, g.nfy, t, i, j);
    const bool on_h = j == 0 || j == g.nfy - 1;
    const int c = on_h ? i : j;           // fine coordinate along the line
    const int side = on_h ? (j != 0) : (i != 0);
    const bool odd = c & 1;
    // lane r: stencil point (c - 1)/2 - 1 + r of an odd node; the coincident
    // parent node (lane 0) of an even one
    const int k = odd ? (c - 1) / 2 - 1 + r : c / 2;
    C m[6];
#pragma unroll
    for (int s = 0; s < 6; ++s) m[s] = C(0);
    if (node && (odd || r == 0)) {
        const int e = on_h ? entry_h(g, g.X0 + k, side) : entry_v(g, g.Y0 + k, side);
        C m1[6];
        if (q.first) {
            const int x = on_h ? g.X0 + k : g.X0 + side * g.Wc, y = on_h ? g.Y0 + side * g.Hc : g.Y0 + k;
            streamed_moments_2d<S>((const S *)q.parent_old, q.parent_links, g.nxc, g.nyc, x, y, m1);
        } else {
#pragma unroll
            for (int s = 0; s < 6; ++s) m1[s] = ((const C *)q.M1)[6 * e + s];
        }
        const C a = C(q.a);
#pragma unroll
        for (int s = 0; s < 6; ++s) m[s] = (C(1) - a) * ((const C *)q.M0)[6 * e + s] + a * m1[s];
    }
    C v[6];
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        const C t1 = __shfl_down_sync(0xffffffffu, m[s], 1), t2 = __shfl_down_sync(0xffffffffu, m[s], 2),
                t3 = __shfl_down_sync(0xffffffffu, m[s], 3);
        v[s] = odd ? (-m[s] + C(9) * t1 + C(9) * t2 - t3) * C(0.0625) : m[s];
    }
    if (node && r == 0)
        store_rebuilt_2d<S>(ff, (int64_t)g.nfx * g.nfy, i + (int64_t)g.nfx * j, v, C(q.alpha_down), C(q.omega_down));
}

template <class S>
__device__ __forceinline__ void level_restrict(const LevelStep2D &q, int lane_id, const S *ff_prev)
{
    using C = CT<S>;
    const RefineGeom &g = q.g;
    const int w = g.Wc - 1, h = g.Hc - 1;  // ring of the rectangle [X0+1, X0+Wc-1] x [Y0+1, Y0+Hc-1]
    const int t = lane_id >> 4, l = lane_id & 15;
    const bool node = t < ring_count(w, h);  // other lanes still join the shuffles
    int a = 0, b = 0;
    if (node) ring_coord(w, h, t, a, b);
    const int x = g.X0 + 1 + a, y = g.Y0 + 1 + b;
    C m[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) m[k] = C(0);
    if (node && l < 9)
        streamed_moments_2d<S>(ff_prev, q.level_links, g.nfx, g.nfy, 2 * (x - g.X0) + l % 3 - 1,
                               2 * (y - g.Y0) + l / 3 - 1, m);
    C mc[6] = {C(0), C(0), C(0), C(0), C(0), C(0)};
#pragma unroll
    for (int k = 0; k < 3; ++k) mc[k] = __shfl_sync(0xffffffffu, m[k], 4, 16);
#pragma unroll
    for (int s = 0; s < 9; ++s) {
        const C wt = C((s % 3 == 1 ? 2 : 1) * (s / 3 == 1 ? 2 : 1)) * C(0.0625);
#pragma unroll
        for (int k = 3; k < 6; ++k) mc[k] += wt * __shfl_sync(0xffffffffu, m[k], s, 16);
    }
    if (node && l == 0)
        store_rebuilt_2d<S>((S *)q.parent_new, (int64_t)g.nxc * g.nyc, x + (int64_t)g.nxc * y, mc, C(q.alpha_up),
                            C(q.omega_up));
}

template <class S, int MASK>
__global__ void __launch_bounds__(256)
    k_level_step_2d(const __grid_constant__ StepParams p, const __grid_constant__ LevelStep2D q)
{
    using C = CT<S>;
    int b = blockIdx.x;
    const int tid = threadIdx.x, nt = blockDim.x;
    if (b < q.nline) return level_line<S>(q, b * nt + tid);
    b -= q.nline;
    if (b < q.nring) return level_ring<S>(q, b * nt + tid, (S *)p.out[0]);
    b -= q.nring;
    if (b < q.nrestrict) return level_restrict<S>(q, b * nt + tid, (const S *)p.in[0]);
    b -= q.nrestrict;
    const unsigned t = (unsigned)b * nt + tid;
    if (t >= (unsigned)p.ncell) return;
    const unsigned nx = p.n[0], y = t / nx;
    update_cell<D2Q9, S, C, false, MASK>(p, p.in, p.out, (int)(t - y * nx), (int)y, 0);
}

// Launch one substep of a refined 2D level (fin read, fout written; block: a multiple of 32 up to 256)
template <class S>
cudaError_t launch_level_step_2d(const StepParams &p, const LevelStep2D &q0, const void *fin, void *fout, int block,
                                 cudaStream_t st)
{
    StepParams s = p;
    set_bases<D2Q9, S>(s, fin, fout);
    LevelStep2D q = q0;
    auto blocks = [block](int64_t threads) { return (int)((threads + block - 1) / block); };
    q.nline = q.first ? blocks(line_count(q.g)) : 0;
    q.nring = blocks(4 * (int64_t)ring_count(q.g.nfx, q.g.nfy));
    q.nrestrict = q.first ? 0 : blocks(16 * (int64_t)ring_count(q.g.Wc - 1, q.g.Hc - 1));
    const unsigned grid = (unsigned)(q.nline + q.nring + q.nrestrict + blocks(p.ncell));
    if (p.any_solid)
        k_level_step_2d<S, kMaskLinks><<<grid, block, 0, st>>>(s, q);
    else
        k_level_step_2d<S, kMaskSkip><<<grid, block, 0, st>>>(s, q);
    return cudaGetLastError();
}

// ===========================================================================
// D3Q19 and D3Q27 patches.  The fine patch covers the coarse nodes X0..X0+Wc,
// Y0..Y0+Hc, Z0..Z0+Dc; fine node (i, j, k) sits at (X0 + i/2, Y0 + j/2,
// Z0 + k/2).  The fine boundary shell is rebuilt from coarse data, the first
// shell of covered coarse nodes from fine data.  Interface moments m = (rho -
// 1, ux, uy, uz, Pxx, Pxy, Pxz, Pyy, Pyz, Pzz) of the coarse nodes on the six
// face planes of the patch box (extended by one node past every edge) are
// kept in a dense box array over [X0-1, X0+Wc+1] x [Y0-1, Y0+Hc+1] x
// [Z0-1, Z0+Dc+1] (10 values of the compute type per node; off-plane entries
// unused).
//   k_plane_moments3 : coarse moments on the six planes
//   k_fill_shell3    : fine shell from plane moments mixed in time and
//                      interpolated along every axis on which the fine node is
//                      odd by (-1, 9, 9, -1)/16 (tensor product on the planes)
//   k_restrict3      : covered coarse shell from the coincident fine node's
//                      rho, u and its (1,2,1)^3 / 64 full-weighted Pi^neq
// ===========================================================================
__host__ __device__ inline int64_t box3_entries(const RefineGeom &g)
{
    return (int64_t)(g.Wc + 3) * (g.Hc + 3) * (g.Dc + 3);
}
__device__ inline int64_t box3_index(const RefineGeom &g, int x, int y, int z)
{
    return (x - g.X0 + 1) + (int64_t)(g.Wc + 3) * ((y - g.Y0 + 1) + (int64_t)(g.Hc + 3) * (z - g.Z0 + 1));
}
// number of plane entries (edge nodes shared by two planes are listed twice)
__host__ __device__ inline int plane3_count(const RefineGeom &g)
{
    return 2 * (g.Hc + 3) * (g.Dc + 3) + 2 * (g.Wc + 3) * (g.Dc + 3) + 2 * (g.Wc + 3) * (g.Hc + 3);
}
__device__ inline void plane3_coord(const RefineGeom &g, int t, int &x, int &y, int &z)
{
    const int A = (g.Hc + 3) * (g.Dc + 3), B = (g.Wc + 3) * (g.Dc + 3);
    if (t < 2 * A) {
        const int side = t / A, r = t - side * A;
        x = g.X0 + side * g.Wc; y = g.Y0 - 1 + r % (g.Hc + 3); z = g.Z0 - 1 + r / (g.Hc + 3);
    } else if (t < 2 * A + 2 * B) {
        t -= 2 * A;
        const int side = t / B, r = t - side * B;
        y = g.Y0 + side * g.Hc; x = g.X0 - 1 + r % (g.Wc + 3); z = g.Z0 - 1 + r / (g.Wc + 3);
    } else {
        t -= 2 * A + 2 * B;
        const int Cn = (g.Wc + 3) * (g.Hc + 3);
        const int side = t / Cn, r = t - side * Cn;
        z = g.Z0 + side * g.Dc; x = g.X0 - 1 + r % (g.Wc + 3); y = g.Y0 - 1 + r / (g.Wc + 3);
    }
}

template <class C>
__device__ inline void pack_moments3(const Mom<C> &mo, C m[10])
{
    const C rho = C(1) + mo.dr;
    const C ux = mo.jx / rho, uy = mo.jy / rho, uz = mo.jz / rho;
    const Sym2<C> p = pi_neq<C>(mo, mo.dr, rho, ux, uy, uz, 3);
    m[0] = mo.dr; m[1] = ux; m[2] = uy; m[3] = uz;
    m[4] = p.xx; m[5] = p.xy; m[6] = p.xz; m[7] = p.yy; m[8] = p.yz; m[9] = p.zz;
}

// Pre-collision moments at (x, y, z) of a 3D lattice: pull with periodic
// wrap and halfway bounce-back on mask == 1.
template <class L, class S>
__device__ void streamed_moments_3d(const S *__restrict__ f, const uint8_t *__restrict__ mask, int nx, int ny,
                                    int nz, int x, int y, int z, CT<S> m[10])
{
    using C = CT<S>;
    const int64_t N = (int64_t)nx * ny * nz;
    const int64_t cell = x + (int64_t)nx * (y + (int64_t)ny * z);
    C g[L::Q];
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        int sx = x - L::cx(i), sy = y - L::cy(i), sz = z - L::cz(i);
        sx = sx < 0 ? sx + nx : (sx >= nx ? sx - nx : sx);
        sy = sy < 0 ? sy + ny : (sy >= ny ? sy - ny : sy);
        sz = sz < 0 ? sz + nz : (sz >= nz ? sz - nz : sz);
        const int64_t src = sx + (int64_t)nx * (sy + (int64_t)ny * sz);
        if (mask && i != 0 && (mask[src] & MASK_TYPE) == MASK_SOLID)
            g[i] = Store<S>::ld(f + (int64_t)opp<L>(i) * N + cell);
        else
            g[i] = Store<S>::ld(f + (int64_t)i * N + src);
    }
    pack_moments3<C>(moments_pairs<L, C>(g), m);
}

template <class L, class S>
__device__ void local_moments_3d(const S *__restrict__ f, int64_t N, int64_t cell, CT<S> m[10])
{
    using C = CT<S>;
    C g[L::Q];
#pragma unroll
    for (int i = 0; i < L::Q; ++i) g[i] = Store<S>::ld(f + (int64_t)i * N + cell);
    pack_moments3<C>(moments_pairs<L, C>(g), m);
}

// Store feqH(rho, u) + omega fneqH(u, alpha Pi^neq) at a cell, omega = 1 - 1/tau
// (alpha and omega come from the host in the compute type: no FP64
// arithmetic on the device)
template <class L, class S>
__device__ void store_rebuilt_3d(S *__restrict__ f, int64_t N, int64_t cell, const CT<S> m[10], CT<S> alpha,
                                 CT<S> omega)
{
    using C = CT<S>;
    Coef<C> k{};
    const C rho = C(1) + m[0];
    add_eq<C, 3, true, full_third_order<L>()>(k, C(1), m[0], rho, m[1], m[2], m[3]);
    Sym2<C> p;
    p.xx = alpha * m[4]; p.xy = alpha * m[5]; p.xz = alpha * m[6];
    p.yy = alpha * m[7]; p.yz = alpha * m[8]; p.zz = alpha * m[9];
    add_neq<C, 3, true, full_third_order<L>()>(k, omega, m[1], m[2], m[3], p);
    const RebuildPre<C> r = rebuild_prep<L, C>(k);
    Store<S>::st(f + cell, rebuild_rest<L, C>(k, r));
#pragma unroll
    for (int i = 1; i <= L::HALF; ++i) {
        C gp, gm;
        rebuild_pair<L, C>(k, r, i, gp, gm);
        Store<S>::st(f + (int64_t)i * N + cell, gp);
        Store<S>::st(f + (int64_t)(i + L::HALF) * N + cell, gm);
    }
}

// Interface moments of the coarse plane nodes, stored in the compute type
// (10 per node: rho - 1, u, Pi^neq)
template <class L, class S>
__global__ void k_plane_moments3(RefineGeom g, const S *__restrict__ fc, const uint8_t *__restrict__ mask,
                                 int streamed, CT<S> *__restrict__ M)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= plane3_count(g)) return;
    int x, y, z;
    plane3_coord(g, t, x, y, z);
    CT<S> m[10];
    if (streamed)
        streamed_moments_3d<L, S>(fc, mask, g.nxc, g.nyc, g.nzc, x, y, z, m);
    else
        local_moments_3d<L, S>(fc, (int64_t)g.nxc * g.nyc * g.nzc, x + (int64_t)g.nxc * (y + (int64_t)g.nyc * z), m);
    const int64_t b = box3_index(g, x, y, z);
#pragma unroll
    for (int k = 0; k < 10; ++k) M[10 * b + k] = m[k];
}

// Point q of the 1D stencil of fine coordinate c on an axis with coarse
// origin o: the coincident node (even c, q = 0), or the centred cubic
// (-1, 9, 9, -1) / 16 between o + (c-1)/2 and o + (c+1)/2 (odd c, q = 0..3).
// No index arrays: a runtime index into a per-thread array would go through
// local memory.
template <class C>
__device__ inline void stencil_point(int c, int o, int q, int &idx, C &w)
{
    if ((c & 1) == 0) {
        idx = o + c / 2;
        w = C(1);
    } else {
        idx = o + (c - 1) / 2 - 1 + q;
        w = (q == 0 || q == 3) ? C(-0.0625) : C(0.5625);
    }
}

__host__ __device__ inline int shell3_count(int nx, int ny, int nz)
{
    return nx * ny * nz - (nx - 2) * (ny - 2) * (nz - 2);
}
// node t of the boundary shell of an nx x ny x nz box
__device__ inline void shell3_coord(int nx, int ny, int nz, int t, int &i, int &j, int &k)
{
    const int A = nx * ny, B = nx * (nz - 2);
    if (t < 2 * A) {
        const int side = t / A, r = t - side * A;
        k = side ? nz - 1 : 0; i = r % nx; j = r / nx;
    } else if (t < 2 * A + 2 * B) {
        t -= 2 * A;
        const int side = t / B, r = t - side * B;
        j = side ? ny - 1 : 0; i = r % nx; k = 1 + r / nx;
    } else {
        t -= 2 * A + 2 * B;
        const int Cn = (ny - 2) * (nz - 2);
        const int side = t / Cn, r = t - side * Cn;
        i = side ? nx - 1 : 0; j = 1 + r % (ny - 2); k = 1 + r / (ny - 2);
    }
}

// Fine shell node values at t + a (Sec. II.B, coarse to fine): the coarse
// plane moments interpolated linearly in time and by the tensor cubic in
// space, f^neq rescaled by alpha, rebuilt.  A shell node's stencil has 1, 4
// or 16 coarse points.  Four lanes take one node (lane r its points r, r + 4,
// r + 8, r + 12), the weighted moments are summed over the four by shuffles,
// and the node's first lane rebuilds and stores it: the loads are spread
// over more threads than one per node, while the rebuild is still shared by
// eight nodes per warp.
template <class L, class S>
__global__ void __launch_bounds__(256) k_fill_shell3(RefineGeom g, const CT<S> *__restrict__ M0,
                                                     const CT<S> *__restrict__ M1, CT<S> a, CT<S> alpha,
                                                     CT<S> omega, S *__restrict__ ff)
{
    using C = CT<S>;
    const int count = shell3_count(g.nfx, g.nfy, g.nfz);
    // block-strided over the nodes (every thread of a block takes the same
    // number of turns), so that a grid smaller than the work can leave room
    // on the SMs for a kernel running beside it
    for (int64_t b0 = blockIdx.x * (int64_t)blockDim.x; b0 < 4 * (int64_t)count;
         b0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t gt = b0 + threadIdx.x;
        const int t = (int)(gt >> 2), r = (int)(gt & 3);
        const bool node = t < count;  // lanes past the last node still join the shuffles
        int i = 0, j = 0, k = 0;
        if (node) shell3_coord(g.nfx, g.nfy, g.nfz, t, i, j, k);
        // per axis: 1 point (even fine coordinate) or 4 (odd); lx = log2 of the count
        const int lx = (i & 1) << 1, ly = (j & 1) << 1, lz = (k & 1) << 1;
        const int npts = node ? 1 << (lx + ly + lz) : 0;
        const C am = a, bm = C(1) - a;
        C m[10];
#pragma unroll
        for (int e = 0; e < 10; ++e) m[e] = C(0);
#pragma unroll
        for (int s4 = 0; s4 < 4; ++s4) {
            const int q = r + 4 * s4;  // stencil point (qx, qy, qz) of the node's stencil
            if (q < npts) {
                const int qx = q & ((1 << lx) - 1), qy = (q >> lx) & ((1 << ly) - 1), qz = q >> (lx + ly);
                int cx, cy, cz;
                C wx, wy, wz;
                stencil_point<C>(i, g.X0, qx, cx, wx);
                stencil_point<C>(j, g.Y0, qy, cy, wy);
                stencil_point<C>(k, g.Z0, qz, cz, wz);
                const int64_t e0 = 10 * box3_index(g, cx, cy, cz);
                const C wt = wx * wy * wz;
                if (a == C(1)) {  // at t + 1 the moments at t do not enter (uniform: a kernel argument)
#pragma unroll
                    for (int e = 0; e < 10; ++e) m[e] = fmac(wt, M1[e0 + e], m[e]);
                } else {
#pragma unroll
                    for (int e = 0; e < 10; ++e) m[e] = fmac(wt, bm * M0[e0 + e] + am * M1[e0 + e], m[e]);
                }
            }
        }
#pragma unroll
        for (int o = 2; o > 0; o >>= 1) {
#pragma unroll
            for (int e = 0; e < 10; ++e) m[e] += __shfl_xor_sync(0xffffffffu, m[e], o);
        }
        if (node && r == 0)
            store_rebuilt_3d<L, S>(ff, (int64_t)g.nfx * g.nfy * g.nfz, i + (int64_t)g.nfx * (j + (int64_t)g.nfy * k), m,
                                alpha, omega);
    }
}

// Covered coarse shell (Sec. II.B, fine to coarse): rho, u of the coincident
// fine node and the (1,2,1)^3 / 64 filtered Pi^neq of its 27 neighbours,
// rescaled by alpha, rebuilt.  One warp per coarse node: lane l < 27 pulls
// the streamed moments of stencil point l, the filtered sum is taken by
// shuffles, and the centre lane (13) supplies rho and u.
template <class L, class S>
__global__ void __launch_bounds__(256) k_restrict3(RefineGeom g, const S *__restrict__ ff_prev,
                                                   const uint8_t *__restrict__ fmask, CT<S> alpha, CT<S> omega,
                                                   S *__restrict__ fc)
{
    using C = CT<S>;
    const int w = g.Wc - 1, h = g.Hc - 1, d = g.Dc - 1;  // shell of [X0+1, X0+Wc-1] x ...
    const int count = shell3_count(w, h, d);
    // block-strided over the nodes, as k_fill_shell3
    for (int64_t b0 = blockIdx.x * (int64_t)blockDim.x; b0 < 32 * (int64_t)count;
         b0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t gt = b0 + threadIdx.x;
        const int t = (int)(gt >> 5), l = (int)(gt & 31);
        const bool node = t < count;  // lanes past the last node still join the shuffles
        int a = 0, b = 0, c = 0;
        if (node) shell3_coord(w, h, d, t, a, b, c);
        const int x = g.X0 + 1 + a, y = g.Y0 + 1 + b, z = g.Z0 + 1 + c;
        const int i = 2 * (x - g.X0), j = 2 * (y - g.Y0), k = 2 * (z - g.Z0);
        C m[10];
#pragma unroll
        for (int e = 0; e < 10; ++e) m[e] = C(0);
        if (node && l < 27) {
            const int p = l % 3 - 1, q = (l / 3) % 3 - 1, r = l / 9 - 1;
            streamed_moments_3d<L, S>(ff_prev, fmask, g.nfx, g.nfy, g.nfz, i + p, j + q, k + r, m);
            const C wt = C((p ? 1 : 2) * (q ? 1 : 2) * (r ? 1 : 2)) * C(1.0 / 64.0);
#pragma unroll
            for (int e = 4; e < 10; ++e) m[e] *= wt;
        }
        C mc[10];
#pragma unroll
        for (int e = 0; e < 4; ++e) mc[e] = __shfl_sync(0xffffffffu, m[e], 13);
#pragma unroll
        for (int e = 4; e < 10; ++e) {
            C v = m[e];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            mc[e] = v;
        }
        if (node && l == 0)
            store_rebuilt_3d<L, S>(fc, (int64_t)g.nxc * g.nyc * g.nzc, x + (int64_t)g.nxc * (y + (int64_t)g.nyc * z), mc,
                                alpha, omega);
    }
}

}  // namespace rr
