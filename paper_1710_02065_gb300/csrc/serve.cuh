// serve.cuh -- batched multi-domain update for the serving engine.
//
// Many independent lattices advance in one launch: a tile list enumerates
// warp work items (domain, row, first cell); a persistent grid strides over
// them and every lane updates its cells with the device functions of the
// single-lattice kernels (update_cell one cell per lane; two cells per lane
// the vector loads, collision and stores of step_vec.cuh on rows that wrap
// around), so a domain's arithmetic does not depend on what it is batched
// with.  A launch holds the domains of one lattice, storage format, cells per
// lane and streaming pattern.  Each domain has its own parameters and buffers
// (two lattices, or one with the in-place AA pattern); which of them a step
// reads, and whether the domain still runs, follows from the step's number s
// within the round, the domain's lattice at the round's start (cur) and its
// remaining steps, so the steps of a round need no bookkeeping between them;
// k_batch_advance does it once at the end of the round.
#pragma once

#include <algorithm>

#include "step_vec.cuh"

namespace rr {

struct BatchDomain {
    char *f[2];        // the two lattices (the same lattice twice for AA)
    int nx, ny, nz;
    unsigned dstride;  // bytes from one direction's array to the next (two cells per lane: < 2 GB in all)
    double omega;      // 1 - 1/tau
    int64_t remaining; // steps left at the start of the round
    int cur;           // at the start of the round; pull: the lattice holding the state; AA: 1 after a gather-push step
    int pad;
    StepParams p;
    char *base[2][kMaxQ];  // per-direction base addresses of the two lattices
};

// Work item of one warp: 32 V consecutive cells, from x0, of one row of one domain.
struct BatchTile {
    int domain;
    int y, z;
    int x0;
};

// Resident 256-thread blocks per SM asked of the compiler: as the
// single-lattice kernel, 16-bit storage with two cells per lane is latency-
// bound and gets 64 registers (32 resident warps per SM) on D2Q9 / D3Q19, 80
// for the in-place steps of D3Q19, whose two step types spill 180 bytes at 64;
// the other groups keep the registers they need.
template <class L, class S, int V, bool AA>
struct BatchMinBlocks {
    static constexpr int value = (sizeof(S) == 2 && V == 2 && L::Q <= 19) ? (AA && L::Q == 19 ? 3 : 4) : 0;
};

// Warps per SM that a group's persistent grid asks for: 32, as many as can be
// resident, unless more rows at a time cost more in the caches than their
// latency hides.  GB300, G cell updates/s, two cells per lane, by warps per SM:
//   D3Q19 FP32 pull, 8 x 128^3 32 40.2, 24 40.4, 20 40.5, 16 41.1, 14 42.8, 12 44.6,
//     10 41.3; rows that fill their last tile in part are best with as many
//     cells at a time: 160^3 (0.83 full) 32 37.4, 16 41.1, 14 41.7, 12 39.6, 8 x 96^3
//     (0.75 full) 32 38.8, 16 42.5, 12 38.2.  A group within twice the L2's bytes
//     does not gain: 4 x 64^3 (159 MB) 32 43.8, 12 39.9, 1 x 128^3 (319 MB) 38.5, 41.6.
//   D3Q19 FP16 in place (80 registers), a batch of 60^3 to 128^3 32 56.5, 24 64.4,
//     20 62.8, 16 58.8 (at 64 registers 55.9 to 58.1, at 100 60.8).
// cells, tiles: of the group's domains; its lattices' bytes are elem 2 Q cells.
inline int batch_warps_per_sm(bool d3q19, size_t elem, int v, bool aa, int64_t cells, int64_t tiles, int64_t l2_bytes)
{
    if (!d3q19 || v != 2) return 32;
    if (aa) return elem == 2 ? 24 : 32;
    if (elem != 4 || 2 * 19 * 4 * cells <= 2 * l2_bytes) return 32;
    return (int)std::min<int64_t>(32, (12 * 64 * tiles + cells / 2) / cells);
}

// V cells of a row of a fully periodic domain, all of them bulk cells: the
// vector update of step_vec.cuh without its boundary roles.  Compiled for one
// streaming step type; with the pull and both AA step types (and the roles)
// in one kernel the D3Q19 FP32 group took 106 registers and the FP16 group
// spilled 104 bytes at its 64.
template <class L, class S, class C, int V, int SP>
__device__ __forceinline__ void update_served(const BatchDomain &d, const char *fin, char *fout, int x0, int y, int z)
{
    using RW = Raw<S, V>;
    const int nx = d.nx, ny = d.ny, nz = d.nz, nxy = nx * ny;
    if (x0 >= nx) return;  // lanes past the row end
    RowOff ro;
    ro.ym = y == 0 ? (ny - 1) * nx : -nx;
    ro.yp = y == ny - 1 ? -(ny - 1) * nx : nx;
    ro.zm = L::D == 2 ? 0 : (z == 0 ? (nz - 1) * nxy : -nxy);
    ro.zp = L::D == 2 ? 0 : (z == nz - 1 ? -(nz - 1) * nxy : nxy);
    const unsigned cell = (unsigned)x0 + (unsigned)nx * y + (unsigned)nxy * z;
    // cells just left / right of the vector, relative to x0 (wrapped around)
    const int dl = x0 > 0 ? -1 : nx - 1;
    const int dr = x0 + V < nx ? V : -x0;
#ifdef LBM_BOUNDS_CHECK
    {
        const int64_t N = (int64_t)nxy * nz;
        bool bad = (int64_t)cell + V > N;
        for (int i = 0; i < L::Q; ++i) {
            const int64_t src = (int64_t)cell + pull_off<L>(ro, i);
            bad = bad || src < 0 || src + V > N || src + dl < 0 || src + dl >= N || src + dr < 0 || src + dr >= N;
        }
        if (index_fault(d.p, bad)) return;
    }
#endif
    const char *bin = fin + (size_t)cell * sizeof(S);
    char *bout = fout + (size_t)cell * sizeof(S);
    const unsigned dstride = d.dstride;
    VecIn<L, S, C, V> r;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        if (SP == kAALocal) {
            r.v[i] = RW::ld(reinterpret_cast<const S *>(bin + (size_t)opp<L>(i) * dstride));
        } else {
            const S *row = vec_row_ptr<L, S, SP>(bin, i, ro, dstride);
            r.v[i] = RW::ld(row);
            if (L::cx(i) > 0) r.e[i] = Store<S>::ld(row + dl);
            if (L::cx(i) < 0) r.e[i] = Store<S>::ld(row + dr);
        }
    }
    const C om = C(d.omega);
    C o[V][L::Q];
#pragma unroll
    for (int k = 0; k < V; ++k) {
        C g[L::Q];
        gather_vec<L, S, C, V, SP>(r, k, g);
        const Mom<C> m = moments_pairs<L, C>(g);
        if constexpr (has_fp64_form<L, C>())
            collide_fp64<L, false>(m, om, C(0), o[k]);
        else
            rebuild_all<L, C, false>(coef_interior<L, C, false>(m, om, C(0)), o[k]);
    }
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        C w[V];
#pragma unroll
        for (int k = 0; k < V; ++k) w[k] = o[k][i];
        if (SP != kAAPush) {
            GroupSt<S, V>::st(reinterpret_cast<S *>(bout + (size_t)i * dstride), w);
            continue;
        }
        // gather-push: o_i goes to P_opp(i)[x + xi_i], wrapped around
        const int j = opp<L>(i);
        S *dst = reinterpret_cast<S *>(bout + ((unsigned)j * dstride + (unsigned)(pull_off<L>(ro, j) * (int)sizeof(S))));
        if (L::cx(i) == 0) {
            GroupSt<S, V>::st(dst, w);
        } else {
#pragma unroll
            for (int k = 0; k < V; ++k) {
                const bool wrap = L::cx(i) > 0 ? (k == V - 1 && x0 + V >= nx) : (k == 0 && x0 == 0);
                Store<S>::st(dst + k + L::cx(i) + (wrap ? -L::cx(i) * nx : 0), w[k]);
            }
        }
    }
}

// Step s of a round for the domains of one group.  tiles: the group's list;
// the next item is fetched while the current one is updated.
template <class L, class S, class C, int V, bool AA>
__global__ void __launch_bounds__(256, (BatchMinBlocks<L, S, V, AA>::value))
    k_batched(const BatchDomain *__restrict__ doms, const int4 *__restrict__ tiles, int ntiles, int s)
{
    const int wpb = blockDim.x >> 5, lane = threadIdx.x & 31;
    int t = blockIdx.x * wpb + (threadIdx.x >> 5);
    if (t >= ntiles) return;
    int4 next = __ldg(tiles + t);
    while (t < ntiles) {
        const int4 tl = next;  // domain, y, z, x0
        t += gridDim.x * wpb;
        if (t < ntiles) next = __ldg(tiles + t);
        const BatchDomain &d = doms[tl.x];
        if (s >= d.remaining) continue;  // uniform across the warp: one domain per tile
        const int cur = d.cur ^ (s & 1);
        const int x0 = tl.w + lane * V;
        if constexpr (V == 1) {
            if (x0 >= d.nx) continue;
            if constexpr (AA) {
                if (cur)
                    update_cell_aa<L, S, C, false, kMaskNone, true>(d.p, d.base[0], x0, tl.y, tl.z);
                else
                    update_cell_aa<L, S, C, false, kMaskNone, false>(d.p, d.base[0], x0, tl.y, tl.z);
            } else {
                update_cell<L, S, C, false, kMaskNone>(d.p, d.base[cur], d.base[1 - cur], x0, tl.y, tl.z);
            }
        } else if constexpr (AA) {
            if (cur)
                update_served<L, S, C, V, kAALocal>(d, d.f[0], d.f[0], x0, tl.y, tl.z);
            else
                update_served<L, S, C, V, kAAPush>(d, d.f[0], d.f[0], x0, tl.y, tl.z);
        } else {
            update_served<L, S, C, V, kPull>(d, d.f[cur], d.f[1 - cur], x0, tl.y, tl.z);
        }
    }
}

// End of a round of `steps` steps: lattice, step count and remaining steps of every domain
__global__ void k_batch_advance(BatchDomain *__restrict__ doms, int ndom, int64_t steps)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= ndom) return;
    BatchDomain &d = doms[k];
    const int64_t adv = d.remaining < steps ? d.remaining : steps;
    if (adv <= 0) return;
    d.cur ^= (int)(adv & 1);
    d.p.step += adv;
    d.remaining -= adv;
}

}  // namespace rr
