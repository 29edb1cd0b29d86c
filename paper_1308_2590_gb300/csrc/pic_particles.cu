// Particle state outside the step: conversion of loaded global positions into
// (cell, offsets), deposit of the moments at rest (after a load or a field
// overwrite, Eq. 3), and export of the particles in the library's order.
// Particles are stored per species, structure-of-arrays, in tile bins
// (pic_internal.cuh).
#include <math.h>

#include <algorithm>

#include "pic_internal.cuh"

namespace pic {

int scan_tiles(pic_t *h, const int32_t *in, int32_t *out);

template <typename R>
struct DepArgs {
    GridArgs<R> g;
    const int32_t *cell;
    const R *ox, *oy, *ux, *uy, *uz, *w;
    const int32_t *bstart, *useg, *segn;
    const V4<R> *B;
    R *M;
    unsigned long long *Mfix;
    FixScale fs;
    R q, m;
    R kb, cq2, hq;    // q dt / (2 m) over the stored B's scale of 4, q^2 dt^2 / (4 m), q dt^2 / (4 m): per species, from the host (as for the push)
    int32_t *flags;   // checks build: FLAG_CHECK on a broken invariant
    double *cr;       // FP64 form: the carried quantities of the bins ([NCARRY][ccap]), else nullptr
    int64_t ccap;
    double *Mc;       // FP64 L2-reduction form: the cell sums the push deposits into (else nullptr)
    int tnx, tny, ntx;  // tiles (FP64: the block's tile of B in cell form, in shared memory)
    const int2 *items;  // work items (tile, run of REST_SEGS segments)
    const int32_t *nitems;
    int32_t *ticket;
};

// Work items of a deposit at rest: the runs of ch segments (REST_SEGS, the FP32
// cell deposit more: rest_segs) of every occupied bin, in any order; resident blocks take them from a queue.  (A grid
// of four blocks per tile started mostly empty blocks: 0.72 ms per species for
// 0.16M particles in 131,072 tiles, whatever they held.)
constexpr int REST_SEGS = 32;
__global__ void k_rest_items(const int32_t *__restrict__ useg, int ntiles, int ch, int2 *__restrict__ items,
                             int32_t *__restrict__ nitems) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int n = t < ntiles ? (useg[t] + ch - 1) / ch : 0;
    // one queue reservation per warp
    const int lane = threadIdx.x & 31;
    int incl = n;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    int base = 0;
    if (lane == 31 && incl) base = atomicAdd(nitems, incl);
    base = __shfl_sync(0xffffffffu, base, 31) + incl - n;
    for (int k = 0; k < n; ++k) items[base + k] = make_int2(t, k);
}

// The block's next item (false: none left); every thread of the block.
__device__ inline bool next_item(const int2 *items, int nitems, int32_t *ticket, int2 *s_item, int2 &it) {
    __syncthreads();   // the previous item (and its shared tables) is done
    if (threadIdx.x == 0) {
        const int k = atomicAdd(ticket, 1);
        *s_item = k < nitems ? items[k] : make_int2(-1, 0);
    }
    __syncthreads();
    it = *s_item;
    return it.x >= 0;
}

// Moments (Eq. 3) of particles at rest with the current node B, a warp per
// segment of the block's item: the FP64 forms and the exact FP32 deposit (the
// plain FP32 one: k_deposit_cells).  FP32: lanes whose particles share a cell (at
// least 6 of them; bins are in cell order, so most segments hold one or two
// cells) first sum their 52 corner products with the butterfly reduce-scatter
// and add 26 values per corner pair; the other lanes add their own products.
// FP64: every lane adds its own products (the butterfly's FP64 adds would cost
// more of the scarce FP64 pipe than the L2 reductions they save), as the push
// does (deposit_fp64).  Global atomics (floating point, or exact fixed point
// when kFix).
template <typename R>
constexpr int min_group_at_rest() { return sizeof(R) == 4 ? 6 : 33; }

template <typename R, bool kFix>
__device__ inline void add_moment(const DepArgs<R> &a, int k, int64_t node, R v) {
    if (kFix)
        atomicAdd(&a.Mfix[(int64_t)k * a.g.nnode + node], (unsigned long long)fix_of(v, a.fs, mom_class(k)));
    else
        atomicAdd(&a.M[(int64_t)k * a.g.nnode + node], v);
}

template <typename R, bool kFix>
__global__ void k_deposit_bins(DepArgs<R> a) {
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ int2 s_item;
    constexpr bool kTab = sizeof(R) == 8;   // FP64: B of the tile's cells in cell form, as the push gathers it
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const GridArgs<R> &g = a.g;
    const int nitems = *a.nitems;
    int2 it;
    while (next_item(a.items, nitems, a.ticket, &s_item, it)) {
    const int t = it.x;
    const int64_t b0 = a.bstart[t];
    const int j0 = it.y * REST_SEGS, u = min(j0 + REST_SEGS, a.useg[t]);
    CellC<R> *tab = (CellC<R> *)dsm;
    const int X0 = (t % a.ntx) * a.tnx, Y0 = (t / a.ntx) * a.tny;
    const int tw = min(a.tnx, g.nx - X0), th = min(a.tny, g.ny - Y0);
    if constexpr (kTab) {
        for (int i = threadIdx.x; i < tw * th; i += blockDim.x) {
            const int ly = i / tw, lx = i - ly * tw;
            const int64_t p00 = pidx(g, X0 + lx, Y0 + ly);
            cell_coef(a.B[p00], a.B[p00 + 1], a.B[p00 + g.nxp], a.B[p00 + g.nxp + 1], tab[i]);
        }
        __syncthreads();
    }
    for (int j = j0 + wid; j < u; j += nw) {
        const int n = a.segn[b0 / SEG + j];
        bool valid = lane < n;
        const int64_t p = b0 + (int64_t)j * SEG + lane;
        if (kChecks && valid) {
            const int32_t cc = a.cell[p];
            const R ofx = a.ox[p], ofy = a.oy[p];
            if (cc < 0 || cc >= g.nx * g.ny || !(ofx >= R(0) && ofx < R(1)) || !(ofy >= R(0) && ofy < R(1))) {
                atomicOr(a.flags, FLAG_CHECK);
                valid = false;
            }
        }
        int32_t c = -1;
        R fx = R(0), fy = R(0);
        R val[NMOM];   // FP32: the moment values; FP64: their parts, with the class factors fr, fS, fj
        for (int k = 0; k < NMOM; ++k) val[k] = R(0);
        R fr = R(0), fS = R(0), fj = R(0);
        if (valid) {
            c = a.cell[p];
            const int cx = c % g.nx, cy = c / g.nx;
            fx = a.ox[p];
            fy = a.oy[p];
            R Bx, By, Bz;
            const int lx = cx - X0, ly = cy - Y0;
            if (kTab && lx >= 0 && lx < tw && ly >= 0 && ly < th) {   // the same bits as gather4
                const CellC<R> &cb = tab[ly * tw + lx];
                const R fxy = fx * fy;
                Bx = cell_eval(cb.k[0], fx, fy, fxy);
                By = cell_eval(cb.k[1], fx, fy, fxy);
                Bz = cell_eval(cb.k[2], fx, fy, fxy);
            } else {
                gather4(a.B, g, cx, cy, fx, fy, Bx, By, Bz);
            }
            R ig, bx, by, bz, inv;
            if (sizeof(R) == 8 && (kFix || !a.Mc))   // FP64 corner form: class factors and parts
                particle_moment_parts(a.q, a.kb, a.cq2, a.w[p], a.ux[p], a.uy[p], a.uz[p], Bx, By, Bz, val, fr, fS, fj,
                                      ig, bx, by, bz, inv);
            else   // the 13 moment values (the FP64 cell form as the push makes them)
                particle_moments_c(a.q, a.kb, a.hq, a.w[p], a.ux[p], a.uy[p], a.uz[p], Bx, By, Bz, val, ig, bx, by,
                                   bz, inv);
            if (sizeof(R) == 8 && a.cr) {   // what the next push needs of this B (carried, FP64 form)
                a.cr[p] = (double)ig;
                a.cr[a.ccap + p] = (double)bx;
                a.cr[2 * a.ccap + p] = (double)by;
                a.cr[3 * a.ccap + p] = (double)bz;
                a.cr[4 * a.ccap + p] = (double)inv;
            }
        }
        const R W[4] = {(R(1) - fx) * (R(1) - fy), fx * (R(1) - fy), (R(1) - fx) * fy, fx * fy};
        unsigned rem = __ballot_sync(0xffffffffu, valid);
        while (rem) {
            const int cand = __shfl_sync(0xffffffffu, c, __ffs(rem) - 1);
            const unsigned grp = __ballot_sync(0xffffffffu, valid && c == cand) & rem;
            if (__popc(grp) < min_group_at_rest<R>()) break;
            const bool mem = (grp >> lane) & 1u;
            const int ccx = cand % g.nx, ccy = cand / g.nx;
            const int idx = rs26_index(lane);
#pragma unroll
            for (int pass = 0; pass < 2; ++pass) {
                R v[26];
#pragma unroll
                for (int c2 = 0; c2 < 2; ++c2)
#pragma unroll
                    for (int k = 0; k < NMOM; ++k) v[c2 * NMOM + k] = mem ? W[2 * pass + c2] * val[k] : R(0);
                const R r = reduce_scatter26(v, lane);
                if (idx >= 0 && r != R(0)) {
                    const int corner = 2 * pass + idx / NMOM, k = idx % NMOM;
                    add_moment<R, kFix>(a, k, node_of(g, ccx, ccy, corner & 1, corner >> 1), r);
                }
            }
            rem &= ~grp;
        }
        if ((rem >> lane) & 1u) {
            const int cx = c % g.nx, cy = c / g.nx;
            if constexpr (sizeof(R) == 8) {
                // the push's own FP64 deposit (cell sums, or node moments for the exact form)
                if (!kFix && a.Mc)
                    deposit_fp64_cell(a.Mc, c, (double)fx, (double)fy, (const double *)val, lane);
                else
                    deposit_fp64<kFix>((double *)a.M, a.Mfix, a.fs, g, cx, cy, (double)fx, (double)fy,
                                       (const double *)val, (double)fr, (double)fS, (double)fj, lane);
            } else {
                const int64_t nd[4] = {node_of(g, cx, cy, 0, 0), node_of(g, cx, cy, 1, 0), node_of(g, cx, cy, 0, 1),
                                       node_of(g, cx, cy, 1, 1)};
#pragma unroll
                for (int k = 0; k < 4; ++k)
#pragma unroll
                    for (int q = 0; q < NMOM; ++q) add_moment<R, kFix>(a, q, nd[k], W[k] * val[q]);
            }
        }
    }
    }
}

// FP64 cell sums of a list of particles at rest, a thread per particle, with the
// weights' sign given (-1: particles that have left the species); cr (or nullptr): the
// carried quantities of the list.  An ionisation pass moves a few per cent of the
// particles from species to species, so it adds their moments and takes the old
// ones off instead of depositing every particle anew: four deposits of 219 us a
// pass over a carbon foil of 0.8M ions -> five lists of 42 us.
struct DepList {
    const int32_t *cell;
    const double *ox, *oy, *ux, *uy, *uz, *w;
    int64_t n;
    double sign, q, kb, hq;
    double *cr;
    int64_t ccap;
};
__global__ void __launch_bounds__(256) k_deposit_list(GridArgs<double> g, const V4<double> *__restrict__ B, DepList a,
                                                      double *__restrict__ Mc) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.n) return;
    const int32_t c = a.cell[p];
    const double fx = a.ox[p], fy = a.oy[p];
    double Bx, By, Bz, val[NMOM], ig, bx, by, bz, inv;
    gather4(B, g, c % g.nx, c / g.nx, fx, fy, Bx, By, Bz);
    particle_moments_c(a.q, a.kb, a.hq, a.sign * a.w[p], a.ux[p], a.uy[p], a.uz[p], Bx, By, Bz, val, ig, bx, by, bz, inv);
    if (a.cr) {
        const double v[NCARRY] = {ig, bx, by, bz, inv};
#pragma unroll
        for (int k = 0; k < NCARRY; ++k) a.cr[k * a.ccap + p] = v[k];
    }
    deposit_fp64_cell(Mc, c, fx, fy, val, threadIdx.x & 31);
}

static int deposit_list(pic_t *h, int s, DepList a) {
    if (a.n == 0) return 0;
    const SpeciesBuf &S = h->sp[s];
    const double dt = h->cfg.dt;
    a.q = S.q;
    a.kb = 0.25 * (S.q * dt / (2.0 * S.m));
    a.hq = S.q * dt * dt / (4.0 * S.m);
    k_deposit_list<<<(unsigned)((a.n + 255) / 256), 256, 0, h->st>>>(grid_args<double>(h), (const V4<double> *)h->B[h->bcur],
                                                                    a, h->Mc);
    count_launch(h);
    return check_launch("k_deposit_list");
}

// The first n particles of species s's spare set, with what they carry.
int deposit_spare(pic_t *h, int s, int64_t n) {
    SpeciesBuf &S = h->sp[s];
    const int b = S.spare;
    return deposit_list(h, s, DepList{S.cell[b], (const double *)S.ox[b], (const double *)S.oy[b], (const double *)S.ux[b],
                                      (const double *)S.uy[b], (const double *)S.uz[b], (const double *)S.w[b], n, 1.0, 0.0,
                                      0.0, 0.0, S.carry[b], S.cap});
}

// n particles that have left species s, in the checkpoint form (planes of `plane` values: offsets, u, w).
int deposit_leavers(pic_t *h, int s, int64_t n, const int32_t *cell, const double *v, int64_t plane) {
    return deposit_list(h, s, DepList{cell, v, v + plane, v + 2 * plane, v + 3 * plane, v + 4 * plane, v + 5 * plane, n, -1.0,
                                      0.0, 0.0, 0.0, nullptr, 0});
}

// FP32 sums of a cell's particles times its corner weights, in a warp's registers:
// the particles' 13 values and 4 weights go to rows in shared memory, and 8 lanes,
// (4 moments) x (2 corners), add every fourth row, the four groups of 8 rows of
// their own: 10 instructions a lane and 4 rows, where lanes that each took 2
// moments of a corner and every row spent 16, and half the shared memory
// wavefronts that bound it.  The groups meet when the warp goes on to another cell.
struct CellDep {
    static constexpr int RS = 20;   // a row: 13 values, 3 of padding, weights (0,0), (1,0), (0,1), (1,1)
    static constexpr int kWarpBytes = 32 * RS * (int)sizeof(float);
    float *rows, *acc;              // acc: the block's tile, RN nodes of W per row and moment
    int W, RN;
    int node;                       // first node of the warp's cell, or -1
    float s[8];                     // moments 4 (lane % 4) + .. of corner 2 (lane / 4 % 2), then of the next

    __device__ inline void init(void *mem, float *tile, int w, int rn) {
        rows = (float *)mem;
        acc = tile;
        W = w;
        RN = rn;
        node = -1;
#pragma unroll
        for (int k = 0; k < 8; ++k) s[k] = 0.f;
    }

    __device__ inline void flush(int lane) {
        if (node < 0) return;
        const bool h16 = lane & 16, h8 = lane & 8;
        float r[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float send = h16 ? s[k] : s[4 + k], own = h16 ? s[4 + k] : s[k];
            r[k] = own + __shfl_xor_sync(0xffffffffu, send, 16);
        }
        const int m = 4 * (lane & 3) + (h8 ? 2 : 0);
        float *a = acc + m * RN + node + (lane & 4 ? W : 0) + (h16 ? 1 : 0);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const float send = h8 ? r[k] : r[2 + k], own = h8 ? r[2 + k] : r[k];
            const float t = own + __shfl_xor_sync(0xffffffffu, send, 8);
            if (m + k < NMOM && t != 0.f) atomicAdd(a + k * RN, t);
        }
        node = -1;
#pragma unroll
        for (int k = 0; k < 8; ++k) s[k] = 0.f;
    }

    // All lanes: the particle of every valid lane, in the cell with first node n0.  Neighbouring lanes of
    // a cell form a run (the bins are in cell order).
    __device__ inline void add(bool valid, int n0, float fx, float fy, const float *val, int lane) {
        const unsigned full = 0xffffffffu;
        const int key = valid ? n0 : -1, prev = __shfl_up_sync(full, key, 1);
        const bool head = valid && (lane == 0 || prev != key);
        unsigned heads = __ballot_sync(full, head);
        const unsigned ends = heads | __ballot_sync(full, !valid);
        __syncwarp();   // the previous segment's rows have been read
        if (valid) {
            float4 *d = (float4 *)(rows + lane * RS);
            d[0] = make_float4(val[0], val[1], val[2], val[3]);
            d[1] = make_float4(val[4], val[5], val[6], val[7]);
            d[2] = make_float4(val[8], val[9], val[10], val[11]);
            d[3] = make_float4(val[12], 0.f, 0.f, 0.f);
            d[4] = make_float4((1.f - fx) * (1.f - fy), fx * (1.f - fy), (1.f - fx) * fy, fx * fy);
        }
        __syncwarp();
        const float *mine = rows + (lane >> 3) * RS;
        const int ov = 4 * (lane & 3), ow = 16 + ((lane >> 1) & 2);
        while (heads) {
            const int p0 = __ffs(heads) - 1;
            heads &= heads - 1;
            const unsigned after = ends & ~((2u << p0) - 1u);
            const int n = (after ? __ffs(after) - 1 : 32) - p0 - (lane >> 3);
            const int k = __shfl_sync(full, key, p0);
            if (k != node) {
                flush(lane);
                node = k;
            }
#pragma unroll 2
            for (int p = 0; p < n; p += 4) {
                const float *r = mine + (p0 + p) * RS;
                const float4 v = *(const float4 *)(r + ov);
                const float2 w = *(const float2 *)(r + ow);
                s[0] = fmaf(w.x, v.x, s[0]);
                s[1] = fmaf(w.x, v.y, s[1]);
                s[2] = fmaf(w.x, v.z, s[2]);
                s[3] = fmaf(w.x, v.w, s[3]);
                s[4] = fmaf(w.y, v.x, s[4]);
                s[5] = fmaf(w.y, v.y, s[5]);
                s[6] = fmaf(w.y, v.z, s[6]);
                s[7] = fmaf(w.y, v.w, s[7]);
            }
        }
    }
};

// FP32 deposit with area weights from cell-ordered bins (at rest, and in the
// steps that deposit after the regroup): a block takes an item (species, tile,
// run of ch segments); its warps take contiguous segments and add them up cell
// by cell (CellDep) into an accumulator over the tile's nodes in shared memory,
// which goes to the global moments once per item with a TwoSum compensation term.
// Every particle lies in its bin's tile, so nothing leaves the accumulator's nodes.
// 33.5M particles, 32 per cell: per species at rest 0.87 ms with a butterfly per
// segment and cell; a step's two species 1.34 ms with a stencil's sums dealt over the
// lanes, 1.35 with CellDep, 1.11 with the next segment's loads in flight as well
// (issue 56 % and loads waited for before).
struct CellDepSp {
    const int32_t *cell, *bstart, *useg, *segn;
    const float *ox, *oy, *ux, *uy, *uz, *w;
    float q, kb, hq;
};
struct CellDepArgs {
    GridArgs<float> g;
    CellDepSp sp[PIC_MAX_SPECIES];
    const V4<float> *B;
    float *M, *Mlo;
    int tnx, tny, ntx, ntiles, ch;
    uint32_t magic_nx;
    const int2 *items;              // (species * ntiles + tile, run)
    const int32_t *nitems;
    int32_t *ticket;
    const int32_t *guard0, *guard1; // flags words: set, the deposit does nothing
    int32_t *flags;
};

__host__ __device__ inline int cell_dep_nodes(int tnx, int tny) { return (tnx + 1) * (tny + 1); }
__host__ __device__ inline int cell_dep_smem(int tnx, int tny) {
    return cell_dep_nodes(tnx, tny) * (int)(sizeof(V4<float>) + NMOM * sizeof(float)) + 8 * CellDep::kWarpBytes;
}

__global__ void __launch_bounds__(256, 3) k_deposit_cells(const __grid_constant__ CellDepArgs a) {
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ int2 s_item;
    if ((a.guard0 && (*a.guard0 & 3)) || (a.guard1 && (*a.guard1 & 3))) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const GridArgs<float> &g = a.g;
    const int W = a.tnx + 1, RN = W * (a.tny + 1);
    V4<float> *sB = (V4<float> *)dsm;
    float *acc = (float *)((unsigned char *)(sB + RN) + 8 * CellDep::kWarpBytes);
    CellDep dep;
    dep.init((unsigned char *)(sB + RN) + wid * CellDep::kWarpBytes, acc, W, RN);
    const int nitems = *a.nitems;
    int2 it;
    while (next_item(a.items, nitems, a.ticket, &s_item, it)) {
        const int s = it.x / a.ntiles, t = it.x - s * a.ntiles;
        const CellDepSp &P = a.sp[s];
        const int X0 = (t % a.ntx) * a.tnx, Y0 = (t / a.ntx) * a.tny;
        const int tw = min(a.tnx, g.nx - X0), th = min(a.tny, g.ny - Y0);
        for (int i = threadIdx.x; i < RN; i += 256) {
            const int ly = i / W, lx = i - ly * W;
            sB[i] = a.B[pidx(g, X0 + lx, Y0 + ly)];   // the ghost ring holds tile + halo + 1 nodes
        }
        for (int i = threadIdx.x; i < NMOM * RN; i += 256) acc[i] = 0.f;
        __syncthreads();
        const int64_t b0 = P.bstart[t];
        const int j0 = it.y * a.ch, j1 = min(j0 + a.ch, P.useg[t]);
        const int per = (j1 - j0 + 7) / 8, m0 = j0 + wid * per, m1 = min(m0 + per, j1);
        // the next segment's particles are in flight while this one's are added up (slots past a segment's
        // count are allocated, their values unused)
        struct {
            int n;
            int32_t c;
            float fx, fy, ux, uy, uz, w;
        } next = {0, 0, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        auto fetch = [&](int j) {
            const int64_t p = b0 + (int64_t)j * SEG + lane;
            next.n = P.segn[b0 / SEG + j];
            next.c = P.cell[p];
            next.fx = P.ox[p];
            next.fy = P.oy[p];
            next.ux = P.ux[p];
            next.uy = P.uy[p];
            next.uz = P.uz[p];
            next.w = P.w[p];
        };
        if (m0 < m1) fetch(m0);
        for (int j = m0; j < m1; ++j) {
            bool valid = lane < next.n;
            const int32_t c = valid ? next.c : 0;
            const float fx = next.fx, fy = next.fy, ux = next.ux, uy = next.uy, uz = next.uz, w = next.w;
            if (j + 1 < m1) fetch(j + 1);
            int cx, cy;
            cell_split(c, g.nx, a.magic_nx, cx, cy);
            const int lx = cx - X0, ly = cy - Y0;
            if (valid && (lx < 0 || lx >= tw || ly < 0 || ly >= th ||
                          (kChecks && !(fx >= 0.f && fx < 1.f && fy >= 0.f && fy < 1.f)))) {
                atomicOr(a.flags, 16);   // outside its bin's tile: skipped
                valid = false;
            }
            float val[NMOM];
            if (valid) {
                const V4<float> *r0 = sB + ly * W + lx, *r1 = r0 + W;
                const V4<float> n00 = r0[0], n10 = r0[1], n01 = r1[0], n11 = r1[1];
                const float w00 = (1.f - fx) * (1.f - fy), w10 = fx * (1.f - fy), w01 = (1.f - fx) * fy, w11 = fx * fy;
                const float Bx = w00 * n00.x + w10 * n10.x + w01 * n01.x + w11 * n11.x;
                const float By = w00 * n00.y + w10 * n10.y + w01 * n01.y + w11 * n11.y;
                const float Bz = w00 * n00.z + w10 * n10.z + w01 * n01.z + w11 * n11.z;
                float ig, bx, by, bz, inv;
                particle_moments_c(P.q, P.kb, P.hq, w, ux, uy, uz, Bx, By, Bz, val, ig, bx, by, bz, inv);
            }
            dep.add(valid, ly * W + lx, fx, fy, val, lane);
        }
        dep.flush(lane);   // (the next item's tile has other nodes)
        __syncthreads();
        for (int r = threadIdx.x; r < RN; r += 256) {
            const int ly = r / W, lx = r - ly * W;
            int gx = X0 + lx, gy = Y0 + ly;
            if (lx > tw || ly > th) continue;   // a ragged tile's unused nodes
            if (gy >= g.ny) gy -= g.ny;
            if (g.periodic_x && gx >= g.nx) gx -= g.nx;
            const int64_t gn = (int64_t)gy * g.nxn + gx;
            float v[NMOM], old[NMOM];
#pragma unroll
            for (int k = 0; k < NMOM; ++k) {
                v[k] = acc[k * RN + r];
                old[k] = v[k] != 0.f ? atomicAdd(&a.M[(int64_t)k * g.nnode + gn], v[k]) : 0.f;
            }
#pragma unroll
            for (int k = 0; k < NMOM; ++k) {
                const float sum = old[k] + v[k], bb = sum - old[k];
                const float err = (old[k] - (sum - bb)) + (v[k] - bb);
                if (err != 0.f) atomicAdd(&a.Mlo[(int64_t)k * g.nnode + gn], err);
            }
        }
    }
}

// Moments at rest with a spline shape of degree N: the gather (gather_s),
// moments and deposit (SplineDep; the exact form lane by lane, so that a
// deposit at rest repeats the push's products bitwise) of the spline-shape
// push; each warp takes a run of the item's segments.
template <typename R, bool kFix, int N>
__global__ void __launch_bounds__(256) k_deposit_s(DepArgs<R> a) {
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ int2 s_item;
    constexpr bool kParts = sizeof(R) == 8 && kFix;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const GridArgs<R> &g = a.g;
    const int nitems = *a.nitems;
    SplineDep<R, N> dep;
    if (!kFix) dep.init(dsm + wid * SplineDep<R, N>::kWarpBytes, lane);
    int2 it;
    while (next_item(a.items, nitems, a.ticket, &s_item, it)) {
        const int64_t b0 = a.bstart[it.x];
        const int j0 = it.y * REST_SEGS, j1 = min(j0 + REST_SEGS, a.useg[it.x]);
        const int per = (j1 - j0 + nw - 1) / nw;
        for (int j = j0 + wid * per; j < min(j0 + (wid + 1) * per, j1); ++j) {
            const int n = a.segn[b0 / SEG + j];
            const int64_t p = b0 + (int64_t)j * SEG + lane;
            bool valid = lane < n;
            int32_t c = 0;
            R fx = R(0), fy = R(0);
            if (valid) {
                c = a.cell[p];
                fx = a.ox[p];
                fy = a.oy[p];
            }
            if (kChecks && valid && (c < 0 || c >= g.nx * g.ny || !(fx >= R(0) && fx < R(1)) || !(fy >= R(0) && fy < R(1)))) {
                atomicOr(a.flags, FLAG_CHECK);
                valid = false;
            }
            R val[NMOM];
            SplineN<R, N> sp;
            if (valid) {
                sp = spline_n<R, N>(c % g.nx, c / g.nx, fx, fy);
                R Bx, By, Bz;
                gather_s(a.B, g, sp, Bx, By, Bz);
                R fr = R(1), fS = R(1), fj = R(1), ig, bx, by, bz, inv;
                if constexpr (kParts)
                    particle_moment_parts(a.q, a.kb, a.cq2, a.w[p], a.ux[p], a.uy[p], a.uz[p], Bx, By, Bz, val, fr, fS,
                                          fj, ig, bx, by, bz, inv);
                else
                    particle_moments_c(a.q, a.kb, a.hq, a.w[p], a.ux[p], a.uy[p], a.uz[p], Bx, By, Bz, val, ig, bx, by,
                                       bz, inv);
                if (sizeof(R) == 8 && a.cr) {   // what the next push needs of this B (carried, FP64 form)
                    a.cr[p] = (double)ig;
                    a.cr[a.ccap + p] = (double)bx;
                    a.cr[2 * a.ccap + p] = (double)by;
                    a.cr[3 * a.ccap + p] = (double)bz;
                    a.cr[4 * a.ccap + p] = (double)inv;
                }
                if constexpr (kFix) deposit_s_fix<R, kParts, N>(a.Mfix, a.fs, g, sp, val, fr, fS, fj, lane);
            }
            if constexpr (!kFix) dep.add(GlobalSink<R>{g, a.M}, g.nx, g.ny, valid, sp, val, lane);
        }
    }
    if constexpr (!kFix) dep.flush(GlobalSink<R>{g, a.M}, lane);
}

// Fixed-point sums -> floating-point moments: FP64 M, or the FP32 pair (M, Mlo)
// with M + Mlo the sum to about 2^-48 relative.
template <typename R>
__global__ void k_fix_to_moments(const unsigned long long *__restrict__ fix, R *__restrict__ M, R *__restrict__ Mlo,
                                 int64_t nnode, FixScale fs) {
    const int64_t n = (int64_t)NMOM * nnode;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double d = (double)(long long)fix[i] * fs.inv[mom_class((int)(i / nnode))];
        const R hi = (R)d;
        M[i] = hi;
        if (sizeof(R) == 4) Mlo[i] = (R)(d - (double)hi);
    }
}

// Global positions -> (cell, offset): s = x/dx, cell = floor(s), offset = s - cell
// (a coordinate rounding onto the far edge folds back or stays in the last cell;
// an FP32 offset that rounds to 1 moves to the next cell with offset 0).
// Positions outside [0, Lx) x [0, Ly) or non-finite momenta / weights are
// rejected: the smallest such index goes to *bad (the load is then dropped).
struct LoadSrc {
    const double *a[6];   // x, y, ux, uy, uz, w: device memory or device-accessible host memory
};

constexpr int LOAD_BS = 256;
constexpr int LOAD_SM_PERMILLE = 500;   // conversion blocks per 1000 SMs (measured: 76 x 256 on GB300
                                        // reads the link at full rate beside a regroup at nearly full speed)

// x / d from the correctly rounded reciprocal rd of d: with q = x rd and the
// remainder r = x - q d (one FMA), q + r rd is the correctly rounded quotient
// (P. Markstein, "Computation of elementary functions on the IBM RISC
// System/6000 processor", 1990) but for quotients within a few 2^-53 of an ulp
// of a rounding boundary or in the denormal range.  Three operations of the FP64
// pipe, which bounds the conversion, instead of a division's dozen.
__device__ inline double div_by(double x, double d, double rd) {
    const double q = x * rd;
    return fma(fma(-q, d, x), rd, q);
}

// floor(x) of 0 <= x < 2^31 as a double and an integer, from the bits.
__device__ inline double floor_cell(double x, int &c) {
    const long long b = __double_as_longlong(x);
    const int e = (int)(b >> 52) - 1023;
    if (e < 0) {
        c = 0;
        return 0.0;
    }
    const int sh = 52 - e;
    c = (int)(((b & 0xFFFFFFFFFFFFFll) | 0x10000000000000ll) >> sh);
    return __longlong_as_double((b >> sh) << sh);
}

// 0 <= x < L of a position: false for NaN, infinities and negative values but
// -0, by integer compares (FP64 compares issue on the FP64 pipe).
__device__ inline bool in_box(double x, double L) {
    const long long b = __double_as_longlong(x);
    return (b >= 0 && b < __double_as_longlong(L)) || b == (long long)0x8000000000000000ull;
}
__device__ inline bool finite_bits(double x) {
    return (__double2hiint(x) & 0x7FF00000) != 0x7FF00000;   // (the 64-bit form compiles to an FP64 compare)
}

template <typename R>
__global__ void __launch_bounds__(LOAD_BS) k_load_convert(GridArgs<double> g, double Lx, double Ly, LoadSrc src, int64_t n,
                               int32_t *cell, R *ox, R *oy, R *ux, R *uy, R *uz, R *w,
                               unsigned long long *bad) {
    // grid-stride.  Arrays read over the CPU-GPU link: one small block on
    // half of the SMs keeps enough reads in flight for the link, while the
    // regroup of the species converted before runs beside it at nearly full
    // speed (a conversion grid over every SM slowed that regroup about
    // threefold).  Arrays in device memory: a full grid.
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const double x = src.a[0][t], y = src.a[1][t];
        const double vx = src.a[2][t], vy = src.a[3][t], vz = src.a[4][t], vw = src.a[5][t];
        if (!in_box(x, Lx) || !in_box(y, Ly) || !finite_bits(vx) || !finite_bits(vy) || !finite_bits(vz) ||
            !finite_bits(vw)) {
            atomicMin(bad, (unsigned long long)t);
            // an in-range placeholder, so that a regroup queued before the check stays in bounds
            cell[t] = 0;
            ox[t] = oy[t] = ux[t] = uy[t] = uz[t] = w[t] = R(0);
            continue;
        }
        const double sxx = div_by(x, g.dx, g.inv_dx), syy = div_by(y, g.dy, g.inv_dy);
        int cx, cy;
        const double flx = floor_cell(sxx, cx), fly = floor_cell(syy, cy);
        double fx = sxx - flx, fy = syy - fly;
        // x < Lx whose x/dx rounds to nx (walls): the last cell, at the largest offset below 1 of the
        // form's precision, so that every stored offset lies in [0, 1)
        if (cx >= g.nx) { if (g.periodic_x) cx -= g.nx; else { cx = g.nx - 1; fx = 0x1.fffffffffffffp-1; } }
        if (cy >= g.ny) cy -= g.ny;
        R rfx = stored<R>(fx), rfy = stored<R>(fy);
        if (sizeof(R) == 4) {
            if (rfx >= R(1)) {
                if (g.periodic_x || cx + 1 < g.nx) { rfx = R(0); cx = (cx + 1 == g.nx) ? 0 : cx + 1; }
                else rfx = (R)0.99999994;
            }
            if (rfy >= R(1)) { rfy = R(0); cy = (cy + 1 == g.ny) ? 0 : cy + 1; }
        }
        cell[t] = cy * g.nx + cx;
        ox[t] = rfx;
        oy[t] = rfy;
        ux[t] = stored<R>(vx);
        uy[t] = stored<R>(vy);
        uz[t] = stored<R>(vz);
        w[t] = stored<R>(vw);
    }
}

// Checkpoint form (cell index, in-cell offsets, u, w) -> the species' spare
// buffer set, checked like a load: cell in range, offsets in [0, 1), all
// finite.  FP32 form: the offsets, u and w are rounded to FP32 (exact for
// values saved by an FP32 handle); an offset that rounds to 1 moves to the
// next cell with offset 0, as in a load.
template <typename R>
__global__ void __launch_bounds__(LOAD_BS) k_restore_convert(GridArgs<double> g, LoadSrc src, const int32_t *csrc,
                                                             int64_t n, int32_t *cell, R *ox, R *oy, R *ux, R *uy,
                                                             R *uz, R *w, unsigned long long *bad) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = csrc[t];
        const double fx = src.a[0][t], fy = src.a[1][t];
        const double vx = src.a[2][t], vy = src.a[3][t], vz = src.a[4][t], vw = src.a[5][t];
        if (c < 0 || (int64_t)c >= (int64_t)g.nx * g.ny || !(fx >= 0.0 && fx < 1.0) || !(fy >= 0.0 && fy < 1.0) ||
            !isfinite(vx) || !isfinite(vy) || !isfinite(vz) || !isfinite(vw)) {
            atomicMin(bad, (unsigned long long)t);
            cell[t] = 0;   // in-range placeholder (a regroup may run before the check is read)
            ox[t] = oy[t] = ux[t] = uy[t] = uz[t] = w[t] = R(0);
            continue;
        }
        int cx = c % g.nx, cy = c / g.nx;
        R rfx = (R)fx, rfy = (R)fy;
        if (sizeof(R) == 4) {
            if (rfx >= R(1)) {
                if (g.periodic_x || cx + 1 < g.nx) { rfx = R(0); cx = (cx + 1 == g.nx) ? 0 : cx + 1; }
                else rfx = (R)0.99999994;
            }
            if (rfy >= R(1)) { rfy = R(0); cy = (cy + 1 == g.ny) ? 0 : cy + 1; }
        }
        cell[t] = cy * g.nx + cx;
        ox[t] = rfx;
        oy[t] = rfy;
        ux[t] = (R)vx;
        uy[t] = (R)vy;
        uz[t] = (R)vz;
        w[t] = (R)vw;
    }
}

// Bins -> compact FP64 staging [x | y | ux | uy | uz | w | cell(int32)], in the
// particle order (tiles, then segments, then the valid prefix of each).
template <typename R>
__global__ void k_bins_to_stage(GridArgs<double> g, const int32_t *bstart, const int32_t *useg, const int32_t *segn,
                                const int32_t *cstart, int64_t n, const int32_t *cell, const R *ox, const R *oy,
                                const R *ux, const R *uy, const R *uz, const R *w, double *st, bool raw) {
    __shared__ int wcnt[32];
    __shared__ int run;
    const int t = blockIdx.x;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int64_t b0 = bstart[t], sb = b0 / SEG;
    const int u = useg[t];
    if (u == 0) return;
    if (threadIdx.x == 0) run = 0;
    __syncthreads();
    for (int j0 = 0; j0 < u; j0 += nw) {
        const int j = j0 + wid;
        const int nseg = (j < u) ? segn[sb + j] : 0;
        if (lane == 0) wcnt[wid] = nseg;
        __syncthreads();
        int before = 0, tot = 0;
        for (int q = 0; q < nw; ++q) {
            if (q < wid) before += wcnt[q];
            tot += wcnt[q];
        }
        if (lane < nseg) {
            const int64_t p = b0 + (int64_t)j * SEG + lane;
            const int64_t o = (int64_t)cstart[t] + run + before + lane;
            const int32_t c = cell[p];
            const int cx = c % g.nx, cy = c / g.nx;
            st[o] = raw ? (double)ox[p] : ((double)cx + (double)ox[p]) * g.dx;
            st[n + o] = raw ? (double)oy[p] : ((double)cy + (double)oy[p]) * g.dy;
            st[2 * n + o] = (double)ux[p];
            st[3 * n + o] = (double)uy[p];
            st[4 * n + o] = (double)uz[p];
            st[5 * n + o] = (double)w[p];
            ((int32_t *)(st + 6 * n))[o] = c;
        }
        __syncthreads();
        if (threadIdx.x == 0) run += tot;
        __syncthreads();
    }
}

// --------------------------------------------------------------------------- host side

// Resident blocks of 256 threads over the work items.
template <typename R>
static int rest_launch(pic_t *h, void (*kernel)(DepArgs<R>), const DepArgs<R> &a, size_t smem) {
    int dev = 0, nsm = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (smem > 32 * 1024) allow_smem((const void *)kernel, smem);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, 256, smem) != cudaSuccess || per < 1) {
        cudaGetLastError();
        per = 1;
    }
    kernel<<<(unsigned)(per * (nsm > 0 ? nsm : 1)), 256, smem, h->st>>>(a);
    count_launch(h);
    return check_launch("deposit at rest");
}

// Species s of the FP32 cell deposit.
static CellDepSp cell_dep_species(const pic_t *h, int s) {
    const SpeciesBuf &S = h->sp[s];
    const int b = S.bins;
    const double dt = h->cfg.dt;
    return CellDepSp{S.cell[b], S.bstart, S.useg[S.scur], S.segn[S.scur], (const float *)S.ox[b], (const float *)S.oy[b],
                     (const float *)S.ux[b], (const float *)S.uy[b], (const float *)S.uz[b], (const float *)S.w[b],
                     (float)S.q, 0.25f * (float)(S.q * dt / (2.0 * S.m)), (float)(S.q * dt * dt / (4.0 * S.m))};
}

static CellDepArgs cell_dep_args(const pic_t *h) {
    CellDepArgs a;
    a.g = grid_args<float>(h);
    a.B = (const V4<float> *)h->B[h->bcur];
    a.M = (float *)h->M;
    a.Mlo = (float *)h->Mlo;
    a.tnx = h->tnx;
    a.tny = h->tny;
    a.ntx = h->ntx;
    a.ntiles = h->ntiles;
    a.magic_nx = (uint32_t)((0x100000000ull + (uint64_t)h->nx - 1) / (uint64_t)h->nx);
    a.items = h->items;
    a.guard0 = a.guard1 = nullptr;
    a.flags = h->d_flags;
    return a;
}

static int cell_dep_launch(pic_t *h, const CellDepArgs &a) {
    const int smem = cell_dep_smem(h->tnx, h->tny);
    int dev = 0, nsm = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (smem > 32 * 1024) allow_smem((const void *)k_deposit_cells, smem);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_deposit_cells, 256, smem) != cudaSuccess || per < 1) {
        cudaGetLastError();
        per = 1;
    }
    k_deposit_cells<<<(unsigned)(per * (nsm > 0 ? nsm : 1)), 256, smem, h->st>>>(a);
    count_launch(h);
    return check_launch("k_deposit_cells");
}

// Steps whose moments are deposited after the regroup, from cell-ordered bins:
// the FP32 form with the time-centred solve.  That solve allows steps in which
// thermal particles cross cells (c dt/dx = 25 on the uniform plasmas); in the
// push a segment's particles then end in some twenty cells and most of its
// lanes went to the global moments one by one, 52 L2 reductions each.  The
// literal solve (c dt <= dx, few crossings) runs beside the regroup and needs
// the moments before it, so its steps keep the deposit in the push.  1024 x
// 1024 periodic plasma, 67M particles, per step: push with deposit 5.26 ms ->
// push 1.09 + deposit 1.11 ms.
bool post_deposit(const pic_t *h) {
    return h->fp32 && !h->det && h->shape == 1 && h->cfg.field_mode == PIC_FIELD_CN;
}

int deposit_step(pic_t *h, const int32_t *guard0, const int32_t *guard1) {
    CellDepArgs a = cell_dep_args(h);
    a.B = (const V4<float> *)h->B[1 - h->bcur];   // the new node B (the step's flip follows)
    for (int s = 0; s < h->nsp; ++s) a.sp[s] = cell_dep_species(h, s);
    a.ch = push_item_segs(h);
    a.nitems = list_counters(h, h->lists) + LC_ITEMS;
    a.ticket = list_counters(h, h->lists) + LC_DEPOSIT;
    a.guard0 = guard0;
    a.guard1 = guard1;
    return cell_dep_launch(h, a);
}

// Segments per item of the FP32 cell deposit at rest: an item ends with the tile's
// nodes going to the global moments (13 pairs of reductions each), so an item is
// as long as leaves every resident block about four of them (the capacity is
// about twice the particles).  With that and the loads ahead, 33.5M particles:
// 0.88 ms in items of 32 -> 0.47 ms in items of 256; 3.3M: 85 -> 66 us.
static int rest_segs(const SpeciesBuf &S) {
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int64_t ch = S.cap / SEG / 2 / (12 * (nsm > 0 ? nsm : 1));
    return (int)std::min<int64_t>(std::max<int64_t>(ch, REST_SEGS), 256);
}

template <typename R>
static int deposit_only_t(pic_t *h, int s) {
    SpeciesBuf &S = h->sp[s];
    if (S.cap == 0) return 0;
    DepArgs<R> a;
    a.g = grid_args<R>(h);
    int b = S.bins;
    a.cell = S.cell[b];
    a.ox = (const R *)S.ox[b]; a.oy = (const R *)S.oy[b];
    a.ux = (const R *)S.ux[b]; a.uy = (const R *)S.uy[b]; a.uz = (const R *)S.uz[b]; a.w = (const R *)S.w[b];
    a.bstart = S.bstart;
    a.useg = S.useg[S.scur];
    a.segn = S.segn[S.scur];
    a.B = (const V4<R> *)h->B[h->bcur];
    a.M = (R *)h->M;
    a.Mfix = h->Mfix;
    if (h->det)
        if (int rc = fix_scale(h, &a.fs)) return rc;
    a.q = (R)S.q;
    a.m = (R)S.m;
    a.kb = R(0.25) * (R)(S.q * h->cfg.dt / (2.0 * S.m));
    a.cq2 = (R)(S.q * S.q * h->cfg.dt * h->cfg.dt / (4.0 * S.m));
    a.hq = (R)(S.q * h->cfg.dt * h->cfg.dt / (4.0 * S.m));
    a.flags = h->d_flags;
    a.cr = S.carry[b];
    a.ccap = S.cap;
    a.Mc = h->Mc;   // node moments after cell_moments
    a.tnx = h->tnx;
    a.tny = h->tny;
    a.ntx = h->ntx;
    // the work items (words 0 and 1 of the queue's counters)
    if (int rc = ensure_items(h)) return rc;
    a.items = h->items;
    a.nitems = h->ticket;
    a.ticket = h->ticket + 1;
    cudaMemsetAsync(h->ticket, 0, 2 * sizeof(int32_t), h->st);
    const bool cells = h->fp32 && !h->det && h->shape == 1;
    const int ch = cells ? rest_segs(S) : REST_SEGS;
    k_rest_items<<<(h->ntiles + 255) / 256, 256, 0, h->st>>>(a.useg, h->ntiles, ch, h->items, h->ticket);
    count_launch(h);
    const size_t tab = h->fp32 ? 0 : (size_t)h->tnx * h->tny * sizeof(CellC<double>);   // B in cell form
    if (cells) {
        CellDepArgs c = cell_dep_args(h);
        c.sp[0] = cell_dep_species(h, s);
        c.ch = ch;
        c.nitems = a.nitems;
        c.ticket = a.ticket;
        return cell_dep_launch(h, c);
    }
    switch (h->shape >= 2 ? h->shape * 2 + (h->det ? 1 : 0) : (h->det ? 1 : 0)) {
        case 0:
            if constexpr (sizeof(R) == 8) return rest_launch(h, k_deposit_bins<R, false>, a, tab);
            break;   // FP32: k_deposit_cells above
        case 1: return rest_launch(h, k_deposit_bins<R, true>, a, tab);
        case 4: return rest_launch(h, k_deposit_s<R, false, 2>, a, 8 * SplineDep<R, 2>::kWarpBytes);
        case 5: return rest_launch(h, k_deposit_s<R, true, 2>, a, 0);
        case 6: return rest_launch(h, k_deposit_s<R, false, 3>, a, 8 * SplineDep<R, 3>::kWarpBytes);
        case 7: return rest_launch(h, k_deposit_s<R, true, 3>, a, 0);
        case 8: return rest_launch(h, k_deposit_s<R, false, 4>, a, 8 * SplineDep<R, 4>::kWarpBytes);
        case 9: return rest_launch(h, k_deposit_s<R, true, 4>, a, 0);
    }
    return PIC_ERR_STATE;
}

int deposit_only(pic_t *h, int s) {
    h->touch_all = true;   // the touched-tile map describes a push, not a deposit at rest
    return h->fp32 ? deposit_only_t<float>(h, s) : deposit_only_t<double>(h, s);
}

// Zero the 13 moment planes (and the FP32 compensation) on the nodes of the
// touched tiles only: a fixed grid takes the tiles of the touched list in
// turn (every tile after a far move).  Node column i belongs to tile min(i / tnx, ntx - 1), so a wall's last
// column joins the last tile.
template <typename R>
__global__ void __launch_bounds__(128) k_clear_touched(const int32_t *__restrict__ list, const int32_t *__restrict__ list_n,
                                                       const int32_t *__restrict__ far, int ntiles, int tnx, int tny,
                                                       int ntx, int nx, int ny, int nxn, int64_t nnode, R *__restrict__ M,
                                                       R *__restrict__ Mlo) {
    const bool all = far && (*far & 1);
    const int n = all ? ntiles : *list_n;
    for (int li = blockIdx.x; li < n; li += gridDim.x) {
        const int T = all ? li : list[li];
        const int tx = T % ntx, ty = T / ntx;
        const int i0 = tx * tnx, j0 = ty * tny;
        const int i1 = (tx == ntx - 1) ? nxn : min(i0 + tnx, nx);
        const int j1 = min(j0 + tny, ny);
        const int w = i1 - i0, nn = w * (j1 - j0);
        for (int k = threadIdx.x; k < nn * NMOM; k += blockDim.x) {
            const int m = k / nn, r = k - m * nn;
            const int jj = r / w, ii = r - jj * w;
            const int64_t o = (int64_t)m * nnode + (int64_t)(j0 + jj) * nxn + i0 + ii;
            M[o] = R(0);
            if (Mlo) Mlo[o] = R(0);
        }
    }
}

int clear_moments(pic_t *h) {
    size_t b = (size_t)NMOM * h->nnode * h->rs;
    if (cudaMemsetAsync(h->M, 0, b, h->st) != cudaSuccess) return check_launch("clear M");
    if (h->Mlo && cudaMemsetAsync(h->Mlo, 0, b, h->st) != cudaSuccess) return check_launch("clear Mlo");
    if (h->Mfix && cudaMemsetAsync(h->Mfix, 0, (size_t)NMOM * h->nnode * 8, h->st) != cudaSuccess)
        return check_launch("clear Mfix");
    return 0;
}

// A step's deposit adds into Mfix (deterministic) or into M and Mlo; the
// conversion after a deterministic deposit overwrites M and Mlo whole.  M is
// zero everywhere before each push: the previous push wrote only inside its
// touched tiles, and those are cleared here (everything after a deposit at
// rest, which keeps no touched-tile map).
int clear_step_moments(pic_t *h) {
    if (!h->det) {
        if (h->moments_cleared) {   // zeroed by the field solve that read them
            h->moments_cleared = false;
            return 0;
        }
        if (h->touch_all) return clear_moments(h);
        int dev = 0, nsm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        unsigned grid = (unsigned)(nsm > 0 ? 8 * nsm : 1024);
        if (grid > (unsigned)h->ntiles) grid = (unsigned)h->ntiles;
        const int32_t *list = h->touch_list + (size_t)h->touch_cur * h->ntiles;
        const int32_t *n = list_counters(h, h->touch_cur) + LC_TOUCH;
        if (h->fp32)
            k_clear_touched<float><<<grid, 128, 0, h->st>>>(list, n, h->touch_far, h->ntiles, h->tnx, h->tny, h->ntx,
                                                            h->nx, h->ny, h->nxn, h->nnode, (float *)h->M,
                                                            (float *)h->Mlo);
        else
            k_clear_touched<double><<<grid, 128, 0, h->st>>>(list, n, h->touch_far, h->ntiles, h->tnx, h->tny, h->ntx,
                                                             h->nx, h->ny, h->nxn, h->nnode, (double *)h->M, nullptr);
        count_launch(h);
        return check_launch("k_clear_touched");
    }
    if (cudaMemsetAsync(h->Mfix, 0, (size_t)NMOM * h->nnode * 8, h->st) != cudaSuccess)
        return check_launch("clear Mfix");
    return 0;
}

// Shares of a sum of |w|: thread and block totals in a fixed order.
__global__ void __launch_bounds__(256) k_abs_sum(const double *__restrict__ w, int64_t n, double *__restrict__ part) {
    __shared__ double sh[256];
    double a = 0.0;
    for (int64_t p = (int64_t)blockIdx.x * 256 + threadIdx.x; p < n; p += (int64_t)gridDim.x * 256) a += fabs(w[p]);
    sh[threadIdx.x] = a;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

int abs_sum(pic_t *h, const double *w, int64_t n, double *part) {
    k_abs_sum<<<ABS_SUM_BLOCKS, 256, 0, h->st>>>(w, n, part);
    count_launch(h);
    return check_launch("k_abs_sum");
}

// Class bounds from the weights loaded so far (see FixScale).
int fix_scale(const pic_t *h, FixScale *out) {
    double B[3] = {0, 0, 0};
    const double dt = h->cfg.dt;
    for (int s = 0; s < h->nsp; ++s) {
        const double q = h->sp[s].q, m = h->sp[s].m;
        B[0] += fabs(q) * h->wabs[s];
        B[1] += q * q * dt * dt / (4.0 * m) * h->wabs[s];
    }
    B[2] = B[0];
    for (int c = 0; c < 3; ++c) {
        int e = 0;
        if (B[c] > 0) {
            int x = 0;
            // B <= 2^x; a bound that is a power of two but for the order its sum was taken in (on the host or
            // the device) is taken as one
            frexp(B[c] * (1.0 + 0x1p-30), &x);
            e = 62 - x;
        }
        if (e < -120) {
            set_error("deterministic deposit: moment bound %g is too large for 64-bit fixed point", B[c]);
            return PIC_ERR_ARG;
        }
        if (e > 120) e = 120;
        out->e[c] = e;
        out->s[c] = ldexpf(1.0f, e);
        out->inv[c] = ldexp(1.0, -e);
    }
    return 0;
}

template <typename R>
static int fix_to_moments_t(pic_t *h) {
    FixScale fs;
    if (int rc = fix_scale(h, &fs)) return rc;
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int64_t n = (int64_t)NMOM * h->nnode;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 8 * (int64_t)nsm) blocks = 8 * (int64_t)nsm;
    k_fix_to_moments<R><<<(unsigned)blocks, 256, 0, h->st>>>(h->Mfix, (R *)h->M, (R *)h->Mlo, h->nnode, fs);
    count_launch(h);
    return check_launch("k_fix_to_moments");
}

int fix_to_moments(pic_t *h) { return h->fp32 ? fix_to_moments_t<float>(h) : fix_to_moments_t<double>(h); }

template <typename R>
static int load_convert_t(pic_t *h, int s, int buf, int64_t n, const double *const src[6], unsigned long long *bad,
                          bool over_link, const int32_t *csrc) {
    SpeciesBuf &S = h->sp[s];
    const double Lx = h->nx * h->cfg.dx, Ly = h->ny * h->cfg.dy;
    LoadSrc ls;
    for (int k = 0; k < 6; ++k) ls.a[k] = src[k];
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    // arrays read over the CPU-GPU link: half of the SMs; arrays in device memory: eight blocks per SM
    const int64_t cap = over_link ? LOAD_SM_PERMILLE * (int64_t)nsm / 1000 : 8 * (int64_t)nsm;
    int64_t blocks = (n + LOAD_BS - 1) / LOAD_BS;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    if (csrc)
        k_restore_convert<R><<<(unsigned)blocks, LOAD_BS, 0, h->st>>>(
            grid_args<double>(h), ls, csrc, n, S.cell[buf], (R *)S.ox[buf], (R *)S.oy[buf], (R *)S.ux[buf],
            (R *)S.uy[buf], (R *)S.uz[buf], (R *)S.w[buf], bad);
    else
        k_load_convert<R><<<(unsigned)blocks, LOAD_BS, 0, h->st>>>(
            grid_args<double>(h), Lx, Ly, ls, n, S.cell[buf], (R *)S.ox[buf], (R *)S.oy[buf], (R *)S.ux[buf],
            (R *)S.uy[buf], (R *)S.uz[buf], (R *)S.w[buf], bad);
    count_launch(h);
    return check_launch("k_load_convert");
}

int load_convert(pic_t *h, int s, int buf, int64_t n, const double *const src[6], unsigned long long *bad,
                 bool over_link, const int32_t *csrc) {
    if (n == 0) return 0;
    return h->fp32 ? load_convert_t<float>(h, s, buf, n, src, bad, over_link, csrc)
                   : load_convert_t<double>(h, s, buf, n, src, bad, over_link, csrc);
}

// *total += the particles of the tiles, a warp per tile.
__global__ void __launch_bounds__(256) k_count(const int32_t *__restrict__ bstart, const int32_t *__restrict__ useg,
                                               const int32_t *__restrict__ segn, int ntiles, int32_t *__restrict__ total) {
    __shared__ int sum;
    if (threadIdx.x == 0) sum = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    int c = 0;
    for (int t = blockIdx.x * 8 + (threadIdx.x >> 5); t < ntiles; t += gridDim.x * 8) {
        const int64_t sb = bstart[t] / SEG;
        const int u = useg[t];
        for (int j = lane; j < u; j += 32) c += segn[sb + j];
    }
    for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
    if (lane == 0 && c) atomicAdd(&sum, c);
    __syncthreads();
    if (threadIdx.x == 0 && sum) atomicAdd(total, sum);
}

static int read_count(pic_t *h, SpeciesBuf &S, const int32_t *src, int64_t *n_out) {
    int32_t tot = 0;
    cudaError_t e = cudaMemcpyAsync(&tot, src, sizeof(int32_t), cudaMemcpyDeviceToHost, h->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->st);
    if (e != cudaSuccess) {
        set_error("count readback: %s", cudaGetErrorString(e));
        return PIC_ERR_CUDA;
    }
    *n_out = tot;
    S.n = tot;
    S.n_exact = true;
    return 0;
}

// Live particles of a species (known on the host unless a step ran since): one sum over the segment
// counts (counts per tile and their scan, which only the export needs, took five launches: 23 us
// against 4 us on 8192 tiles, five times in an ionisation pass).
int count_species(pic_t *h, int s, int64_t *n_out) {
    SpeciesBuf &S = h->sp[s];
    if (S.cap == 0 || S.n_exact) {
        *n_out = S.cap == 0 ? 0 : S.n;
        return 0;
    }
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    int32_t *total = h->ticket + 2;   // (words 0 and 1: a deposit at rest)
    cudaMemsetAsync(total, 0, sizeof(int32_t), h->st);
    const int blocks = std::min((h->ntiles + 7) / 8, 8 * (nsm > 0 ? nsm : 1));
    k_count<<<blocks, 256, 0, h->st>>>(S.bstart, S.useg[S.scur], S.segn[S.scur], h->ntiles, total);
    count_launch(h);
    if (int rc = check_launch("k_count")) return rc;
    return read_count(h, S, total, n_out);
}

// The same with the tiles' compact starts in cstart.
static int count_starts(pic_t *h, int s, int64_t *n_out) {
    SpeciesBuf &S = h->sp[s];
    *n_out = 0;
    if (S.cap == 0) return 0;
    if (int rc = tile_counts(h, s)) return rc;
    if (int rc = scan_tiles(h, S.tcount, S.cstart)) return rc;
    return read_count(h, S, S.cstart + h->ntiles, n_out);
}

int ensure_stage_doubles(pic_t *h, int64_t ndoubles);

template <typename R>
static int to_stage_t(pic_t *h, int s, int64_t n, bool raw) {
    SpeciesBuf &S = h->sp[s];
    int b = S.bins;
    k_bins_to_stage<R><<<h->ntiles, 256, 0, h->st>>>(grid_args<double>(h), S.bstart, S.useg[S.scur], S.segn[S.scur],
                                                     S.cstart, n, S.cell[b],
                                                     (const R *)S.ox[b], (const R *)S.oy[b], (const R *)S.ux[b],
                                                     (const R *)S.uy[b], (const R *)S.uz[b], (const R *)S.w[b],
                                                     h->stage, raw);
    count_launch(h);
    return check_launch("k_bins_to_stage");
}

// Compact copy of species s into the staging buffer; *n_out = live count.
// raw: the stored in-cell offsets instead of global positions.
int particles_to_stage(pic_t *h, int s, int64_t *n_out, bool raw) {
    int64_t n = 0;
    if (int rc = count_starts(h, s, &n)) return rc;
    *n_out = n;
    if (n == 0) return 0;
    if (int rc = ensure_stage_doubles(h, 7 * n)) return rc;
    return h->fp32 ? to_stage_t<float>(h, s, n, raw) : to_stage_t<double>(h, s, n, raw);
}

}  // namespace pic
