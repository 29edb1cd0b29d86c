// Binary Coulomb collisions (the paper names collisions, with ionisation, as
// what drives its growing particle counts, Sections 4 and 5; it states no
// model).  Reading: the binary collision model of Takizuka and Abe (J. Comput.
// Phys. 25, 205, 1977) applied to u = p/(m c) as the velocity, with the weight
// rule of Nanbu and Yonemura (1998).  A pass runs, for each (species a,
// species b) of its list in turn, over the cells: the particles of a cell are
// consecutive in a species' order (tile, then cell), so a cell is a run of
// indices.  Like particles pair as (0,1), (2,3), ... (odd N >= 3: the first
// three as (0,1), (1,2), (2,0) at half the variance); unlike ones pair the
// driving species' particle i (the species with more particles in the cell, a
// on a tie) with particle i mod N_other of the other.  The pairs of a cell act as
// if run in that order, each seeing the previous pairs' updates: pairs that
// share no particle run in the lanes of the cell's warp at once.  Per pair
// (1, 2): g = u1 - u2, mu = m1 m2 / (m1 + m2), n_L = the cell density of the
// species (like) or the lower of the two (sum of w over dx dy), variance
// s2 = q1^2 q2^2 n_L lnL kappa dt / (2 mu^2 |g|^3) (kappa = r_e omega / c),
// delta = sqrt(s2) sqrt(-2 ln(1 - v0)) cos(2 pi v1), phi = 2 pi v2 and the
// rotation of g by the angle 2 atan(delta) about a random axis; u1 moves by
// m2/(m1+m2) dg when v3 < w2 / max(w1, w2), u2 by -m1/(m1+m2) dg when v3 <
// w1 / max(w1, w2).  v0..v3: Philox-4x64-10 at counter (index of the pair's
// first particle in its species' order, 16 + list position, step, 1), key
// (seed, 0).  Momentum and the kinetic energy sum m |u|^2 / 2 are conserved by
// every pair of equal weights.  The pass changes only u; the moments are
// redeposited at rest before they are next used.
#include <math.h>

#include "pic_internal.cuh"
#include "pic_philox.cuh"

namespace pic {

// A species seen cell by cell.  The particles of a tile are stored in cell
// order, so a cell's particles are one run [first[c], end[c]) of indices in the
// species' order (end[c] = 0: an empty cell).
template <typename R>
struct ColSpecies {
    const int32_t *first, *end;     // per grid cell
    const int32_t *tbase;           // per tile: index of its first particle
    const int32_t *bstart, *useg;
    const int32_t *pre;             // per segment: particles of its tile before it
    const uint8_t *dense;           // per tile: every segment but the last is full
    R *ux, *uy, *uz;
    const R *w;
};

// Cell runs of a species: per tile (one block), the segments' exclusive
// prefix, whether the tile is dense, and, where the cell changes, the ends of
// the runs.  list (or nullptr): the cells that hold particles, in any order.
__global__ void __launch_bounds__(256) k_col_cells(const int32_t *__restrict__ bstart, const int32_t *__restrict__ useg,
                                                   const int32_t *__restrict__ segn, const int32_t *__restrict__ cell,
                                                   const int32_t *__restrict__ tbase, int32_t *__restrict__ pre,
                                                   uint8_t *__restrict__ dense, int32_t *__restrict__ first,
                                                   int32_t *__restrict__ end, int32_t *__restrict__ list,
                                                   int32_t *__restrict__ list_n) {
    __shared__ int wsum[8], s_run, s_dense;
    const int t = blockIdx.x, u = useg[t];
    if (u == 0) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t b0 = bstart[t], sb = b0 / SEG;
    const int32_t base = tbase[t];
    if (threadIdx.x == 0) {
        s_run = 0;
        s_dense = 1;
    }
    __syncthreads();
    for (int j0 = 0; j0 < u; j0 += 256) {
        const int j = j0 + threadIdx.x;
        const int n = j < u ? segn[sb + j] : 0;
        if (j < u - 1 && n != SEG) s_dense = 0;
        int incl = n;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wsum[wid] = incl;
        __syncthreads();
        int before = s_run, tot = 0;
        for (int q = 0; q < 8; ++q) {
            if (q < wid) before += wsum[q];
            tot += wsum[q];
        }
        if (j < u) pre[sb + j] = before + incl - n;
        __syncthreads();
        if (threadIdx.x == 0) s_run += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) dense[t] = s_dense;
    // a warp per segment; the particles before and after a segment's ends lie in the nearest
    // non-empty segments of the tile
    for (int j = wid; j < u; j += 8) {
        const int n = segn[sb + j];
        if (n == 0) continue;
        const int64_t slot = b0 + (int64_t)j * SEG + lane;
        const int32_t c = lane < n ? cell[slot] : -1;
        int32_t cp = __shfl_up_sync(0xffffffffu, c, 1), cn = __shfl_down_sync(0xffffffffu, c, 1);
        if (lane == 0) {
            int k = j - 1;
            while (k >= 0 && segn[sb + k] == 0) --k;
            cp = k >= 0 ? cell[b0 + (int64_t)k * SEG + segn[sb + k] - 1] : -1;
        }
        if (lane == n - 1) {
            int k = j + 1;
            while (k < u && segn[sb + k] == 0) ++k;
            cn = k < u ? cell[b0 + (int64_t)k * SEG] : -1;
        }
        const int32_t i = base + pre[sb + j] + lane;
        const bool starts = lane < n && cp != c;
        if (starts) first[c] = i;
        if (lane < n && cn != c) end[c] = i + 1;
        if (list) {
            const unsigned m = __ballot_sync(0xffffffffu, starts);
            int at = 0;
            if (lane == 0 && m) at = atomicAdd(list_n, __popc(m));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (starts) list[at + __popc(m & ((1u << lane) - 1u))] = c;
        }
    }
}

template <typename R>
struct ColArgs {
    ColSpecies<R> A, B;
    const int32_t *list, *list_n;   // the cells holding particles of species a
    int like;
    int nx, tnx, tny, ntx;
    double f1, f2;                  // m_b / (m_a + m_b), m_a / (m_a + m_b)
    double cvar;                    // q_a^2 q_b^2 lnL kappa dt / (2 mu^2)
    double inv_area;
    int spec;
    int64_t step;
    uint64_t seed;
    unsigned long long *pairs;
    int *ticket;                    // batches taken (zero at the launch)
};

// A tile's part of the index -> slot map (the warp's cell lies in one tile).
struct ColTile {
    int32_t base, u;
    int64_t b0;
    const int32_t *pre;   // nullptr: dense
};

template <typename R>
__device__ inline ColTile col_tile(const ColSpecies<R> &S, int t) {
    ColTile k;
    k.base = S.tbase[t];
    k.b0 = S.bstart[t];
    k.u = S.useg[t];
    k.pre = S.dense[t] ? nullptr : S.pre + k.b0 / SEG;
    return k;
}

__device__ inline int64_t col_slot(const ColTile &k, int32_t index) {
    const int32_t i = index - k.base;
    if (!k.pre) return k.b0 + i;
    int lo = 0, hi = k.u;   // the last segment with pre <= i (an empty one shares its successor's pre)
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (k.pre[mid] <= i) lo = mid;
        else hi = mid;
    }
    return k.b0 + (int64_t)lo * SEG + (i - k.pre[lo]);
}

// One pair (1, 2), in FP64: particle 1 is driven, its index keys the draws.
// The FP64 pipe bounds the pass, so a pair takes two reciprocal square roots,
// one square root, one reciprocal and no further divisions: |g| and 1/|g|^3
// from rsqrt(g.g), one root of the product s2 (-2 ln(1 - v0)),
// 1 - cos = delta sin, the species' constants from the host, and the weight
// ratio only where the weights differ (of w1/wmax and w2/wmax one is 1, which
// a draw is always below).
template <typename R>
__device__ inline void col_pair(const ColSpecies<R> &S1, int64_t s1, const ColSpecies<R> &S2, int64_t s2, int32_t index,
                                const ColArgs<R> &a, double f1, double f2, double nL, bool half) {
    const double u1[3] = {(double)S1.ux[s1], (double)S1.uy[s1], (double)S1.uz[s1]};
    const double u2[3] = {(double)S2.ux[s2], (double)S2.uy[s2], (double)S2.uz[s2]};
    const double w1 = (double)S1.w[s1], w2 = (double)S2.w[s2];
    const double g[3] = {u1[0] - u2[0], u1[1] - u2[1], u1[2] - u2[2]};
    const double gp2 = g[0] * g[0] + g[1] * g[1], g2 = gp2 + g[2] * g[2];
    if (g2 == 0.0 || nL <= 0.0) return;
    uint64_t x[4] = {(uint64_t)index, (uint64_t)(16 + a.spec), (uint64_t)a.step, 1ull};
    philox4x64_10(x, a.seed, 0ull);
    const double ig = rsqrt(g2), gm = g2 * ig;
    double var = a.cvar * nL * (ig * ig * ig);
    if (half) var *= 0.5;
    const double de = sqrt(var * (-2.0 * log(1.0 - philox_uniform(x[0])))) * cospi(2.0 * philox_uniform(x[1]));
    double sp, cp;
    sincospi(2.0 * philox_uniform(x[2]), &sp, &cp);
    const double sT = 2.0 * de * rcp_r(1.0 + de * de), cT1 = de * sT;
    double dg[3];
    if (gp2 > 0.0) {
        const double igp = rsqrt(gp2), nx = g[0] * igp, ny = g[1] * igp;
        const double sc = sT * cp, ss = sT * sp * gm;
        dg[0] = nx * g[2] * sc - ny * ss - g[0] * cT1;
        dg[1] = ny * g[2] * sc + nx * ss - g[1] * cT1;
        dg[2] = -(gp2 * igp) * sc - g[2] * cT1;
    } else {
        dg[0] = gm * sT * cp;
        dg[1] = gm * sT * sp;
        dg[2] = -gm * cT1;
    }
    bool move1 = true, move2 = true;
    if (!(w1 == w2 && w1 > 0.0)) {
        const double wmax = w1 > w2 ? w1 : w2, v3 = philox_uniform(x[3]);
        move1 = v3 < w2 / wmax;
        move2 = v3 < w1 / wmax;
    }
    if (move1) {
        S1.ux[s1] = (R)(u1[0] + f1 * dg[0]);
        S1.uy[s1] = (R)(u1[1] + f1 * dg[1]);
        S1.uz[s1] = (R)(u1[2] + f1 * dg[2]);
    }
    if (move2) {
        S2.ux[s2] = (R)(u2[0] - f2 * dg[0]);
        S2.uy[s2] = (R)(u2[1] - f2 * dg[1]);
        S2.uz[s2] = (R)(u2[2] - f2 * dg[2]);
    }
}

// A cell of a warp's batch: the driving species (d) and the other (o): index
// of the first particle, count, slot of the first particle (-1: the tile is not
// dense, slots come from the segment prefix).  Like pairs: both are the species.
struct ColCell {
    double nL;
    int32_t sd, nd, ld, so, no, lo, tile, swapped;
};
constexpr int COL_BATCH = 16;
constexpr int COL_WARPS = 8;

template <typename R>
__device__ inline void col_run(const ColSpecies<R> &S, int t, int32_t s, int32_t n, int32_t &slot0, double &w) {
    const ColTile k = col_tile(S, t);
    slot0 = k.pre ? -1 : (int32_t)(k.b0 + (s - k.base));
    w = 0.0;
    for (int32_t i = 0; i < n; ++i) w += (double)S.w[slot0 >= 0 ? slot0 + i : col_slot(k, s + i)];
}

template <typename R>
__device__ inline int64_t col_at(const ColSpecies<R> &S, int32_t slot0, int32_t s, int32_t i, int t) {
    return slot0 >= 0 ? (int64_t)slot0 + i : col_slot(col_tile(S, t), s + i);
}

// A warp takes COL_BATCH cells of the list at a time and runs their pairs in
// phases of pairs that share no particle, the phase's pairs of all its cells
// spread over the lanes.  Like pairs: (0,1) of the odd cells' triple with every
// other pair, then the triples' (1,2), then their (2,0).  Unlike pairs: phase r
// takes the driving particles r n_o .. (r + 1) n_o - 1 (particle t meets the
// other species' t mod n_o).  The FP64 pipe bounds the pass and is busy for a
// whole warp however few lanes take part, so the lanes are kept full: one warp
// per cell (16 pairs in 32 lanes, the triple alone for two thirds of an odd
// cell's time) took 0.83 ms per entry on a foil of 51,200 cells x 32 particles,
// one thread per cell 0.91 ms.
template <typename R>
__global__ void __launch_bounds__(32 * COL_WARPS) k_collide(const __grid_constant__ ColArgs<R> a) {
    __shared__ ColCell s_cell[COL_WARPS][COL_BATCH];
    __shared__ int s_pfx[COL_WARPS][COL_BATCH + 1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nc = *a.list_n;
    ColCell *cells = s_cell[wid];
    int *pfx = s_pfx[wid];
    unsigned long long np = 0;
    for (;;) {
        int b = 0;
        if (lane == 0) b = atomicAdd(a.ticket, 1);
        b = __shfl_sync(0xffffffffu, b, 0);
        if ((int64_t)b * COL_BATCH >= nc) break;
        const int n = min(COL_BATCH, nc - b * COL_BATCH);
        int32_t nd = 0, no = 0;   // lane l < n: counts of cell l
        if (lane < n) {
            const int32_t c = a.list[b * COL_BATCH + lane];
            const int cx = c % a.nx, cy = c / a.nx;
            ColCell k;
            k.tile = (cy / a.tny) * a.ntx + cx / a.tnx;
            k.swapped = 0;
            const int32_t s = a.A.first[c], na = a.A.end[c] - s;
            double wa = 0.0, wb = 0.0;
            if (a.like) {
                col_run(a.A, k.tile, s, na, k.ld, wa);
                k.sd = k.so = s;
                k.nd = k.no = na;
                k.lo = k.ld;
                k.nL = wa * a.inv_area;
            } else {
                const int32_t eb = a.B.end[c];
                const int32_t sb = eb ? a.B.first[c] : 0, nb = eb - sb;
                int32_t la = -1, lb = -1;
                if (nb > 0) {
                    col_run(a.A, k.tile, s, na, la, wa);
                    col_run(a.B, k.tile, sb, nb, lb, wb);
                }
                k.nL = (wa < wb ? wa : wb) * a.inv_area;
                k.swapped = na < nb;
                k.sd = k.swapped ? sb : s;
                k.nd = nb == 0 ? 0 : k.swapped ? nb : na;
                k.ld = k.swapped ? lb : la;
                k.so = k.swapped ? s : sb;
                k.no = k.swapped ? na : nb;
                k.lo = k.swapped ? la : lb;
            }
            nd = k.nd;
            no = k.no;
            cells[lane] = k;
        }
        for (int phase = 0;; ++phase) {
            int m;   // pairs of lane l's cell in this phase
            if (a.like) {
                const bool odd = (nd & 1) && nd >= 3;
                m = phase == 0 ? (odd ? 1 + (nd - 3) / 2 : nd / 2) : (odd ? 1 : 0);
            } else {
                const int64_t left = (int64_t)nd - (int64_t)phase * no;
                m = left <= 0 ? 0 : left < no ? (int)left : no;
            }
            int incl = m;
            for (int o = 1; o < COL_BATCH; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const int total = __shfl_sync(0xffffffffu, incl, COL_BATCH - 1);
            if (total == 0 || (a.like && phase == 3)) break;
            if (lane < COL_BATCH) pfx[lane + 1] = incl;
            if (lane == 0) pfx[0] = 0;
            __syncwarp();   // the cells, the prefix and the pairs of the phase before
            for (int p = lane; p < total; p += 32) {
                int q = 0;   // the largest cell with pfx[q] <= p
#pragma unroll
                for (int h = COL_BATCH / 2; h > 0; h >>= 1)
                    if (pfx[q + h] <= p) q += h;
                const ColCell &k = cells[q];
                const int j = p - pfx[q];
                if (a.like) {
                    const bool odd = k.nd & 1, three = odd && (phase > 0 || j == 0);
                    const int32_t i = three ? phase : odd ? 2 * j + 1 : 2 * j, i2 = phase == 2 ? 0 : i + 1;
                    col_pair(a.A, col_at(a.A, k.ld, k.sd, i, k.tile), a.A, col_at(a.A, k.ld, k.sd, i2, k.tile), k.sd + i,
                             a, a.f1, a.f2, k.nL, three);
                } else {
                    const int32_t i = phase * k.no + j;
                    const ColSpecies<R> &D = k.swapped ? a.B : a.A, &O = k.swapped ? a.A : a.B;
                    col_pair(D, col_at(D, k.ld, k.sd, i, k.tile), O, col_at(O, k.lo, k.so, j, k.tile), k.sd + i, a,
                             k.swapped ? a.f2 : a.f1, k.swapped ? a.f1 : a.f2, k.nL, false);
                }
            }
            np += total;
            __syncwarp();   // before the prefix is rewritten, and the phases in order
        }
        __syncwarp();   // before the cells are rewritten
    }
    if (lane == 0 && np) atomicAdd(a.pairs, np);
}

// Cell runs of one species in stream-ordered scratch (one allocation).
struct ColMaps {
    char *mem = nullptr;
    int32_t *first = nullptr, *end = nullptr, *list = nullptr, *list_n = nullptr, *pre = nullptr, *tbase = nullptr;
    uint8_t *dense = nullptr;
};

static int col_maps(pic_t *h, int s, ColMaps &m) {
    SpeciesBuf &S = h->sp[s];
    const size_t nc = (size_t)h->nx * h->ny, nseg = (size_t)(S.cap / SEG), nt = (size_t)h->ntiles + 1;
    // end and list_n (cleared), first, list, pre, tbase, dense
    const size_t words = 3 * nc + 1 + nseg + nt + (nt + 3) / 4;
    if (cudaMallocAsync((void **)&m.mem, words * sizeof(int32_t), h->st) != cudaSuccess) {
        cudaGetLastError();
        set_error("pic_collide: scratch allocation failed");
        return PIC_ERR_OOM;
    }
    m.end = (int32_t *)m.mem;
    m.list_n = m.end + nc;
    m.first = m.list_n + 1;
    m.list = m.first + nc;
    m.pre = m.list + nc;
    m.tbase = m.pre + nseg;
    m.dense = (uint8_t *)(m.tbase + nt);
    cudaMemsetAsync(m.end, 0, (nc + 1) * sizeof(int32_t), h->st);
    if (int rc = tile_counts(h, s)) return rc;
    if (int rc = scan_tiles(h, S.tcount, m.tbase)) return rc;
    k_col_cells<<<h->ntiles, 256, 0, h->st>>>(S.bstart, S.useg[S.scur], S.segn[S.scur], S.cell[S.bins], m.tbase, m.pre,
                                              m.dense, m.first, m.end, m.list, m.list_n);
    count_launch(h);
    return check_launch("k_col_cells");
}

template <typename R>
static ColSpecies<R> col_species(pic_t *h, int s, const ColMaps &m) {
    SpeciesBuf &S = h->sp[s];
    ColSpecies<R> c;
    const int b = S.bins;
    c.first = m.first;
    c.end = m.end;
    c.tbase = m.tbase;
    c.bstart = S.bstart;
    c.useg = S.useg[S.scur];
    c.pre = m.pre;
    c.dense = m.dense;
    c.ux = (R *)S.ux[b];
    c.uy = (R *)S.uy[b];
    c.uz = (R *)S.uz[b];
    c.w = (const R *)S.w[b];
    return c;
}

template <typename R>
static int collide_t(pic_t *h, const pic_collisions *p, unsigned long long *d_pairs) {
    // a pass changes only u: each species' cell runs are made once, for all the entries that use it
    ColMaps maps[PIC_MAX_SPECIES];
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    int rc = 0;
    for (int k = 0; k < p->n_pairs && !rc; ++k) {
        const int sa = p->a[k], sb = p->b[k];
        if (h->sp[sa].cap == 0 || h->sp[sb].cap == 0) continue;
        for (int s : {sa, sb})
            if (!rc && !maps[s].mem) rc = col_maps(h, s, maps[s]);
        if (rc) break;
        const double m1 = h->sp[sa].m, m2 = h->sp[sb].m, q1 = h->sp[sa].q, q2 = h->sp[sb].q;
        const double mu = m1 * m2 / (m1 + m2);
        ColArgs<R> a;
        a.A = col_species<R>(h, sa, maps[sa]);
        a.B = col_species<R>(h, sb, maps[sb]);
        a.list = maps[sa].list;
        a.list_n = maps[sa].list_n;
        a.like = (sb == sa) ? 1 : 0;
        a.nx = h->nx;
        a.tnx = h->tnx;
        a.tny = h->tny;
        a.ntx = h->ntx;
        a.f1 = m2 / (m1 + m2);
        a.f2 = m1 / (m1 + m2);
        a.cvar = q1 * q1 * q2 * q2 * p->ln_lambda * p->kappa * h->cfg.dt / (2.0 * mu * mu);
        a.inv_area = 1.0 / (h->cfg.dx * h->cfg.dy);
        a.spec = k;
        a.step = h->step;
        a.seed = p->seed;
        a.pairs = d_pairs;
        a.ticket = (int *)(d_pairs + 1) + k;
        k_collide<R><<<(unsigned)(2 * (nsm > 0 ? nsm : 128)), 32 * COL_WARPS, 0, h->st>>>(a);
        count_launch(h);
        rc = check_launch("k_collide");
    }
    for (ColMaps &m : maps)
        if (m.mem) cudaFreeAsync(m.mem, h->st);
    return rc;
}

int collide(pic_t *h, const pic_collisions *p, unsigned long long *d_pairs) {
    return h->fp32 ? collide_t<float>(h, p, d_pairs) : collide_t<double>(h, p, d_pairs);
}

}  // namespace pic
