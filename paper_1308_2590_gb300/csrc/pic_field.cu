// Field solve (Section 2, Eqs. 4-5; Section 3.3 steps 3-9 without the
// inter-processor messages): E at the nodes, H at the cell centres.
//
// literal mode: per node (I + S) E^{n+1} = (I - S) E^n + dt (curl_h H - dj)
//               with a closed-form 3x3 inverse, walls by a first-order Mur
//               condition and the incident plane wave at x = 0, then
//               H^{n+3/2} = H^{n+1/2} - dt curl_e E^{n+1}.
// CN mode:      (I + S) X + (dt/2)^2 curl_h curl_e X = E^n + (dt/2)(curl_h H^n - dj)
//               solved inside one kernel (a cooperative grid or one cluster)
//               by FP64 iterative refinement around FP32 corrections
//               (preconditioned BiCGSTAB, or the preconditioner alone), then
//               E^{n+1} = 2X - E^n, H^{n+1} = H^n - dt curl_e X.
// All kernels are bandwidth-bound stencils over node/cell arrays of V4.
#include <cooperative_groups.h>
#include <math.h>
#include <stdio.h>

#include "pic_internal.cuh"

namespace cg = cooperative_groups;

namespace pic {

// Closed-form solution of A z = r (A 3x3) by the adjugate.
template <typename R>
__device__ inline void solve3(const R a[9], const R r[3], R z[3]) {
    R c00 = a[4] * a[8] - a[5] * a[7];
    R c01 = a[5] * a[6] - a[3] * a[8];
    R c02 = a[3] * a[7] - a[4] * a[6];
    R det = a[0] * c00 + a[1] * c01 + a[2] * c02;
    R id = R(1) / det;
    z[0] = (c00 * r[0] + (a[2] * a[7] - a[1] * a[8]) * r[1] + (a[1] * a[5] - a[2] * a[4]) * r[2]) * id;
    z[1] = (c01 * r[0] + (a[0] * a[8] - a[2] * a[6]) * r[1] + (a[2] * a[3] - a[0] * a[5]) * r[2]) * id;
    z[2] = (c02 * r[0] + (a[1] * a[6] - a[0] * a[7]) * r[1] + (a[0] * a[4] - a[1] * a[3]) * r[2]) * id;
}

// curl_h of cell-centred H at interior node (i, j): centred differences over
// the four cells sharing the node (a = (i,j), b = (i-1,j), c = (i,j-1),
// d = (i-1,j-1)), averaged transversely.  With the diagonal differences
// p = a.z - d.z and q = b.z - c.z the two Hz derivatives are (p + q)/(2 dy)
// and (p - q)/(2 dx): returned are u = p + q, v = q - p, sy = 2 dx dHy/dx and
// sx = 2 dy dHx/dy (10 FP64 operations), so that
// curl_h H = (u/(2 dy), v/(2 dx), sy/(2 dx) - sx/(2 dy)).  The FP64 pipe, not
// memory, bounds the FP64 field kernels on this GPU.
template <typename R>
__device__ inline void curl_h_parts(const GridArgs<R> &g, const V4<R> *__restrict__ H, int i, int j, R &u, R &v, R &sy,
                                    R &sx) {
    int im = (i == 0) ? g.nx - 1 : i - 1;
    int jm = (j == 0) ? g.ny - 1 : j - 1;
    V4<R> a = H[(int64_t)j * g.nx + i], b = H[(int64_t)j * g.nx + im];
    V4<R> c = H[(int64_t)jm * g.nx + i], d = H[(int64_t)jm * g.nx + im];
    const R pz = a.z - d.z, qz = b.z - c.z;
    u = pz + qz;
    v = qz - pz;
    sy = (a.y - d.y) + (c.y - b.y);
    sx = (a.x - d.x) + (b.x - c.x);
}

// Node tiles of the touched-tile map (nullptr: every tile may hold moments).
// clr / clr_lo (or nullptr): the moment planes (and compensation planes)
// that the E solve zeroes on the touched tiles once it has read them, so that
// the next push deposits into cleared moments without a pass of its own.
template <typename R>
struct TouchArgs {
    const uint8_t *touched;
    const int32_t *far;    // (or nullptr) the push's flags: bit 0, a far move, and every tile may hold moments
    int tnx, tny, ntx;
    R *clr, *clr_lo;
};

template <typename R>
__device__ inline void clear_node_moments(const GridArgs<R> &g, const TouchArgs<R> &tm, int64_t node) {
#pragma unroll
    for (int k = 0; k < NMOM; ++k) {
        tm.clr[(int64_t)k * g.nnode + node] = R(0);
        if (tm.clr_lo) tm.clr_lo[(int64_t)k * g.nnode + node] = R(0);
    }
}

// A padded node's value with its images in the ghost ring: periodic copies in y
// (and x when periodic); beyond a wall the ring stays zero.
template <typename R>
__device__ inline void store_padded(V4<R> *__restrict__ F, const GridArgs<R> &g, int i, int j, const V4<R> &v) {
    F[pidx(g, i, j)] = v;
    const bool edge_y = j < g.G || j >= g.ny - g.G, edge_x = g.periodic_x && (i < g.G || i >= g.nxn - g.G);
    if (!edge_y && !edge_x) return;
    int j0 = j, i0 = i;   // the first images inside the ring
    while (j0 - g.ny >= -g.G) j0 -= g.ny;
    if (g.periodic_x)
        while (i0 - g.nxn >= -g.G) i0 -= g.nxn;
    for (int jj = j0; jj < g.ny + g.G; jj += g.ny)
        for (int ii = i0; ii < g.nxn + g.G; ii += g.nxn) {
            F[pidx(g, ii, jj)] = v;
            if (!g.periodic_x) break;
        }
}

struct Inc {
    double new0[3], old0[3], new1[3], old1[3];
};

// Eq. 4 at the nodes, a thread per node (a walk down the rows that shares the
// curl's vertical halves left the few warps over the plasma, which read moments
// and solve, running alone: 540 us).  The FP64 pipe bounds the FP64 form, so the
// factors dt/(2 dx), dt/(2 dy) go into the update's FMAs and the sum E^n + E^{n+1}
// that the push gathers is stored without its half (the push's factor has it):
// 17 operations per vacuum node instead of 23.  The FP32 form is bound by memory and
// forms the change first, so that E rounds once (chained FMAs round at its size
// two to three times).  4096 x 2048 nodes FP64, vacuum but
// for a thin foil: 472 -> 300 us (the two passes of H and B: 425 -> 339 us).
//
// Walls (reading of the missing boundary and source equations): the wall node is
// vacuum; Ex advances with the one-sided dHz/dy, Ey and Ez follow a first-order Mur
// condition on the outgoing field -- at x = 0 on the field minus the incident
// wave, which is added back.  The thread of the neighbour column does them.
template <typename R>
__global__ void __launch_bounds__(128, 6) k_field_E_literal(GridArgs<R> g, const V4<R> *__restrict__ E,
                                                         const V4<R> *__restrict__ H, const R *M, const R *Mlo,
                                                         V4<R> *__restrict__ Enew, V4<R> *__restrict__ Esum,
                                                         TouchArgs<R> tm, Inc inc, R kap) {
    const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x) + (g.periodic_x ? 0 : 1), j = blockIdx.y;
    if (i >= g.nx) return;
    const int64_t node = (int64_t)j * g.nxn + i;
    const uint8_t *map = tm.touched && !(tm.far && (*tm.far & 1)) ? tm.touched + (j / tm.tny) * tm.ntx : nullptr;
    const bool touched = !map || map[min(i / tm.tnx, tm.ntx - 1)];
    R u, v, sy, sx;
    curl_h_parts(g, H, i, j, u, v, sy, sx);   // curl_h H = (u/(2 dy), v/(2 dx), sy/(2 dx) - sx/(2 dy))
    const V4<R> e = E[node];
    V4<R> z;
    if (!touched) {
        // vacuum (S = 0, dj = 0 on every node of the tile): Eq. 4 reduces to E^{n+1} = E^n + dt curl_h H,
        // with no moment read and no 3x3 solve.  The same operations as the solve below on such a node
        // (where the 3x3 solve returns its right-hand side exactly), so a node's bits do not depend on
        // whether its tile was marked.
        if constexpr (sizeof(R) == 8) {
            z.x = fma_r(g.khy, u, e.x);
            z.y = fma_r(g.khx, v, e.y);
            z.z = fma_r(g.khx, sy, fma_r(-g.khy, sx, e.z));
        } else {
            z.x = fma_r(g.dt, u * g.hy, e.x);
            z.y = fma_r(g.dt, v * g.hx, e.y);
            z.z = fma_r(g.dt, fma_r(sy, g.hx, -(sx * g.hy)), e.z);
        }
    } else {
        const R ia = g.inv_dx * g.inv_dy;
        const R ev[3] = {e.x, e.y, e.z};
        R a[9], r[3], w[3];
#pragma unroll
        for (int row = 0; row < 3; ++row) {
            R s_e = R(0);
#pragma unroll
            for (int col = 0; col < 3; ++col) {
                const int64_t mi = (int64_t)(1 + 3 * row + col) * g.nnode + node;
                const R S = (Mlo ? M[mi] + Mlo[mi] : M[mi]) * ia;
                a[3 * row + col] = (row == col ? R(1) : R(0)) + S;
                s_e += ((row == col ? R(1) : R(0)) - S) * ev[col];
            }
            const int64_t ji = (int64_t)(10 + row) * g.nnode + node;
            const R m = Mlo ? M[ji] + Mlo[ji] : M[ji];
            if constexpr (sizeof(R) == 8) {
                r[row] = fma_r(-g.dt, m * ia, s_e);
            } else {
                const R c = row == 0 ? u * g.hy : row == 1 ? v * g.hx : fma_r(sy, g.hx, -(sx * g.hy));
                r[row] = fma_r(g.dt, fma_r(-m, ia, c), s_e);
            }
        }
        if constexpr (sizeof(R) == 8) {
            r[0] = fma_r(g.khy, u, r[0]);
            r[1] = fma_r(g.khx, v, r[1]);
            r[2] = fma_r(g.khx, sy, fma_r(-g.khy, sx, r[2]));
        }
        if (tm.clr) clear_node_moments(g, tm, node);   // read above by this thread only
        solve3(a, r, w);
        z.x = w[0];
        z.y = w[1];
        z.z = w[2];
    }
    z.w = R(0);
    Enew[node] = z;
    store_padded(Esum, g, i, j, V4<R>{e.x + z.x, e.y + z.y, e.z + z.z, R(0)});
    if (g.periodic_x) return;
    const int jm = (j == 0) ? g.ny - 1 : j - 1;
    if (i == 1) {
        const V4<R> e0 = E[node - 1];
        const R dz = H[(int64_t)j * g.nx].z - H[(int64_t)jm * g.nx].z;
        const R s0y = e0.y - (R)inc.old0[1], s1y = e.y - (R)inc.old1[1], n1y = z.y - (R)inc.new1[1];
        const R s0z = e0.z - (R)inc.old0[2], s1z = e.z - (R)inc.old1[2], n1z = z.z - (R)inc.new1[2];
        const V4<R> w{fma_r(g.dt, dz * g.inv_dy, e0.x), (R)inc.new0[1] + s1y + kap * (n1y - s0y),
                      (R)inc.new0[2] + s1z + kap * (n1z - s0z), R(0)};
        Enew[node - 1] = w;
        store_padded(Esum, g, 0, j, V4<R>{e0.x + w.x, e0.y + w.y, e0.z + w.z, R(0)});
        if (tm.clr && (!map || map[0])) clear_node_moments(g, tm, node - 1);   // (its moments are not read)
    }
    if (i == g.nx - 1) {
        const V4<R> eN = E[node + 1];
        const R dz = H[(int64_t)j * g.nx + g.nx - 1].z - H[(int64_t)jm * g.nx + g.nx - 1].z;
        const V4<R> w{fma_r(g.dt, dz * g.inv_dy, eN.x), e.y + kap * (z.y - eN.y), e.z + kap * (z.z - eN.z), R(0)};
        Enew[node + 1] = w;
        store_padded(Esum, g, g.nx, j, V4<R>{eN.x + w.x, eN.y + w.y, eN.z + w.z, R(0)});
        if (tm.clr && (!map || map[tm.ntx - 1])) clear_node_moments(g, tm, node + 1);
    }
}

// Differences of a row's y and z to the next column's (the next lane's).
template <typename R>
struct RowDiff {
    R y, z;
};
template <typename R>
__device__ inline RowDiff<R> row_diff(const V4<R> &e) {
    return RowDiff<R>{__shfl_down_sync(0xffffffffu, e.y, 1) - e.y, __shfl_down_sync(0xffffffffu, e.z, 1) - e.z};
}

constexpr int FIELD_WARPS = 4;   // warps of a block of k_field_HB, each with rows of its own
constexpr int HB_COLS = 30;      // columns a warp produces: the outer two lanes are their neighbours' only

// Eq. 5 and the node B of the new H in one pass: a warp walks down rows of
// HB_COLS columns, lane l holding E column c0 + l.  H_out = H_in - dt curl_e(Ec)
// at the cells (kx = dt/(2 dx), ky = dt/(2 dy), the right neighbour's values by
// shuffles: 12 FP64 operations per cell).  Differences of neighbours come before
// any sum, as they are exact where the field is smooth: sums of two rows first
// would round at twice the size of E (FP32, fields of 1.5: H off by 1.5 half ulps
// instead of 1).  B = the sum
// of the four cells sharing the node, without its quarter (the deposits' factor
// has it; on a wall column twice the two inside cells): 6 operations per node
// instead of 12, and H is not read again.  A row of H above the strip is formed
// twice.  4096 x 2048 FP64: 227 + 198 us for the two
// passes before -> 339 us.
template <typename R, typename RE>
__global__ void __launch_bounds__(32 * FIELD_WARPS) k_field_HB(GridArgs<R> g, const V4<RE> *__restrict__ Ec,
                                                               const V4<R> *__restrict__ Hin, V4<R> *__restrict__ Hout,
                                                               V4<R> *__restrict__ Bp, RE kx, RE ky, int rows) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int i = (int)blockIdx.x * HB_COLS - 1 + lane;   // column of this lane's nodes and cells
    const int y0 = ((int)blockIdx.y * FIELD_WARPS + wid) * rows, y1 = min(y0 + rows, g.ny);
    if (y0 >= g.ny) return;   // (whole warps)
    int n = i, c = i;         // loaded columns of E and H
    if (g.periodic_x) {
        n = n < 0 ? g.nx - 1 : n >= g.nx ? n - g.nx : n;   // (i <= nx + 29: lanes past the end are not used,
        if (n >= g.nx) n = 0;                              //  but for column nx, which is column 0)
        c = n;
    } else {
        n = min(max(n, 0), g.nx);
        c = min(max(c, 0), g.nx - 1);
    }
    const bool node = lane > 0 && lane <= HB_COLS && i < g.nxn, cell = lane > 0 && lane <= HB_COLS && i < g.nx;
    const int jb = y0 == 0 ? g.ny - 1 : y0 - 1;
    V4<RE> eb = Ec[(int64_t)jb * g.nxn + n], en = Ec[(int64_t)y0 * g.nxn + n];
    V4<R> hn = Hin[(int64_t)jb * g.nx + c];
    RowDiff<RE> db = row_diff(eb);
    V4<R> below{R(0), R(0), R(0), R(0)};   // the new H of the row above the strip, then of the previous row
    for (int j = y0 - 1; j < y1; ++j) {
        const V4<RE> ea = en;               // E rows j + 1 (ea) and j (eb), H row j
        const V4<R> h = hn;
        if (j + 1 < y1) {
            en = Ec[(int64_t)(j + 2 >= g.ny ? j + 2 - g.ny : j + 2) * g.nxn + n];
            hn = Hin[(int64_t)(j + 1) * g.nx + c];
        }
        // 2 dy dEz/dy and 2 dy dEx/dy over columns i and i + 1, 2 dx dEz/dx and 2 dx dEy/dx over rows j and j + 1
        const RowDiff<RE> da = row_diff(ea);
        const RE vz = ea.z - eb.z, vx = ea.x - eb.x;
        const RE zy = vz + __shfl_down_sync(0xffffffffu, vz, 1), xy = vx + __shfl_down_sync(0xffffffffu, vx, 1);
        const RE zx = da.z + db.z, yx = da.y + db.y;
        eb = ea;
        db = da;
        auto in = [](R x) -> RE {
            if constexpr (sizeof(RE) == 8) return widen(x);
            else return x;
        };
        auto out = [](RE x) -> R {
            if constexpr (sizeof(RE) == 8) return stored<R>(x);
            else return x;
        };
        const V4<R> w{out(fma(-ky, zy, in(h.x))), out(fma(kx, zx, in(h.y))), out(fma(ky, xy, fma(-kx, yx, in(h.z)))), R(0)};
        if (j >= y0) {
            if (cell) Hout[(int64_t)j * g.nx + i] = w;
            const V4<R> s{below.x + w.x, below.y + w.y, below.z + w.z, R(0)};   // cells (i, j - 1) and (i, j)
            const R lx = __shfl_up_sync(0xffffffffu, s.x, 1), ly = __shfl_up_sync(0xffffffffu, s.y, 1);
            const R lz = __shfl_up_sync(0xffffffffu, s.z, 1);
            if (node) {
                // the columns i - 1 and i of cells; on a wall the inside one twice (selected before the additions)
                const bool w0 = !g.periodic_x && i == 0, wn = !g.periodic_x && i == g.nx;
                store_padded(Bp, g, i, j, V4<R>{(wn ? lx : s.x) + (w0 ? s.x : lx), (wn ? ly : s.y) + (w0 ? s.y : ly),
                                                (wn ? lz : s.z) + (w0 ? s.z : lz), R(0)});
            }
        }
        below = w;
    }
}

// Node B of a given H (an overwritten field), in the same form: the sums of k_field_HB.
template <typename R>
__global__ void k_node_average(GridArgs<R> g, const V4<R> *__restrict__ Hc, V4<R> *__restrict__ Bp) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y;
    if (i >= g.nxn || j >= g.ny) return;
    int jm = (j == 0) ? g.ny - 1 : j - 1;
    auto column = [&](int c) {
        const V4<R> a = Hc[(int64_t)jm * g.nx + c], b = Hc[(int64_t)j * g.nx + c];
        return V4<R>{a.x + b.x, a.y + b.y, a.z + b.z, R(0)};
    };
    V4<R> o;
    if (!g.periodic_x && (i == 0 || i == g.nx)) {
        const V4<R> s = column(i == 0 ? 0 : g.nx - 1);
        o = V4<R>{R(2) * s.x, R(2) * s.y, R(2) * s.z, R(0)};
    } else {
        const V4<R> s = column(i), l = column((i == 0) ? g.nx - 1 : i - 1);
        o = V4<R>{s.x + l.x, s.y + l.y, s.z + l.z, R(0)};
    }
    store_padded(Bp, g, i, j, o);
}

// --------------------------------------------------------------------------- CN solver

// Mixed-precision solve.  The outer loop is iterative refinement in FP64:
// r = b - A x with FP64 moments and FP64 iterate, stop when |r| <= tol |b|;
// otherwise an FP32 block-Jacobi BiCGSTAB solves A d = r to a relative
// residual of CN_INNER_RTOL and x += d.  The FP32 operator differs from A
// by rounding (~1e-7 relative), far below 1/cond(A), so every refinement cuts
// the FP64 residual by about the inner tolerance.
// One axis of the spectral preconditioner's transforms: n points, lg = log2 n, or
// -1 where n is no power of two; then n is the product of the nf factors f.
constexpr int FFT_FACTORS = 12;
struct FftAxis {
    int n, lg, nf, f[FFT_FACTORS];
};

struct CNVec {
    V4<double> *x, *b;                              // FP64 iterate and right-hand side
    V4<double> *cc;                                 // FP64 residual: curl_e x at the cells
    V4<float> *d, *r, *r0, *p, *v, *s, *t, *ph, *sh;  // FP32 inner solve of A d = r
    float *minv;                                    // [9][nnode] block-Jacobi inverse
    float *S;                                       // [9][nnode] S / dA
    // spectral preconditioner (periodic): complex work arrays of nnode entries
    // and twiddles e^{-2 pi i t / n}, t <= n/2, for x and y
    float2 *FA, *FB, *GA, *GB, *twx, *twy;
    int fft, ly;
    FftAxis ax, ay;
    // line preconditioner (walls, ny a power of two): per column means of the
    // diagonal of S ([3][nxn]), the factors ([10][nxn][ny/2 + 1]) and the sweep
    // work ([6][nxn][ny/2 + 1]) of the per-mode block-tridiagonal solves
    float *scol, *lf, *lw;
    int line;
};

constexpr float CN_INNER_RTOL = 1e-4f;
constexpr int CN_MAX_OUTER = 30;

// A box with walls (the wall node is vacuum): the x row is X_x + (dt/2)^2
// (curl_h curl_e X)_x with the wall column's one-sided curl_h, i.e.
// 2 hy (Cz(ic, j) - Cz(ic, j-1)) of the inside cell column ic; the y and z
// rows are the time-centred Mur condition cw X_w + cv X_v (v the neighbour
// column, cw = 1/dt + 1/dx, cv = 1/dt - 1/dx).
struct WallRows {
    double cw, cv;
};

template <typename T>
__device__ inline T cell_curl_z(const V4<T> &e00, const V4<T> &e10, const V4<T> &e01, const V4<T> &e11, T hx, T hy) {
    return ((e10.y + e11.y) - (e00.y + e01.y)) * hx - ((e01.x + e11.x) - (e00.x + e10.x)) * hy;
}

template <typename T>
__device__ inline V4<T> apply_A_wall(const GridArgs<double> &g, const V4<T> *__restrict__ X, T c2, T hx, T hy, T cw,
                                     T cv, int i, int j) {
    const int ic = (i == 0) ? 0 : g.nx - 1, iv = (i == 0) ? 1 : g.nx - 1;
    const int jm = (j == 0) ? g.ny - 1 : j - 1, jp = (j + 1 == g.ny) ? 0 : j + 1;
    auto at = [&](int a, int b) { return X[(int64_t)b * g.nxn + a]; };
    const V4<T> m0 = at(ic, jm), m1 = at(ic + 1, jm), c0 = at(ic, j), c1 = at(ic + 1, j), p0 = at(ic, jp),
                p1 = at(ic + 1, jp);
    const T up = cell_curl_z(c0, c1, p0, p1, hx, hy), dn = cell_curl_z(m0, m1, c0, c1, hx, hy);
    const V4<T> xw = at(i, j), xv = at(iv, j);
    return V4<T>{xw.x + c2 * ((up - dn) * (T(2) * hy)), cw * xw.y + cv * xv.y, cw * xw.z + cv * xv.z, T(0)};
}

// (I + S) X + (dt/2)^2 curl_h curl_e X at node (i, j) (wall nodes: apply_A_wall);
// S9 points at the 9 planar S rows (stride nnode), each scaled by sc.
template <typename T>
__device__ inline V4<T> apply_A(const GridArgs<double> &g, const V4<T> *__restrict__ X, const T *__restrict__ S9,
                                T sc, T c2, T hx, T hy, int i, int j, T cw = T(0), T cv = T(0)) {
    if (!g.periodic_x && (i == 0 || i == g.nx)) return apply_A_wall<T>(g, X, c2, hx, hy, cw, cv, i, j);
    int im = (i == 0) ? g.nx - 1 : i - 1, ip = (g.periodic_x && i + 1 == g.nx) ? 0 : i + 1;
    int jm = (j == 0) ? g.ny - 1 : j - 1, jp = (j + 1 == g.ny) ? 0 : j + 1;
    const int xs[3] = {im, i, ip};
    const int ys[3] = {jm, j, jp};
    V4<T> n[3][3];
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int a = 0; a < 3; ++a) n[b][a] = X[(int64_t)ys[b] * g.nxn + xs[a]];
    // curl_e at the four cells around the node; cell (ci, cj) has corners n[cj][ci..ci+1], n[cj+1][...]
    T Cx[2][2], Cy[2][2], Cz[2][2];
#pragma unroll
    for (int cj = 0; cj < 2; ++cj)
#pragma unroll
        for (int ci = 0; ci < 2; ++ci) {
            const V4<T> &e00 = n[cj][ci], &e10 = n[cj][ci + 1], &e01 = n[cj + 1][ci], &e11 = n[cj + 1][ci + 1];
            T dEz_dy = ((e01.z + e11.z) - (e00.z + e10.z)) * hy;
            T dEz_dx = ((e10.z + e11.z) - (e00.z + e01.z)) * hx;
            T dEy_dx = ((e10.y + e11.y) - (e00.y + e01.y)) * hx;
            T dEx_dy = ((e01.x + e11.x) - (e00.x + e10.x)) * hy;
            Cx[cj][ci] = dEz_dy;
            Cy[cj][ci] = -dEz_dx;
            Cz[cj][ci] = dEy_dx - dEx_dy;
        }
    // curl_h at the node from cells a = [1][1], b = [1][0], c = [0][1], d = [0][0]
    T kx = ((Cz[1][1] + Cz[1][0]) - (Cz[0][1] + Cz[0][0])) * hy;
    T ky = -(((Cz[1][1] + Cz[0][1]) - (Cz[1][0] + Cz[0][0])) * hx);
    T kz = ((Cy[1][1] + Cy[0][1]) - (Cy[1][0] + Cy[0][0])) * hx - ((Cx[1][1] + Cx[1][0]) - (Cx[0][1] + Cx[0][0])) * hy;
    int64_t node = (int64_t)j * g.nxn + i;
    const V4<T> &xc = n[1][1];
    T S[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) S[k] = S9[(int64_t)k * g.nnode + node] * sc;
    V4<T> y;
    y.x = xc.x + (S[0] * xc.x + S[1] * xc.y + S[2] * xc.z) + c2 * kx;
    y.y = xc.y + (S[3] * xc.x + S[4] * xc.y + S[5] * xc.z) + c2 * ky;
    y.z = xc.z + (S[6] * xc.x + S[7] * xc.y + S[8] * xc.z) + c2 * kz;
    y.w = T(0);
    return y;
}

// The FP64 residual's operator in two passes: curl_e of X once per cell (cell
// (ci, cj) has corners (ci, cj), (ci+1, cj), (ci, cj+1), (ci+1, cj+1),
// periodic), then per node curl_h of those cell values, S X and X.  The FP64 pipe
// bounds the residual, so the derivatives come from diagonal differences
// (curl_h_parts), the factors of curl_h and (dt/2)^2 are one constant per axis,
// and the moments are scaled by the inverse area once per row.
__device__ inline V4<double> cell_curl_e(const GridArgs<double> &g, const V4<double> *__restrict__ X, double hx,
                                         double hy, int ci, int cj) {
    const int ip = (g.periodic_x && ci + 1 == g.nx) ? 0 : ci + 1, jp = (cj + 1 == g.ny) ? 0 : cj + 1;
    const V4<double> e00 = X[(int64_t)cj * g.nxn + ci], e10 = X[(int64_t)cj * g.nxn + ip];
    const V4<double> e01 = X[(int64_t)jp * g.nxn + ci], e11 = X[(int64_t)jp * g.nxn + ip];
    const double pz = e11.z - e00.z, qz = e01.z - e10.z;
    const double sy = (e11.y - e00.y) + (e10.y - e01.y);   // 2 dx dEy/dx
    const double sx = (e11.x - e00.x) + (e01.x - e10.x);   // 2 dy dEx/dy
    return V4<double>{(pz + qz) * hy, (qz - pz) * hx, fma(sy, hx, -(sx * hy)), 0.0};
}

// kx = c2 hx, ky = c2 hy
__device__ inline V4<double> apply_A_from_cells(const GridArgs<double> &g, const V4<double> *__restrict__ X,
                                                const V4<double> *__restrict__ Cc, const double *__restrict__ S9,
                                                double sc, double kx, double ky, int i, int j, double cw, double cv) {
    if (!g.periodic_x && (i == 0 || i == g.nx)) {   // wall node (apply_A_wall with the cells' curls)
        const int jm = (j == 0) ? g.ny - 1 : j - 1;
        const int ic = (i == 0) ? 0 : g.nx - 1, iv = (i == 0) ? 1 : g.nx - 1;
        const double up = Cc[(int64_t)j * g.nx + ic].z, dn = Cc[(int64_t)jm * g.nx + ic].z;
        const V4<double> xw = X[(int64_t)j * g.nxn + i], xv = X[(int64_t)j * g.nxn + iv];
        return V4<double>{fma(up - dn, 2.0 * ky, xw.x), cw * xw.y + cv * xv.y, cw * xw.z + cv * xv.z, 0.0};
    }
    double u, v, sy, sx;
    curl_h_parts(g, Cc, i, j, u, v, sy, sx);
    const int64_t node = (int64_t)j * g.nxn + i;
    const V4<double> xc = X[node];
    const double *q = S9 + node;
    const int64_t st = g.nnode;
    V4<double> y;
    y.x = fma(fma(q[2 * st], xc.z, fma(q[st], xc.y, q[0] * xc.x)), sc, fma(u, ky, xc.x));
    y.y = fma(fma(q[5 * st], xc.z, fma(q[4 * st], xc.y, q[3 * st] * xc.x)), sc, fma(v, kx, xc.y));
    y.z = fma(fma(q[8 * st], xc.z, fma(q[7 * st], xc.y, q[6 * st] * xc.x)), sc, fma(sy, kx, fma(-sx, ky, xc.z)));
    y.w = 0.0;
    return y;
}

__device__ inline V4<float> apply_minv(const float *__restrict__ mi, int64_t nnode, int64_t node, const V4<float> &v) {
    float a[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) a[k] = mi[(int64_t)k * nnode + node];
    return V4<float>{a[0] * v.x + a[1] * v.y + a[2] * v.z, a[3] * v.x + a[4] * v.y + a[5] * v.z,
                     a[6] * v.x + a[7] * v.y + a[8] * v.z, 0.f};
}

template <typename T>
__device__ inline T dot(const V4<T> &a, const V4<T> &b) { return a.x * b.x + a.y * b.y + a.z * b.z; }

// ---- spectral preconditioner ------------------------------------------------
// On a periodic grid the operator (1 + s) X + c2 curl_h curl_e X with a
// uniform s is diagonal in Fourier space: for the mode e^{i(a i + b j)}, with
// p = (e^{ia} - 1)(1 + e^{ib}) / (2 dx) and q = (1 + e^{ia})(e^{ib} - 1) / (2 dy)
// (the symbols of d/dx and d/dy from nodes to cells), curl_h curl_e acts as
// [[|q|^2, -q* p, 0], [-p* q, |p|^2, 0], [0, 0, |p|^2 + |q|^2]].  The
// preconditioner solves that 3x3 system per mode with s = the grid mean of the
// diagonal of S, using FP32 FFTs; x and y share one complex transform (x + i y).

__device__ inline float2 cmul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }

// Barrier over all the blocks of the solve: a grid barrier (cooperative launch),
// or, when the whole grid is one thread-block cluster (small grids), the
// cluster barrier, which costs a fraction of it.
template <bool kCluster>
struct SolveBarrier {
    __device__ inline void sync() const {
        if constexpr (kCluster) cg::this_cluster().sync();
        else cg::this_grid().sync();
    }
};

// Twiddles of an n-point transform by stage, in shared memory: entries L - 1 +
// k, k < L, hold e^{-2 pi i k / (2 L)} for L = 1, 2, ..., n/2 (n - 1 entries),
// so that neighbouring threads of a stage read neighbouring words.
__device__ inline void fft_twiddles(float2 *tws, const float2 *__restrict__ tw, int n) {
    const int nh = n >> 1;
    for (int t = threadIdx.x; t < n - 1; t += blockDim.x) {
        const int lg = 31 - __clz(t + 1), L = 1 << lg, k = t - (L - 1);
        tws[t] = tw[k * (nh >> lg)];
    }
}

// FFT of nrow rows of n = 2^logn complex values (row r at r * rs of x), by the
// Stockham autosort form with radix-4 stages (and one of radix 2 first when
// logn is odd) between the two shared buffers x and y; on return x holds the
// result.  Stage L reads x[j + r n/4] (r = 0 .. 3, j = q L + k < n/4) and writes
// y[4 q L + k + s L].  Input and output in natural order; the inverse is not
// scaled.  Ends with a block barrier.
template <bool kInv>
__device__ inline void fft_core(float2 *&x, float2 *&y, int nrow, int rs, int n, int logn, const float2 *tws) {
    auto tw = [&](int i) {
        float2 w = tws[i];
        if (kInv) w.y = -w.y;
        return w;
    };
    int lg = 0;
    if (logn & 1) {
        const int nh = n >> 1;
        for (int e = threadIdx.x; e < nrow * nh; e += blockDim.x) {
            const int r = e >> (logn - 1), j = e & (nh - 1);
            const float2 a = x[r * rs + j], t = x[r * rs + j + nh];
            y[r * rs + 2 * j] = make_float2(a.x + t.x, a.y + t.y);
            y[r * rs + 2 * j + 1] = make_float2(a.x - t.x, a.y - t.y);
        }
        __syncthreads();
        float2 *z = x;
        x = y;
        y = z;
        lg = 1;
    }
    const int n4 = n >> 2;
    for (; lg < logn; lg += 2) {
        const int L = 1 << lg;
        for (int e = threadIdx.x; e < nrow * n4; e += blockDim.x) {
            const int r = e >> (logn - 2), j = e & (n4 - 1), k = j & (L - 1);
            const float2 *xr = x + r * rs + j;
            float2 *yo = y + r * rs + ((j >> lg) << (lg + 2)) + k;
            const float2 w1 = tw(2 * L - 1 + k), w2 = tw(L - 1 + k), w3 = cmul(w1, w2);
            const float2 a0 = xr[0], a1 = cmul(w1, xr[n4]), a2 = cmul(w2, xr[2 * n4]), a3 = cmul(w3, xr[3 * n4]);
            const float2 t0 = make_float2(a0.x + a2.x, a0.y + a2.y), t1 = make_float2(a0.x - a2.x, a0.y - a2.y);
            const float2 t2 = make_float2(a1.x + a3.x, a1.y + a3.y), t3 = make_float2(a1.x - a3.x, a1.y - a3.y);
            yo[0] = make_float2(t0.x + t2.x, t0.y + t2.y);
            yo[2 * L] = make_float2(t0.x - t2.x, t0.y - t2.y);
            const float2 m = make_float2(t1.x + t3.y, t1.y - t3.x), q = make_float2(t1.x - t3.y, t1.y + t3.x);   // t1 -+ i t3
            yo[L] = kInv ? q : m;
            yo[3 * L] = kInv ? m : q;
        }
        __syncthreads();
        float2 *z = x;
        x = y;
        y = z;
    }
}

// The same for any n = f[0] f[1] ...: a stage of radix r after those of product
// L takes y[q L r + k + t L] = sum over s of x[q L + k + s n/r] e^{-2 pi i s (k + t
// L) / (L r)}, an output at a time.  tws: e^{-2 pi i t / n}, t < n.
template <bool kInv>
__device__ inline void fft_core_any(float2 *&x, float2 *&y, int nrow, int rs, const FftAxis &ax, const float2 *tws) {
    const int n = ax.n;
    for (int st = 0, L = 1; st < ax.nf; ++st) {
        const int r = ax.f[st], Lr = L * r, step = n / r, ws = n / Lr;   // root ws k' of unity for k' of Lr
        for (int e = threadIdx.x; e < nrow * n; e += blockDim.x) {
            const int row = e / n, o = e - row * n, q = o / Lr, kt = o - q * Lr, k = kt % L;
            const float2 *xr = x + row * rs + q * L + k;
            float2 acc = xr[0];
            int w = 0;
            for (int s = 1; s < r; ++s) {
                w += kt * ws;
                if (w >= n) w -= n;
                float2 c = tws[w];
                if (kInv) c.y = -c.y;
                const float2 t = cmul(c, xr[s * step]);
                acc.x += t.x;
                acc.y += t.y;
            }
            y[row * rs + o] = acc;
        }
        __syncthreads();
        float2 *z = x;
        x = y;
        y = z;
        L = Lr;
    }
}

template <bool kInv>
__device__ inline void fft_axis(float2 *&x, float2 *&y, int nrow, int rs, const FftAxis &ax, const float2 *tws) {
    if (ax.lg >= 0) fft_core<kInv>(x, y, nrow, rs, ax.n, ax.lg, tws);
    else fft_core_any<kInv>(x, y, nrow, rs, ax, tws);
}

// Twiddles of an axis in shared memory (n entries), and e^{2 pi i k / n}, 0 <= k < n, from them.
__device__ inline void axis_twiddles(float2 *tws, const float2 *__restrict__ tw, const FftAxis &ax) {
    if (ax.lg >= 0) {
        fft_twiddles(tws, tw, ax.n);
        return;
    }
    for (int t = threadIdx.x; t < ax.n; t += blockDim.x) {
        float2 w = tw[min(t, ax.n - t)];
        if (2 * t > ax.n) w.y = -w.y;
        tws[t] = w;
    }
}
__device__ inline float2 axis_unit(const float2 *tws, const FftAxis &ax, int k) {
    if (ax.lg < 0) return make_float2(tws[k].x, -tws[k].y);
    const int h = ax.n >> 1;   // the last stage's entries
    const float2 w = tws[h - 1 + (k < h ? k : k - h)];
    return k < h ? make_float2(w.x, -w.y) : make_float2(-w.x, w.y);
}
__device__ inline int axis_div(int e, const FftAxis &ax) { return ax.lg >= 0 ? e >> ax.lg : e / ax.n; }
__device__ inline int axis_neg(int k, const FftAxis &ax) { return k == 0 ? 0 : ax.n - k; }

// Values of one row group of the transforms (short rows are taken several at
// a time, so that the threads have work between two barriers).
constexpr int FFT_GROUP = 2048;
__host__ __device__ inline int fft_buffer(int n, int columns) {   // float2 entries of one of the two buffers
    const int need = columns ? 2 * (n + 1) : n;
    return need > FFT_GROUP ? need : FFT_GROUP;
}

// In-place FFT of nrows rows of n values (row r of the first nrows_a rows in
// A, the rest in B); the line preconditioner's transforms.
__device__ inline void fft_rows(float2 *A, float2 *B, int nrows_a, int n, int logn, const float2 *__restrict__ tw,
                                bool inverse, float2 *sm) {
    const int G = fft_buffer(n, 0);
    float2 *tws = sm + 2 * G;
    fft_twiddles(tws, tw, n);
    __syncthreads();
    const int nrows = 2 * nrows_a;
    const int share = (nrows + gridDim.x - 1) / gridDim.x;
    const int rpb = max(1, min(G >> logn, share));
    for (int row0 = blockIdx.x * rpb; row0 < nrows; row0 += gridDim.x * rpb) {
        const int nr = min(rpb, nrows - row0);
        auto at = [&](int e) {
            const int row = row0 + (e >> logn);
            return (row < nrows_a ? A + (int64_t)row * n : B + (int64_t)(row - nrows_a) * n) + (e & (n - 1));
        };
        float2 *x = sm, *y = sm + G;
        for (int e = threadIdx.x; e < nr * n; e += blockDim.x) x[e] = *at(e);
        __syncthreads();
        if (inverse) fft_core<true>(x, y, nr, n, n, logn, tws);
        else fft_core<false>(x, y, nr, n, n, logn, tws);
        for (int e = threadIdx.x; e < nr * n; e += blockDim.x) *at(e) = x[e];
        __syncthreads();
    }
}

// out_a = in_a^T, out_b = in_b^T for R x C row-major arrays (32 x 32 tiles).
__device__ inline void transpose2(const float2 *in_a, const float2 *in_b, float2 *out_a, float2 *out_b, int R, int C,
                                  float2 *sm) {
    const int tr_n = (R + 31) / 32, tc_n = (C + 31) / 32, ntile = tr_n * tc_n;
    for (int tile = blockIdx.x; tile < 2 * ntile; tile += gridDim.x) {
        const float2 *in = tile < ntile ? in_a : in_b;
        float2 *out = tile < ntile ? out_a : out_b;
        const int tt = tile < ntile ? tile : tile - ntile;
        const int tr = tt / tc_n, tc = tt - tr * tc_n;
        for (int e = threadIdx.x; e < 1024; e += blockDim.x) {
            const int ty = e >> 5, tx = e & 31, r = tr * 32 + ty, c = tc * 32 + tx;
            if (r < R && c < C) sm[ty * 33 + tx] = in[(int64_t)r * C + c];
        }
        __syncthreads();
        for (int e = threadIdx.x; e < 1024; e += blockDim.x) {
            const int ty = e >> 5, tx = e & 31, c = tc * 32 + ty, r = tr * 32 + tx;
            if (r < R && c < C) out[(int64_t)c * R + r] = sm[tx * 33 + ty];
        }
        __syncthreads();
    }
}

// One application takes three passes over the grid, with a barrier between
// them: transforms along x of x + i y and z row by row (the first pass also
// forms the vector, load(n) = its value at node n); then, column by column, the
// transform along y, the modes' 3x3 systems and the transform back; then the
// transforms back along x.  The columns kx and -kx, which the modes of the two
// real fields in x + i y couple, are taken by the same block.  (Transposing the
// arrays around the transforms along y, with passes of their own, took five
// barriers and four more passes.)  Shared memory: two buffers, then the
// twiddles of x and of y (fft_tables).
struct FftShared {
    float2 *buf0, *buf1, *twx, *twy;
    int G;
};

__host__ __device__ inline int spectral_buffer(int nx, int ny) {
    const int a = fft_buffer(2 * nx, 0), b = fft_buffer(ny, 1);
    return a > b ? a : b;
}

__device__ inline FftShared fft_shared(const GridArgs<double> &g, float2 *sm) {
    FftShared f;
    f.G = spectral_buffer(g.nx, g.ny);
    f.buf0 = sm;
    f.buf1 = sm + f.G;
    f.twx = sm + 2 * f.G;
    f.twy = f.twx + g.nx;
    return f;
}

template <typename Load>
__device__ inline void spectral_rows(const GridArgs<double> &g, const CNVec &v, const FftShared &f, const Load &load) {
    const int nx = g.nx;
    const int rpb = max(1, min(f.G / (2 * nx), (g.ny + (int)gridDim.x - 1) / (int)gridDim.x));
    for (int y0 = blockIdx.x * rpb; y0 < g.ny; y0 += gridDim.x * rpb) {
        const int nr = min(rpb, g.ny - y0), m = nr * nx;
        const int64_t n0 = (int64_t)y0 * nx;
        float2 *x = f.buf0, *y = f.buf1;
        for (int e = threadIdx.x; e < m; e += blockDim.x) {
            const V4<float> q = load(n0 + e);
            x[e] = make_float2(q.x, q.y);
            x[m + e] = make_float2(q.z, 0.f);
        }
        __syncthreads();
        fft_axis<false>(x, y, 2 * nr, nx, v.ax, f.twx);
        for (int e = threadIdx.x; e < m; e += blockDim.x) {
            v.FA[n0 + e] = x[e];
            v.FB[n0 + e] = x[m + e];
        }
        __syncthreads();
    }
}

template <typename Store>
__device__ inline void spectral_rows_back(const GridArgs<double> &g, const CNVec &v, const FftShared &f, const Store &store) {
    const int nx = g.nx;
    const int rpb = max(1, min(f.G / (2 * nx), (g.ny + (int)gridDim.x - 1) / (int)gridDim.x));
    for (int y0 = blockIdx.x * rpb; y0 < g.ny; y0 += gridDim.x * rpb) {
        const int nr = min(rpb, g.ny - y0), m = nr * nx;
        const int64_t n0 = (int64_t)y0 * nx;
        float2 *x = f.buf0, *y = f.buf1;
        for (int e = threadIdx.x; e < m; e += blockDim.x) {
            x[e] = v.FA[n0 + e];
            x[m + e] = v.FB[n0 + e];
        }
        __syncthreads();
        fft_axis<true>(x, y, 2 * nr, nx, v.ax, f.twx);
        for (int e = threadIdx.x; e < m; e += blockDim.x) store(n0 + e, V4<float>{x[e].x, x[e].y, x[m + e].x, 0.f});
        __syncthreads();
    }
}

__device__ inline void spectral_columns(const GridArgs<double> &g, const CNVec &v, const FftShared &f, float c2, float sx,
                                        float sy, float sz) {
    const int nx = g.nx, ny = g.ny, rs = ny + 1, npair = nx / 2 + 1;
    const int per = max(1, min(f.G / (2 * rs), (npair + (int)gridDim.x - 1) / (int)gridDim.x));
    const float ihx = 0.5f * (float)g.inv_dx, ihy = 0.5f * (float)g.inv_dy, inv_n = 1.f / (float)((int64_t)nx * ny);
    // p = (e^{ia} - 1)(1 + e^{ib}) / (2 dx), q = (1 + e^{ia})(e^{ib} - 1) / (2 dy)
    auto symbols = [&](int kx, int ky, float2 &p, float2 &q) {
        const float2 a = axis_unit(f.twx, v.ax, kx), b = axis_unit(f.twy, v.ay, ky);
        p = cmul(make_float2(a.x - 1.f, a.y), make_float2(b.x + 1.f, b.y));
        q = cmul(make_float2(a.x + 1.f, a.y), make_float2(b.x - 1.f, b.y));
        p = make_float2(p.x * ihx, p.y * ihx);
        q = make_float2(q.x * ihy, q.y * ihy);
    };
    for (int c0 = blockIdx.x * per; c0 < npair; c0 += gridDim.x * per) {
        const int nc = min(per, npair - c0), ns = 2 * nc;   // slots: columns c0 .. c0 + nc - 1, then their partners
        auto column = [&](int s) { return s < nc ? c0 + s : axis_neg(c0 + s - nc, v.ax); };
        auto own = [&](int s) { return s < nc || column(s) != c0 + s - nc; };   // (0 and, for an even nx, nx/2 are their own partners)
        // both fields at once where the buffers hold them (short columns: fewer rounds of latency)
        const int nf = 2 * ns * rs <= f.G ? 2 : 1;
        for (int f0 = 0; f0 < 2; f0 += nf) {
            float2 *x = f.buf0, *y = f.buf1;
            for (int e = threadIdx.x; e < nf * ny * ns; e += blockDim.x) {
                const int r = e / ns, s = e - r * ns, fl = r >= ny ? 1 : 0, rr = r - fl * ny;
                x[(fl * ns + s) * rs + rr] = ((f0 + fl) ? v.FB : v.FA)[(int64_t)rr * nx + column(s)];
            }
            __syncthreads();
            fft_axis<false>(x, y, nf * ns, rs, v.ay, f.twy);
            if (f0 == 0) {
                for (int e = threadIdx.x; e < nc * ny; e += blockDim.x) {
                    const int s = axis_div(e, v.ay), ky = e - s * ny, mky = axis_neg(ky, v.ay), kx = c0 + s;
                    const bool self = column(nc + s) == kx;
                    if (self && ky > mky) continue;   // taken with its conjugate
                    float2 *F0 = x + s * rs + ky, *F1 = x + (self ? s : nc + s) * rs + mky;
                    const float2 Fk = *F0, Fm = *F1;
                    // X = (F + conj(Fm)) / 2, Y = (F - conj(Fm)) / (2i)
                    const float2 X = make_float2(0.5f * (Fk.x + Fm.x), 0.5f * (Fk.y - Fm.y));
                    const float2 Y = make_float2(0.5f * (Fk.y + Fm.y), -0.5f * (Fk.x - Fm.x));
                    float2 p, q;
                    symbols(kx, ky, p, q);
                    const float pp = p.x * p.x + p.y * p.y, qq = q.x * q.x + q.y * q.y;
                    const float2 cqp = cmul(make_float2(q.x, -q.y), p);   // conj(q) p
                    const float A11 = 1.f + sx + c2 * qq, A22 = 1.f + sy + c2 * pp;
                    const float2 A12 = make_float2(-c2 * cqp.x, -c2 * cqp.y), A21 = make_float2(A12.x, -A12.y);
                    const float idet = inv_n / (A11 * A22 - (A12.x * A12.x + A12.y * A12.y));
                    const float2 a12y = cmul(A12, Y), a21x = cmul(A21, X);
                    const float2 Xs = make_float2((A22 * X.x - a12y.x) * idet, (A22 * X.y - a12y.y) * idet);
                    const float2 Ys = make_float2((A11 * Y.x - a21x.x) * idet, (A11 * Y.y - a21x.y) * idet);
                    *F0 = make_float2(Xs.x - Ys.y, Xs.y + Ys.x);                       // X' + i Y'
                    if (F1 != F0) *F1 = make_float2(Xs.x + Ys.y, Ys.x - Xs.y);         // conj(X') + i conj(Y')
                }
            }
            if (f0 + nf == 2) {
                float2 *xb = x + (nf - 1) * ns * rs;
                for (int e = threadIdx.x; e < ns * ny; e += blockDim.x) {
                    const int s = axis_div(e, v.ay), ky = e - s * ny;
                    float2 p, q;
                    symbols(column(s), ky, p, q);
                    const float iz = inv_n / (1.f + sz + c2 * ((p.x * p.x + p.y * p.y) + (q.x * q.x + q.y * q.y)));
                    float2 &Z = xb[s * rs + ky];
                    Z = make_float2(Z.x * iz, Z.y * iz);
                }
            }
            __syncthreads();
            fft_axis<true>(x, y, nf * ns, rs, v.ay, f.twy);
            for (int e = threadIdx.x; e < nf * ny * ns; e += blockDim.x) {
                const int r = e / ns, s = e - r * ns, fl = r >= ny ? 1 : 0, rr = r - fl * ny;
                if (own(s)) ((f0 + fl) ? v.FB : v.FA)[(int64_t)rr * nx + column(s)] = x[(fl * ns + s) * rs + rr];
            }
            __syncthreads();
        }
    }
}

// store(n, .) = P^{-1} of the vector that load makes (all blocks take part).
// mid(): between the first pass and its barrier; more(): after that barrier,
// false ends the application there.
template <bool kCluster, typename Load, typename Mid, typename More, typename Store>
__device__ inline bool apply_spectral(const SolveBarrier<kCluster> &grid, const GridArgs<double> &g, const CNVec &v,
                                      const FftShared &f, const Load &load, const Mid &mid, const More &more,
                                      const Store &store, float c2, float sx, float sy, float sz) {
    spectral_rows(g, v, f, load);
    mid();
    grid.sync();
    if (!more()) return false;
    spectral_columns(g, v, f, c2, sx, sy, sz);
    grid.sync();
    spectral_rows_back(g, v, f, store);
    return true;
}

// ---- line preconditioner (walls) -----------------------------------------
// In a box with walls x is not periodic, y is.  For the y-mode e^{i b j}
// (j the node row) the operator (1 + s_i) X + c2 curl_h curl_e X couples a
// node column only to its two neighbours.  With ax = 1/(2 dx), ay = 1/(2 dy),
// A = 4 ay^2 sin^2(b/2), B = 4 ax^2 cos^2(b/2), sg = 2 ax ay sin b and
// Yt = i Y, the interior rows are real:
//   X:  (1 + sx_i + 2 c2 A) X_i + c2 A (X_{i-1} + X_{i+1}) + c2 sg (Yt_{i+1} - Yt_{i-1})
//   Yt: (1 + sy_i + 2 c2 B) Yt_i - c2 B (Yt_{i-1} + Yt_{i+1}) - c2 sg (X_{i+1} - X_{i-1})
//   Z:  (1 + sz_i + 2 c2 (A + B)) Z_i + c2 (A - B) (Z_{i-1} + Z_{i+1})
// and the wall rows (vacuum, the one-sided curl_h of the inside cell column,
// the time-centred Mur condition) are, at i = 0 (v = 1; at i = nx, v = nx - 1
// and the sign of the sg terms flipped):
//   X:  (1 + 2 c2 A) X_w + 2 c2 A X_v - 2 c2 sg (Yt_w - Yt_v),  Yt: cw Yt_w + cv Yt_v,  Z: cw Z_w + cv Z_v.
// s_i = the mean over the column of the diagonal of S (0 on the walls).  The
// preconditioner solves these block-tridiagonal systems exactly, mode by mode
// (block Thomas, factored once per solve): FP32 FFTs along y of x + i y and
// z, one thread per mode b = 0 .. ny/2 sweeping the columns (the modes -b are
// the conjugates: the fields are real), and the inverse FFTs.  Without a
// plasma (S = 0) it inverts the vacuum operator.
struct LineCoef {
    float A, B, sg;
};

__device__ inline LineCoef line_coef(const GridArgs<double> &g, int b) {
    float sn, cs, sh, ch;
    sincospif((float)b / (float)g.ny, &sh, &ch);          // b/2 of the mode angle 2 pi b / ny
    sincospif(2.f * (float)b / (float)g.ny, &sn, &cs);
    const float ax = 0.5f * (float)g.inv_dx, ay = 0.5f * (float)g.inv_dy;
    return LineCoef{4.f * ay * ay * sh * sh, 4.f * ax * ax * ch * ch, 2.f * ax * ay * sn};
}

// The 2 x 2 (X, Yt) blocks of row i: diagonal D, left L (column i - 1), right U (column i + 1).
__device__ inline void line_blocks(const GridArgs<double> &g, const LineCoef &k, float c2, float cw, float cv,
                                   const float *scol, int i, float (&D)[4], float (&L)[4], float (&U)[4], float &dz,
                                   float &lz, float &uz) {
    const int nxn = g.nxn;
    const float a = c2 * k.A, bb = c2 * k.B, s = c2 * k.sg;
    if (i == 0 || i == g.nx) {
        const float sgn = (i == 0) ? 1.f : -1.f;   // Yt_w - Yt_v at x = 0, the opposite at x = Lx
        const float D_[4] = {1.f + 2.f * a, -2.f * s * sgn, 0.f, cw};
        const float O_[4] = {2.f * a, 2.f * s * sgn, 0.f, cv};
        const float Z_[4] = {0.f, 0.f, 0.f, 0.f};
        for (int q = 0; q < 4; ++q) {
            D[q] = D_[q];
            L[q] = (i == 0) ? Z_[q] : O_[q];
            U[q] = (i == 0) ? O_[q] : Z_[q];
        }
        dz = cw;
        lz = (i == 0) ? 0.f : cv;
        uz = (i == 0) ? cv : 0.f;
        return;
    }
    D[0] = 1.f + scol[i] + 2.f * a;
    D[1] = 0.f;
    D[2] = 0.f;
    D[3] = 1.f + scol[nxn + i] + 2.f * bb;
    L[0] = a;  L[1] = -s; L[2] = s;  L[3] = -bb;
    U[0] = a;  U[1] = s;  U[2] = -s; U[3] = -bb;
    dz = 1.f + scol[2 * nxn + i] + 2.f * (a + bb);
    lz = uz = a - bb;
}

__device__ inline void inv2(const float (&m)[4], float (&o)[4]) {
    const float id = 1.f / (m[0] * m[3] - m[1] * m[2]);
    o[0] = m[3] * id;
    o[1] = -m[1] * id;
    o[2] = -m[2] * id;
    o[3] = m[0] * id;
}

__device__ inline void mul2(const float (&p)[4], const float (&q)[4], float (&o)[4]) {
    o[0] = p[0] * q[0] + p[1] * q[2];
    o[1] = p[0] * q[1] + p[1] * q[3];
    o[2] = p[2] * q[0] + p[3] * q[2];
    o[3] = p[2] * q[1] + p[3] * q[3];
}

// Per-column means of the diagonal of S, then the factors of every mode: for
// column i, Dp_i = D_i - M_i U_{i-1} with M_i = L_i Dp_{i-1}^{-1}; stored, mode
// by mode (lf[b][q][i]), are Dp_i^{-1} (q = 0..3), M_i (4..7), 1/dp_i and m_i
// of the Z row (8, 9).  nbm = ny/2 + 1 modes.
template <bool kCluster>
__device__ inline void line_setup(const SolveBarrier<kCluster> &grid, const GridArgs<double> &g, const CNVec &v, float c2, float cw,
                                  float cv) {
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    const int nxn = g.nxn, nbm = g.ny / 2 + 1;
    const int64_t N = g.nnode;
    for (int64_t i = tid; i < nxn; i += stride) {
        float a0 = 0.f, a1 = 0.f, a2 = 0.f;
        if (i != 0 && i != g.nx)
            for (int j = 0; j < g.ny; ++j) {
                const int64_t n = (int64_t)j * nxn + i;
                a0 += v.S[n];
                a1 += v.S[4 * N + n];
                a2 += v.S[8 * N + n];
            }
        const float inv = 1.f / (float)g.ny;
        v.scol[i] = a0 * inv;
        v.scol[nxn + i] = a1 * inv;
        v.scol[2 * nxn + i] = a2 * inv;
    }
    const int hyn = g.ny / 2;
    for (int64_t t = tid; t < hyn; t += stride) {
        double sn, cs;
        sincospi(-2.0 * (double)t / g.ny, &sn, &cs);
        v.twy[t] = make_float2((float)cs, (float)sn);
    }
    grid.sync();
    for (int64_t b = tid; b < nbm; b += stride) {
        const LineCoef k = line_coef(g, (int)b);
        float *lf = v.lf + b * 10 * (int64_t)nxn;
        float Dp[4], Dpi[4], Up[4], dpz = 0.f, upz = 0.f;
        for (int i = 0; i < nxn; ++i) {
            float D[4], L[4], U[4], dz, lz, uz, M[4] = {0.f, 0.f, 0.f, 0.f}, mz = 0.f;
            line_blocks(g, k, c2, cw, cv, v.scol, i, D, L, U, dz, lz, uz);
            if (i > 0) {
                mul2(L, Dpi, M);
                float MU[4];
                mul2(M, Up, MU);
                for (int q = 0; q < 4; ++q) Dp[q] = D[q] - MU[q];
                mz = lz / dpz;
                dpz = dz - mz * upz;
            } else {
                for (int q = 0; q < 4; ++q) Dp[q] = D[q];
                dpz = dz;
            }
            inv2(Dp, Dpi);
            for (int q = 0; q < 4; ++q) lf[q * nxn + i] = Dpi[q];
            for (int q = 0; q < 4; ++q) lf[(4 + q) * nxn + i] = M[q];
            lf[8 * nxn + i] = 1.f / dpz;
            lf[9 * nxn + i] = mz;
            for (int q = 0; q < 4; ++q) Up[q] = U[q];
            upz = uz;
        }
    }
}

// Shared memory of one mode's sweep: the mode's factors and the 6 right-hand-
// side and solution streams (3 complex values per column).
__host__ __device__ inline size_t line_sweep_bytes(int nxn) { return (size_t)nxn * 16 * sizeof(float); }

// out = P^{-1} in (all blocks of the cooperative grid take part; ends with out written).
template <bool kCluster>
__device__ inline void apply_line(const SolveBarrier<kCluster> &grid, const GridArgs<double> &g, const CNVec &v,
                                  const V4<float> *in, V4<float> *out, float c2, float cw, float cv, float2 *sm) {
    const int nxn = g.nxn, ny = g.ny, nbm = ny / 2 + 1;
    const int64_t N = g.nnode;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    // columns as rows: GA[i][j] = x + i y, GB[i][j] = z
    for (int64_t e = tid; e < N; e += stride) {
        const int i = (int)(e / ny), j = (int)(e - (int64_t)i * ny);
        const V4<float> q = in[(int64_t)j * nxn + i];
        v.GA[e] = make_float2(q.x, q.y);
        v.GB[e] = make_float2(q.z, 0.f);
    }
    grid.sync();
    fft_rows(v.GA, v.GB, nxn, ny, v.ly, v.twy, false, sm);   // along y: [column][mode]
    grid.sync();
    transpose2(v.GA, v.GB, v.FA, v.FB, nxn, ny, sm);           // -> [mode][column]
    grid.sync();
    const float inv_n = 1.f / (float)ny;
    float *s_lf = (float *)sm;                 // [10][nxn]
    float *s_xr = s_lf + 10 * (size_t)nxn;     // (X, Yt) real parts, interleaved [nxn][2]
    float *s_xi = s_xr + 2 * (size_t)nxn;      // (X, Yt) imaginary parts
    float *s_zr = s_xi + 2 * (size_t)nxn, *s_zi = s_zr + nxn;
    for (int b = blockIdx.x; b < nbm; b += gridDim.x) {
        const int bm = (ny - b) & (ny - 1);
        const LineCoef k = line_coef(g, b);
        const float *lf = v.lf + (int64_t)b * 10 * nxn;
        for (int e = threadIdx.x; e < 10 * nxn; e += blockDim.x) s_lf[e] = lf[e];
        for (int i = threadIdx.x; i < nxn; i += blockDim.x) {
            const float2 F = v.FA[(int64_t)b * nxn + i], Fm = v.FA[(int64_t)bm * nxn + i], Z = v.FB[(int64_t)b * nxn + i];
            const float Xr = 0.5f * (F.x + Fm.x), Xi = 0.5f * (F.y - Fm.y);       // X_b = (F + conj(Fm)) / 2
            const float Yr = 0.5f * (F.y + Fm.y), Yi = -0.5f * (F.x - Fm.x);      // Y_b = (F - conj(Fm)) / (2i)
            s_xr[2 * i] = Xr;                                                      // (X, i Y): real parts
            s_xr[2 * i + 1] = -Yi;
            s_xi[2 * i] = Xi;                                                      // imaginary parts
            s_xi[2 * i + 1] = Yr;
            s_zr[i] = Z.x;
            s_zi[i] = Z.y;
        }
        __syncthreads();
        // four independent recurrences: (X, Yt) real and imaginary parts (threads 0, 1), Z real and
        // imaginary parts (threads 32, 33: another warp, so that the two kinds do not diverge in one)
        const int t = threadIdx.x;
        if (t < 2) {
            float *x = t == 0 ? s_xr : s_xi;
            float y0 = 0.f, y1 = 0.f;
            for (int i = 0; i < nxn; ++i) {   // y_i = r_i - M_i y_{i-1}
                float r0 = x[2 * i], r1 = x[2 * i + 1];
                if (i > 0) {
                    r0 -= s_lf[4 * nxn + i] * y0 + s_lf[5 * nxn + i] * y1;
                    r1 -= s_lf[6 * nxn + i] * y0 + s_lf[7 * nxn + i] * y1;
                }
                y0 = r0;
                y1 = r1;
                x[2 * i] = y0;
                x[2 * i + 1] = y1;
            }
            float x0 = 0.f, x1 = 0.f;
            for (int i = nxn - 1; i >= 0; --i) {   // x_i = Dp_i^{-1} (y_i - U_i x_{i+1})
                float t0 = x[2 * i], t1 = x[2 * i + 1];
                if (i < nxn - 1) {
                    float D[4], L[4], U[4], dz, lz, uz;
                    line_blocks(g, k, c2, cw, cv, v.scol, i, D, L, U, dz, lz, uz);
                    t0 -= U[0] * x0 + U[1] * x1;
                    t1 -= U[2] * x0 + U[3] * x1;
                }
                x0 = s_lf[i] * t0 + s_lf[nxn + i] * t1;
                x1 = s_lf[2 * nxn + i] * t0 + s_lf[3 * nxn + i] * t1;
                x[2 * i] = x0;
                x[2 * i + 1] = x1;
            }
        } else if (t == 32 || t == 33) {
            float *z = t == 32 ? s_zr : s_zi;
            float y = 0.f;
            for (int i = 0; i < nxn; ++i) {
                float r = z[i];
                if (i > 0) r -= s_lf[9 * nxn + i] * y;
                y = r;
                z[i] = y;
            }
            const float uz = c2 * (k.A - k.B);
            float xz = 0.f;
            for (int i = nxn - 1; i >= 0; --i) {
                float t = z[i];
                if (i < nxn - 1) t -= ((i == 0) ? cv : uz) * xz;   // row 0: the wall's Mur coefficient
                xz = s_lf[8 * nxn + i] * t;
                z[i] = xz;
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < nxn; i += blockDim.x) {
            // X' = xr[0] + i xi[0]; i Y' = xr[1] + i xi[1], so Y' = xi[1] - i xr[1]
            const float Xr = s_xr[2 * i], Xi = s_xi[2 * i], Yr = s_xi[2 * i + 1], Yi = -s_xr[2 * i + 1];
            const float zr = s_zr[i], zi = s_zi[i];
            // F' = X' + i Y' (mode b), conj(X') + i conj(Y') (mode -b); Z' and conj(Z')
            v.FA[(int64_t)b * nxn + i] = make_float2((Xr - Yi) * inv_n, (Xi + Yr) * inv_n);
            v.FB[(int64_t)b * nxn + i] = make_float2(zr * inv_n, zi * inv_n);
            if (bm != b) {
                v.FA[(int64_t)bm * nxn + i] = make_float2((Xr + Yi) * inv_n, (Yr - Xi) * inv_n);
                v.FB[(int64_t)bm * nxn + i] = make_float2(zr * inv_n, -zi * inv_n);
            }
        }
        __syncthreads();
    }
    grid.sync();
    transpose2(v.FA, v.FB, v.GA, v.GB, ny, nxn, sm);           // -> [column][mode]
    grid.sync();
    fft_rows(v.GA, v.GB, nxn, ny, v.ly, v.twy, true, sm);    // back along y
    grid.sync();
    for (int64_t e = tid; e < N; e += stride) {
        const int j = (int)(e / nxn), i = (int)(e - (int64_t)j * nxn);
        const float2 a = v.GA[(int64_t)i * ny + j], z = v.GB[(int64_t)i * ny + j];
        out[e] = V4<float>{a.x, a.y, z.x, 0.f};
    }
}

// RHS, initial guess (E^n), FP32 S / dA and FP32 block-Jacobi inverse.  A
// wall node (a box with walls) is vacuum: its x row has the one-sided curl_h of
// the inside cell column, its y and z rows are the time-centred Mur condition
// with right-hand side (E_w + E_v)/dt, at x = 0 for the field minus the
// incident wave (inc: the wave at the wall node and its neighbour at the old
// and new times), whose centred values move to the right-hand side.
//
// FP32 form: the moments are FP64 for the solver, the sum of each and its
// compensation term; the pass writes the planes of S that the solve reads (Md)
// and zeroes what it has read (clr), so that neither a conversion of all 13
// planes nor a clear follows.  The FP64 pipe bounds it: values change their width
// by their bits (narrow, widen), and the block inverses (45 operations and a
// division) are left out where another preconditioner is used (jac = 0).
// 1024 x 1024 FP32: 222 us, 75 us of conversions and 38 us of clears -> 112 us.
template <typename R>
__global__ void k_cn_setup(GridArgs<double> g, const V4<R> *__restrict__ E, const V4<R> *__restrict__ H, R *M, R *Mlo,
                           double *__restrict__ Md, int clr, int jac, CNVec v, double c2, WallRows wr, Inc inc) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y;
    if (i >= g.nxn || j >= g.ny) return;
    int64_t node = (int64_t)j * g.nxn + i;
    double m[NMOM];   // (rho is read to be zeroed only)
    if constexpr (sizeof(R) == 4) {
        R hi[NMOM], lo[NMOM];
#pragma unroll
        for (int k = 0; k < NMOM; ++k) {
            hi[k] = M[(int64_t)k * g.nnode + node];
            lo[k] = Mlo[(int64_t)k * g.nnode + node];
        }
#pragma unroll
        for (int k = 0; k < NMOM; ++k) {
            m[k] = widen(hi[k]) + widen(lo[k]);
            if (k >= 1 && k <= 9) Md[(int64_t)k * g.nnode + node] = m[k];
            if (clr && hi[k] != R(0)) M[(int64_t)k * g.nnode + node] = R(0);
            if (clr && lo[k] != R(0)) Mlo[(int64_t)k * g.nnode + node] = R(0);
        }
    } else {
#pragma unroll
        for (int k = 1; k < NMOM; ++k) m[k] = M[(int64_t)k * g.nnode + node];
    }
    int im = (i == 0) ? g.nx - 1 : i - 1;
    int jm = (j == 0) ? g.ny - 1 : j - 1;
    if (!g.periodic_x && (i == 0 || i == g.nx)) {
        const int ic = (i == 0) ? 0 : g.nx - 1, iv = (i == 0) ? 1 : g.nx - 1;
        const V4<R> e = E[node], ev = E[(int64_t)j * g.nxn + iv];
        const V4<R> up = H[(int64_t)j * g.nx + ic], dn = H[(int64_t)jm * g.nx + ic];
        double ry = ((double)e.y + (double)ev.y) / g.dt, rz = ((double)e.z + (double)ev.z) / g.dt;
        if (i == 0) {
            ry += -(inc.old0[1] + inc.old1[1]) / g.dt + wr.cw * 0.5 * (inc.old0[1] + inc.new0[1]) +
                  wr.cv * 0.5 * (inc.old1[1] + inc.new1[1]);
            rz += -(inc.old0[2] + inc.old1[2]) / g.dt + wr.cw * 0.5 * (inc.old0[2] + inc.new0[2]) +
                  wr.cv * 0.5 * (inc.old1[2] + inc.new1[2]);
        }
        v.b[node] = V4<double>{(double)e.x + 0.5 * g.dt * (((double)up.z - (double)dn.z) * g.inv_dy), ry, rz, 0.0};
        v.x[node] = V4<double>{(double)e.x, (double)e.y, (double)e.z, 0.0};
        for (int k = 0; k < 9; ++k) v.S[(int64_t)k * g.nnode + node] = 0.f;
        if (!jac) return;
        for (int k = 0; k < 9; ++k) v.minv[(int64_t)k * g.nnode + node] = 0.f;
        // diagonal of the wall rows: 1 + (dt/2)^2 / dy^2 (x), cw (y, z)
        v.minv[node] = (float)(1.0 / (1.0 + c2 * g.inv_dy * g.inv_dy));
        v.minv[4 * g.nnode + node] = (float)(1.0 / wr.cw);
        v.minv[8 * g.nnode + node] = (float)(1.0 / wr.cw);
        return;
    }
    V4<R> ha = H[(int64_t)j * g.nx + i], hb = H[(int64_t)j * g.nx + im];
    V4<R> hc = H[(int64_t)jm * g.nx + i], hd = H[(int64_t)jm * g.nx + im];
    const double hy = 0.5 * g.inv_dy, hx = 0.5 * g.inv_dx;
    const double az = widen(ha.z), bz = widen(hb.z), cz_ = widen(hc.z), dz = widen(hd.z);
    double cx = ((az + bz) - (cz_ + dz)) * hy;
    double cy = -(((az + cz_) - (bz + dz)) * hx);
    double cz = ((widen(ha.y) + widen(hc.y)) - (widen(hb.y) + widen(hd.y))) * hx -
                ((widen(ha.x) + widen(hb.x)) - (widen(hc.x) + widen(hd.x))) * hy;
    double ia = g.inv_dx * g.inv_dy;
    const V4<R> er = E[node];
    const V4<double> e{widen(er.x), widen(er.y), widen(er.z), 0.0};
    double hdt = 0.5 * g.dt;
    v.b[node] = V4<double>{e.x + hdt * (cx - m[10] * ia), e.y + hdt * (cy - m[11] * ia), e.z + hdt * (cz - m[12] * ia), 0.0};
    v.x[node] = e;
    double A[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        A[k] = m[1 + k] * ia;
        v.S[(int64_t)k * g.nnode + node] = narrow(A[k]);
    }
    if (!jac) return;
    // diagonal of (dt/2)^2 curl_h curl_e: (1/dy^2, 1/dx^2, 1/dx^2 + 1/dy^2)
    A[0] += 1.0 + c2 * g.inv_dy * g.inv_dy;
    A[4] += 1.0 + c2 * g.inv_dx * g.inv_dx;
    A[8] += 1.0 + c2 * (g.inv_dx * g.inv_dx + g.inv_dy * g.inv_dy);
    double c00 = A[4] * A[8] - A[5] * A[7], c01 = A[5] * A[6] - A[3] * A[8], c02 = A[3] * A[7] - A[4] * A[6];
    double det = A[0] * c00 + A[1] * c01 + A[2] * c02;
    double id = 1.0 / det;
    double inv[9] = {c00 * id, (A[2] * A[7] - A[1] * A[8]) * id, (A[1] * A[5] - A[2] * A[4]) * id,
                     c01 * id, (A[0] * A[8] - A[2] * A[6]) * id, (A[2] * A[3] - A[0] * A[5]) * id,
                     c02 * id, (A[1] * A[6] - A[0] * A[7]) * id, (A[0] * A[4] - A[1] * A[3]) * id};
#pragma unroll
    for (int k = 0; k < 9; ++k) v.minv[(int64_t)k * g.nnode + node] = narrow(inv[k]);
}

// Block sum of up to 3 values; thread 0 writes them to part[k * nb + block].
// The threads' values meet in shared memory and warp 0 adds them (strided
// lanes, then a butterfly), so that the FP64 adds run in one warp.
constexpr int CN_BS = 256;            // threads of a block of the cooperative solve
constexpr int CN_CLUSTER_BS = 256;    // and of the single-cluster solve
constexpr int CN_CLUSTER = 16;        // its blocks
template <int BS>
__device__ inline void block_partials(double a0, double a1, double a2, int nv, double *part, int nb) {
    __shared__ double sh[3][BS];
    const double v[3] = {a0, a1, a2};
    for (int k = 0; k < nv; ++k) sh[k][threadIdx.x] = v[k];
    __syncthreads();
    if (threadIdx.x < 32) {
        for (int k = 0; k < nv; ++k) {
            double s[4] = {0.0, 0.0, 0.0, 0.0};   // independent chains
            for (int j = threadIdx.x; j < BS; j += 128)
#pragma unroll
                for (int u = 0; u < 4; ++u) s[u] += sh[k][j + 32 * u];
            double t = (s[0] + s[1]) + (s[2] + s[3]);
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (threadIdx.x == 0) part[(int64_t)k * nb + blockIdx.x] = t;
        }
    }
    __syncthreads();
}

// Fixed-order sum of the partials, identical in every block: lane l of warp 0
// adds partials l, l + 32, ..., then a butterfly over the lanes; thread 0 then
// runs next(sums), the solve's scalar arithmetic (every block the same), and the
// block goes on.  All of it in one warp: the FP64 pipe takes 16 cycles for a
// warp's instruction, so that a division done by every thread of a block costs
// as much as a pass over its nodes.  The partials come from other blocks: read
// through L2.
template <typename Next>
__device__ inline void reduce_partials(const double *part, int nb, int nv, const Next &next) {
    if (threadIdx.x < 32) {
        double t[3];
        for (int k = 0; k < nv; ++k) {
            const double *q = part + (int64_t)k * nb;
            double s[4] = {0.0, 0.0, 0.0, 0.0};
            for (int b = threadIdx.x; b < nb; b += 128)
#pragma unroll
                for (int u = 0; u < 4; ++u) s[u] += b + 32 * u < nb ? __ldcg(q + b + 32 * u) : 0.0;
            t[k] = (s[0] + s[1]) + (s[2] + s[3]);
            for (int o = 16; o > 0; o >>= 1) t[k] += __shfl_xor_sync(0xffffffffu, t[k], o);
        }
        if (threadIdx.x == 0) next(t);
    }
    __syncthreads();
}

// Largest of the block's three values (threads of one warp, then shared memory).
__device__ inline void block_largest(float a, float b, float c, double *part, int nb) {
    __shared__ float sh[3][32];
    float v[3] = {a, b, c};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        for (int o = 16; o > 0; o >>= 1) v[k] = fmaxf(v[k], __shfl_xor_sync(0xffffffffu, v[k], o));
        if ((threadIdx.x & 31) == 0) sh[k][threadIdx.x >> 5] = v[k];
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        float m = sh[threadIdx.x][0];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, sh[threadIdx.x][w]);
        part[(int64_t)threadIdx.x * nb + blockIdx.x] = (double)m;
    }
    __syncthreads();
}
// and of the blocks' (thread 0 of warp 0 gets them).
__device__ inline void grid_largest(const double *part, int nb, double *out) {
    if (threadIdx.x >= 32) return;
    for (int k = 0; k < 3; ++k) {
        float m = -INFINITY;
        for (int b = threadIdx.x; b < nb; b += 32) m = fmaxf(m, (float)__ldcg(part + (int64_t)k * nb + b));
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        out[k] = (double)m;
    }
}

// The solve's scalars (shared memory, written by thread 0 of every block alike).
struct SolveScalars {
    double bnorm, res, rr, rr_prev, rr_root, stop;   // of the refinement
    double rho, alpha, omega;               // of BiCGSTAB
    float beta, alphaf, omegaf;
    float sx, sy, sz;                       // grid means of the diagonal of S
    float rate;                             // bound on (or measured) reduction per spectral correction
    int sweep;                              // the refinements' corrections by the preconditioner alone
    int go;                                 // goes on after this reduction
};

// The spectral preconditioner's corrections converge by themselves, as d += P^{-1} r,
// r -= A P^{-1} r, where S varies little: the error is multiplied by at most
// rho = max |S - mean| / (1 + mean).  Below CN_SWEEP_RHO the solve takes them
// instead of BiCGSTAB: no dot products, half the vectors, four barriers per
// application instead of four and a half.  The field solve of uniform plasmas of
// growing density, corrections / BiCGSTAB (us, FP64; FP32 alike): 64 x 64 rho 0.05
// 157 / 203, 0.13 216 / 246, 0.20 250 / 277; 256 x 256 0.10 317 / 419, 0.17 416 /
// 420, 0.25 490 / 471; 512 x 512 0.08 676 / 768, 0.13 722 / 873, 0.19 1053 / 926,
// 0.26 1205 / 1030.  They meet between 0.16 (large grids) and above 0.2 (small).
constexpr float CN_SWEEP_RHO = 0.2f;

// The whole solve in one launch (grid-wide barriers between the dependent
// phases).  Thread partial sums of the FP32 phases are FP32 (a few nodes per
// thread), block and grid sums FP64 in a fixed order.
// out = [FP32 iterations, relative FP64 residual, refinements].
// Launch times, against BiCGSTAB throughout with grid barriers, transposes and FP64
// scalars in every thread: 64 x 64 periodic 303 -> 150 us; 1024 x 1024, FP32, 2.56 ->
// 1.58 ms; 1024 x 512 with walls (block-Jacobi) 1.04 -> 0.80 ms.
template <bool kCluster, int BS>
__global__ void __launch_bounds__(BS, kCluster ? 1 : 3) k_cn_solve(GridArgs<double> g, const double *__restrict__ Md, CNVec v, double c2, double tol,
                           int max_iter, double *part, double *out, WallRows wr) {
    const SolveBarrier<kCluster> grid;
    const int N = (int)g.nnode, NC = g.nx * g.ny;   // (at most 2^30 cells; a wall adds a column)
    const int tid = blockIdx.x * BS + threadIdx.x, stride = gridDim.x * BS;
    const int nb = gridDim.x;
    const double ia = g.inv_dx * g.inv_dy;
    const double hx = 0.5 * g.inv_dx, hy = 0.5 * g.inv_dy;
    const float c2f = (float)c2, hxf = (float)hx, hyf = (float)hy, cwf = (float)wr.cw, cvf = (float)wr.cv;
    double *pa = part, *pb = part + 3 * (int64_t)nb;  // alternating partial buffers
    int flip = 0;
    auto P = [&]() { double *q = flip ? pb : pa; flip ^= 1; return q; };
    int total = 0, outer = 0;
    extern __shared__ float2 cn_sm[];
    __shared__ SolveScalars sc;
    const FftShared fs = fft_shared(g, cn_sm);   // (spectral preconditioner)
    if (v.fft) {
        // twiddles, and the grid means of the diagonal of S for the preconditioner
        const int hxn = g.nx / 2 + 1, hyn = g.ny / 2 + 1;
        for (int t = tid; t < hxn + hyn; t += stride) {
            double sn, cs;
            if (t < hxn) {
                sincospi(-2.0 * (double)t / g.nx, &sn, &cs);
                v.twx[t] = make_float2((float)cs, (float)sn);
            } else {
                sincospi(-2.0 * (double)(t - hxn) / g.ny, &sn, &cs);
                v.twy[t - hxn] = make_float2((float)cs, (float)sn);
            }
        }
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, lo = INFINITY, hi = -INFINITY, off = 0.f;
        for (int n = tid; n < N; n += stride) {
            float S[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) S[k] = v.S[(int64_t)k * N + n];
            a0 += S[0];
            a1 += S[4];
            a2 += S[8];
            lo = fminf(lo, fminf(S[0], fminf(S[4], S[8])));
            hi = fmaxf(hi, fmaxf(S[0], fmaxf(S[4], S[8])));
            // |off-diagonal part| <= its largest row or column sum
            const float b1 = fabsf(S[1]), b2 = fabsf(S[2]), b3 = fabsf(S[3]), b5 = fabsf(S[5]), b6 = fabsf(S[6]),
                        b7 = fabsf(S[7]);
            off = fmaxf(off, fmaxf(fmaxf(b1 + b2, fmaxf(b3 + b5, b6 + b7)), fmaxf(b3 + b6, fmaxf(b1 + b7, b2 + b5))));
        }
        double *q0 = P(), *q1 = P();
        block_partials<BS>(a0, a1, a2, 3, q0, nb);
        block_largest(-lo, hi, off, q1, nb);
        grid.sync();
        double ext[3];
        grid_largest(q1, nb, ext);
        reduce_partials(q0, nb, 3, [&](const double *red) {
            sc.sx = (float)(red[0] / N);
            sc.sy = (float)(red[1] / N);
            sc.sz = (float)(red[2] / N);
            const float smin = fminf(sc.sx, fminf(sc.sy, sc.sz)), smax = fmaxf(sc.sx, fmaxf(sc.sy, sc.sz));
            sc.rate = (fmaxf((float)ext[1] - smin, smax + (float)ext[0]) + (float)ext[2]) / (1.f + smin);
            sc.sweep = smin >= 0.f && sc.rate < CN_SWEEP_RHO;
        });
        axis_twiddles(fs.twx, v.twx, v.ax);
        axis_twiddles(fs.twy, v.twy, v.ay);
        __syncthreads();
    } else if (v.line) {
        line_setup(grid, g, v, c2f, cwf, cvf);
        grid.sync();
    }
    auto split = [&](int n, int &i, int &j) {
        j = (int)((unsigned)n / (unsigned)g.nxn);
        i = n - j * g.nxn;
    };
    for (;;) {
        // FP64 residual r = b - A x, handed to the FP32 solve (r0 = r)
        double s_rr = 0, s_bb = 0;
        for (int c = tid; c < NC; c += stride) {
            const int cj = (int)((unsigned)c / (unsigned)g.nx), ci = c - cj * g.nx;
            v.cc[c] = cell_curl_e(g, v.x, hx, hy, ci, cj);
        }
        grid.sync();
        for (int n = tid; n < N; n += stride) {
            int i, j;
            split(n, i, j);
            V4<double> ax = apply_A_from_cells(g, v.x, v.cc, Md + N, ia, c2 * hx, c2 * hy, i, j, wr.cw, wr.cv);
            V4<double> b = v.b[n];
            V4<double> r{b.x - ax.x, b.y - ax.y, b.z - ax.z, 0.0};
            V4<float> rf{narrow(r.x), narrow(r.y), narrow(r.z), 0.f};
            v.r[n] = rf;
            if (!(v.fft && sc.sweep)) v.r0[n] = rf;
            s_rr += dot(r, r);
            if (outer == 0) s_bb += dot(b, b);
        }
        double *q = P();
        block_partials<BS>(s_rr, s_bb, 0.0, 2, q, nb);
        grid.sync();
        reduce_partials(q, nb, 2, [&](const double *red) {
            if (outer == 0) sc.bnorm = sqrt(red[1]);
            sc.rr = red[0];
            sc.res = sc.bnorm == 0.0 ? 0.0 : sqrt(sc.rr) / sc.bnorm;
            // converged, out of budget, or no longer improving (FP64 rounding floor)
            sc.go = !(sc.bnorm == 0.0 || sc.res <= tol || total >= max_iter || outer >= CN_MAX_OUTER ||
                      (outer > 0 && sc.rr > 0.25 * sc.rr_prev));
            sc.rr_prev = sc.rr;
            sc.rr_root = sqrt(sc.rr);
            sc.stop = (double)CN_INNER_RTOL * sc.rr_root;
            sc.rho = sc.rr;
            sc.alpha = sc.omega = 1.0;
            sc.beta = sc.omegaf = 0.f;
        });
        if (!sc.go) {
            if (sc.bnorm == 0.0)
                for (int n = tid; n < N; n += stride) v.x[n] = V4<double>{0, 0, 0, 0};
            break;
        }
        ++outer;
        if (v.fft && sc.sweep) {
            // corrections by the preconditioner (CN_SWEEP_RHO) until r is below the stop; where the
            // reduction seen so far says that one more will do, that one goes straight into x and the
            // next FP64 residual judges it
            bool first = true;   // d = 0 before it
            int last = sc.rate * sc.rr_root <= sc.stop || total + 1 >= max_iter;
            for (;;) {
                auto keep = [&](int64_t n, const V4<float> &z) { v.ph[n] = z; };
                auto finish = [&](int64_t n, const V4<float> &z) {
                    V4<float> d{0.f, 0.f, 0.f, 0.f};
                    if (!first) d = v.d[n];
                    const V4<double> x = v.x[n];
                    v.x[n] = V4<double>{x.x + widen(d.x + z.x), x.y + widen(d.y + z.y), x.z + widen(d.z + z.z), 0.0};
                };
                auto load_r = [&](int64_t n) { return v.r[n]; };
                ++total;
                if (last) {
                    apply_spectral(grid, g, v, fs, load_r, [] {}, [] { return true; }, finish, c2f, sc.sx, sc.sy, sc.sz);
                    break;
                }
                apply_spectral(grid, g, v, fs, load_r, [] {}, [] { return true; }, keep, c2f, sc.sx, sc.sy, sc.sz);
                grid.sync();
                float s_r = 0.f;
                for (int n = tid; n < N; n += stride) {
                    int i, j;
                    split(n, i, j);
                    const V4<float> az = apply_A<float>(g, v.ph, v.S, 1.f, c2f, hxf, hyf, i, j, cwf, cvf), z = v.ph[n];
                    V4<float> r = v.r[n], d = z;
                    if (!first) {
                        d = v.d[n];
                        d = V4<float>{d.x + z.x, d.y + z.y, d.z + z.z, 0.f};
                    }
                    r = V4<float>{r.x - az.x, r.y - az.y, r.z - az.z, 0.f};
                    v.r[n] = r;
                    v.d[n] = d;
                    s_r += dot(r, r);
                }
                first = false;
                q = P();
                block_partials<BS>(s_r, 0, 0, 1, q, nb);
                grid.sync();
                reduce_partials(q, nb, 1, [&](const double *red) {
                    const double r = sqrt(red[0]), next = r * (r / sc.rr_root);
                    // 0: below the stop; 1: at least two more; 2: one more will do (or is all that may be taken)
                    sc.go = r <= sc.stop ? 0 : (next <= 0.3 * sc.stop || total + 1 >= max_iter) ? 2 : 1;
                    sc.rr_root = r;
                });
                if (sc.go == 0) {
                    for (int n = tid; n < N; n += stride) {
                        const V4<double> x = v.x[n];
                        const V4<float> d = v.d[n];
                        v.x[n] = V4<double>{x.x + widen(d.x), x.y + widen(d.y), x.z + widen(d.z), 0.0};
                    }
                    break;
                }
                last = sc.go == 2;
            }
            grid.sync();
            continue;
        }
        // FP32 BiCGSTAB (right preconditioned) on A d = r
        bool first = true;   // p = r, d = 0 before it
        while (total < max_iter) {
            const float beta = sc.beta, omf = sc.omegaf;
            auto next_p = [&](int n) {
                V4<float> pn = v.r[n];
                if (!first) {
                    const V4<float> p = v.p[n], vv = v.v[n];
                    pn = V4<float>{pn.x + beta * (p.x - omf * vv.x), pn.y + beta * (p.y - omf * vv.y),
                                   pn.z + beta * (p.z - omf * vv.z), 0.f};
                }
                v.p[n] = pn;
                return pn;
            };
            if (v.fft)
                apply_spectral(grid, g, v, fs, next_p, [] {}, [] { return true; },
                               [&](int64_t n, const V4<float> &z) { v.ph[n] = z; }, c2f, sc.sx, sc.sy, sc.sz);
            else
                for (int n = tid; n < N; n += stride) {
                    const V4<float> pn = next_p(n);
                    if (!v.line) v.ph[n] = apply_minv(v.minv, N, n, pn);
                }
            if (v.line) {
                grid.sync();
                apply_line(grid, g, v, v.p, v.ph, c2f, cwf, cvf, cn_sm);
            }
            grid.sync();
            float s_r0v = 0.f;
            for (int n = tid; n < N; n += stride) {
                int i, j;
                split(n, i, j);
                V4<float> av = apply_A<float>(g, v.ph, v.S, 1.f, c2f, hxf, hyf, i, j, cwf, cvf);
                v.v[n] = av;
                s_r0v += dot(v.r0[n], av);
            }
            q = P();
            block_partials<BS>(s_r0v, 0, 0, 1, q, nb);
            grid.sync();
            reduce_partials(q, nb, 1, [&](const double *red) {
                sc.go = red[0] != 0.0;
                sc.alpha = sc.rho / red[0];
                sc.alphaf = (float)sc.alpha;
            });
            if (!sc.go) break;
            const float af = sc.alphaf;
            float s_ss = 0.f;
            auto next_s = [&](int n) {
                V4<float> r = v.r[n], vv = v.v[n];
                V4<float> s{r.x - af * vv.x, r.y - af * vv.y, r.z - af * vv.z, 0.f};
                v.s[n] = s;
                s_ss += dot(s, s);
                return s;
            };
            q = P();
            auto partial = [&] { block_partials<BS>(s_ss, 0, 0, 1, q, nb); };
            auto larger = [&] {
                reduce_partials(q, nb, 1, [&](const double *red) { sc.go = sqrt(red[0]) > sc.stop; });
                ++total;
                return sc.go != 0;
            };
            bool go_on;
            if (v.fft) {
                go_on = apply_spectral(grid, g, v, fs, next_s, partial, larger,
                                       [&](int64_t n, const V4<float> &z) { v.sh[n] = z; }, c2f, sc.sx, sc.sy, sc.sz);
            } else {
                for (int n = tid; n < N; n += stride) {
                    const V4<float> s = next_s(n);
                    if (!v.line) v.sh[n] = apply_minv(v.minv, N, n, s);
                }
                partial();
                grid.sync();
                go_on = larger();
            }
            if (!go_on) {
                for (int n = tid; n < N; n += stride) {
                    const V4<float> d = first ? V4<float>{0.f, 0.f, 0.f, 0.f} : v.d[n], ph = v.ph[n];
                    v.d[n] = V4<float>{d.x + af * ph.x, d.y + af * ph.y, d.z + af * ph.z, 0.f};
                }
                first = false;
                break;
            }
            if (v.line) apply_line(grid, g, v, v.s, v.sh, c2f, cwf, cvf, cn_sm);
            if (v.fft || v.line) grid.sync();
            float s_ts = 0.f, s_tt = 0.f;
            for (int n = tid; n < N; n += stride) {
                int i, j;
                split(n, i, j);
                V4<float> at = apply_A<float>(g, v.sh, v.S, 1.f, c2f, hxf, hyf, i, j, cwf, cvf);
                v.t[n] = at;
                V4<float> s = v.s[n];
                s_ts += dot(at, s);
                s_tt += dot(at, at);
            }
            q = P();
            block_partials<BS>(s_ts, s_tt, 0, 2, q, nb);
            grid.sync();
            reduce_partials(q, nb, 2, [&](const double *red) {
                sc.go = red[1] != 0.0;
                sc.omega = red[0] / red[1];
                sc.omegaf = (float)sc.omega;
            });
            if (!sc.go) break;
            const float of = sc.omegaf;
            float s_r0r = 0.f, s_rr2 = 0.f;
            for (int n = tid; n < N; n += stride) {
                V4<float> ph = v.ph[n], sh = v.sh[n], s = v.s[n], t = v.t[n];
                const V4<float> d = first ? V4<float>{0.f, 0.f, 0.f, 0.f} : v.d[n];
                v.d[n] = V4<float>{d.x + af * ph.x + of * sh.x, d.y + af * ph.y + of * sh.y,
                                   d.z + af * ph.z + of * sh.z, 0.f};
                V4<float> r{s.x - of * t.x, s.y - of * t.y, s.z - of * t.z, 0.f};
                v.r[n] = r;
                s_r0r += dot(v.r0[n], r);
                s_rr2 += dot(r, r);
            }
            first = false;
            q = P();
            block_partials<BS>(s_r0r, s_rr2, 0, 2, q, nb);
            grid.sync();
            reduce_partials(q, nb, 2, [&](const double *red) {
                sc.go = !(sqrt(red[1]) <= sc.stop || red[0] == 0.0 || sc.omega == 0.0);
                sc.beta = (float)((red[0] / sc.rho) * (sc.alpha / sc.omega));
                sc.rho = red[0];
            });
            if (!sc.go) break;
        }
        // x += d in FP64 (nothing was added where the first iteration broke down)
        if (!first)
            for (int n = tid; n < N; n += stride) {
                V4<double> x = v.x[n];
                V4<float> d = v.d[n];
                v.x[n] = V4<double>{x.x + widen(d.x), x.y + widen(d.y), x.z + widen(d.z), 0.0};
            }
        grid.sync();
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        out[0] = (double)total;
        out[1] = sc.res;
        out[2] = (double)outer;
    }
}

// E^{n+1} = 2X - E^n, E^n + E^{n+1} = 2X (padded, for the push).
template <typename R>
__global__ void k_cn_finish(GridArgs<R> g, const V4<double> *__restrict__ X, const V4<R> *__restrict__ E,
                            V4<R> *__restrict__ Enew, V4<R> *__restrict__ Esum) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y;
    if (i >= g.nxn || j >= g.ny) return;
    int64_t node = (int64_t)j * g.nxn + i;
    V4<double> x = X[node];
    V4<R> e = E[node];
    // (widths changed by their bits: 1024 x 1024 FP32 32 -> 16 us, and k_field_HB 52 -> 37)
    Enew[node] = V4<R>{stored<R>(2.0 * x.x - widen(e.x)), stored<R>(2.0 * x.y - widen(e.y)),
                       stored<R>(2.0 * x.z - widen(e.z)), R(0)};
    store_padded(Esum, g, i, j, V4<R>{stored<R>(2.0 * x.x), stored<R>(2.0 * x.y), stored<R>(2.0 * x.z), R(0)});
}

// --------------------------------------------------------------------------- host side

static dim3 node_grid(const pic_t *h, int bs) { return dim3((h->nxn + bs - 1) / bs, h->ny); }

template <typename R>
static int node_average_t(pic_t *h, int hsrc, int bdst) {
    GridArgs<R> g = grid_args<R>(h);
    k_node_average<R><<<node_grid(h, 128), 128, 0, h->st>>>(g, (const V4<R> *)h->H[hsrc], (V4<R> *)h->B[bdst]);
    count_launch(h);
    return check_launch("k_node_average");
}

int node_average(pic_t *h, int hsrc, int bdst) {
    return h->fp32 ? node_average_t<float>(h, hsrc, bdst) : node_average_t<double>(h, hsrc, bdst);
}

double host_laser(double t, double a0, double omega, double tau, double t0);

// The incident plane wave (reading of the missing source equation) at the x = 0
// wall node and its neighbour, at the times of E^n and E^{n+1} of this step, in
// the polarised component (y or z).
static Inc incident(const pic_t *h) {
    const pic_config &c = h->cfg;
    double t_new = (double)(h->step + 1) * c.dt, t_old = t_new - c.dt;
    Inc inc;
    int pc = (c.laser_pol == 0) ? 1 : 2;
    for (int k = 0; k < 3; ++k) {
        bool on = (k == pc) && !h->periodic_x;
        inc.new0[k] = on ? host_laser(t_new, c.laser_a0, c.laser_omega, c.laser_tau, c.laser_t0) : 0.0;
        inc.old0[k] = on ? host_laser(t_old, c.laser_a0, c.laser_omega, c.laser_tau, c.laser_t0) : 0.0;
        inc.new1[k] = on ? host_laser(t_new - c.dx, c.laser_a0, c.laser_omega, c.laser_tau, c.laser_t0) : 0.0;
        inc.old1[k] = on ? host_laser(t_old - c.dx, c.laser_a0, c.laser_omega, c.laser_tau, c.laser_t0) : 0.0;
    }
    return inc;
}

// Rows a warp of k_field_HB walks down: up to 32 (it forms a row of H more than
// it stores), fewer where that leaves the GPU short of warps.
static int field_rows(const pic_t *h, int xw) {
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int64_t r = (int64_t)h->ny * xw / (24 * (int64_t)(nsm > 0 ? nsm : 128));
    return r < 2 ? 2 : r > 32 ? 32 : (int)r;
}

template <typename R, typename RE>
static int field_HB(pic_t *h, const void *Ec) {
    const int hn = 1 - h->hcur, xw = (h->nxn + HB_COLS - 1) / HB_COLS, rows = field_rows(h, xw);
    k_field_HB<R, RE><<<dim3(xw, (h->ny + rows * FIELD_WARPS - 1) / (rows * FIELD_WARPS)), 32 * FIELD_WARPS, 0, h->st>>>(
        grid_args<R>(h), (const V4<RE> *)Ec, (const V4<R> *)h->H[h->hcur], (V4<R> *)h->H[hn], (V4<R> *)h->B[1 - h->bcur],
        (RE)(0.5 * h->cfg.dt / h->cfg.dx), (RE)(0.5 * h->cfg.dt / h->cfg.dy), rows);
    count_launch(h);
    return check_launch("k_field_HB");
}

template <typename R>
static int field_literal_t(pic_t *h) {
    int en = 1 - h->ecur;
    // the exact deposit rewrites every moment from its fixed-point sums; the others deposit into the
    // moments this solve has read and zeroed
    TouchArgs<R> tm{h->touch_all ? nullptr : h->touched + (size_t)h->touch_cur * h->ntiles, h->touch_far, h->tnx, h->tny, h->ntx, h->det ? nullptr : (R *)h->M,
                    h->det ? nullptr : (R *)h->Mlo};
    const pic_config &c = h->cfg;
    const int cols = h->periodic_x ? h->nx : h->nx - 1;   // (the walls' columns by their neighbours' threads)
    k_field_E_literal<R><<<dim3((cols + 127) / 128, h->ny), 128, 0, h->st>>>(
        grid_args<R>(h), (const V4<R> *)h->E[h->ecur], (const V4<R> *)h->H[h->hcur], (const R *)h->M, (const R *)h->Mlo,
        (V4<R> *)h->E[en], (V4<R> *)h->Ehalf, tm, incident(h), (R)((c.dt - c.dx) / (c.dt + c.dx)));
    count_launch(h);
    if (int rc = check_launch("k_field_E_literal")) return rc;
    h->moments_cleared = !h->det;
    return field_HB<R, R>(h, h->E[en]);
}

int field_literal(pic_t *h) { return h->fp32 ? field_literal_t<float>(h) : field_literal_t<double>(h); }

// Factors of an axis of the spectral preconditioner: 4s, then primes; false
// where a prime is too large for direct sums (or n for the shared buffers).
constexpr int FFT_MAX_PRIME = 61;
static bool fft_factors(int n, FftAxis *ax) {
    if (n < 2 || n > 4096) return false;
    *ax = FftAxis{};
    ax->n = n;
    ax->lg = -1;
    if ((n & (n - 1)) == 0)
        for (ax->lg = 0; (1 << ax->lg) < n;) ++ax->lg;
    int m = n;
    while (m % 4 == 0) {
        ax->f[ax->nf++] = 4;
        m /= 4;
    }
    for (int p = 2; p <= FFT_MAX_PRIME && m > 1; ++p)
        while (m % p == 0) {
            ax->f[ax->nf++] = p;
            m /= p;
        }
    return m == 1;
}

// The spectral preconditioner applies to periodic grids whose sides have no
// prime factor above FFT_MAX_PRIME (at most 4096), the line preconditioner to
// boxes with walls whose ny is a power of two.  Without it such a grid takes
// some three hundred block-Jacobi iterations at c dt / dx = 25 (90 x 64: 6.6 ms
// a solve; 0.27 ms with it).
static bool cn_spectral(const pic_t *h) {
    FftAxis a, b;
    return h->cfg.cn_precond != PIC_CN_PRECOND_JACOBI && h->periodic_x && fft_factors(h->nx, &a) && fft_factors(h->ny, &b);
}

static bool cn_line(const pic_t *h) {
    if (h->cfg.cn_precond == PIC_CN_PRECOND_JACOBI || h->periodic_x || (h->ny & (h->ny - 1)) != 0 || h->ny < 2 ||
        h->ny > 4096 || line_sweep_bytes(h->nxn) > 200 * 1024)   // a mode's sweep must fit in shared memory
        return false;
    // automatic: block-Jacobi (on the 1024 x 512 foil the line preconditioner cuts the iterations from
    // 6 to 3 at c dt/dx = 0.4 and from 19 to 6 at 2, but each application costs ~7 block-Jacobi ones)
    return h->cfg.cn_precond == PIC_CN_PRECOND_FFT;
}

// floats of the line preconditioner's arrays: column means, factors, sweep work
static size_t cn_line_floats(const pic_t *h) {
    return (size_t)h->nxn * (3 + 16 * (size_t)(h->ny / 2 + 1));
}

static CNVec cn_views(pic_t *h, double **Md) {
    char *base = (char *)h->cn;
    const size_t n = (size_t)h->nnode;
    CNVec v;
    v.x = (V4<double> *)base;
    v.b = v.x + n;
    v.cc = v.b + n;                  // cells: nx * ny = n (periodic x)
    V4<float> *f = (V4<float> *)(v.cc + n);
    V4<float> **slots[9] = {&v.d, &v.r, &v.r0, &v.p, &v.v, &v.s, &v.t, &v.ph, &v.sh};
    for (int k = 0; k < 9; ++k) *slots[k] = f + k * n;
    v.minv = (float *)(f + 9 * n);
    v.S = v.minv + 9 * n;
    *Md = (double *)(v.S + 9 * n);   // 312 n bytes from the base: 8-byte aligned
    v.FA = (float2 *)(*Md + (size_t)NMOM * n);
    v.FB = v.FA + n;
    v.GA = v.FB + n;
    v.GB = v.GA + n;
    v.twx = v.GB + n;
    v.twy = v.twx + h->nx / 2 + 1;
    auto log2i = [](int x) { int l = 0; while ((1 << l) < x) ++l; return l; };
    v.fft = cn_spectral(h) ? 1 : 0;
    fft_factors(h->nx, &v.ax);
    fft_factors(h->ny, &v.ay);
    v.ly = log2i(h->ny);
    v.line = cn_line(h) ? 1 : 0;
    v.scol = (float *)(v.twy + h->ny / 2 + 1);
    v.lf = v.scol + 3 * (size_t)h->nxn;
    v.lw = v.lf + 10 * (size_t)h->nxn * (h->ny / 2 + 1);
    return v;
}

// dynamic shared memory of the CN solve: two FFT row buffers and the
// per-stage twiddles (spectral preconditioner), else one transpose tile
static size_t cn_smem(const pic_t *h) {
    size_t nmax = (size_t)(h->nx > h->ny ? h->nx : h->ny);
    const size_t tile = 32 * 33 * sizeof(float2);
    if (cn_line(h)) nmax = (size_t)h->ny;   // its FFTs run along y only
    else if (!cn_spectral(h)) return tile;
    // two row-group buffers and the per-stage twiddles (spectral: of both axes)
    size_t fft = cn_line(h) ? (2 * (size_t)fft_buffer((int)nmax, 0) + nmax) * sizeof(float2)
                            : (2 * (size_t)spectral_buffer(h->nx, h->ny) + h->nx + h->ny) * sizeof(float2);
    if (cn_line(h) && line_sweep_bytes(h->nxn) > fft) fft = line_sweep_bytes(h->nxn);
    return fft > tile ? fft : tile;
}

size_t cn_bytes(const pic_t *h) {
    const size_t n = (size_t)h->nnode;
    return 3 * n * sizeof(V4<double>) + 9 * n * sizeof(V4<float>) + 18 * n * sizeof(float) +
           (size_t)NMOM * n * sizeof(double) + 4 * n * sizeof(float2) + (size_t)(h->nx + h->ny + 4) * sizeof(float2) +
           cn_line_floats(h) * sizeof(float) + 16;
}

// Grids of up to CN_CLUSTER_NODES nodes are solved by one cluster of CN_CLUSTER
// blocks, whose barrier is much cheaper than a grid barrier (a solve has some
// thirty of them); larger grids need more SMs (field solve on one cluster / on
// the grid, us: 64 x 64 163 / 192, 96 x 64 with walls 255 / 256, 128 x 64 206 /
// 197, 128 x 128 312 / 209).
constexpr int64_t CN_CLUSTER_NODES = 6144;

static void cn_cluster_config(cudaLaunchConfig_t &lc, cudaLaunchAttribute *at, size_t smem, cudaStream_t st) {
    lc.gridDim = dim3(CN_CLUSTER);
    lc.blockDim = dim3(CN_CLUSTER_BS);
    lc.dynamicSmemBytes = smem;
    lc.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CN_CLUSTER;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
}

static bool cn_single_cluster(const pic_t *h, size_t smem) {
    if (h->nnode > CN_CLUSTER_NODES || h->cn_red_cap < CN_CLUSTER) return false;
    const void *k = (const void *)k_cn_solve<true, CN_CLUSTER_BS>;
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute at[1];
    cn_cluster_config(lc, at, smem, h->st);
    int n = 0;   // (clusters of more than 8 blocks are opt-in, and may not fit a partitioned GPU)
    if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        allow_smem(k, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, k, &lc) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n >= 1;
}

template <typename R>
static int field_cn_t(pic_t *h) {
    GridArgs<R> g = grid_args<R>(h);
    GridArgs<double> gd = grid_args<double>(h);
    double *Md = nullptr;
    CNVec v = cn_views(h, &Md);
    const double *Msrc = h->fp32 ? Md : (const double *)h->M;   // planes 1 .. 9: S
    const bool clr = h->fp32 && !h->det;
    double c2 = 0.25 * h->cfg.dt * h->cfg.dt;
    WallRows wr{1.0 / h->cfg.dt + 1.0 / h->cfg.dx, 1.0 / h->cfg.dt - 1.0 / h->cfg.dx};
    Inc inc = incident(h);
    k_cn_setup<R><<<node_grid(h, 128), 128, 0, h->st>>>(gd, (const V4<R> *)h->E[h->ecur], (const V4<R> *)h->H[h->hcur],
                                                         (R *)h->M, (R *)h->Mlo, Md, clr ? 1 : 0, v.fft || v.line ? 0 : 1,
                                                         v, c2, wr, inc);
    count_launch(h);
    h->moments_cleared = clr;
    if (int rc = check_launch("k_cn_setup")) return rc;
    int dev = 0, nsm = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    double tol = h->cfg.cn_tol > 0 ? h->cfg.cn_tol : (h->fp32 ? 1e-10 : 1e-12);
    int maxit = h->cfg.cn_max_iter > 0 ? h->cfg.cn_max_iter : 400;
    void *args[] = {(void *)&gd, (void *)&Msrc, (void *)&v, (void *)&c2, (void *)&tol, (void *)&maxit,
                    (void *)&h->cn_red, (void *)&h->cn_out, (void *)&wr};
    const size_t smem = cn_smem(h);
    cudaError_t e;
    if (cn_single_cluster(h, smem)) {
        const void *k = (const void *)k_cn_solve<true, CN_CLUSTER_BS>;
        cudaLaunchConfig_t lc = {};
        cudaLaunchAttribute at[1];
        cn_cluster_config(lc, at, smem, h->st);
        e = cudaLaunchKernelExC(&lc, k, args);
    } else {
        const void *k = (const void *)k_cn_solve<false, CN_BS>;
        // the whole grid must be resident: fix the shared-memory split before asking how many blocks fit
        allow_smem(k, smem);
        cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, CN_BS, smem);
        int nb = per_sm * nsm;
        int need = (int)((h->nnode + CN_BS - 1) / CN_BS);
        if (nb > need) nb = need;
        if (nb < 1) nb = 1;
        if (nb > h->cn_red_cap) {
            set_error("CN reduction scratch too small (%d < %d)", h->cn_red_cap, nb);
            return PIC_ERR_STATE;
        }
        e = cudaLaunchCooperativeKernel(k, dim3(nb), dim3(CN_BS), args, smem, h->st);
    }
    count_launch(h);
    if (e != cudaSuccess) {
        set_error("launch of k_cn_solve: %s", cudaGetErrorString(e));
        return PIC_ERR_CUDA;
    }
    int en = 1 - h->ecur;
    k_cn_finish<R><<<node_grid(h, 128), 128, 0, h->st>>>(g, v.x, (const V4<R> *)h->E[h->ecur], (V4<R> *)h->E[en],
                                                          (V4<R> *)h->Ehalf);
    count_launch(h);
    if (int rc = check_launch("k_cn_finish")) return rc;
    return field_HB<R, double>(h, v.x);
}

int field_cn(pic_t *h) { return h->fp32 ? field_cn_t<float>(h) : field_cn_t<double>(h); }

// --------------------------------------------------------------------------- host <-> device field transfer

template <typename R>
__global__ void k_planar_to_v4(const double *__restrict__ src, int64_t n, V4<R> *__restrict__ dst) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) dst[t] = V4<R>{(R)src[t], (R)src[n + t], (R)src[2 * n + t], R(0)};
}

template <typename R>
__global__ void k_v4_to_planar(const V4<R> *__restrict__ src, int64_t n, double *__restrict__ dst) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) {
        V4<R> v = src[t];
        dst[t] = (double)v.x;
        dst[n + t] = (double)v.y;
        dst[2 * n + t] = (double)v.z;
    }
}

template <typename R>
static int upload_fields_t(pic_t *h, const double *E3, const double *H3) {
    if (E3) {
        int64_t n = h->nnode;
        if (cudaMemcpyAsync(h->stage, E3, 3 * n * sizeof(double), cudaMemcpyHostToDevice, h->st) != cudaSuccess)
            return check_launch("upload E");
        k_planar_to_v4<R><<<(unsigned)((n + 255) / 256), 256, 0, h->st>>>(h->stage, n, (V4<R> *)h->E[h->ecur]);
        count_launch(h);
        if (int rc = check_launch("k_planar_to_v4(E)")) return rc;
    }
    if (H3) {
        int64_t n = h->ncell;
        if (cudaMemcpyAsync(h->stage, H3, 3 * n * sizeof(double), cudaMemcpyHostToDevice, h->st) != cudaSuccess)
            return check_launch("upload H");
        k_planar_to_v4<R><<<(unsigned)((n + 255) / 256), 256, 0, h->st>>>(h->stage, n, (V4<R> *)h->H[h->hcur]);
        count_launch(h);
        if (int rc = check_launch("k_planar_to_v4(H)")) return rc;
        cudaMemcpyAsync(h->H[1 - h->hcur], h->H[h->hcur], n * sizeof(V4<R>), cudaMemcpyDeviceToDevice, h->st);
    }
    return 0;
}

int upload_fields(pic_t *h, const double *E3, const double *H3) {
    return h->fp32 ? upload_fields_t<float>(h, E3, H3) : upload_fields_t<double>(h, E3, H3);
}

template <typename R>
static int download_fields_t(pic_t *h, double *E3, double *H3) {
    if (E3) {
        int64_t n = h->nnode;
        k_v4_to_planar<R><<<(unsigned)((n + 255) / 256), 256, 0, h->st>>>((const V4<R> *)h->E[h->ecur], n, h->stage);
        count_launch(h);
        if (int rc = check_launch("k_v4_to_planar(E)")) return rc;
        cudaMemcpyAsync(E3, h->stage, 3 * n * sizeof(double), cudaMemcpyDeviceToHost, h->st);
        if (cudaStreamSynchronize(h->st) != cudaSuccess) return check_launch("download E");
    }
    if (H3) {
        int64_t n = h->ncell;
        k_v4_to_planar<R><<<(unsigned)((n + 255) / 256), 256, 0, h->st>>>((const V4<R> *)h->H[h->hcur], n, h->stage);
        count_launch(h);
        if (int rc = check_launch("k_v4_to_planar(H)")) return rc;
        cudaMemcpyAsync(H3, h->stage, 3 * n * sizeof(double), cudaMemcpyDeviceToHost, h->st);
        if (cudaStreamSynchronize(h->st) != cudaSuccess) return check_launch("download H");
    }
    return 0;
}

int download_fields(pic_t *h, double *E3, double *H3) {
    return h->fp32 ? download_fields_t<float>(h, E3, H3) : download_fields_t<double>(h, E3, H3);
}

}  // namespace pic
