// Internal definitions of libpic: the handle, device buffers, small vector
// type, device helpers shared by the kernels, and host launch entry points.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string>

#include <vector>

#include "pic.h"

namespace pic {

constexpr int NMOM = 13;          // rho, S (9, row-major), dj (3)

// Checks build (compiled with PIC_CHECKS): the kernels test their invariants
// (cell indices in range, offsets in [0, 1), destinations inside their bin,
// the shared-memory canary after the push's accumulator) and record a broken
// one in the sticky flags (FLAG_CHECK) instead of touching memory out of
// range.  In the normal build every check compiles away.
#ifdef PIC_CHECKS
constexpr bool kChecks = true;
#else
constexpr bool kChecks = false;
#endif
constexpr int32_t FLAG_CHECK = 32;
constexpr uint32_t CANARY = 0xC0DEC0DEu;
constexpr uint32_t KEY_DEAD = 0xFFFFFFFFu;

// Four-component vector (x, y, z, spare) stored 4*sizeof(T)-aligned so that
// a node's field is one vector load.
template <typename T>
struct alignas(4 * sizeof(T)) V4 {
    T x, y, z, w;
};

void set_error(const char *fmt, ...);

// --------------------------------------------------------------------------- handle

// Particles of one species live in tile bins made of 32-slot segments: bin t
// occupies slots [bstart[t], bstart[t+1]) of the "bins" buffer (multiples of
// SEG), uses its first useg[t] segments, and segment j holds segn[j] valid
// particles at its front.  The species' particle order is: tiles ascending,
// inside a tile its segments in order, inside a segment its valid prefix.
// Three buffer sets rotate roles: bins, mirror (the leavers of the current
// step, kept in the segment they left, at its front, count segml[j]) and spare
// (output of the per-step regroup or of a full rebuild; staging of a load).
constexpr int SEG = 32;

// FP64 form: quantities each deposit computes and the next push needs again.
// The push of step n+1 gathers the node B the moments of step n were made with,
// at the same position and with the same u, so its 1/gamma, b = q dt B /
// (2 m gamma) and 1/(1 + |b|^2) are exactly the deposit's.  They are kept per
// particle (planes of NCARRY values beside the state) instead of recomputed:
// on this GPU's FP64 pipe a B gather, a reciprocal square root and a
// reciprocal cost far more than reading and writing 40 bytes.
constexpr int NCARRY = 5;   // 1/gamma, bx, by, bz, 1/(1 + |b|^2)

struct SpeciesBuf {
    double q = 0, m = 1;
    int64_t cap = 0;   // slots per buffer set (multiple of SEG)
    int64_t n = 0;     // host copy of the live count (exact after a sync)
    bool n_exact = true;   // n is the live count (no step since it was read or set)
    int bins = 0, mir = 1, spare = 2;
    void *mem = nullptr;   // one allocation: the three buffer sets and the segment counts below
    int32_t *cell[3] = {nullptr, nullptr, nullptr};
    void *ox[3] = {nullptr, nullptr, nullptr}, *oy[3] = {nullptr, nullptr, nullptr};
    void *ux[3] = {nullptr, nullptr, nullptr}, *uy[3] = {nullptr, nullptr, nullptr};
    void *uz[3] = {nullptr, nullptr, nullptr}, *w[3] = {nullptr, nullptr, nullptr};
    double *carry[3] = {nullptr, nullptr, nullptr};   // FP64 form: [NCARRY][cap] carried quantities per set
    unsigned long long *segd = nullptr;   // [cap/SEG] leavers per mirror segment and neighbour (8 bits each)
    int32_t *segn[2] = {nullptr, nullptr};  // [cap/SEG] valid particles per bin segment
    int32_t *useg[2] = {nullptr, nullptr};  // [ntiles] segments in use per bin
    int scur = 0;               // segn[scur], useg[scur] describe the bins; the regroup writes the other pair
    int32_t *segml = nullptr;   // [cap/SEG] leavers per mirror segment (this step)
    int32_t *bstart = nullptr;  // [ntiles + 1] slot offsets of the bins
    int32_t *tcount = nullptr;  // [ntiles + 1] scratch: particles per tile
    int32_t *cstart = nullptr;  // [ntiles + 1] scratch: compact starts
    int32_t *cend = nullptr;    // [ntiles + 1] scratch: run ends of a rebuild
};

// Several device arrays in one allocation, 256-byte aligned each: a served run
// spent 0.6 ms in its hundred cudaMalloc calls and 0.55 ms in cudaFree, more than
// in its 40 steps; a burst of 12 takes 31.5 ms with these, 43.7 ms without.
struct Slab {
    struct Part {
        void **p;
        size_t at;
    };
    std::vector<Part> parts;
    size_t bytes = 0;
    template <typename T>
    void add(T **p, size_t n) {
        *p = nullptr;
        if (n == 0) return;
        parts.push_back(Part{(void **)p, bytes});
        bytes += (n + 255) / 256 * 256;
    }
    int commit(void **base, const char *what);   // the allocation (freed by its base alone) and every pointer
};

// Counters of a set of tile lists.
enum { LC_TOUCH = 0, LC_REGROUP = 1, LC_QUEUE = 2, LC_ITEMS = LC_QUEUE + PIC_MAX_SPECIES, LC_TICKET, LC_DEPOSIT, LC_SIZE = 16 };
static_assert(LC_DEPOSIT < LC_SIZE, "counters of a set");

struct Timing {
    bool enabled = false;
    double ms[4] = {0, 0, 0, 0};
    int64_t launches[5] = {0, 0, 0, 0, 0};
};

}  // namespace pic

struct pic_t {
    pic_config cfg;
    cudaStream_t st = nullptr;
    bool fp32 = false;
    size_t rs = 8;                      // sizeof(real)
    bool periodic_x = true;
    int nx = 0, ny = 0, nxn = 0;
    int64_t nnode = 0, ncell = 0;
    int G = 0, nxp = 0, nyp = 0;        // ghost width and padded node-array dims
    int64_t npad = 0;
    int tnx = 16, tny = 16, ntx = 0, nty = 0, ntiles = 0;

    void *mem = nullptr;                // one allocation: the grid arrays, tile lists and bins of the handle
    // fields, all V4<real>
    void *E[2] = {nullptr, nullptr};    // nodes [nnode]; E[ecur] = E^n
    int ecur = 0;
    void *H[2] = {nullptr, nullptr};    // cells [ncell]; H[hcur] current, H[1-hcur] previous
    int hcur = 0;
    void *Ehalf = nullptr;              // padded nodes: E^n + E^{n+1}, twice the E the push sees
    void *B[2] = {nullptr, nullptr};    // padded nodes: B[bcur] = four times the node B the moments were made with
    int bcur = 0;
    void *M = nullptr;                  // raw moment sums, planar [13][nnode] real

    // CN solver work (FP64 V4 vectors of nnode) and reduction scratch
    void *cn = nullptr;
    double *cn_red = nullptr;           // per-block partials
    int cn_red_cap = 0;
    double *cn_out = nullptr;           // [iterations, residual]

    // particles
    int nsp = 0;
    pic::SpeciesBuf sp[PIC_MAX_SPECIES];
    int64_t *d_removed = nullptr;       // [nsp] cumulative wall removals
    int32_t *d_flags = nullptr;         // sticky: bit 0 far mover seen, bit 2 capacity, bit 3 TMA wait timeout
    int32_t *d_step_flags = nullptr;    // [2], one per step parity: bit 0 far mover, bit 1 bin overflow -> full rebuild;
                                        // d_flags is the word after them
    int32_t *h_step_flags = nullptr;    // pinned: [4 p ..] those three words after a step of parity p, [3] d_flags after
                                        // a load
    const int32_t *guard = nullptr;     // steps: the previous step's flags; its particle kernels do nothing if set
    void *h_diag = nullptr;             // pinned host copy of the diagnostics record
    cudaEvent_t ev_flags[2] = {nullptr, nullptr};   // per step parity: that step's flags are on the host
    bool flags_pending = false;         // a step's regroup flags are in flight (its regroup already committed)
    int pending_p = 0;                  // that step's parity
    bool pending_post = false;          // that step deposits after its regroup (nothing if the regroup failed)
    int halo = 1;                       // deposit halo of a tile, in cells
    void *Mlo = nullptr;                // FP32 form: second part of the moment sums (compensation, stragglers)
    bool det = false;                   // deterministic deposit: exact fixed-point sums in Mfix
    unsigned long long *Mfix = nullptr; // [13][nnode] two's-complement fixed-point moment sums
    double *Mc = nullptr;               // FP64 L2-reduction push (linear shape): cell sums [ncell][13][4]
    double wabs[PIC_MAX_SPECIES] = {0, 0, 0, 0, 0, 0, 0, 0};  // sum of |w| loaded per species
    void *tmaps = nullptr;              // host storage of the TMA descriptors
    int2 *items = nullptr;              // work item k of the push -> (species-tile index, run within it)
    int64_t items_cap = 0;
    int32_t *ticket = nullptr;          // work-queue counters of a deposit at rest
    int32_t *nbr = nullptr;             // [ntiles][9] neighbour count, then the neighbour tiles ascending
    // Tile lists, three sets in turn (push_prep): the field solve and the clear of a step read the set of the
    // last push (touch_cur) while the next push's set (lists) is made, which zeroes the third one's counters.
    int32_t *counters = nullptr;        // [3][pic::LC_SIZE]
    uint8_t *touched = nullptr;         // [3][ntiles] node tiles whose moments the push may write
    int32_t *touch_list = nullptr;      // [3][ntiles] the touched tiles, in no particular order
    int32_t *rg_list = nullptr;         // [ntiles] tiles the regroup must visit (an occupied tile or neighbour)
    int lists = 0, touch_cur = 0;
    bool lists_zero[3] = {true, true, true};   // the set's counters are (or will be, in stream order) zero
    const int32_t *touch_far = nullptr; // flags word of the last push: bit 0 (a far move), every tile is touched
    int regroup_blocks = 0;             // blocks per species of the list-driven regroup
    bool touch_all = true;              // no touched-tile map: moments may be non-zero anywhere (after init)
    bool moments_cleared = false;       // the last field solve zeroed the moments it read
    unsigned long long *d_bad = nullptr;  // per species: first invalid particle index of a load
    uint32_t *scan_sums = nullptr;      // per-block totals of the multi-block scans
    bool moments_stale = false;         // particles or B changed since the last deposit at rest
    bool post = false;                  // steps deposit after the regroup (post_deposit)
    bool shared_gpu = false;            // steps beside other runs': no second stream (set_shared)
    cudaEvent_t ev_batch = nullptr;     // a batched step: this run's prologue is queued
    cudaStream_t st2 = nullptr;         // loads: regroups of converted species, beside the next conversion
    cudaEvent_t ev_load = nullptr;      // loads: st2's work joined back to st
    cudaEvent_t ev_conv[PIC_MAX_SPECIES] = {};   // loads: a species' conversion is done (st -> st2)
    cudaStream_t st3 = nullptr;         // loads: the species' sorts, beside the previous species' deposit at rest
    cudaEvent_t ev_sorted[PIC_MAX_SPECIES] = {};   // loads: a species is sorted into its bins (st3 -> st2)
    cudaEvent_t ev_sorts = nullptr;     // loads: every sort is done (st3 -> st2)
    cudaEvent_t ev_push = nullptr;      // steps: the push (and its moments) is done (st -> st2)
    cudaEvent_t ev_field = nullptr;     // steps: the field solve is done (st2 -> st)
    cudaEvent_t ev_cellm = nullptr;     // steps: the push's cell sums are in the node moments (st2 -> st)
    int push_blocks = 0;                // persistent grid size of the push
    int items_ch = 0;                   // segments per work item of the current item table

    // sort scratch
    void *sort_mem = nullptr;           // one allocation: the sort scratch
    uint32_t *keys[2] = {nullptr, nullptr};   // sort scratch, 2*cap entries
    uint32_t *vals[2] = {nullptr, nullptr};
    uint32_t *hist = nullptr;
    int64_t sort_cap = 0, hist_cap = 0;

    // staging for load / readback (device FP64)
    double *stage = nullptr;
    int64_t stage_cap = 0;

    // prefetched loads (pic_prefetch_species): two slots of device copies, loaded in the order filled
    struct Prefetch {
        double *buf = nullptr;          // per species the six arrays, one after another
        int64_t cap = 0;                // doubles
        int nsp = 0;
        int64_t n[PIC_MAX_SPECIES] = {};
        cudaEvent_t copied = nullptr;   // the copy is complete (pf_st -> st)
        cudaEvent_t freed = nullptr;    // the load that read it is complete (st -> pf_st)
    } pf[2];
    int pf_head = 0, pf_count = 0;      // oldest filled slot, filled slots
    cudaStream_t pf_st = nullptr;       // the prefetch copies

    // field ionisation: staging of the ionised particles (checkpoint form) and of multi-source appends
    int32_t *ion_cell = nullptr;
    double *ion_val = nullptr;          // [6][ion_cap]
    int64_t ion_cap = 0;
    int32_t *ion_dcell = nullptr;
    double *ion_dval = nullptr;         // [6][ion_dcap]
    int64_t ion_dcap = 0;

    // diagnostics scratch
    double *d_diag = nullptr;           // partial sums
    int diag_cap = 0;

    int64_t step = 0;
    int64_t rebuilds = 0;               // full regroups run by the step fallback
    int shape = 1;                      // particle shape order: 1 (area weighting) or 2 (quadratic spline)
    int push_blocks_s2 = 0;             // grid of the order-2 push
    int cn_iters_last = 0;
    double cn_res_last = 0.0;
    pic::Timing timing;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
};

namespace pic {

// --------------------------------------------------------------------------- kernels' argument blocks

template <typename R>
struct GridArgs {
    int nx, ny, nxn, G, nxp;
    int periodic_x;
    R dx, dy, dt;
    R inv_dx, inv_dy;
    R hx, hy;       // 1/(2 dx), 1/(2 dy): the centred differences of the curls
    R khx, khy;     // dt/(2 dx), dt/(2 dy)
    int64_t nnode;
};

template <typename R>
GridArgs<R> grid_args(const pic_t *h) {
    GridArgs<R> g;
    g.nx = h->nx; g.ny = h->ny; g.nxn = h->nxn; g.G = h->G; g.nxp = h->nxp;
    g.periodic_x = h->periodic_x ? 1 : 0;
    g.dx = (R)h->cfg.dx; g.dy = (R)h->cfg.dy; g.dt = (R)h->cfg.dt;
    g.inv_dx = (R)(1.0 / h->cfg.dx); g.inv_dy = (R)(1.0 / h->cfg.dy);
    g.hx = (R)(0.5 / h->cfg.dx); g.hy = (R)(0.5 / h->cfg.dy);
    g.khx = (R)(0.5 * h->cfg.dt / h->cfg.dx); g.khy = (R)(0.5 * h->cfg.dt / h->cfg.dy);
    g.nnode = h->nnode;
    return g;
}

template <typename R>
__host__ __device__ inline int64_t pidx(const GridArgs<R> &g, int i, int j) {
    return (int64_t)(j + g.G) * g.nxp + (i + g.G);
}

// --------------------------------------------------------------------------- device helpers

// The FP32 value nearest to v (ties to even) and the FP64 value of f, from
// their bits: a conversion instruction issues on the FP64 pipe.  In 32-bit halves,
// since a mask that takes the sign off the whole word is compiled to an FP64
// operation as well (the load conversion issued 18 of them per particle, 8 of
// which are arithmetic).
__device__ inline float narrow(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v), h = hi & 0x7fffffffu, e = h >> 20;
    unsigned r;
    if (e >= 897) {
        r = __funnelshift_l(lo, hi, 3) - (896u << 23);
        r += (lo & 0x1fffffffu) > 0x10000000u - (r & 1u) ? 1u : 0u;
        if (e > 1150) r = h > 0x7ff00000u || (h == 0x7ff00000u && lo) ? 0x7fffffffu : 0x7f800000u;
    } else {   // FP32 denormals and zero
        const unsigned sh = 926 - e;
        const unsigned long long q = ((unsigned long long)((h & 0xfffffu) | 0x100000u) << 32) | lo;
        r = sh > 54 ? 0u : (unsigned)((q + ((1ull << (sh - 1)) - 1) + ((q >> sh) & 1)) >> sh);
    }
    return __uint_as_float(r | (hi & 0x80000000u));
}
__device__ inline double widen(float f) {
    const unsigned u = __float_as_uint(f), m = u & 0x7fffffffu;
    unsigned long long d = 0;
    if (m >= 0x00800000u) {
        d = ((unsigned long long)m << 29) + ((m >= 0x7f800000u ? 1792ull : 896ull) << 52);
    } else if (m) {
        const int z = __clz(m);
        d = ((unsigned long long)((m << (z - 8)) & 0x7fffffu) << 29) | ((unsigned long long)(905 - z) << 52);
    }
    return __longlong_as_double((long long)(d | (unsigned long long)(u & 0x80000000u) << 32));
}
__device__ inline double widen(double v) { return v; }
// v in the storage type (FP64 or FP32).
template <typename R>
__device__ inline R stored(double v) {
    if constexpr (sizeof(R) == 4) return narrow(v);
    else return v;
}

// 1/sqrt(x) and 1/x: in FP32 the hardware approximations (2 ulp, far below the
// FP32 form's tolerances); in FP64 the library's correctly rounded forms.
__device__ inline float rsqrt_r(float x) { return rsqrtf(x); }
__device__ inline double rsqrt_r(double x) { return rsqrt(x); }
__device__ inline float rcp_r(float x) { return __fdividef(1.0f, x); }
__device__ inline double rcp_r(double x) { return __drcp_rn(x); }

// x >= 1 for a non-negative x.  FP64: an integer compare of the bits (ordered
// like the values for non-negative doubles), which keeps the comparison off
// the narrow FP64 pipe.
__device__ inline bool ge_one(double x) { return __double_as_longlong(x) >= 0x3FF0000000000000ll; }
__device__ inline bool ge_one(float x) { return x >= 1.0f; }

__device__ inline double fma_r(double a, double b, double c) { return fma(a, b, c); }
__device__ inline float fma_r(float a, float b, float c) { return fmaf(a, b, c); }

// (R(b) v)_x = v_x + (v.b) b_x + v_y b_z - v_z b_y (and cyclically) before the
// division by 1 + |b|^2: three FMAs per component.
template <typename R>
__device__ inline R rot_row(R v0, R v1, R v2, R vb, R b0, R b1, R b2) {
    return fma_r(v1, b2, fma_r(-v2, b1, fma_r(vb, b0, v0)));
}

// The implicit push's velocity update and move (Eq. 2) from w = u + k E: the
// rows r of (1 + |b|^2) R(b) w, then u' = 2 ubar - u = r (2 inv) - u and the
// move in cells s = f + dt/dx ubar/gamma = f + r (inv/gamma) dt/dx (one
// product fewer than forming ubar first).
template <typename R>
__device__ inline void push_move(R bx, R by, R bz, R inv, R ig, R wx, R wy, R wz, R ux, R uy, R uz, R fx, R fy,
                                 R sdx, R sdy, R &nux, R &nuy, R &nuz, R &sx, R &sy) {
    const R vb = wx * bx + wy * by + wz * bz;
    const R rx = rot_row(wx, wy, wz, vb, bx, by, bz), ry = rot_row(wy, wz, wx, vb, by, bz, bx);
    const R rz = rot_row(wz, wx, wy, vb, bz, bx, by);
    const R i2 = R(2) * inv, ti = inv * ig;
    nux = fma_r(rx, i2, -ux);
    nuy = fma_r(ry, i2, -uy);
    nuz = fma_r(rz, i2, -uz);
    sx = fma_r(rx, ti * sdx, fx);
    sy = fma_r(ry, ti * sdy, fy);
}

// The 13 moments one particle contributes (Eq. 3): rho = w q,
// S = w q^2 dt^2 / (4 m gamma) R(b), dj = w q R(b) u / gamma, with
// gamma = sqrt(1 + |u|^2) and b = q dt B / (2 m gamma).
// kq = q dt / (2 m) and hq = q dt^2 / (4 m) are per-species constants (the S
// factor w q^2 dt^2 / (4 m gamma (1+|b|^2)) is the dj factor times hq).  Also
// returns 1/gamma, b and 1/(1 + |b|^2) (the FP64 form carries them to the next
// push).
template <typename R>
__device__ inline void particle_moments_c(R q, R kq, R hq, R w, R ux, R uy, R uz, R Bx, R By, R Bz, R *val, R &ig,
                                          R &bx, R &by, R &bz, R &inv) {
    ig = rsqrt_r(R(1) + ux * ux + uy * uy + uz * uz);
    R k = kq * ig;
    bx = k * Bx, by = k * By, bz = k * Bz;
    inv = rcp_r(R(1) + bx * bx + by * by + bz * bz);
    const R gi = ig * inv;
    val[0] = w * q;
    const R cj = val[0] * gi, cs = cj * hq;
    // cs times the rows of (I + [.x b] + b b^T) ((R v)_x = v_x + v_y bz - v_z by + (v.b) bx, ...):
    // with c = cs b each entry is one FMA, e.g. cs (bz + bx by) = cz + cx by
    const R cx = cs * bx, cy = cs * by, cz = cs * bz;
    val[1] = fma_r(cx, bx, cs);
    val[2] = fma_r(cx, by, cz);
    val[3] = fma_r(cx, bz, -cy);
    val[4] = fma_r(cy, bx, -cz);
    val[5] = fma_r(cy, by, cs);
    val[6] = fma_r(cy, bz, cx);
    val[7] = fma_r(cz, bx, cy);
    val[8] = fma_r(cz, by, -cx);
    val[9] = fma_r(cz, bz, cs);
    R vb = ux * bx + uy * by + uz * bz;
    val[10] = cj * rot_row(ux, uy, uz, vb, bx, by, bz);
    val[11] = cj * rot_row(uy, uz, ux, vb, by, bz, bx);
    val[12] = cj * rot_row(uz, ux, uy, vb, bz, bx, by);
}

// The same moments as class factors times unscaled parts (FP64 deposits, which
// fold the factors into the corner weights: 4 products per class instead of
// 13 scalings): rho = fr, S = fS part[1..9], dj = fj part[10..12] (part[0] is
// not set).  Same 1/gamma, b, 1/(1+|b|^2) as particle_moments_c.
template <typename R>
__device__ inline void particle_moment_parts(R q, R kq, R cq2, R w, R ux, R uy, R uz, R Bx, R By, R Bz, R *part,
                                             R &fr, R &fS, R &fj, R &ig, R &bx, R &by, R &bz, R &inv) {
    ig = rsqrt_r(R(1) + ux * ux + uy * uy + uz * uz);
    R k = kq * ig;
    bx = k * Bx, by = k * By, bz = k * Bz;
    inv = rcp_r(R(1) + bx * bx + by * by + bz * bz);
    const R gi = ig * inv;
    fr = w * q;
    fS = (w * cq2) * gi;
    fj = fr * gi;
    part[1] = R(1) + bx * bx;
    part[2] = bz + bx * by;
    part[3] = -by + bx * bz;
    part[4] = -bz + by * bx;
    part[5] = R(1) + by * by;
    part[6] = bx + by * bz;
    part[7] = by + bz * bx;
    part[8] = -bx + bz * by;
    part[9] = R(1) + bz * bz;
    R vb = ux * bx + uy * by + uz * bz;
    part[10] = rot_row(ux, uy, uz, vb, bx, by, bz);
    part[11] = rot_row(uy, uz, ux, vb, by, bz, bx);
    part[12] = rot_row(uz, ux, uy, vb, bz, bx, by);
}

// Deterministic deposit.  Every corner contribution of a particle is rounded
// once to an integer multiple of 2^-e[class] and the integers are summed with
// 64-bit integer additions, which are exact and associative: the sums do not
// depend on the order in which warps, blocks or atomics add them.  The classes
// are rho (moment 0), S (1..9) and dj (10..12).  |rho| and every |dj| component
// of one particle are at most |w q| (|R(b) u| <= |u| < gamma), every |S|
// entry at most |w| q^2 dt^2 / (4 m) (R(b) entries are at most 1 in size, and
// 1/gamma <= 1), and the bilinear weights of one particle on one node are at
// most 1, so a node sum stays below the class bound B = sum over all loaded
// particles; e = 62 - ceil(log2 B) keeps |sum| 2^e <= 2^62.
struct FixScale {
    int e[3];     // exponents of the classes rho, S, dj
    float s[3];   // 2^e (FP32 form)
    double inv[3];  // 2^-e
};

__host__ __device__ constexpr int mom_class(int k) { return k == 0 ? 0 : (k < 10 ? 1 : 2); }

// x 2^e rounded to the nearest integer (ties away from zero), from the bits of
// x with integer operations only.
__device__ inline long long fix_of(double x, const FixScale &f, int cls) {
    const long long b = __double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7ff);
    const long long m = (b & 0xFFFFFFFFFFFFFll) | 0x10000000000000ll;
    const int sh = ex - 1075 + f.e[cls];   // |x| 2^e = m 2^sh
    long long r;
    if (ex == 0 || sh <= -64) r = 0;
    else if (sh >= 0) r = m << sh;          // sh <= 9 while |x| 2^e < 2^62
    else r = (m + (1ll << (-sh - 1))) >> (-sh);
    return b < 0 ? -r : r;
}
__device__ inline long long fix_of(float x, const FixScale &f, int cls) { return __float2ll_rn(x * f.s[cls]); }

// Butterfly reduce-scatter of 26 values over the warp: returns, in every
// lane, the warp sum of one of the 26 (index rs26_index(lane), -1 for the six
// lanes that end up with padding).  26 -> 13 -> 7 -> 4 -> 2 -> 1 values per lane.
template <typename R>
__device__ inline R reduce_scatter26(const R (&v)[26], int lane) {
    R a[14];
    bool b = (lane & 16) != 0;
#pragma unroll
    for (int j = 0; j < 13; ++j) {
        R lo = v[j], hi = v[j + 13];
        R s = b ? lo : hi, k = b ? hi : lo;
        a[j] = k + __shfl_xor_sync(0xffffffffu, s, 16);
    }
    a[13] = R(0);
    R c[8];
    b = (lane & 8) != 0;
#pragma unroll
    for (int j = 0; j < 7; ++j) {
        R lo = a[j], hi = a[j + 7];
        R s = b ? lo : hi, k = b ? hi : lo;
        c[j] = k + __shfl_xor_sync(0xffffffffu, s, 8);
    }
    c[7] = R(0);
    R d[4];
    b = (lane & 4) != 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        R lo = c[j], hi = c[j + 4];
        R s = b ? lo : hi, k = b ? hi : lo;
        d[j] = k + __shfl_xor_sync(0xffffffffu, s, 4);
    }
    R e[2];
    b = (lane & 2) != 0;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        R lo = d[j], hi = d[j + 2];
        R s = b ? lo : hi, k = b ? hi : lo;
        e[j] = k + __shfl_xor_sync(0xffffffffu, s, 2);
    }
    b = (lane & 1) != 0;
    R s = b ? e[0] : e[1], k = b ? e[1] : e[0];
    return k + __shfl_xor_sync(0xffffffffu, s, 1);
}

__device__ inline int rs26_index(int lane) {
    int j2 = (lane & 1) + 2 * ((lane >> 1) & 1) + 4 * ((lane >> 2) & 1);
    if (j2 >= 7) return -1;
    int j1 = j2 + 7 * ((lane >> 3) & 1);
    if (j1 >= 13) return -1;
    return j1 + 13 * ((lane >> 4) & 1);
}

// c = cy * nx + cx split with a multiply-high (magic = ceil(2^32 / nx), c < 2^31).
__device__ inline void cell_split(int32_t c, int nx, uint32_t magic, int &cx, int &cy) {
    int q = (int)__umulhi((uint32_t)c, magic);
    int r = c - q * nx;
    if (r < 0) {
        q -= 1;
        r += nx;
    }
    cx = r;
    cy = q;
}

// a mod n for a in (-n, 2n)
__device__ inline int wrap1(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// Cell form of the bilinear weighting (Section 3.3, area weighting), used by
// every FP64 gather: per component F(fx, fy) = a + fx b + fy c + fx fy d with
// a = F00, b = F10 - F00, c = F01 - F00, d = (F11 - F10) - c -- three FMAs
// per component instead of the four corner weights and four products.  The
// FP64 push makes (a, b, c, d) once per cell of its tile; the coefficients
// and their evaluation come from these two functions alone, so that a
// particle's field is the same bits in the push and at rest.
template <typename R>
struct CellC {
    V4<R> k[3];   // per component: (a, b, c, d)
};

template <typename R>
__device__ inline V4<R> cell_coef1(R f00, R f10, R f01, R f11) {
    V4<R> v;
    v.x = f00;
    v.y = f10 - f00;
    v.z = f01 - f00;
    v.w = (f11 - f10) - v.z;
    return v;
}

template <typename R>
__device__ inline void cell_coef(const V4<R> &f00, const V4<R> &f10, const V4<R> &f01, const V4<R> &f11,
                                 CellC<R> &o) {
    o.k[0] = cell_coef1(f00.x, f10.x, f01.x, f11.x);
    o.k[1] = cell_coef1(f00.y, f10.y, f01.y, f11.y);
    o.k[2] = cell_coef1(f00.z, f10.z, f01.z, f11.z);
}

template <typename R>
__device__ inline R cell_eval(const V4<R> &k, R fx, R fy, R fxy) {
    return fma(fxy, k.w, fma(fy, k.z, fma(fx, k.y, k.x)));
}

// Bilinear gather of a padded V4 node field at cell (cx, cy), offsets (fx, fy)
// (FP64: the cell form above).
template <typename R>
__device__ inline void gather4(const V4<R> *__restrict__ F, const GridArgs<R> &g, int cx, int cy, R fx, R fy,
                               R &ox, R &oy, R &oz) {
    int64_t p00 = pidx(g, cx, cy);
    V4<R> a = F[p00], b = F[p00 + 1], c = F[p00 + g.nxp], d = F[p00 + g.nxp + 1];
    if constexpr (sizeof(R) == 8) {
        CellC<R> k;
        cell_coef(a, b, c, d, k);
        const R fxy = fx * fy;
        ox = cell_eval(k.k[0], fx, fy, fxy);
        oy = cell_eval(k.k[1], fx, fy, fxy);
        oz = cell_eval(k.k[2], fx, fy, fxy);
        return;
    }
    R w00 = (R(1) - fx) * (R(1) - fy), w10 = fx * (R(1) - fy), w01 = (R(1) - fx) * fy, w11 = fx * fy;
    ox = w00 * a.x + w10 * b.x + w01 * c.x + w11 * d.x;
    oy = w00 * a.y + w10 * b.y + w01 * c.y + w11 * d.y;
    oz = w00 * a.z + w10 * b.z + w01 * c.z + w11 * d.z;
}

// Unpadded node index of the corner (cx + di, cy + dj) with wrap.
template <typename R>
__device__ inline int64_t node_of(const GridArgs<R> &g, int cx, int cy, int di, int dj) {
    int i = cx + di, j = cy + dj;
    if (g.periodic_x && i >= g.nx) i -= g.nx;
    if (j >= g.ny) j -= g.ny;
    return (int64_t)j * g.nxn + i;
}

// FP64 deposit of one particle (in the push and at rest alike, so that a
// deposit at rest repeats the push's bitwise): per corner, the weight times
// each class factor, times the parts; every lane adds its own products in L2.
// The lanes of one cell would all add to one address in each instruction, so
// lane l starts at corner l mod 4 and, for the FP64 adds, at moment 3 ((l / 4)
// mod 4): 16 addresses per instruction, two lanes on each (the fixed-point
// adds keep the moment order: their class scale would become a run-time index).
template <bool kFix>
__device__ inline void deposit_fp64(double *M, unsigned long long *Mfix, const FixScale &fs, const GridArgs<double> &g,
                                    int cx, int cy, double fx, double fy, const double *part, double fr, double fS,
                                    double fj, int lane) {
    const double mx = 1.0 - fx, my = 1.0 - fy;
    const int rr = kFix ? 0 : (lane >> 2) & 3;
#pragma unroll
    for (int c0 = 0; c0 < 4; ++c0) {
        const int cc = (c0 + lane) & 3, ox = cc & 1, oy = cc >> 1;
        const double wc = (ox ? fx : mx) * (oy ? fy : my);   // the bilinear weight of corner (ox, oy)
        const int64_t node = node_of(g, cx, cy, ox, oy);
        const double wr = wc * fr, ws = wc * fS, wj = wc * fj;
#pragma unroll
        for (int kk = 0; kk < NMOM; ++kk) {
            if (kFix) {
                const double p = kk == 0 ? wr : (kk < 10 ? ws : wj) * part[kk];
                atomicAdd(&Mfix[(int64_t)kk * g.nnode + node], (unsigned long long)fix_of(p, fs, mom_class(kk)));
            } else {
                // moment (kk + 3 rr) mod 13: its factor and part selected (rho: factor wr, part 1)
                const int k1 = (kk + 3) % NMOM, k2 = (kk + 6) % NMOM, k3 = (kk + 9) % NMOM;
                const int km = rr == 0 ? kk : rr == 1 ? k1 : rr == 2 ? k2 : k3;
                auto fac = [&](int k) { return k == 0 ? wr : (k < 10 ? ws : wj); };
                auto prt = [&](int k) { return k == 0 ? 1.0 : part[k]; };
                const double f = rr == 0 ? fac(kk) : rr == 1 ? fac(k1) : rr == 2 ? fac(k2) : fac(k3);
                const double q = rr == 0 ? prt(kk) : rr == 1 ? prt(k1) : rr == 2 ? prt(k2) : prt(k3);
                atomicAdd(&M[(int64_t)km * g.nnode + node], f * q);
            }
        }
    }
}

// FP64 deposit of the push in cell form.  With P_k the particle's 13 moment
// values (particle_moments_c) and (fx, fy) its offsets in cell c, its
// corner contributions (1-fx)(1-fy) P, fx(1-fy) P, (1-fx) fy P and fx fy P
// (the area weighting of Section 3.3) are sums of A = P, X = fx P, Y = fy P and
// Z = fx fy P: corner (0,0) A - X - Y + Z, (1,0) X - Z, (0,1) Y - Z, (1,1) Z.
// The push adds A, X, Y, Z of every moment into its cell's sums (three
// products per moment instead of four, and no corner weights);
// k_cell_moments then adds every cell's corner values into the node moments.
// A cell's sums are adjacent, the four of a moment in one 32-byte sector; lane l
// starts at moment (l / 4) mod 2 and at sum l mod 4, so that the lanes of one
// cell spread each instruction's reductions over 8 addresses in 2 sectors
// (measured on the 1024 x 512 foil's push: 1, 2, 4, 8 moment offsets
// 2.225, 2.183, 2.191, 2.196 ms; 8 offsets with the sums in separate planes, 32
// sectors per instruction, 5.79 ms).
__device__ inline void deposit_fp64_cell(double *Mc, int64_t cell, double fx, double fy, const double *val, int lane) {
    const double fxy = fx * fy;
    double P[NMOM];
#pragma unroll
    for (int k = 0; k < NMOM; ++k) P[k] = val[k];
    // P rotated by rr: Q[k] = P[(k + rr) mod 13]
    const int rr = (lane >> 2) & 1;
    {
        double Q[NMOM];
#pragma unroll
        for (int k = 0; k < NMOM; ++k) Q[k] = rr ? P[(k + 1) % NMOM] : P[k];
#pragma unroll
        for (int k = 0; k < NMOM; ++k) P[k] = Q[k];
    }
#pragma unroll
    for (int kk = 0; kk < NMOM; ++kk) {
        const int km = kk + rr >= NMOM ? kk + rr - NMOM : kk + rr;
        const double a = P[kk], x = a * fx, y = a * fy, z = a * fxy;
        double *base = Mc + (cell * NMOM + km) * 4;
#pragma unroll
        for (int c0 = 0; c0 < 4; ++c0) {
            const int kind = (c0 + lane) & 3;
            const double v = kind == 0 ? a : kind == 1 ? x : kind == 2 ? y : z;
            atomicAdd(base + kind, v);
        }
    }
}

// ---------------------------------------------------------------- shape orders 2-4
//
// The centred B-spline of degree N (2, 3, 4) over the (N + 1) x (N + 1) nodes
// nearest the particle (the higher-order weightings Section 3.3's last
// paragraph mentions beside the paper's linear one, up to fourth order).  Per
// axis, from the cell c and offset f: the first node is c - (N - 1)/2 for odd
// N, c - N/2 (one more when f >= 1/2, centring on the nearest node) for even
// N; node k weighs B_N of its distance (first + k - c) - f.  Along y and a
// periodic x the node indices wrap; along a walled x a node beyond a wall is
// folded onto the wall node (its weight stays in the box).  N = 1 is the area
// weighting in the same form.
template <typename R, int N>
struct SplineN {
    int ix, iy;                 // first node column and row, not wrapped or folded
    R wx[N + 1], wy[N + 1];
};

// Weights of one axis (the piecewise polynomials of B_N at the N + 1 nodes,
// without branches); returns the first node relative to the cell.
template <typename R, int N>
__device__ inline int spline_axis(R f, R (&w)[N + 1]) {
    if constexpr (N == 3) {
        const R g = R(1) - f, f2 = f * f, g2 = g * g;
        w[0] = g2 * (g * R(1.0 / 6.0));
        w[1] = fma_r(f2, fma_r(R(0.5), f, R(-1)), R(2.0 / 3.0));
        w[2] = fma_r(g2, fma_r(R(0.5), g, R(-1)), R(2.0 / 3.0));
        w[3] = f2 * (f * R(1.0 / 6.0));
        return -1;
    } else {
        const int up = f >= R(0.5) ? 1 : 0;
        const R d = f - R(up), a = R(0.5) - d, b = R(0.5) + d, d2 = d * d;   // nodes at distances k - N/2 - d
        if constexpr (N == 2) {
            w[0] = (R(0.5) * a) * a;
            w[1] = R(0.75) - d2;
            w[2] = (R(0.5) * b) * b;
        } else {
            const R a2 = a * a, b2 = b * b;
            const R xl = R(1) + d, xr = R(1) - d;
            auto mid = [](R x) {   // (55 + 20 x - 120 x^2 + 80 x^3 - 16 x^4) / 96
                R p = fma_r(x, R(-16.0 / 96.0), R(80.0 / 96.0));
                p = fma_r(x, p, R(-120.0 / 96.0));
                p = fma_r(x, p, R(20.0 / 96.0));
                return fma_r(x, p, R(55.0 / 96.0));
            };
            w[0] = (a2 * R(1.0 / 24.0)) * a2;
            w[1] = mid(xl);
            w[2] = fma_r(d2, fma_r(d2, R(0.25), R(-0.625)), R(115.0 / 192.0));
            w[3] = mid(xr);
            w[4] = (b2 * R(1.0 / 24.0)) * b2;
        }
        return up - N / 2;
    }
}

template <typename R, int N>
__device__ inline SplineN<R, N> spline_n(int cx, int cy, R fx, R fy) {
    SplineN<R, N> s;
    s.ix = cx + spline_axis<R, N>(fx, s.wx);
    s.iy = cy + spline_axis<R, N>(fy, s.wy);
    return s;
}

// Column a of the stencil as a real node column: folded onto a wall, wrapped
// in a periodic box (unpadded arrays); rows always wrap.
template <typename R>
__device__ inline int spline_col(const GridArgs<R> &g, int i) {
    if (!g.periodic_x) return i < 0 ? 0 : (i > g.nx ? g.nx : i);
    i %= g.nx;
    return i < 0 ? i + g.nx : i;
}
template <typename R>
__device__ inline int spline_row(const GridArgs<R> &g, int j) {
    j %= g.ny;
    return j < 0 ? j + g.ny : j;
}

// Value of a padded V4 node field at the particle (rows first, then columns).
// The ghost ring (tile + halo + 1 >= 3 nodes) holds the periodic copies that
// the stencil reaches, so only a walled x needs its columns folded.
template <typename R, int N>
__device__ inline void gather_s(const V4<R> *__restrict__ F, const GridArgs<R> &g, const SplineN<R, N> &s, R &ox,
                                R &oy, R &oz) {
    ox = oy = oz = R(0);
    int col[N + 1];
#pragma unroll
    for (int a = 0; a <= N; ++a) col[a] = g.periodic_x ? s.ix + a : min(max(s.ix + a, 0), g.nx);
#pragma unroll
    for (int b = 0; b <= N; ++b) {
        const V4<R> *row = F + (int64_t)(s.iy + b + g.G) * g.nxp + g.G;
        R sx = R(0), sy = R(0), sz = R(0);
#pragma unroll
        for (int a = 0; a <= N; ++a) {
            const V4<R> v = row[col[a]];
            sx += s.wx[a] * v.x;
            sy += s.wx[a] * v.y;
            sz += s.wx[a] * v.z;
        }
        ox += s.wy[b] * sx;
        oy += s.wy[b] * sy;
        oz += s.wy[b] * sz;
    }
}

// Element j of a short register array, by compare and select (no local memory).
template <int M, typename T>
__device__ inline T pick(const T (&v)[M], int j) {
    T r = v[0];
#pragma unroll
    for (int q = 1; q < M; ++q) r = (j == q) ? v[q] : r;
    return r;
}

// Exact deposit of one particle with a spline shape (in the push and at rest
// alike): node by node, every lane adds its own products in fixed point, the
// lanes of a warp starting at different nodes (lane mod (N + 1)^2).  kParts:
// the values are FP64 parts with the class factors fr, fS, fj (as
// deposit_fp64 takes them); otherwise the 13 moment values.
template <typename R, bool kParts, int N>
__device__ inline void deposit_s_fix(unsigned long long *Mfix, const FixScale &fs, const GridArgs<R> &g,
                                     const SplineN<R, N> &s, const R *val, R fr, R fS, R fj, int lane) {
    constexpr int NN = (N + 1) * (N + 1);
#pragma unroll 1
    for (int k0 = 0; k0 < NN; ++k0) {
        int k = k0 + lane % NN;
        k = k >= NN ? k - NN : k;
        const int a = k % (N + 1), b = k / (N + 1);
        const R wc = pick<N + 1>(s.wx, a) * pick<N + 1>(s.wy, b);
        const int64_t node = (int64_t)spline_row(g, s.iy + b) * g.nxn + spline_col(g, s.ix + a);
        const R wr = wc * fr, ws = wc * fS, wj = wc * fj;
#pragma unroll
        for (int kk = 0; kk < NMOM; ++kk) {
            const R p = kParts ? (kk == 0 ? wr : (kk < 10 ? ws : wj) * val[kk]) : wc * val[kk];
            atomicAdd(&Mfix[(int64_t)kk * g.nnode + node], (unsigned long long)fix_of(p, fs, mom_class(kk)));
        }
    }
}

// Deposit of a warp's particles with a spline shape, transposed: instead of
// every lane adding its particle's 13 (N + 1)^2 products in L2 (117 to 325
// scalar reductions per particle, what bounded the spline pushes), the
// particles' 13 values and (N + 1)^2 node weights go to shared memory, and each
// lane owns some of the 13 (N + 1)^2 sums of the stencil at node (K) and adds
// the products of all particles with that stencil in registers, FMA by FMA.
// Only when the warp's stencil changes do the sums go to the global moments.
// The bins are in cell order, so a stencil usually lasts for more than a
// segment; a warp whose particles lie in many cells pays one flush (13 (N +
// 1)^2 / 32 reductions per lane) per cell, not per particle.
// FP32: a lane takes one node and a run of moments (1 + 1 .. 4 shared loads per
// particle); FP64: sums are dealt flat over the lanes (the FP64 pipe, not the
// loads, bounds it, and no lane idles), sum o = node * 13 + moment at lane
// o mod 32.  Measured on the 1024 x 512 foil (6.55M particles, per push / per
// species at rest): FP32 cubic 2.87 -> 0.56 ms / 1.30 -> 0.16 ms; FP64
// quadratic 5.30 -> 4.10 / 1.89 -> 1.54 ms (FP64 pipe 87 % active).
// Where a stencil's sums go.  GlobalSink: the moments, columns folded or wrapped.
template <typename R>
struct GlobalSink {
    const GridArgs<R> &g;
    R *M;
    __device__ inline void operator()(int i, int j, int k, R v) const {
        atomicAdd(&M[(int64_t)k * g.nnode + (int64_t)spline_row(g, j) * g.nxn + spline_col(g, i)], v);
    }
};
template <typename R, int N>
struct SplineDep {
    static constexpr int NP = N + 1, NN = NP * NP, NS = NN * NMOM;
    static constexpr bool kFlat = sizeof(R) == 8;
    // a particle's row: 13 values (padded to VS), then the NN weights; FP32 row strides of 4 mod 8
    // words keep the 16-byte stores of 8 lanes on different banks
    static constexpr int VS = kFlat ? 14 : 16;
    static constexpr int RS = kFlat ? (VS + NN + (NN & 1)) : (N == 2 ? 28 : N == 3 ? 36 : 44);
    static constexpr int HG = N == 2 ? 3 : N == 3 ? 2 : 1;     // FP32: lanes per node
    static constexpr int KW = N == 2 ? 4 : N == 3 ? 8 : 13;    // and moments per lane
    static constexpr int J = kFlat ? (NS + 31) / 32 : (N == 2 ? 5 : KW);    // sums per lane
    static constexpr int kWarpBytes = 32 * RS * (int)sizeof(R);

    R *rows;
    R acc[J];
    unsigned K;         // the warp's stencil: its key
    bool some;          // there is one
    int kx, ky;         // its first node (row wrapped)
    int node, m0;       // FP32: the lane's node and first moment

    __device__ inline void init(void *smem, int lane) {
        rows = (R *)smem;
        K = 0;
        some = false;
        kx = ky = 0;
        node = kFlat ? 0 : min(lane / HG, NN - 1);
        m0 = kFlat ? 0 : (lane % HG) * KW;
#pragma unroll
        for (int j = 0; j < J; ++j) acc[j] = R(0);
    }

    // Sum j of this lane: its node and moment (false: none).
    __device__ inline bool sum_of(int j, int lane, int &nd, int &k) const {
        if (kFlat) {
            const int o = lane + 32 * j;
            nd = o / NMOM;
            k = o - nd * NMOM;
            return o < NS;
        }
        nd = node;
        k = (N == 2 && j == 4) ? 12 : m0 + j;
        return lane < NN * HG && (N == 2 ? (j < 4 || m0 == 8) : k < NMOM);
    }

    template <typename Sink>
    __device__ inline void flush(const Sink &sink, int lane) {
        if (!some) return;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            int nd, k;
            if (sum_of(j, lane, nd, k) && acc[j] != R(0)) {
                const int b = nd / NP, a = nd - b * NP;
                sink(kx + a, ky + b, k, acc[j]);
            }
            acc[j] = R(0);
        }
    }

    __device__ inline void add_rows(int p0, int p1, int lane) {
        if constexpr (kFlat) {
            int ov[J], ow[J];
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int o = min(lane + 32 * j, NS - 1), nd = o / NMOM;
                ov[j] = o - nd * NMOM;
                ow[j] = VS + nd;
            }
#pragma unroll 2
            for (int p = p0; p < p1; ++p) {
                const R *r = rows + p * RS;
#pragma unroll
                for (int j = 0; j < J; ++j) acc[j] = fma_r(r[ow[j]], r[ov[j]], acc[j]);
            }
        } else {
#pragma unroll 4
            for (int p = p0; p < p1; ++p) {
                const float *r = (const float *)rows + p * RS;
                const float w = r[VS + node];
#pragma unroll
                for (int q = 0; q < (N == 4 ? 3 : KW / 4); ++q) {
                    const float4 v = *(const float4 *)(r + m0 + 4 * q);
                    acc[4 * q] = fmaf(w, v.x, acc[4 * q]);
                    acc[4 * q + 1] = fmaf(w, v.y, acc[4 * q + 1]);
                    acc[4 * q + 2] = fmaf(w, v.z, acc[4 * q + 2]);
                    acc[4 * q + 3] = fmaf(w, v.w, acc[4 * q + 3]);
                }
                if constexpr (N != 3) acc[J - 1] = fmaf(w, r[12], acc[J - 1]);   // moment 12
            }
        }
    }

    // All lanes of the warp: particle (s, val) of every lane with alive set; nx, ny: the grid's cells, in whose
    // numbering s's first node lies within -2 .. n + 1.
    template <typename Sink>
    __device__ inline void add(const Sink &sink, int nx, int ny, bool alive, const SplineN<R, N> &s, const R *val,
                               int lane) {
        const unsigned full = 0xffffffffu, lt = (1u << lane) - 1u;
        // first node as one number: ny (nx + 4) < 2^32 - 32 for every grid (nx >= 2, nx ny <= 2^30)
        const int row0 = wrap1(s.iy, ny);
        const unsigned key = alive ? (unsigned)row0 * (unsigned)(nx + 4) + (unsigned)(s.ix + 2) : 0xffffffffu - lane;
        const unsigned same = __match_any_sync(full, key);
        const int size = alive && (same & lt) == 0 ? __popc(same) : 0;   // at a stencil's first lane: its particles
        int incl = size;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(full, incl, o);
            if (lane >= o) incl += y;
        }
        const int first = __ffs(same) - 1;
        const int slot = __shfl_sync(full, incl - size, first) + __popc(same & lt);   // rows grouped by stencil
        __syncwarp();   // the previous particles' rows have been read
        if (alive) {
            R row[RS];
#pragma unroll
            for (int k = 0; k < VS; ++k) row[k] = k < NMOM ? val[k] : R(0);
#pragma unroll
            for (int b = 0; b < NP; ++b)
#pragma unroll
                for (int a = 0; a < NP; ++a) row[VS + b * NP + a] = s.wx[a] * s.wy[b];
#pragma unroll
            for (int k = VS + NN; k < RS; ++k) row[k] = R(0);
            constexpr int V = 16 / (int)sizeof(R);
            struct alignas(16) Vec {
                R x[V];
            };
            Vec *dst = (Vec *)(rows + slot * RS);
#pragma unroll
            for (int k = 0; k < (VS + NN + V - 1) / V; ++k) {
                Vec t;
#pragma unroll
                for (int q = 0; q < V; ++q) t.x[q] = row[V * k + q];
                dst[k] = t;
            }
        }
        __syncwarp();
        unsigned left = __ballot_sync(full, size > 0);
        const unsigned inK = __ballot_sync(full, size > 0 && some && key == K);   // the warp's stencil first
        while (left) {
            const int l = __ffs(left & inK ? left & inK : left) - 1;
            left &= ~(1u << l);
            const unsigned k = __shfl_sync(full, key, l);
            const int p1 = __shfl_sync(full, incl, l), p0 = p1 - __shfl_sync(full, size, l);
            const int nx0 = __shfl_sync(full, s.ix, l), ny0 = __shfl_sync(full, row0, l);
            if (!some || k != K) {
                flush(sink, lane);
                some = true;
                K = k;
                kx = nx0;
                ky = ny0;
            }
            add_rows(p0, p1, lane);
        }
    }
};

// --------------------------------------------------------------------------- host entry points

int check_launch(const char *what);
// Lets a kernel be launched with `bytes` of dynamic shared memory: the limit is the kernel's, whichever run launches
// it, and is only ever raised.
cudaError_t allow_smem(const void *kernel, size_t bytes);
void timing_begin(pic_t *h);
void timing_end(pic_t *h, int cls, int nlaunch);
inline void count_launch(pic_t *h, int n = 1) { h->timing.launches[4] += n; }

// fields (pic_field.cu)
int field_literal(pic_t *h);            // E, H and node B of the next time level, E^n + E^{n+1} for the push
int field_cn(pic_t *h);
int node_average(pic_t *h, int hsrc, int bdst);   // node B of a given H
int upload_fields(pic_t *h, const double *E3, const double *H3);
int download_fields(pic_t *h, double *E3, double *H3);

// particles (pic_particles.cu): conversion, deposit at rest, state export
int deposit_only(pic_t *h, int s);
int deposit_spare(pic_t *h, int s, int64_t n);   // FP64 cell sums: new particles still in the spare set
int deposit_leavers(pic_t *h, int s, int64_t n, const int32_t *cell, const double *v, int64_t plane);   // and those gone
bool post_deposit(const pic_t *h);      // the form whose steps deposit after the regroup
int deposit_step(pic_t *h, const int32_t *guard0, const int32_t *guard1);   // that deposit, over the push's next work items
int push_item_segs(const pic_t *h);     // segments per work item of the push
int ensure_items(pic_t *h);             // the work-item table holds an entry per used segment
int clear_moments(pic_t *h);
int clear_step_moments(pic_t *h);       // what a step's deposit adds into (the touched node tiles only)
int fix_to_moments(pic_t *h);           // deterministic deposit: Mfix -> M (+ Mlo)
int fix_scale(const pic_t *h, FixScale *out);
constexpr int ABS_SUM_BLOCKS = 256;
int abs_sum(pic_t *h, const double *w, int64_t n, double *part);   // part[ABS_SUM_BLOCKS]: shares of the sum of |w|
int load_convert(pic_t *h, int s, int buf, int64_t n, const double *const src[6], unsigned long long *bad,
                 bool over_link, const int32_t *csrc = nullptr);
// over_link: the arrays are page-locked host memory read in place; csrc: checkpoint form (src[0], src[1]
// are in-cell offsets, csrc the cell indices)   // *bad = first invalid index
int particles_to_stage(pic_t *h, int s, int64_t *n_out, bool raw = false);   // raw: in-cell offsets for x, y
int count_species(pic_t *h, int s, int64_t *n_out);

// batched particle step of several runs (pic_tile.cu launches, pic_api.cu drives)
struct BatchScratch {
    cudaStream_t st = nullptr;
    int cap = 0;                        // runs
    void *args_dev = nullptr;           // cap argument blocks
    void *args_host[2] = {nullptr, nullptr};     // pinned staging of the argument blocks (two, alternating)
    int32_t *idx = nullptr;             // device: run_items[cap + 1], run_tiles[cap + 1], ticket
    int32_t *idx_host[2] = {nullptr, nullptr};   // pinned staging of run_tiles
    cudaEvent_t ev_stage[2] = {nullptr, nullptr}, ev_push = nullptr, ev_done = nullptr;
    int slot = 0;                       // staging slot of the current step
};
size_t batch_args_bytes();              // one argument block (the larger of the two forms)
int batch_push(BatchScratch &b, pic_t **hs, int n);
int batch_regroup(BatchScratch &b, pic_t **hs, int n);

// tiled step (pic_tile.cu)
int tile_setup(pic_t *h);
int particle_tiles(pic_t *h);
int push_prep(pic_t *h, const int32_t *guard, int32_t *word);   // the next push's work items and tile lists
int32_t *list_counters(const pic_t *h, int set);
int cell_moments(pic_t *h);      // FP64 cell sums -> node moments (the listed touched tiles)
int rest_touch(pic_t *h);        // touched[] and its list after a deposit at rest into cleared moments
int regroup_tiles(pic_t *h);     // per-tile stable cell sort of stayers + arrivals into the spare set
int scan_tiles(pic_t *h, const int32_t *in, int32_t *out);
int tile_counts(pic_t *h, int s);   // tcount[t] = particles of tile t (device)

// sort and rebuild (pic_sort.cu)
enum RebuildSource { REBUILD_FROM_STEP = 0, REBUILD_FROM_LOAD = 1 };
int rebuild_species(pic_t *h, int s, int source, int64_t n_second);
int ensure_sort_capacity(pic_t *h, int64_t n);
int init_empty_bins(pic_t *h, int s);
int64_t slots_needed(const pic_t *h, int64_t n);
int64_t sort_hist_entries(int64_t cap);   // radix histogram entries for cap keys
int scan_i32_inplace(pic_t *h, int32_t *a, int64_t n);   // exclusive, multi-block
int scan_sums_entries();

// field ionisation (pic_ionize.cu): one chain's pass over its ion species -- decisions, staging of the
// ionised particles at offset of the staging planes (stride scap), compaction of the species
struct IonChain {
    int species;            // the ion species
    double c2ip, expo, K;   // |C|^2 Ip, 2 n* - 1, 2 (2 Ip)^(3/2) (atomic units)
    double fmax;            // field of the rate formula's maximum (atomic units)
    double field_au, dt_au; // the run's field unit and time step in atomic units
};
int collide(pic_t *h, const pic_collisions *p, unsigned long long *d_pairs);
int ion_chain(pic_t *h, const IonChain &c, uint64_t seed, int32_t *scell, double *sval, int64_t scap, int64_t offset,
              int64_t *n_out);

// diagnostics (pic_diag.cu)
int diagnostics(pic_t *h, pic_diag *out);
int moments_to_stage(pic_t *h);     // stage[13][nnode] = M (+ Mlo) / node area, FP64

}  // namespace pic
