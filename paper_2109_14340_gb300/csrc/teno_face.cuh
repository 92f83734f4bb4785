// Face fluxes: for every face i+1/2 of the face grids, Roe average ->
// eigenvectors -> characteristic projection of the 2H-cell stencil ->
// LLF/Rusanov split -> TENO-AA reconstruction of f+ and f- per field ->
// back-projection -> positivity limiter (arXiv 2109.14340, Sec. 3-5).
//
// An FP64 instruction holds its scheduler's FP64 unit for 64 cycles, with one
// lane active or 32 (2 lanes per SM and clock), so a face costs what the warps
// issue, idle lanes included, and the unit idles whenever all warps of a
// scheduler are busy with something else.  The work is therefore cut where
// lanes would diverge, over four kernels that pass values through memory
// (about 1 kB per face at most, of a bandwidth that FP64 work leaves idle):
//
//   sweep   a warp per tile of 32 faces, a lane per face: staging, Roe state,
//           projection, split fluxes.  Reconstructions that quick_large accepts
//           for the largest stencil get their value; the others go to the
//           tile's queue.
//   decide  the queues of several tiles by a warp: the whole filter for each
//           entry, then the values, the large stencils' and the fallback's each
//           on compact lanes.  What the filter leaves open goes to one list.
//   exact   that list through the exact path, a lane or a warp per entry.
//   finish  a lane per face: back-projection, limiter, the flux.
//
// 2 M faces of 128^3 TENO10 (smooth flow): sweep 2.61 ms, its FP64 unit 90 %
// busy with 701 instructions per 32 faces; decide 0.18 to 0.26 ms, bound by the
// instructions it issues (53 % of the slots; FP64 43 %); exact 0.02 to 0.04 ms;
// finish 0.12 ms, FP64 86 % busy: 3.0 ms.  One kernel with its queue in shared
// memory took 3.6 to 3.9 ms (FP64 80 to 84 % busy, 824 to 839 instructions).
//
// The buffers between them are sized for at most kChunkTiles tiles, so a larger
// evaluation goes through them in chunks.  U and F are staged halved (exact: a
// power of two), so that the projections give the halved characteristic
// variables and fluxes w/2, g/2 directly and the split fluxes (g +- alpha w)/2
// need no further scaling.
#pragma once

#include "teno_dev.cuh"
#include "teno_fast.cuh"

namespace teno {

constexpr int kTileFaces = 32;
// Tiles a chunk holds at most: 2 M faces.  Each chunk ends with partly filled
// waves of its four kernels, about 40 us; 65536 tiles of 3D ten-point faces
// take some 2.6 ms and 2 GB.
constexpr int64_t kChunkTiles = 65536;

// One direction's faces.
struct DirArgs {
    double *F;             // face fluxes, [nc][nfaces]
    uint8_t *flags;        // decision record or nullptr
    const uint8_t *frozen; // recorded decisions to apply instead of deciding, or nullptr
    uint16_t *argmax;      // per face: the maximising stencil cells of the splitting
                           // speeds (4 bits each: u-c, u, u+c, |u|+c), or nullptr
    const uint16_t *frozen_argmax;   // recorded maximising cells to apply, or nullptr
    uint8_t *limrec;       // per face: 1 where the positivity limiter bound, or nullptr
    const double *bcs_lo, *bcs_hi;   // Dirichlet boundary-face states or halo arrays, or nullptr
    const double *lam;     // limiter's effective dt/dx for this direction (device)
    int64_t nfaces;
    int bc_lo, bc_hi;      // boundary rules at the two ends of the axis
    int skip_last;         // 1: face n of each line is not computed (periodic axis, no
                           // decision record: its flux is face 0's, bitwise); the fused 1D
                           // stage computes it, but counts nothing there
    // A tile is 2^tps pencils (side by side in x, in y for the x sweep) by 32 >> tps
    // faces; tiles per line of faces, and groups of 2^tps pencils along that axis.
    int tps;
    int own;               // faces a tile owns along the line: all, or one fewer where tiles
                           // overlap by a face (the fused 1D stage)
    int64_t line_tiles, groups;
};

// The evaluation's input.
struct GridArgs {
    const double *U;       // state, [nc][ncell]
    const double *P;       // primitives of U ([PrimRows::NP][ncell], store_prims) or
                           // nullptr: computed while staging
    Status *st;
    int64_t n[3];
    int64_t ncell;
    int fast;              // 1: certified FP32 decision filter first
    int need_ct;           // 1: recorded decision bytes carry their C_T exponent; 0: only
                           // where it decided (the selection bits are exact either way)
    int count_cells;       // 1: count the non-physical cells the x sweep owns (each cell once)
    int limiter;           // 1: positivity limiter
    uint32_t tag;          // top bit of the queue lengths (a batch's scheme)
};

// The buffers between the four kernels; nt: tiles they hold.  Queue entries of
// tile t are q = t per_tile .. + count[t], per_tile = 64 nc.
struct SweepBuf {
    double *qv;            // [2H][nt per_tile] values of the queued reconstructions
    uint16_t *qslot;       // [nt per_tile] (2k+s) 32 + lane
    uint32_t *xlist;       // [nt per_tile] entries left to the exact path
    uint32_t *count;       // [nt] queue lengths
    double *R;             // [2 nc][nt 32] reconstructed values
    double *RO;            // [nd + 4][nt 32] Roe velocity, enthalpy, sound speed, |u|^2, u_d c
    double *RL;            // [4 nc + 1][nt 32] limiter: halved U, F of cells i, i+1, and the
                           // Lax-Friedrichs speed; nullptr without a limiter
    uint8_t *RD;           // [2 nc][nt 32] decision bytes; nullptr without a record
    int64_t nt;
};

inline size_t sweep_align(size_t x) { return (x + 255) & ~(size_t)255; }

// Lays the buffers for nt tiles out from p (null: only measures); W values per
// entry.  queue = false: only what a frozen replay passes on (R, RO, RL), for grids
// whose other evaluations take the single launch (2D 128^2 ten-point: 4 MB in place
// of 28).  Returns the bytes used.
inline size_t sweep_buf_layout(SweepBuf &b, char *p, int64_t nt, int nd, int W, bool limiter,
                               bool queue)
{
    const int nc = nd + 2;
    const size_t q = queue ? (size_t)nt * 64 * nc : 0, f = (size_t)nt * kTileFaces;
    size_t off = 0;
    auto take = [&](size_t bytes) { char *r = p + off; off += sweep_align(bytes); return r; };
    b.nt = nt;
    b.qv = (double *)take(sizeof(double) * W * q);
    b.xlist = (uint32_t *)take(sizeof(uint32_t) * q);
    b.qslot = (uint16_t *)take(sizeof(uint16_t) * q);
    b.count = (uint32_t *)take(queue ? sizeof(uint32_t) * nt : 0);
    b.R = (double *)take(sizeof(double) * 2 * nc * f);
    b.RO = (double *)take(sizeof(double) * (nd + 4) * f);
    b.RD = (uint8_t *)take(queue ? 2 * nc * f : 0);
    b.RL = limiter ? (double *)take(sizeof(double) * (4 * nc + 1) * f) : nullptr;
    return off;
}

// A run of tiles of one direction inside a chunk: tiles first .. first+count-1
// of the chunk are tiles t0 .. of direction d (tile_face_at's order).
struct SweepPart {
    int64_t t0;
    int32_t first, count, d;
};

// The fused 1D stage: a tile's faces also give its cells their update, which the
// tile writes in place of its fluxes (tiles overlap by a face; the input and the
// output are different arrays).
struct FuseArgs {
    const double *Un;      // state at t^n (RK modes), [3][n]
    double *out;           // rhs (mode 0) or next stage state, [3][n]
    const double *dt_dev;  // time step, or nullptr for dt
    double dt, inv_dx;
    int mode;              // -1: not fused; 0: rhs; 1..3: RK stage 0..2
};

struct SweepArgs {
    GridArgs g;
    DirArgs dir[3];
    SweepPart part[3];
    int32_t nparts, tiles;
    int small;                         // 1: the single launch for few tiles
    unsigned *nexact;                  // length of the exact path's list (zeroed beforehand)
    unsigned long long *exact_count;   // adds the exact-path reconstructions, or nullptr
    FuseArgs fuse;
    SweepBuf buf;
    FastK FK;
    Consts K;
};

// Shape of direction D's tiles: the 2^tps pencils (at most 4) that leave the
// fewest lanes without a face, weighed with the cells a tile stages (12 FP64
// instructions per 32 of them beside some 690 for the faces).  Lines of 65
// faces: 3 tiles a line of 1 x 32, 2.25 of 4 x 8.
inline void tile_shape(DirArgs &d, int64_t faces, int64_t pencils, int H)
{
    double best = 0.0;
    for (int tps = 0; tps <= 2; tps++) {
        const int64_t tp = 1 << tps, tf = kTileFaces >> tps;
        const int64_t lt = (faces + tf - 1) / tf, gr = (pencils + tp - 1) / tp;
        const int64_t rounds = (tp * (tf + 2 * H - 1) + 31) / 32;
        const double cost = (double)lt * (double)gr * (690.0 + 12.0 * (double)rounds);
        if (tps == 0 || cost < best) {
            best = cost;
            d.tps = tps;
            d.own = (int)tf;
            d.line_tiles = lt;
            d.groups = gr;
        }
        if (pencils == 1) break;
    }
}

// Whether an evaluation of so many tiles takes the single launch (small_kernel)
// rather than the four kernels.  Measured per right-hand side, four kernels
// against one: 1D 400 cells 58 against 34 us, 100 000 cells (3126 tiles) 163
// against 154; 2D ten-point 128^2 (1088 tiles) 123 against 110, 256^2 (4200) 314
// against 316; 2D twelve-point 96^2 (620) 124 against 107, 160^2 (1640) 151
// against 183; 3D 20^3 (900) 131 against 138, 28^3 216 against 289.  Above the
// line in 1D, three ten-point steps of a tube whose plateaus carry rounding
// noise: 140 000 cells (4376 tiles) 2.13 against 2.15 ms, 200 000 2.75 against
// 3.02, 300 000 3.74 against 4.45, 500 000 5.72 against 7.32.
inline bool small_evaluation(int64_t tiles, int nd, int H)
{
    return tiles <= (nd == 1 ? 4096 : (nd == 2 ? (H == 6 ? 1024 : 3072) : 512));
}

// Tile t of direction D: first face f0 and the position of its first pencil.  x
// runs fastest in the y and z sweeps: neighbouring pencils share the sectors of
// their strided loads.
template <int ND, int D>
__device__ __forceinline__ void tile_at(const int64_t (&n)[3], const DirArgs &da, int64_t t,
                                        int64_t &f0, int64_t &x, int64_t &y, int64_t &z)
{
    x = y = z = 0;
    int64_t ft = t;
    if (ND > 1) {
        const int64_t fast = D == 0 ? da.line_tiles : da.groups;
        const int64_t r = t / fast, i = t - r * fast;
        if (D == 0) {
            ft = i;
            z = ND == 2 ? 0 : r / da.groups;
            y = (r - z * da.groups) << da.tps;
        } else {
            x = i << da.tps;
            const int64_t o = ND == 2 ? 0 : r / da.line_tiles;
            ft = r - o * da.line_tiles;
            if (D == 1) z = o;
            else y = o;
        }
    }
    f0 = ft * da.own;
}

// The lane's face within its tile: pencil p and offset fo along D.
template <int D>
__device__ __forceinline__ void tile_lane(int tps, int lane, int &p, int &fo)
{
    if (D == 0) {
        fo = lane & ((kTileFaces >> tps) - 1);
        p = lane >> (5 - tps);
    } else {
        p = lane & ((1 << tps) - 1);
        fo = lane >> tps;
    }
}

// A record's 16-bit words: a step's records lie back to back, and an odd number
// of bytes each puts the second's words at odd addresses.
__device__ __forceinline__ void put_word(uint16_t *p, unsigned v)
{
    if ((uintptr_t)p & 1) {
        ((uint8_t *)p)[0] = (uint8_t)v;
        ((uint8_t *)p)[1] = (uint8_t)(v >> 8);
    } else {
        *p = (uint16_t)v;
    }
}

__device__ __forceinline__ unsigned get_word(const uint16_t *p)
{
    const uint8_t *b = (const uint8_t *)p;
    return (uintptr_t)p & 1 ? b[0] | (unsigned)b[1] << 8 : *p;
}

// Index of face f of the pencil at (x, y, z) in direction D's face grid.
template <int D>
__device__ __forceinline__ int64_t face_index(const int64_t (&n)[3], int64_t f, int64_t x, int64_t y,
                                              int64_t z)
{
    if (D == 0) return f + (n[0] + 1) * (y + n[1] * z);
    if (D == 1) return x + n[0] * (f + (n[1] + 1) * z);
    return x + n[0] * (y + n[1] * f);
}

// App. A ghost-cell rules along one axis.  Returns the interior cell whose
// state defines the (possibly ghost) cell j, and the rule to apply to it:
// 0 copy, 1 slip-wall mirror (wall-normal momentum negated), 2 no-slip
// mirror (all momentum negated), 3 / 4 Dirichlet reflection about the low /
// high boundary-face state; or, for a side whose ghost cells are a
// neighbouring sub-domain's cells (TENO_BC_HALO), rule 5 / 6 and the plane of
// the side's halo array (0 .. H-1 in ascending position: cell -H + q below,
// n + q above).  The final clamps only matter for padding cells beyond the
// last face of a tile.
__device__ __forceinline__ int64_t map_index(int64_t j, int64_t n, int H, int lo, int hi, int &rule)
{
    rule = 0;
    int64_t r = j;
    if (j < 0) {
        if (lo == 0) r = ((j % n) + n) % n;
        else if (lo == 1) r = 0;
        else if (lo == 5) { rule = 5; r = j + H; return r < 0 ? 0 : r; }
        else { rule = lo == 2 ? 1 : (lo == 3 ? 2 : 3); r = -j - 1; }
    } else if (j >= n) {
        if (hi == 0) r = j % n;
        else if (hi == 1) r = n - 1;
        else if (hi == 5) { rule = 6; r = j - n; return r >= H ? H - 1 : r; }
        else { rule = hi == 2 ? 1 : (hi == 3 ? 2 : 4); r = 2 * n - 1 - j; }
    }
    return r < 0 ? 0 : (r >= n ? n - 1 : r);
}

// Ghost state of a Dirichlet side (App. A.3): the mirror cell's primitives
// phi (with the exact path's arithmetic for p) reflected about the boundary
// face's primitives phi' as 2 phi' - phi, then back to conserved variables.
// st: the side's state array, m faces per primitive, s this face.
template <int ND>
__device__ __forceinline__ void dirichlet_ghost(double (&Uc)[ND + 2], const double *st, int64_t m,
                                                int64_t s, double gm1)
{
    constexpr int nc = ND + 2;
    const double rho = Uc[0], E = Uc[nc - 1];
    const double rinv = 1.0 / rho;
    double u[ND];
#pragma unroll
    for (int a = 0; a < ND; a++) u[a] = Uc[1 + a] * rinv;
    double t = Uc[1] * u[0];
#pragma unroll
    for (int a = 1; a < ND; a++) t = fma(Uc[1 + a], u[a], t);
    const double p = gm1 * (E - 0.5 * t);
    const double rg = 2.0 * st[s] - rho;
    double ug[ND];
#pragma unroll
    for (int a = 0; a < ND; a++) ug[a] = 2.0 * st[(1 + a) * m + s] - u[a];
    const double pg = 2.0 * st[(nc - 1) * m + s] - p;
    Uc[0] = rg;
#pragma unroll
    for (int a = 0; a < ND; a++) Uc[1 + a] = rg * ug[a];
    double k2 = Uc[1] * ug[0];
#pragma unroll
    for (int a = 1; a < ND; a++) k2 = fma(Uc[1 + a], ug[a], k2);
    Uc[nc - 1] = pg / gm1 + 0.5 * k2;
}

// Applies a ghost rule of map_index to the loaded state of the mirror cell.
template <int ND, int D>
__device__ __forceinline__ void apply_ghost_rule(double (&Uc)[ND + 2], int rule, const double *st_lo,
                                                 const double *st_hi, int64_t m, int64_t s,
                                                 double gm1)
{
    if (rule == 1) {
        Uc[1 + D] = -Uc[1 + D];
    } else if (rule == 2) {
#pragma unroll
        for (int a = 0; a < ND; a++) Uc[1 + a] = -Uc[1 + a];
    } else if (rule >= 3) {
        dirichlet_ghost<ND>(Uc, rule == 3 ? st_lo : st_hi, m, s, gm1);
    }
}

// A sweeping warp's slice of shared memory, in doubles: the halved (U_c, F_c)
// pairs of the staged cells, [c][cell], then the quantities that the Roe
// average and the splitting speeds need, [row][cell].
template <int ND, int H>
struct FaceSmem {
    static constexpr int nc = ND + 2;
    static constexpr int NS = 4 * (kTileFaces / 4 + 2 * H - 1);    // cells of the widest shape
    static constexpr int QV = 0, QH = ND, QSR = ND + 1;           // rows of the second part
    static constexpr int QLM = ND + 2, QL0 = ND + 3, QLP = ND + 4, QLR = ND + 5, NT = ND + 6;
    static constexpr int TMP = 2 * nc * NS;
    static constexpr int TOTAL = (TMP + NT * NS + 1) & ~1;         // 16-byte slices
};

// Sweep modes, a compile-time choice so that each kernel holds only its own
// code: a plain sweep, one that writes the decision record (flags, argmax,
// limrec), and one that applies recorded decisions (frozen, frozen_argmax).
enum { kSweepPlain = 0, kSweepRecord = 1, kSweepFrozen = 2 };

// Stages the cells of a tile from f0-H along D, pencil by pencil in the x sweep,
// pencils side by side in the others: cells first, first + step, ...
template <int ND, int H, int D>
__device__ __forceinline__ void stage_cells(const GridArgs &a, const DirArgs &da, const Consts &K,
                                            int64_t f0, int64_t x, int64_t y, int64_t z, double *sm,
                                            int first, int step)
{
    using SL = FaceSmem<ND, H>;
    constexpr int nc = ND + 2, last = nc - 1, NS = SL::NS;
    double2 *UF = (double2 *)sm;
#define TMP(q, j) sm[SL::TMP + (q) * NS + (j)]
    const int64_t n0 = a.n[0], n1 = a.n[1], nD = a.n[D];
    const int tps = ND == 1 ? 0 : da.tps, tp = 1 << tps;
    const int nsf = (kTileFaces >> tps) + 2 * H - 1;   // cells of one pencil
    const int64_t npen = D == 0 ? n1 - y : n0 - x;     // pencils from the first one on
    const int64_t cstride = D == 0 ? 1 : (D == 1 ? n0 : n0 * n1);
    for (int idx = first; idx < tp * nsf; idx += step) {
        int j, pp;
        if (D == 0) {
            pp = (idx >= nsf) + (idx >= 2 * nsf) + (idx >= 3 * nsf);
            j = idx - pp * nsf;
        } else {
            pp = idx & (tp - 1);
            j = idx >> tps;
        }
        if (pp >= npen) continue;
        const int64_t px = D == 0 ? 0 : x + pp, py = D == 0 ? y + pp : y;
        const int64_t cbase = px + n0 * ((D == 1 ? 0 : py) + n1 * (D == 2 ? 0 : z));
        int rule;
        const int64_t gi = map_index(f0 - H + j, nD, H, da.bc_lo, da.bc_hi, rule);
        double Uc[nc];
        CellQ<ND> q;
        if (rule >= 5) {
            // a neighbouring sub-domain's cell from the side's halo array,
            // [nc][H planes][cells of a plane, the other axes x fastest]
            const int64_t m = a.ncell / nD;
            const int64_t sf = (D == 0) ? py + n1 * z : (D == 1 ? px + n0 * z : px + n0 * y);
            const double *hb = rule == 5 ? da.bcs_lo : da.bcs_hi;
            const int64_t ih = gi * m + sf;
            const bool ok = TENO_IN(a.st, ih, H * m);
#pragma unroll
            for (int c = 0; c < nc; c++) Uc[c] = ok ? hb[(int64_t)c * H * m + ih] : 0.0;
            cell_quantities<ND, D>(Uc, K, q);
        } else {
            const int64_t id = cbase + gi * cstride;
            const bool ok = TENO_IN(a.st, id, a.ncell);
#pragma unroll
            for (int c = 0; c < nc; c++) Uc[c] = ok ? a.U[c * a.ncell + id] : 0.0;
            if (rule < 3 && a.P && ok) {
                // stored for this input; a mirror image has its cell's, velocities
                // (all or the wall-normal one) with the other sign, bit for bit
                load_prims<ND>(a.P, a.ncell, id, q);
                apply_ghost_rule<ND, D>(Uc, rule, nullptr, nullptr, 0, 0, K.gm1);
#pragma unroll
                for (int k = 0; k < ND; k++)
                    if (rule == 2 || (rule == 1 && k == D)) q.u[k] = -q.u[k];
            } else {
                if (rule) {
                    // boundary-face index among the faces of this side (other axes, x fastest)
                    const int64_t m = a.ncell / nD;
                    const int64_t sf = (D == 0) ? py + n1 * z : (D == 1 ? px + n0 * z : px + n0 * y);
                    if (rule < 3 || TENO_IN(a.st, sf, m))
                        apply_ghost_rule<ND, D>(Uc, rule, da.bcs_lo, da.bcs_hi, m, sf, K.gm1);
                }
                cell_quantities<ND, D>(Uc, K, q);
            }
        }
        if (D == 0 && a.count_cells) {
            // interior cells of this tile's own face range: each cell once
            const int64_t ci = f0 - H + j;
            if (ci >= f0 && ci < f0 + da.own && ci < nD && nonphysical_cell<ND>(Uc[0], q))
                atomicAdd(&a.st->nonphys, 1ull);
        }
        // halves of U and of the flux along D: each product and sum of
        // cell_quantities' flux with one factor or both terms halved
        double hU[nc], hF[nc];
#pragma unroll
        for (int c = 0; c < nc; c++) hU[c] = half_of(Uc[c]);
        const double hp = half_of(q.p), hm = hU[1 + D];
        hF[0] = hm;
#pragma unroll
        for (int k = 0; k < ND; k++) hF[1 + k] = k == D ? hm * q.u[k] + hp : hm * q.u[k];
        hF[last] = q.u[D] * (hU[last] + hp);
#pragma unroll
        for (int c = 0; c < nc; c++) UF[c * NS + idx] = make_double2(hU[c], hF[c]);
#pragma unroll
        for (int k = 0; k < ND; k++) TMP(SL::QV + k, idx) = q.u[k];
        TMP(SL::QH, idx) = q.H;
        TMP(SL::QSR, idx) = q.sr;
        const double vd = q.u[D], cj = q.c;
        TMP(SL::QLM, idx) = fabs(vd - cj);
        TMP(SL::QL0, idx) = fabs(vd);
        TMP(SL::QLP, idx) = fabs(vd + cj);
        TMP(SL::QLR, idx) = fabs(vd) + cj;
    }
#undef TMP
}

// One tile by one warp: the faces from f0 along D of the pencils from (x, y, z);
// tile: its index in the chunk's buffers; sm: the warp's slice.  Every lane of
// the warp calls it; it returns with the warp in step, its values, queue and
// Roe states in the buffers.
template <int ND, int H, int D, int MODE>
__device__ __forceinline__ void sweep_tile(const GridArgs &a, const DirArgs &da, const FastK &FK,
                                           const Consts &K, const SweepBuf &B, int64_t f0, int64_t x,
                                           int64_t y, int64_t z, int64_t tile, double *sm)
{
    using SL = FaceSmem<ND, H>;
    constexpr int nc = ND + 2, last = nc - 1, W = 2 * H, NS = SL::NS;
    const int lane = threadIdx.x & 31;
    double2 *UF = (double2 *)sm;
#define TMP(q, j) sm[SL::TMP + (q) * NS + (j)]

    const int64_t nD = a.n[D];
    const int tps = ND == 1 ? 0 : da.tps, tp = 1 << tps;
    const int nsf = (kTileFaces >> tps) + 2 * H - 1;   // cells of one pencil
    const int64_t npen = D == 0 ? a.n[1] - y : a.n[0] - x;     // pencils from the first one on

    stage_cells<ND, H, D>(a, da, K, f0, x, y, z, sm, lane, 32);
    __syncwarp();

    int p, fo;
    tile_lane<D>(tps, lane, p, fo);
    const int64_t f = f0 + fo;
    const int64_t nf = B.nt * kTileFaces, cf = tile * kTileFaces + lane;   // in the buffers
    const bool active = f <= nD - da.skip_last && p < npen && TENO_IN(a.st, cf, nf);
    // the lane's first cell, the step to the next, and cells i and i+1
    const int b0 = D == 0 ? p * nsf + fo : lane, bs = D == 0 ? 1 : tp;
    const int bl = b0 + (H - 1) * bs, br = bl + bs;

    RoeScalars<ND> rs;                 // eigenvector rows / columns are built from these
    double am = 0.0, a0 = 0.0, ap = 0.0, ar = 0.0;
    int64_t flin = 0;
    if (active) {
        // Roe average and eigenvectors (Sec. 5).
        double ul[ND], ur[ND];
#pragma unroll
        for (int k = 0; k < ND; k++) { ul[k] = TMP(SL::QV + k, bl); ur[k] = TMP(SL::QV + k, br); }
        const double c2 = roe_state<ND, D>(ul, TMP(SL::QH, bl), TMP(SL::QSR, bl), ur,
                                           TMP(SL::QH, br), TMP(SL::QSR, br), K.gm1, rs);
        if (!(c2 > 0.0)) atomicAdd(&a.st->nonphys, 1ull);
        flin = face_index<D>(a.n, f, D == 0 ? x : x + p, D == 0 ? y + p : y, z);
        if (!TENO_IN(a.st, flin, da.nfaces)) flin = 0;        // debug build: counted, redirected
        // what the finish kernel needs
#pragma unroll
        for (int k = 0; k < ND; k++) B.RO[k * nf + cf] = rs.ut[k];
        B.RO[ND * nf + cf] = rs.Ht;
        B.RO[(ND + 1) * nf + cf] = rs.ct;
        B.RO[(ND + 2) * nf + cf] = rs.q2;
        B.RO[(ND + 3) * nf + cf] = rs.unct;
        if (a.limiter) {
#pragma unroll
            for (int c = 0; c < nc; c++) {
                const double2 cl = UF[c * NS + bl], cr = UF[c * NS + br];
                B.RL[(4 * c) * nf + cf] = cl.x;
                B.RL[(4 * c + 1) * nf + cf] = cl.y;
                B.RL[(4 * c + 2) * nf + cf] = cr.x;
                B.RL[(4 * c + 3) * nf + cf] = cr.y;
            }
            const double al = TMP(SL::QLR, bl), arr = TMP(SL::QLR, br);
            B.RL[4 * nc * nf + cf] = arr > al ? arr : al;
        }
        // Splitting speeds over the stencil (first maximum), or at recorded cells.
        if constexpr (MODE == kSweepFrozen) {
            unsigned w = get_word(da.frozen_argmax + flin);
            if (!TENO_IN(a.st, (int)(w & 15), W) || !TENO_IN(a.st, (int)((w >> 4) & 15), W) ||
                !TENO_IN(a.st, (int)((w >> 8) & 15), W) || !TENO_IN(a.st, (int)(w >> 12), W))
                w = 0;
            am = TMP(SL::QLM, b0 + (int)(w & 15) * bs);
            a0 = TMP(SL::QL0, b0 + (int)((w >> 4) & 15) * bs);
            ap = TMP(SL::QLP, b0 + (int)((w >> 8) & 15) * bs);
            ar = TMP(SL::QLR, b0 + (int)((w >> 12) & 15) * bs);
        } else {
            int jm = 0, j0 = 0, jp = 0, jr_ = 0;
#pragma unroll
            for (int j = 0; j < W; j++) {
                const double em = TMP(SL::QLM, b0 + j * bs), e0 = TMP(SL::QL0, b0 + j * bs);
                const double ep = TMP(SL::QLP, b0 + j * bs), er = TMP(SL::QLR, b0 + j * bs);
                if (j == 0 || speed_gt(em, am)) { am = em; jm = j; }
                if (j == 0 || speed_gt(e0, a0)) { a0 = e0; j0 = j; }
                if (j == 0 || speed_gt(ep, ap)) { ap = ep; jp = j; }
                if (j == 0 || speed_gt(er, ar)) { ar = er; jr_ = j; }
            }
            if constexpr (MODE == kSweepRecord)
                put_word(da.argmax + flin, jm | (j0 << 4) | (jp << 8) | (jr_ << 12));
        }
        if (K.split) am = a0 = ap = ar;               // Rusanov: one speed for every field
    }
    // Split-flux reconstructions of every field and sign.
    const int64_t nq = B.nt * (64 * nc), q0 = tile * (64 * nc);
    int cnt = 0;                                      // queue length (warp-uniform)
#pragma unroll 1
    for (int k = 0; k < nc; k++) {
        double v[W], vm[W];                       // v+ and v-, in stencil order
        if (active) {
            const bool shear = (k >= 2 && k < last);
            const int tax = shear ? shear_axis<ND, D>(k) : 0;
            double lrow[nc];
            l_row<ND, D>(rs, k, lrow);
            const double alpha = k == 0 ? am : (k == last ? ap : a0);
            // hw = w/2 = l.(U/2), hg = g/2 = l.(F/2) from the halved staged values:
            // every product and sum is the unhalved one scaled by 1/2, exactly.
            // f+ on offsets m -> cell i+m; f- mirrored: offset m -> cell i+1-m;
            // v = (g +- alpha w)/2 = fma(+-alpha, w/2, g/2), rounded once.
#pragma unroll
            for (int j = 0; j < W; j++) {
                double wv, gv;
                const double2 c0 = UF[b0 + j * bs];
                if (shear) {
                    const double2 ct = UF[(1 + tax) * NS + b0 + j * bs];
                    wv = ct.x + lrow[0] * c0.x;
                    gv = ct.y + lrow[0] * c0.y;
                } else {
                    wv = lrow[0] * c0.x;
                    gv = lrow[0] * c0.y;
#pragma unroll
                    for (int c = 1; c < nc; c++) {
                        const double2 cc = UF[c * NS + b0 + j * bs];
                        wv = fma(lrow[c], cc.x, wv);
                        gv = fma(lrow[c], cc.y, gv);
                    }
                }
                v[j] = fma(alpha, wv, gv);
                vm[W - 1 - j] = fma(-alpha, wv, gv);
            }
        }
#pragma unroll 1
        for (int s = 0; s < 2; s++) {
            const int slot = (2 * k + s) * kTileFaces + lane;
            bool open = false;
            if (active) {
                double *r = B.R + (2 * k + s) * nf + cf;
                if constexpr (MODE == kSweepFrozen) {
                    *r = frozen_recon<H>(v, da.frozen[(flin * nc + k) * 2 + s]);
                } else {
                    uint8_t fl;
                    open = !(a.fast && quick_large<H>(v, FK, MODE == kSweepRecord && a.need_ct, fl));
                    if (!open) {
                        *r = flux_large<H, H>(v);
                        if constexpr (MODE == kSweepRecord) B.RD[(2 * k + s) * nf + cf] = fl;
                    }
                }
            }
            if constexpr (MODE != kSweepFrozen) {
                const unsigned m = __ballot_sync(0xffffffffu, open);
                const int64_t q = q0 + cnt + __popc(m & ((1u << lane) - 1u));
                if (open && TENO_IN(a.st, q, nq)) {
#pragma unroll
                    for (int kk = 0; kk < W; kk++) B.qv[kk * nq + q] = v[kk];
                    B.qslot[q] = (uint16_t)slot;
                }
                cnt += __popc(m);
            }
#pragma unroll
            for (int kk = 0; kk < W; kk++) v[kk] = vm[kk];
        }
    }
    if (MODE != kSweepFrozen && lane == 0 && TENO_IN(a.st, tile, B.nt)) B.count[tile] = (uint32_t)cnt | a.tag;
    __syncwarp();
#undef TMP
}

// Back-projection of a face and the limiter: the flux Fo (and the limiter's byte
// of the record).  lam: the limiter's dt/dx.
template <int ND, int D, int MODE>
__device__ __forceinline__ void face_flux(const DirArgs &da, int limiter, double lam, const Consts &K,
                                          const SweepBuf &B, int64_t cf, int64_t flin,
                                          double (&Fo)[ND + 2])
{
    constexpr int nc = ND + 2, last = nc - 1;
    const int64_t nf = B.nt * kTileFaces;
    RoeScalars<ND> rs;                 // what r_entry reads
#pragma unroll
    for (int k = 0; k < ND; k++) rs.ut[k] = B.RO[k * nf + cf];
    rs.Ht = B.RO[ND * nf + cf];
    rs.ct = B.RO[(ND + 1) * nf + cf];
    rs.q2 = B.RO[(ND + 2) * nf + cf];
    rs.unct = B.RO[(ND + 3) * nf + cf];
    // F = sum_k r_k (f+_k + f-_k), fields ascending; the zero and unit entries
    // of the shear columns are skipped.
#pragma unroll
    for (int k = 0; k < nc; k++) {
        const double hsum = B.R[(2 * k) * nf + cf] + B.R[(2 * k + 1) * nf + cf];
        if (k == 0) {
#pragma unroll
            for (int c = 0; c < nc; c++) Fo[c] = r_entry<ND, D>(rs, c, 0) * hsum;
        } else if (k >= 2 && k < last) {
            const int tax = shear_axis<ND, D>(k);
#pragma unroll
            for (int aa = 0; aa < ND; aa++)
                if (aa == tax) Fo[1 + aa] = Fo[1 + aa] + hsum;
            Fo[last] = fma(r_entry<ND, D>(rs, last, k), hsum, Fo[last]);
        } else {
#pragma unroll
            for (int c = 0; c < nc; c++) Fo[c] = fma(r_entry<ND, D>(rs, c, k), hsum, Fo[c]);
        }
    }

    if (limiter) {
        // Positivity-preserving flux limiter (cited in Sec. 5.3): blend toward
        // the Lax-Friedrichs flux so that the one-sided half updates of cells i
        // and i+1 keep rho >= eps and p >= eps.
        const double eps = K.lim_eps, lam2 = 2.0 * lam, af = B.RL[4 * nc * nf + cf];
        double FL[nc], dF[nc], UL[nc], UR[nc], dUL[nc], dUR[nc];
#pragma unroll
        for (int c = 0; c < nc; c++) {
            // staged halves: FL = (F_l + F_r)/2 - af (U_r - U_l)/2 exactly as
            // ((F_l + F_r) - af (U_r - U_l)) / 2; a doubled half joins a sum in one fma
            const double hUl = B.RL[(4 * c) * nf + cf], hFl = B.RL[(4 * c + 1) * nf + cf];
            const double hUr = B.RL[(4 * c + 2) * nf + cf], hFr = B.RL[(4 * c + 3) * nf + cf];
            FL[c] = (hFl + hFr) - af * (hUr - hUl);
            dF[c] = Fo[c] - FL[c];
            UL[c] = fma(2.0, hUl, -(lam2 * fma(-2.0, hFl, FL[c])));
            UR[c] = fma(2.0, hUr, lam2 * fma(-2.0, hFr, FL[c]));
            dUR[c] = lam2 * dF[c];
            dUL[c] = -dUR[c];
        }
        double th = 1.0;
#pragma unroll
        for (int side = 0; side < 2; side++) {
            const double r0 = side ? UR[0] : UL[0];
            const double r1 = r0 + (side ? dUR[0] : dUL[0]);
            if (r1 < eps) {
                double t = (r0 - eps) / (r0 - r1);
                if (!(t > 0.0)) t = 0.0;
                if (t < th) th = t;
            }
        }
        double thp = th;
#pragma unroll
        for (int side = 0; side < 2; side++) {
            double Us[nc], Ut[nc];
#pragma unroll
            for (int c = 0; c < nc; c++) {
                Us[c] = side ? UR[c] : UL[c];
                const double dU = side ? dUR[c] : dUL[c];
                Ut[c] = Us[c] + (th == 1.0 ? dU : th * dU);
            }
            const double pt = pressure_of<ND>(Ut, K.gm1);
            if (pt < eps) {
                const double p0 = pressure_of<ND>(Us, K.gm1);
                double t = th * ((p0 - eps) / (p0 - pt));
                if (!(t > 0.0)) t = 0.0;
                if (t < thp) thp = t;
            }
        }
        if (thp < 1.0) {
#pragma unroll
            for (int c = 0; c < nc; c++) Fo[c] = FL[c] + thp * dF[c];
        }
        if constexpr (MODE == kSweepRecord) da.limrec[flin] = thp < 1.0 ? 1 : 0;
    } else if constexpr (MODE == kSweepRecord) {
        da.limrec[flin] = 0;
    }

}

// That and what else the face leaves: the flux in its array and (BYTES) its
// decision bytes in the record.
template <int ND, int D, int MODE, bool BYTES = true>
__device__ __forceinline__ void finish_face(const DirArgs &da, int limiter, const Consts &K,
                                            const SweepBuf &B, int64_t cf, int64_t flin, Status *st)
{
    constexpr int nc = ND + 2;
    const int64_t nf = B.nt * kTileFaces;
    if (!TENO_IN(st, flin, da.nfaces) || !TENO_IN(st, cf, nf)) return;
    double Fo[nc];
    face_flux<ND, D, MODE>(da, limiter, limiter ? *da.lam : 0.0, K, B, cf, flin, Fo);
    if constexpr (MODE == kSweepRecord && BYTES) {
#pragma unroll
        for (int q = 0; q < 2 * nc; q++) da.flags[flin * nc * 2 + q] = B.RD[q * nf + cf];
    }
#pragma unroll
    for (int c = 0; c < nc; c++) da.F[c * da.nfaces + flin] = Fo[c];
}

// Warps per block of the sweep (pencils side by side in the y and z sweeps) and
// the blocks per SM that its registers are bounded for: 16 warps keep the FP64
// unit 90 % busy; 20 (102 registers) gain nothing (128^3 TENO10 +0.7 %, TENO8
// -0.1 %).
constexpr int kSweepWarps = 4;
constexpr int kSweepBlocks = 4;

template <int ND, int H, int MODE>
__global__ void __launch_bounds__(32 * kSweepWarps, kSweepBlocks) sweep_kernel(const SweepArgs a)
{
    extern __shared__ double sm[];
    chain_next();
    chain_wait();
    const int w = threadIdx.x >> 5;
    const int32_t tile = (int32_t)blockIdx.x * kSweepWarps + w;
    if (tile >= a.tiles) return;
    double *slice = sm + (size_t)w * FaceSmem<ND, H>::TOTAL;
    int i = 0;
    while (i + 1 < a.nparts && tile >= a.part[i + 1].first) i++;
    const int64_t t = a.part[i].t0 + (tile - a.part[i].first);
    const int d = a.part[i].d;
    int64_t f0, x, y, z;
    if (d == 0) {
        tile_at<ND, 0>(a.g.n, a.dir[0], t, f0, x, y, z);
        sweep_tile<ND, H, 0, MODE>(a.g, a.dir[0], a.FK, a.K, a.buf, f0, x, y, z, tile, slice);
    }
    if constexpr (ND >= 2) {
        if (d == 1) {
            tile_at<ND, 1>(a.g.n, a.dir[1], t, f0, x, y, z);
            sweep_tile<ND, H, 1, MODE>(a.g, a.dir[1], a.FK, a.K, a.buf, f0, x, y, z, tile, slice);
        }
    }
    if constexpr (ND >= 3) {
        if (d == 2) {
            tile_at<ND, 2>(a.g.n, a.dir[2], t, f0, x, y, z);
            sweep_tile<ND, H, 2, MODE>(a.g, a.dir[2], a.FK, a.K, a.buf, f0, x, y, z, tile, slice);
        }
    }
}

// What the decide and exact kernels need beside the buffers.  Arguments of both
// schemes of a batch; a single problem uses one.
struct DecideArgs {
    SweepBuf B;
    int32_t tiles;
    int nc, fast, need_ct;
    int group, split;      // tiles per warp, warps per group of tiles
    unsigned *nexact[2];   // lengths of the exact path's lists (zeroed beforehand),
    uint32_t *xlist[2];    // one per scheme
    unsigned long long *exact_count;   // adds the exact-path reconstructions, or nullptr
    Status *st;
    FastK FK;
    Consts K;
};

// A decided entry's value, to its owner's place.
template <int H, bool RECORD>
__device__ __forceinline__ void decided_out(const SweepBuf &B, int64_t nq, int64_t nf, uint32_t per,
                                            bool fallback, uint32_t q, uint8_t f, int nc, Status *st)
{
    constexpr int W = 2 * H;
    double v[W];
#pragma unroll
    for (int kk = 0; kk < W; kk++) v[kk] = B.qv[kk * nq + q];
    const int slot = B.qslot[q];
    const int64_t o = (slot >> 5) * nf + (int64_t)(q / per) * kTileFaces + (slot & 31);
    if (!TENO_IN(st, o, 2 * nc * nf)) return;
    if (fallback) B.R[o] = fallback_value<H>(v, (f >> 2) & 7);
    else B.R[o] = large_value<H>(v, H == 6 && (f & 31) == 0 ? 6 : (f & 3) + 2);
    if (RECORD) B.RD[o] = f;
}

constexpr int kDecideWarps = 4, kDecideMostTiles = 16;

// The queued reconstructions of `group` consecutive tiles, by `split` warps that
// take every split-th round of 32 entries.  A round takes one entry per lane
// through the filter; its outcomes gather by kind in shared memory, and a
// kind's values are evaluated when it has a warp's worth, the rest at the end.
// Few tiles per warp and split > 1 shorten a small evaluation, many fill the
// lanes of a large one.  RECORD: decision bytes are kept.  mixed: -1, or in a
// batch of both schemes the top bit of the lengths of the tiles to take.
template <int H, bool RECORD>
__device__ __forceinline__ void decide_unit(const DecideArgs &a, int64_t unit, int mixed,
                                            uint32_t (*list)[64], uint8_t (*code)[64])
{
    constexpr int W = 2 * H;
    const SweepBuf &B = a.B;
    const int lane = threadIdx.x & 31, nc = a.nc, group = a.group, split = a.split;
    const int64_t t0 = unit / split * group;
    if (t0 >= a.tiles) return;
    const uint32_t per = 64u * nc;
    const int64_t nq = B.nt * per, nf = B.nt * kTileFaces;
    const int which = mixed > 0;
    // entries before each tile of the group: lane i holds tile i's
    int before = 0, total;
    {
        uint32_t c = lane < group && t0 + lane < a.tiles ? B.count[t0 + lane] : 0u;
        if (mixed >= 0 && (int)(c >> 31) != mixed) c = 0u;
        int sum = (int)(c & 0x7fffffffu);
        const int own = sum;
#pragma unroll
        for (int o = 1; o < kDecideMostTiles; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, sum, o);
            if (lane >= o) sum += u;
        }
        before = sum - own;
        total = __shfl_sync(0xffffffffu, sum, kDecideMostTiles - 1);
    }
    int n0 = 0, n1 = 0;                                // gathered, per kind (warp-uniform)
    for (int base = (int)(unit % split) * 32; base < total; base += 32 * split) {
        const int e = base + lane;
        uint32_t q = (uint32_t)(t0 * per) + (uint32_t)e;
        if (group > 1) {                               // the entry's tile in the group
            int i = 0;
#pragma unroll
            for (int b = kDecideMostTiles / 2; b > 0; b >>= 1) {
                const int f = __shfl_sync(0xffffffffu, before, i + b);
                if (i + b < group && e >= f) i += b;
            }
            q = (uint32_t)((t0 + i) * per) + (uint32_t)(e - __shfl_sync(0xffffffffu, before, i));
        }
        int kind = -1;                                 // 0 large stencil, 1 fallback, 2 exact path
        uint8_t fl = 0;
        if (e < total) {
            kind = 2;
            if (a.fast && TENO_IN(a.st, q, nq)) {
                double v[W];
#pragma unroll
                for (int kk = 0; kk < W; kk++) v[kk] = B.qv[kk * nq + q];
                if (fast_decide<H>(v, a.FK, fl, a.need_ct != 0))
                    kind = (fl & 3) != 0 || (H == 6 && (fl & 31) == 0) ? 0 : 1;
            }
        }
        const unsigned below = (1u << lane) - 1u;
        const unsigned m0 = __ballot_sync(0xffffffffu, kind == 0);
        const unsigned m1 = __ballot_sync(0xffffffffu, kind == 1);
        const unsigned m2 = __ballot_sync(0xffffffffu, kind == 2);
        if (kind == 0 || kind == 1) {
            const int at = kind ? n1 + __popc(m1 & below) : n0 + __popc(m0 & below);
            list[kind][at] = q;
            code[kind][at] = fl;
        }
        n0 += __popc(m0);
        n1 += __popc(m1);
        if (m2) {
            int at = 0;
            if (lane == 0) at = (int)atomicAdd(a.nexact[which], __popc(m2));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(m2 & below);
            if (kind == 2 && TENO_IN(a.st, at, nq)) a.xlist[which][at] = q;
        }
        __syncwarp();
        const bool end = base + 32 * split >= total;
        if (n0 >= 32 || (end && n0 > 0)) {
            const int n = min(n0, 32);
            n0 -= n;
            if (lane < n)
                decided_out<H, RECORD>(B, nq, nf, per, false, list[0][n0 + lane], code[0][n0 + lane], nc, a.st);
        }
        if (n1 >= 32 || (end && n1 > 0)) {
            const int n = min(n1, 32);
            n1 -= n;
            if (lane < n)
                decided_out<H, RECORD>(B, nq, nf, per, true, list[1][n1 + lane], code[1][n1 + lane], nc, a.st);
        }
        __syncwarp();
    }
    // at most 31 of a kind are left after the last round's pass
    if (lane < n0) decided_out<H, RECORD>(B, nq, nf, per, false, list[0][lane], code[0][lane], nc, a.st);
    if (lane < n1) decided_out<H, RECORD>(B, nq, nf, per, true, list[1][lane], code[1][lane], nc, a.st);
}

// MIX = 0: scheme 2 H; 1: a batch of eight- and ten-point problems, every other
// unit for each scheme.
template <int H, bool RECORD, int MIX>
__global__ void __launch_bounds__(32 * kDecideWarps, 6) decide_kernel(const DecideArgs a, int mixed)
{
    __shared__ uint32_t list_[kDecideWarps][2][64];    // gathered entries: large stencil, fallback
    __shared__ uint8_t code_[kDecideWarps][2][64];
    chain_next();
    chain_wait();
    const int warp = threadIdx.x >> 5;
    const int64_t unit = (int64_t)blockIdx.x * kDecideWarps + warp;
    if constexpr (MIX == 0) {
        decide_unit<H, RECORD>(a, unit, mixed, list_[warp], code_[warp]);
    } else if (unit & 1) {
        decide_unit<5, RECORD>(a, unit >> 1, 1, list_[warp], code_[warp]);
    } else {
        decide_unit<4, RECORD>(a, unit >> 1, 0, list_[warp], code_[warp]);
    }
}

// One reconstruction through the exact path by a whole warp, bitwise
// teno_recon: an FP64 instruction costs the warp the same for one lane as for
// 32, and a lane on its own goes through some 280 of them, 17 divisions
// among them.  Here the rows of the quadratic forms, the four eta_j, the
// small indicators, the separations gamma and the chi run side by side, about
// 100 instructions in all.  Lanes 0 .. 2H-2 hold the rows of S_H's form, the
// next 2H-3 those of S_(H-1), and so on (32 in all for H = 6); qc: the lane's
// row of coefficients.  Every lane returns the value.
// first lane of S_L's rows
template <int H>
__host__ __device__ constexpr int exact_first(int L)
{
    int f = 0;
    for (int l = H; l > L; l--) f += 2 * l - 1;
    return f;
}

template <int H, int L>
__device__ __forceinline__ void exact_row(int lane, int &row, double (&qc)[2 * H])
{
    constexpr int f = exact_first<H>(L), n = 2 * L - 1;
    if (lane >= f && lane < f + n) {
        // rows in ascending offset without offset 0 (index L - 1)
        const int r = lane - f + (lane - f >= L - 1 ? 1 : 0);
        row = r + (H - L);                             // its value index in the 2H stencil
#pragma unroll
        for (int c = 0; c < 2 * L; c++) {
            double q = 0.0;
#pragma unroll
            for (int rr = 0; rr <= c; rr++)
                if (rr == r) q = qcoef<L>(rr, c);
            qc[c + H - L] = q;
        }
    }
    if constexpr (L > 3) exact_row<H, L - 1>(lane, row, qc);
}

// The sum over the rows, in order, as beta_large_s forms it.
template <int H, int L>
__device__ __forceinline__ double exact_sum(double sr, double inner)
{
    constexpr int f = exact_first<H>(L);
    double acc = 0.0;
#pragma unroll
    for (int i = 0; i < 2 * L - 1; i++) {
        const double s = __shfl_sync(0xffffffffu, sr, f + i);
        const double t = __shfl_sync(0xffffffffu, inner, f + i);
        acc = i == 0 ? s * t : fma(s, t, acc);
    }
    return acc;
}

template <int H>
__device__ __forceinline__ double exact_warp(const double (&v)[2 * H], int row, const double (&qc)[2 * H],
                                             const Consts &K, uint8_t &flag)
{
    constexpr int W = 2 * H;
    const unsigned all = 0xffffffffu;
    const int lane = threadIdx.x & 31;
#define V(m) v[(m) + H - 1]
    // rows: inner_r = q_rr s_r + sum_{c > r} q_rc s_c, ascending c, offset 0 left out
    double sr = 0.0, inner = 0.0;
    bool begun = false;
#pragma unroll
    for (int c = 0; c < W; c++) {
        if (c == H - 1) continue;
        const double s = v[c] - V(0);
        if (c == row) {
            sr = s;
            inner = qc[c] * s;
            begun = true;
        } else if (begun && c < W) {
            const double t = fma(qc[c], s, inner);
            inner = qc[c] != 0.0 ? t : inner;          // beyond the row's stencil: no term
        }
    }
    double b3 = exact_sum<H, 3>(sr, inner), b4 = exact_sum<H, 4>(sr, inner), b5 = 0.0, b6 = 0.0;
    if constexpr (H >= 5) b5 = exact_sum<H, 5>(sr, inner);
    if constexpr (H >= 6) b6 = exact_sum<H, 6>(sr, inner);
    // small indicators k = 0, 1, 2: b = (x - 2 y) + z; a_0 = V(-1) - V(1),
    // a_1 = (3 V(0) - 4 V(1)) + V(2), a_2 = (V(-2) - 4 V(-1)) + 3 V(0)
    const int k3 = lane % 3;
    const double t3 = 3.0 * V(0);
    const double ax = k3 == 0 ? V(-1) : (k3 == 1 ? t3 : V(-2));
    const double ay = k3 == 2 ? V(-1) : V(1);
    const double ab = fma(k3 == 0 ? -1.0 : -4.0, ay, ax);
    const double az = k3 == 1 ? V(2) : t3;
    const double a = k3 == 0 ? ab : ab + az;
    const double bx = k3 == 0 ? V(-1) : (k3 == 1 ? V(0) : V(-2));
    const double by = k3 == 0 ? V(0) : (k3 == 1 ? V(1) : V(-1));
    const double bz = k3 == 0 ? V(1) : (k3 == 1 ? V(2) : V(0));
    const double b = fma(-2.0, by, bx) + bz;
    const double bs = 0.25 * (a * a) + (13.0 / 12.0) * (b * b);
    // lanes 0-2: gamma of the small stencils; 3..H: of S_3..S_H; 8-11: eta_j, j = -1..2
    const int j = (lane & 3) - 1;
    const double vp = j < 0 ? V(0) : (j == 0 ? V(1) : (j == 1 ? V(2) : V(3)));
    const double vo = j < 0 ? V(-1) : (j == 0 ? V(0) : (j == 1 ? V(1) : V(2)));
    const double vn = j < 0 ? V(-2) : (j == 0 ? V(-1) : (j == 1 ? V(0) : V(1)));
    const double dp = vp - vo, dm = vo - vn;
    const double num = fabs((2.0 * dp) * dm) + K.eps_eta;
    const double den = (dp * dp + dm * dm) + K.eps_eta;
    const double beta = lane < 3 ? bs : (lane == 3 ? b3 : (lane == 4 ? b4 : (lane == 5 ? b5 : b6)));
    const double x = beta + K.eps_beta, x2 = x * x, x4 = x2 * x2, x7 = (x4 * x2) * x;
    const bool eta = lane >= 8;
    const double q1 = (eta ? num : 1.0) / (eta ? den : x7);
    const double g0 = __shfl_sync(all, q1, 0), g1 = __shfl_sync(all, q1, 1), g2 = __shfl_sync(all, q1, 2);
    double emin = __shfl_sync(all, q1, 8);
#pragma unroll
    for (int i = 1; i < 4; i++) {
        const double e = __shfl_sync(all, q1, 8 + i);
        if (e < emin) emin = e;
    }
    const double g012 = (g0 + g1) + g2;
    // lanes 0-2: g_k / g012; 3..H: chi of S_3..S_H; 8: eta / C_r
    const double q2 = (eta ? emin : q1) / (eta ? K.cr : (lane < 3 ? g012 : g012 + q1));
    const double r = __shfl_sync(all, q2, 8);
    const double m = 1.0 - (r < 1.0 ? r : 1.0);
    const double om = 1.0 - m, om2 = om * om;
    const double g = (om2 * om2) * (1.0 + 4.0 * m);
    const double bct = K.alpha1 - K.alpha2 * (1.0 - g);
    const double fln = floor(bct);
    const int nexp = fln < 0.0 ? 0 : (fln > 22.0 ? 22 : (int)fln);
    const unsigned keep = __ballot_sync(all, !(q2 < TENO_TENPOW[nexp]));
    const uint8_t fct = (uint8_t)(((nexp - 7) & 7) << 5);
    int sel = 0;
#pragma unroll
    for (int L = 3; L <= H; L++)
        if (keep >> L & 1u) sel = L;
    if (sel) {
        flag = (uint8_t)(large_code(sel) | fct);
        return large_value<H>(v, sel);
    }
    flag = (uint8_t)((keep & 7u) << 2 | fct);
    return fallback_value<H>(v, (int)(keep & 7u));
#undef V
}

// The listed reconstructions through the exact path: a warp for each while they
// are few (at most kExactFew), a lane for each when they fill warps.  Bound by
// the FP64 pipe (86 % busy).
constexpr unsigned kExactFew = 152 * 16;

// Entries of a long list that the largest stencil's test rejected, with what the
// other tests need, until a warp of them is together: some 3 % reject in smooth
// flow, spread over two thirds of the warps, whose lanes would all wait for the
// smaller stencils' forms.
struct ExactRest {
    ReconTests t[64];
    uint32_t q[64];
};

// Value (and, RECORD, decision byte) of entry q to its owner's place.
template <bool RECORD>
__device__ __forceinline__ void exact_out(const DecideArgs &a, uint32_t q, double val, uint8_t fl)
{
    const SweepBuf &B = a.B;
    const uint32_t per = 64u * a.nc;
    const int64_t nf = B.nt * kTileFaces;
    const int slot = B.qslot[q];
    const int64_t o = (slot >> 5) * nf + (int64_t)(q / per) * kTileFaces + (slot & 31);
    if (!TENO_IN(a.st, o, 2 * a.nc * nf)) return;
    B.R[o] = val;
    if (RECORD) B.RD[o] = fl;
}

template <int H>
__device__ __forceinline__ void exact_in(const SweepBuf &B, int64_t nq, uint32_t q, double (&v)[2 * H])
{
#pragma unroll
    for (int kk = 0; kk < 2 * H; kk++) v[kk] = B.qv[kk * nq + q];
}

// which: the list; kExactAll: every queued entry, where there is no filter to make
// a list (the queues' lanes are nearly all filled then).
constexpr int kExactAll = -1;

template <int H, bool RECORD>
__device__ __forceinline__ void exact_list(const DecideArgs &a, int which, unsigned block,
                                           unsigned blocks, ExactRest &rest)
{
    const SweepBuf &B = a.B;
    const uint32_t per = 64u * a.nc;
    const int64_t nq = B.nt * per;
    const bool all = which == kExactAll;
    const unsigned n = all ? (unsigned)a.tiles * per : *a.nexact[which];
    if (n == 0) return;
    if (a.exact_count && !all && block == 0 && threadIdx.x == 0)
        atomicAdd(a.exact_count, (unsigned long long)n);
    const int lane = threadIdx.x & 31;
    const unsigned warp = block * (blockDim.x >> 5) + (threadIdx.x >> 5), warps = blocks * (blockDim.x >> 5);
    if (!all && n <= kExactFew) {
        int row = -1;
        double qc[2 * H];
#pragma unroll
        for (int c = 0; c < 2 * H; c++) qc[c] = 0.0;   // beyond the row's stencil
        exact_row<H, H>(lane, row, qc);
        for (unsigned i = warp; i < n; i += warps) {
            const uint32_t q = a.xlist[which][i];
            if (!TENO_IN(a.st, q, nq)) continue;
            double v[2 * H];
            exact_in<H>(B, nq, q, v);
            uint8_t fl;
            const double val = exact_warp<H>(v, row, qc, a.K, fl);
            if (lane == 0) exact_out<RECORD>(a, q, val, fl);
        }
        return;
    }
    int held = 0;                                      // gathered (warp-uniform)
    for (unsigned base = warp * 32; base < n; base += warps * 32) {
        const bool last = base + warps * 32 >= n;
        bool rejected = false;
        uint32_t q = 0;
        ReconTests t;
        bool have = base + lane < n;
        if (have && all) {
            q = base + lane;
            const uint32_t tile = q / per;
            have = q - tile * per < (B.count[tile] & 0x7fffffffu);
        } else if (have) {
            q = a.xlist[which][base + lane];
        }
        if (all && a.exact_count) {
            const unsigned m = __ballot_sync(0xffffffffu, have);
            if (lane == 0 && m) atomicAdd(a.exact_count, (unsigned long long)__popc(m));
        }
        if (have) {
            if (TENO_IN(a.st, q, nq)) {
                double v[2 * H], val;
                uint8_t fl;
                exact_in<H>(B, nq, q, v);
                rejected = !recon_largest<H>(v, a.K, t, val, fl);
                if (!rejected) exact_out<RECORD>(a, q, val, fl);
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, rejected);
        if (rejected) {
            const int at = held + __popc(m & ((1u << lane) - 1u));
            rest.t[at] = t;
            rest.q[at] = q;
        }
        held += __popc(m);
        __syncwarp();
        while (held >= 32 || (last && held > 0)) {
            const int k = min(held, 32);
            held -= k;
            if (lane < k) {
                const ReconTests tr = rest.t[held + lane];
                const uint32_t qr = rest.q[held + lane];
                double v[2 * H];
                uint8_t fl;
                exact_in<H>(B, nq, qr, v);
                const double val = recon_smaller<H>(v, a.K, tr, fl);
                exact_out<RECORD>(a, qr, val, fl);
            }
        }
        __syncwarp();
    }
}

template <int H, bool RECORD, int MIX>
__global__ void __launch_bounds__(128) exact_kernel(const DecideArgs a, int which)
{
    __shared__ ExactRest rest_[4];
    ExactRest &rest = rest_[threadIdx.x >> 5];
    chain_next();
    chain_wait();
    if constexpr (MIX == 0) {
        exact_list<H, RECORD>(a, which, blockIdx.x, gridDim.x, rest);
    } else if (blockIdx.x & 1) {
        exact_list<5, RECORD>(a, 1, blockIdx.x >> 1, gridDim.x >> 1, rest);
    } else {
        exact_list<4, RECORD>(a, 0, blockIdx.x >> 1, gridDim.x >> 1, rest);
    }
}

template <int ND, int D, int MODE>
__device__ __forceinline__ void finish_lane(const SweepArgs &a, int64_t t, int lane, int64_t cf)
{
    const DirArgs &da = a.dir[D];
    int64_t f0, x, y, z;
    int p, fo;
    tile_at<ND, D>(a.g.n, da, t, f0, x, y, z);
    tile_lane<D>(ND == 1 ? 0 : da.tps, lane, p, fo);
    if (D == 0) y += p;
    else x += p;
    if (f0 + fo > a.g.n[D] - da.skip_last || x >= a.g.n[0] || y >= a.g.n[1]) return;
    finish_face<ND, D, MODE>(da, a.g.limiter, a.K, a.buf, cf, face_index<D>(a.g.n, f0 + fo, x, y, z),
                             a.g.st);
}

template <int ND, int MODE>
__global__ void __launch_bounds__(128) finish_kernel(const SweepArgs a)
{
    chain_next();
    chain_wait();
    const int32_t tile = (int32_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (tile >= a.tiles) return;
    int i = 0;
    while (i + 1 < a.nparts && tile >= a.part[i + 1].first) i++;
    const int64_t t = a.part[i].t0 + (tile - a.part[i].first), cf = (int64_t)tile * kTileFaces + lane;
    const int d = a.part[i].d;
    if (d == 0) finish_lane<ND, 0, MODE>(a, t, lane, cf);
    if constexpr (ND >= 2) {
        if (d == 1) finish_lane<ND, 1, MODE>(a, t, lane, cf);
    }
    if constexpr (ND >= 3) {
        if (d == 2) finish_lane<ND, 2, MODE>(a, t, lane, cf);
    }
}

// Few tiles: a block per tile, a warp per field and sign, everything in one
// launch.  Where tiles do not fill the chip, what counts is the longest chain
// of one warp: a lane of the sweep goes through all fields one after the other
// (some 390 FP64 instructions in 1D, 64 cycles each), and the decide, exact and
// finish kernels follow it with a launch each.  Here the warps share a tile's
// fields and signs: Roe state and splitting speeds by one warp each, w by the
// f+ warp of a field and g by its f- warp, then each its reconstruction.  Lanes
// of a warp may want different kinds of value, which costs FP64 instructions
// that the four kernels save: those are the better ones for more tiles.
template <int ND, int H>
struct SmallSmem {
    static constexpr int nc = ND + 2, W = 2 * H;
    static constexpr int NW = 2 * nc;                  // warps
    static constexpr int CELLS = 0;                    // FaceSmem
    static constexpr int ROE = FaceSmem<ND, H>::TOTAL; // [nd + 9][32] Roe scalars, finish's rows first
    static constexpr int SPD = ROE + (ND + 9) * 32;    // [4][32] splitting speeds
    static constexpr int PRJ = SPD + 4 * 32;           // [2 nc][W][32] halved w and g
    static constexpr int VAL = PRJ + NW * W * 32;      // [2 nc][32] values
    static constexpr int BYTES = 8 * (VAL + NW * 32);
    static constexpr int ARG = 4 * 32 * 2;             // maximising cells, small_tile's own array
    // the limiter's rows [4 nc + 1][32] take the projections' room once those were read
    static_assert(4 * nc + 1 <= NW * W, "limiter rows fit in the projections' room");
};

// Flux difference of one component of a cell and the stage's combination, as
// combine_kernel forms them.
__device__ __forceinline__ double stage_value(int mode, double acc, double U, double Un, double dt)
{
    if (mode == 0) return acc;
    const double t = U + dt * acc;
    if (mode == 1) return t;
    if (mode == 2) return 0.75 * Un + 0.25 * t;
    return (1.0 / 3.0) * Un + (2.0 / 3.0) * t;
}

// Roe state, its rows for the projections and the finish, and the splitting
// speeds of a tile: warp 0 the first, warps 1-4 a speed each.
template <int ND, int H, int D, int MODE>
__device__ __forceinline__ void small_states(const GridArgs &a, const DirArgs &da, const Consts &K,
                                             int warp, int b0, int bs, bool active, bool own,
                                             double *sm, uint16_t *arg)
{
    using SL = FaceSmem<ND, H>;
    using SS = SmallSmem<ND, H>;
    constexpr int W = 2 * H, NS = SL::NS;
    const int lane = threadIdx.x & 31;
#define TMP(q, j) sm[SL::TMP + (q) * NS + (j)]
    if (!active) return;
    if (warp == 0) {
        const int bl = b0 + (H - 1) * bs, br = bl + bs;
        RoeScalars<ND> rs;
        double ul[ND], ur[ND];
#pragma unroll
        for (int k = 0; k < ND; k++) { ul[k] = TMP(SL::QV + k, bl); ur[k] = TMP(SL::QV + k, br); }
        const double c2 = roe_state<ND, D>(ul, TMP(SL::QH, bl), TMP(SL::QSR, bl), ur, TMP(SL::QH, br),
                                           TMP(SL::QSR, br), K.gm1, rs);
        if (own && !(c2 > 0.0)) atomicAdd(&a.st->nonphys, 1ull);
        double *r = sm + SS::ROE + lane;
#pragma unroll
        for (int k = 0; k < ND; k++) r[k * 32] = rs.ut[k];
        r[ND * 32] = rs.Ht;
        r[(ND + 1) * 32] = rs.ct;
        r[(ND + 2) * 32] = rs.q2;
        r[(ND + 3) * 32] = rs.unct;
        r[(ND + 4) * 32] = rs.cinv;
        r[(ND + 5) * 32] = rs.b1;
        r[(ND + 6) * 32] = rs.b2;
        r[(ND + 7) * 32] = rs.unc;
        r[(ND + 8) * 32] = rs.bu;
    } else if (warp <= 4) {
        const int row = warp == 1 ? SL::QLM : (warp == 2 ? SL::QL0 : (warp == 3 ? SL::QLP : SL::QLR));
        double m = 0.0;
        int jm = 0;
#pragma unroll
        for (int j = 0; j < W; j++) {
            const double e = TMP(row, b0 + j * bs);
            if (j == 0 || speed_gt(e, m)) { m = e; jm = j; }
        }
        sm[SS::SPD + (warp - 1) * 32 + lane] = m;
        if (MODE == kSweepRecord) arg[(warp - 1) * 32 + lane] = (uint16_t)jm;
    }
#undef TMP
}

// This warp's row of L applied to U (f+ warps) or F (f- warps) of the stencil.
template <int ND, int H, int D>
__device__ __forceinline__ void small_project(int k, int s, int b0, int bs, const double *sm, double *out)
{
    using SL = FaceSmem<ND, H>;
    using SS = SmallSmem<ND, H>;
    constexpr int nc = ND + 2, last = nc - 1, W = 2 * H, NS = SL::NS;
    const int lane = threadIdx.x & 31;
    const double *r = sm + SS::ROE + lane;
    RoeScalars<ND> rs;
#pragma unroll
    for (int i = 0; i < ND; i++) rs.ut[i] = r[i * 32];
    rs.cinv = r[(ND + 4) * 32];
    rs.b1 = r[(ND + 5) * 32];
    rs.b2 = r[(ND + 6) * 32];
    rs.unc = r[(ND + 7) * 32];
    rs.bu = r[(ND + 8) * 32];
    const bool shear = (k >= 2 && k < last);
    const int tax = shear ? shear_axis<ND, D>(k) : 0;
    double lrow[nc];
    l_row<ND, D>(rs, k, lrow);
#pragma unroll
    for (int j = 0; j < W; j++) {
        const double *c = sm + 2 * (b0 + j * bs) + s;  // the pair's U or F
        double w;
        if (shear) {
            w = c[2 * (1 + tax) * NS] + lrow[0] * c[0];
        } else {
            w = lrow[0] * c[0];
#pragma unroll
            for (int i = 1; i < nc; i++) w = fma(lrow[i], c[2 * i * NS], w);
        }
        out[j * 32 + lane] = w;
    }
}

// One tile at the pencils from (x, y, z), faces from f0 of direction d, by a block.
template <int ND, int H, int MODE>
__device__ __forceinline__ void small_tile(const GridArgs &a, const DirArgs &da, const FastK &FK,
                                           const Consts &K, int d, int64_t f0, int64_t x, int64_t y,
                                           int64_t z, unsigned long long *exact_count, double *sm,
                                           const FuseArgs &fuse)
{
    using SL = FaceSmem<ND, H>;
    using SS = SmallSmem<ND, H>;
    constexpr int nc = ND + 2, last = nc - 1, W = 2 * H, NS = SL::NS, NT = 32 * SS::NW;
    const bool fused = ND == 1 && fuse.mode >= 0;
    __shared__ uint16_t arg[SS::ARG / 2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, k = warp >> 1, s = warp & 1;
    const int tps = ND == 1 ? 0 : da.tps;
    int p, fo, b0, bs;
    int64_t flin, npen;
    const double2 *UF = (const double2 *)sm;
    if (d == 0) {
        tile_lane<0>(tps, lane, p, fo);
        b0 = p * ((kTileFaces >> tps) + 2 * H - 1) + fo;
        bs = 1;
        npen = a.n[1] - y;
        flin = face_index<0>(a.n, f0 + fo, x, y + p, z);
    } else {
        tile_lane<1>(tps, lane, p, fo);
        b0 = lane;
        bs = 1 << tps;
        npen = a.n[0] - x;
        flin = d == 1 ? face_index<1>(a.n, f0 + fo, x + p, y, z) : face_index<2>(a.n, f0 + fo, x + p, y, z);
    }
    const int64_t last_face = (d == 0 ? a.n[0] : (d == 1 ? a.n[1] : a.n[2])) - da.skip_last;
    // the fused update of the last cell takes face n also where skip_last leaves it out
    const bool active = f0 + fo <= (fused ? a.n[0] : last_face) && p < npen;
    if (active && !TENO_IN(a.st, flin, da.nfaces)) flin = 0;     // debug build: counted, redirected
    // counted here: all, unless tiles overlap or face n is the periodic image of face 0
    const bool own = f0 + fo <= last_face && (fo < da.own || f0 + fo == a.n[0]);
    // the fused update's inputs, on their way while the fluxes are computed
    double Uk[nc], Un[nc], dt = 0.0;
    const int64_t ic = f0 + lane;                                 // the lane's cell
    const bool mine = fused && warp == 0 && lane < da.own && ic < a.n[0];
    if (fused && warp == 0) dt = fuse.dt_dev ? *fuse.dt_dev : fuse.dt;
    if (mine) {
#pragma unroll
        for (int c = 0; c < nc; c++) {
            Uk[c] = fuse.mode > 0 ? a.U[c * a.ncell + ic] : 0.0;
            Un[c] = fuse.mode > 1 ? fuse.Un[c * a.ncell + ic] : 0.0;
        }
    }

    if (ND == 1 || d == 0) stage_cells<ND, H, 0>(a, da, K, f0, x, y, z, sm, threadIdx.x, NT);
    if constexpr (ND >= 2) {
        if (d == 1) stage_cells<ND, H, 1>(a, da, K, f0, x, y, z, sm, threadIdx.x, NT);
    }
    if constexpr (ND >= 3) {
        if (d == 2) stage_cells<ND, H, 2>(a, da, K, f0, x, y, z, sm, threadIdx.x, NT);
    }
    __syncthreads();
    if (ND == 1 || d == 0) small_states<ND, H, 0, MODE>(a, da, K, warp, b0, bs, active, own, sm, arg);
    if constexpr (ND >= 2) {
        if (d == 1) small_states<ND, H, 1, MODE>(a, da, K, warp, b0, bs, active, own, sm, arg);
    }
    if constexpr (ND >= 3) {
        if (d == 2) small_states<ND, H, 2, MODE>(a, da, K, warp, b0, bs, active, own, sm, arg);
    }
    __syncthreads();
    double *prj = sm + SS::PRJ + warp * W * 32;
    if (active) {
        if (ND == 1 || d == 0) small_project<ND, H, 0>(k, s, b0, bs, sm, prj);
        if constexpr (ND >= 2) {
            if (d == 1) small_project<ND, H, 1>(k, s, b0, bs, sm, prj);
        }
        if constexpr (ND >= 3) {
            if (d == 2) small_project<ND, H, 2>(k, s, b0, bs, sm, prj);
        }
    }
    __syncthreads();
    double v[W], val = 0.0;
    uint8_t fl = 0;
    bool open = false;
    if (active) {
        const double *hw = sm + SS::PRJ + 2 * k * W * 32 + lane, *hg = hw + W * 32;
        const int sp = K.split ? 3 : (k == 0 ? 0 : (k == last ? 2 : 1));
        const double al = sm[SS::SPD + sp * 32 + lane], sa = s ? -al : al;
#pragma unroll
        for (int kk = 0; kk < W; kk++) {
            const int j = s ? W - 1 - kk : kk;
            v[kk] = fma(sa, hw[j * 32], hg[j * 32]);
        }
        const bool need_ct = MODE == kSweepRecord && a.need_ct;
        open = true;
        if (a.fast) {
            open = !quick_large<H>(v, FK, need_ct, fl) && !fast_decide<H>(v, FK, fl, need_ct);
            if (!open) val = decided_value<H>(v, fl);
        }
    }
    unsigned left = __ballot_sync(0xffffffffu, open);
    if (left) {
        const unsigned owned = __ballot_sync(0xffffffffu, own);
        if (exact_count && lane == 0) atomicAdd(exact_count, (unsigned long long)__popc(left & owned));
        if (__popc(left) > 3) {                        // a lane each costs about as much as three
            if (open) val = teno_recon<H>(v, K, fl);
        } else {
            int row = -1;
            double qc[W];
#pragma unroll
            for (int c = 0; c < W; c++) qc[c] = 0.0;
            exact_row<H, H>(lane, row, qc);
            while (left) {
                const int src = __ffs(left) - 1;
                left &= left - 1;
                double u[W];
#pragma unroll
                for (int kk = 0; kk < W; kk++) u[kk] = __shfl_sync(0xffffffffu, v[kk], src);
                uint8_t f;
                const double r = exact_warp<H>(u, row, qc, K, f);
                if (lane == src) {
                    val = r;
                    fl = f;
                }
            }
        }
    }
    sm[SS::VAL + warp * 32 + lane] = val;
    if (MODE == kSweepRecord && active) da.flags[flin * nc * 2 + 2 * k + s] = fl;
    __syncthreads();
    if (warp) return;
    double Fo[nc];
    if (active) {
        SweepBuf B;
        B.nt = 1;                                      // rows of 32
        B.R = sm + SS::VAL;
        B.RO = sm + SS::ROE;
        B.RL = sm + SS::PRJ;
        if (a.limiter) {
            const int bl = b0 + (H - 1) * bs, br = bl + bs;
#pragma unroll
            for (int c = 0; c < nc; c++) {
                const double2 cl = UF[c * NS + bl], cr = UF[c * NS + br];
                B.RL[(4 * c) * 32 + lane] = cl.x;
                B.RL[(4 * c + 1) * 32 + lane] = cl.y;
                B.RL[(4 * c + 2) * 32 + lane] = cr.x;
                B.RL[(4 * c + 3) * 32 + lane] = cr.y;
            }
            const double sl = sm[SL::TMP + SL::QLR * NS + bl], sr = sm[SL::TMP + SL::QLR * NS + br];
            B.RL[4 * nc * 32 + lane] = sr > sl ? sr : sl;
        }
        if (MODE == kSweepRecord)
            put_word(da.argmax + flin, arg[lane] | (arg[32 + lane] << 4) | (arg[64 + lane] << 8) |
                                           (arg[96 + lane] << 12));
        // the fused stage's limiter forms dt/dx itself (1D)
        const double lam = fused ? dt * fuse.inv_dx : (a.limiter ? *da.lam : 0.0);
        if (ND == 1 || d == 0) face_flux<ND, 0, MODE>(da, a.limiter, lam, K, B, lane, flin, Fo);
        if constexpr (ND >= 2) {
            if (d == 1) face_flux<ND, 1, MODE>(da, a.limiter, lam, K, B, lane, flin, Fo);
        }
        if constexpr (ND >= 3) {
            if (d == 2) face_flux<ND, 2, MODE>(da, a.limiter, lam, K, B, lane, flin, Fo);
        }
        if (!fused) {
#pragma unroll
            for (int c = 0; c < nc; c++) da.F[c * da.nfaces + flin] = Fo[c];
        }
    }
    if (ND == 1 && fused) {
#pragma unroll
        for (int c = 0; c < nc; c++) {
            const double Fr = __shfl_down_sync(0xffffffffu, Fo[c], 1);
            const double t = (Fr - Fo[c]) * fuse.inv_dx;
            const double acc = zero_minus(t);
            if (mine && TENO_IN(a.st, ic, a.ncell))
                fuse.out[c * a.ncell + ic] = stage_value(fuse.mode, acc, Uk[c], Un[c], dt);
        }
    }
}

// 24 warps per SM at least (30 in 1D, 20 in 3D), 80 registers (64, 96).
template <int ND, int H, int MODE>
__global__ void __launch_bounds__(64 * (ND + 2), ND == 1 ? 5 : (ND == 2 ? 3 : 2))
    small_kernel(const SweepArgs a)
{
    extern __shared__ double sm[];
    chain_next();
    chain_wait();
    const int32_t tile = (int32_t)blockIdx.x;
    int i = 0;
    while (i + 1 < a.nparts && tile >= a.part[i + 1].first) i++;
    const int64_t t = a.part[i].t0 + (tile - a.part[i].first);
    const int d = a.part[i].d;
    int64_t f0, x, y, z;
    if (ND == 1 || d == 0) tile_at<ND, 0>(a.g.n, a.dir[0], t, f0, x, y, z);
    if constexpr (ND >= 2) {
        if (d == 1) tile_at<ND, 1>(a.g.n, a.dir[1], t, f0, x, y, z);
    }
    if constexpr (ND >= 3) {
        if (d == 2) tile_at<ND, 2>(a.g.n, a.dir[2], t, f0, x, y, z);
    }
    small_tile<ND, H, MODE>(a.g, a.dir[d], a.FK, a.K, d, f0, x, y, z, a.exact_count, sm, a.fuse);
}

// Blocks of the exact kernel: 128 lanes for every possible entry, at most a wave.
inline int64_t exact_blocks(const DecideArgs &a)
{
    const int64_t most = ((int64_t)a.tiles * a.nc + 1) / 2;
    return most < 608 ? most : 608;
}

// The decide and exact kernels of one chunk (a's group and split are set here).
// mixed: in a batch of both schemes, the one to take (MIX = 0).
template <int H, bool RECORD, int MIX>
cudaError_t launch_decisions(DecideArgs &a, cudaStream_t s, int mixed = -1)
{
    // at least four waves of warps (24 on each of 152 SMs) before tiles share
    // one; a small evaluation's rounds go to a warp each while that is about two
    // waves (a round takes some 5 us, alone or beside 23 others)
    const int64_t fill = 152 * 24, sides = MIX ? 2 : 1;
    a.group = a.split = 1;
    while (a.group < kDecideMostTiles && a.tiles * sides >= 8 * fill * a.group) a.group *= 2;
    while (a.group == 1 && a.split < 2 * a.nc && a.tiles * sides * a.split <= fill) a.split *= 2;
    const int64_t units = (int64_t)((a.tiles + a.group - 1) / a.group) * a.split * sides;
    cudaError_t e = launch_chained(a.tiles <= kChainTiles, decide_kernel<H, RECORD, MIX>,
                                   (unsigned)((units + kDecideWarps - 1) / kDecideWarps),
                                   32 * kDecideWarps, 0, s, a, mixed);
    if (e != cudaSuccess) return e;
    return launch_chained(a.tiles <= kChainTiles, exact_kernel<H, RECORD, MIX>,
                          (unsigned)(sides * exact_blocks(a)), 128, 0, s, a, (int)(mixed > 0));
}

template <int ND, int H, int MODE>
cudaError_t launch_chunk_mode(const SweepArgs &a, cudaStream_t s)
{
    constexpr size_t smem = sizeof(double) * (size_t)FaceSmem<ND, H>::TOTAL * kSweepWarps;
    static_assert(smem <= (size_t)48 << 10, "launched without allow_shared");
    if constexpr (MODE != kSweepFrozen) {
        if (a.small) {
            constexpr size_t bytes = SmallSmem<ND, H>::BYTES;
            const cudaError_t e = allow_shared(small_kernel<ND, H, MODE>, bytes, SmallSmem<ND, H>::ARG);
            if (e != cudaSuccess) return e;
            return launch_chained(a.tiles <= kChainTiles, small_kernel<ND, H, MODE>, (unsigned)a.tiles,
                                  64 * (ND + 2), bytes, s, a);
        }
    }
    const unsigned blocks = (unsigned)((a.tiles + kSweepWarps - 1) / kSweepWarps);
    cudaError_t e = launch_chained(a.tiles <= kChainTiles, sweep_kernel<ND, H, MODE>, blocks, 32 * kSweepWarps, smem, s, a);
    if (e != cudaSuccess) return e;
    if (MODE != kSweepFrozen) {
        DecideArgs d;
        d.B = a.buf;
        d.tiles = a.tiles;
        d.nc = ND + 2;
        d.fast = a.g.fast;
        d.need_ct = a.g.need_ct;
        d.nexact[0] = d.nexact[1] = a.nexact;
        d.xlist[0] = d.xlist[1] = a.buf.xlist;
        d.exact_count = a.exact_count;
        d.st = a.g.st;
        d.FK = a.FK;
        d.K = a.K;
        // no filter: the exact kernel takes the queues as they are (a pass of the decide
        // kernel that only lists them costs 0.45 ms per 2 M faces)
        e = d.fast ? launch_decisions<H, MODE == kSweepRecord, 0>(d, s)
                   : launch_chained(a.tiles <= kChainTiles, exact_kernel<H, MODE == kSweepRecord, 0>,
                                    (unsigned)exact_blocks(d), 128, 0, s, d, kExactAll);
        if (e != cudaSuccess) return e;
    }
    return launch_chained(a.tiles <= kChainTiles, finish_kernel<ND, MODE>, (unsigned)((a.tiles + 3) / 4), 128, 0,
                          s, a);
}

// One chunk's fluxes, in the mode its arguments ask for (a decision record to
// write, recorded decisions to apply, or neither).
template <int ND, int H>
cudaError_t launch_chunk(const SweepArgs &a, cudaStream_t s)
{
    for (int i = 0; i < a.nparts; i++) {
        const DirArgs &d = a.dir[a.part[i].d];
        if ((d.flags && d.frozen) || (d.flags && (!d.argmax || !d.limrec)) ||
            (d.frozen && !d.frozen_argmax))
            return cudaErrorInvalidValue;
    }
    if (a.dir[0].flags) return launch_chunk_mode<ND, H, kSweepRecord>(a, s);
    if (a.dir[0].frozen) return launch_chunk_mode<ND, H, kSweepFrozen>(a, s);
    return launch_chunk_mode<ND, H, kSweepPlain>(a, s);
}

}  // namespace teno
