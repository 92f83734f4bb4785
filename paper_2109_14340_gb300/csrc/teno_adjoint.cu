// Adjoint (vector-Jacobian product) of the TENO-AA right-hand side and of the
// SSP-RK3 step, with the forward's discrete decisions frozen.
//
// With the stencil selection and the small-stencil cut-offs of every face,
// field and sign fixed (the decision record of the forward), the TENO-AA
// reconstruction (Sec. 3.3) is a fixed linear combination of the split
// characteristic fluxes, so L(U) is differentiable: the Roe average,
// eigenvectors, projection, splitting speeds (their maximising cell fixed),
// back-projection and the flux difference are smooth.  The positivity limiter
// is not differentiated (the adjoint calls reject limiter = 1).
//
// Per direction, three kernels (the FP64 pipe bounds them all):
//
//   adj_face     a warp per tile of 32 faces, as in the sweep: the face's forward
//                values from the state and its stored primitives, then the
//                reverse of each step.  Where every field has the same frozen
//                coefficients (smooth regions), a face's part in the adjoint of
//                its 2H cells is a product: (c+_j - c-_j) M for U and
//                (c+_j + c-_j) N for the flux, M = sum_k l_k alpha_k h_k / 2 and
//                N = sum_k l_k h_k / 2, so M and N are all that is written.
//   adj_mixed    the other faces, from a list, a lane each: their parts written
//                out per stencil position.
//   adj_gather   a lane per cell: the parts of the faces whose stencils contain
//                it (ghost positions mapped back by the boundary rules).  What
//                faces contribute to a cell's velocity, pressure, sound speed,
//                enthalpy and sqrt(rho) is summed over faces and directions
//                first, and taken to the conserved variables once.
//
// 512^2 TENO8, per direction: adj_face 0.23 ms (FP64 85 % busy), adj_mixed 0.06 to
// 0.07 (a chain of dependent FP64 work, few faces), adj_gather 0.11 to 0.13 (FP64
// 74 to 80 %).  One kernel that wrote every face's part per stencil position took
// 0.49 to 0.54 ms and its gather 0.07 to 0.10.
//
// The result is deterministic (a list's order only says which lane does a face).
#include <cstring>

#include "teno.h"
#include "teno_face.cuh"

namespace teno {

// Rows of a face's part, [row][nfaces]: M, N; the Roe state's adjoints of
// velocity, enthalpy and sqrt(rho) of cells i and i+1; the splitting speeds'.
template <int ND>
struct AdjRows {
    static constexpr int nc = ND + 2;
    static constexpr int M = 0, N = nc, LEFT = 2 * nc, RIGHT = LEFT + ND + 2, SPEED = RIGHT + ND + 2;
    static constexpr int NR = SPEED + 3;
};

// Rows summed over directions per cell, [row][ncell]: adjoints of U, velocity,
// pressure, sound speed, enthalpy, sqrt(rho).
template <int ND>
struct AdjSums {
    static constexpr int nc = ND + 2;
    static constexpr int U = 0, V = nc, P = nc + ND, C = P + 1, H = P + 2, S = P + 3, NR = P + 4;
};

// Kinds of face in the gather.
enum { kAdjLarge = 0, kAdjUniform = 1, kAdjMixed = 2 };

struct AdjArgs {
    GridArgs g;             // state and its primitives
    DirArgs d;
    const double *lam;      // adjoint of L(U) [nc][ncell]
    const uint8_t *flags;   // decision record of this direction
    double *rows;           // AdjRows
    double *slots;          // [W][2 nc][nfaces]: mixed faces' parts per stencil position, the
                            // adjoint of U then of F
    uint16_t *words;        // [nfaces] maximising cells of the splitting speeds
    uint8_t *kind;          // [nfaces]
    uint32_t *list;         // mixed faces
    unsigned *count;        // their number
    double *sums;           // AdjSums
    int64_t tiles;
    double inv_dx;
    Consts K;
};

// Adjoints of a cell gathered from its faces.
template <int ND>
struct CellBar {
    double U[ND + 2], F[ND + 2], u[ND], p, c, H, s;
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int k = 0; k < ND + 2; k++) U[k] = F[k] = 0.0;
#pragma unroll
        for (int k = 0; k < ND; k++) u[k] = 0.0;
        p = c = H = s = 0.0;
    }
};

// Reverse of the physical flux F_D = (m_D, m_D u + p e_D, u_D (E + p)), b.F onto U,
// velocity and pressure.
template <int ND, int D>
__device__ __forceinline__ void flux_bar(const double (&U)[ND + 2], const double (&u)[ND], double p,
                                         CellBar<ND> &b)
{
    constexpr int last = ND + 1;
    double md = b.F[0];
#pragma unroll
    for (int a = 0; a < ND; a++) {
        md = fma(b.F[1 + a], u[a], md);
        b.u[a] = fma(b.F[1 + a], U[1 + D], b.u[a]);
    }
    b.U[1 + D] += md;
    b.u[D] = fma(b.F[last], U[last] + p, b.u[D]);
    b.U[last] = fma(b.F[last], u[D], b.U[last]);
    b.p += fma(b.F[last], u[D], b.F[1 + D]);
}

// Reverse of the primitive variables (cell_quantities): adjoints of velocity,
// pressure, sound speed, enthalpy and sqrt(rho) onto U.
template <int ND>
__device__ __forceinline__ void prim_bar(const double (&U)[ND + 2], const double (&u)[ND], double p,
                                         double c, double sr, double gamma, double gm1, CellBar<ND> &b)
{
    constexpr int last = ND + 1;
    const double rinv = 1.0 / U[0], cinv = 1.0 / c;
    double rb = b.s * 0.5 * (sr * rinv);                 // 1 / sqrt(rho) = sqrt(rho) / rho
    const double Epb = b.H * rinv;                       // H = (E + p) / rho
    double rinvb = b.H * (U[last] + p);
    double pb = b.p + Epb;
    const double zb = b.c * 0.5 * cinv;                  // c = sqrt(gamma p / rho)
    pb = fma(gamma * rinv, zb, pb);
    rinvb = fma(gamma * p, zb, rinvb);
    const double pg = gm1 * pb;                          // p = gm1 (E - m.u / 2)
    b.U[last] += Epb + pg;
    const double tb = -0.5 * pg;
#pragma unroll
    for (int a = 0; a < ND; a++) {
        const double ub = fma(tb, U[1 + a], b.u[a]);
        b.U[1 + a] += fma(tb, u[a], ub * rinv);          // u_a = m_a / rho
        rinvb = fma(ub, U[1 + a], rinvb);
    }
    rb = fma(-rinv * rinv, rinvb, rb);
    b.U[0] += rb;
}

template <int ND>
__global__ void __launch_bounds__(256) adj_prims_kernel(const double *U, int64_t ncell, Consts K, double *P)
{
    constexpr int nc = ND + 2;
    for (int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; id < ncell;
         id += (int64_t)gridDim.x * blockDim.x) {
        double Uc[nc];
#pragma unroll
        for (int c = 0; c < nc; c++) Uc[c] = U[c * ncell + id];
        CellQ<ND> q;
        cell_quantities<ND, 0>(Uc, K, q);
        store_prims<ND>(q, P, ncell, id);
    }
}

__device__ __forceinline__ double sign_of(double x) { return x > 0.0 ? 1.0 : (x < 0.0 ? -1.0 : 0.0); }

// The two cells beside a face and its splitting speeds, maximising cells
// included (first maximum, as the forward): v and c there.
template <int ND>
struct FaceSides {
    double ul[ND], ur[ND], Hl, Hr, sl, sr;
    double am, a0, ap, ar;
    double vm, cm, v0, vp, cp, vr;                       // u_D and c at the maximising cells
    int jm, j0, jp, jr;
};

// Reverse of one face.  cell(c, j): the halved (U_c, F_c) of stencil cell j.
// UNIFORM: every field's decision bytes have the low five bits of fl[0], fl[1];
// otherwise the parts per stencil position go to the slots.  coef: the frozen
// coefficients [32][W] by those bits (lanes with different decisions read it
// side by side, where constant memory would serve one after the other).
template <int ND, int H, int D, bool UNIFORM, class Cell>
__device__ __forceinline__ void reverse_face(const AdjArgs &a, int64_t flin, const FaceSides<ND> &f,
                                             const double (&Fb)[ND + 2], const uint8_t (&fl)[2 * (ND + 2)],
                                             const double *coef, Cell cell)
{
    using R = AdjRows<ND>;
    constexpr int nc = ND + 2, last = nc - 1, W = 2 * H;
    const double gm1 = a.K.gm1;
    const int64_t fs = a.d.nfaces;
    RoeScalars<ND> rs;
    roe_state<ND, D>(f.ul, f.Hl, f.sl, f.ur, f.Hr, f.sr, gm1, rs);
    const double un = rs.ut[D], ct = rs.ct, cinv = rs.cinv, b1 = rs.b1;

    // With P_j = (c+_j + c-_j)/2 and Q_j = (c+_j - c-_j)/2 the frozen reconstruction
    // gives h_k = alpha sum_j Q_j w_j + sum_j P_j g_j; with A_c = sum_j Q_j U_cj and
    // B_c = sum_j P_j F_cj (w = l.U, g = l.F): sum_j Q_j w_j = l.A, h_k = alpha l.A
    // + l.B, and the adjoint of the row l is hb_k (alpha A + B).
    double A[nc], B[nc];
    auto sums = [&](uint8_t flp, uint8_t flm) {
#pragma unroll
        for (int c = 0; c < nc; c++) A[c] = B[c] = 0.0;
        const double *tp = coef + (flp & 31) * W, *tm = coef + (flm & 31) * W;
#pragma unroll
        for (int j = 0; j < W; j++) {
            const double cp = tp[j], cm = tm[W - 1 - j];     // v+ index j, v- index W-1-j
            const double Pc = cp + cm, Qc = cp - cm;
#pragma unroll
            for (int c = 0; c < nc; c++) {
                const double2 u = cell(c, j);
                A[c] = fma(Qc, u.x, A[c]);
                B[c] = fma(Pc, u.y, B[c]);
            }
        }
    };
    if (UNIFORM) sums(fl[0], fl[1]);

    double b1b = 0.0, b2b = 0.0, uncb = 0.0, cinvb = 0.0, bub = 0.0, Htb = 0.0, q2b = 0.0;
    double ctb = 0.0, unb = 0.0, unctb = 0.0, utb[ND], M[nc], N[nc];
    double ab_m = 0.0, ab_0 = 0.0, ab_p = 0.0;
#pragma unroll
    for (int k = 0; k < ND; k++) utb[k] = 0.0;
#pragma unroll
    for (int c = 0; c < nc; c++) M[c] = N[c] = 0.0;
    double Lk[UNIFORM ? 1 : nc][nc], swk[UNIFORM ? 1 : nc], sgk[UNIFORM ? 1 : nc];
#pragma unroll
    for (int k = 0; k < nc; k++) {
        const bool shear = (k >= 2 && k < last);
        const int t = shear ? shear_axis<ND, D>(k) : 0;
        double l[nc];
        l_row<ND, D>(rs, k, l);
        // hb = sum_c R[c][k] Fb_c
        double hb;
        if (shear) {
            hb = 0.0;
#pragma unroll
            for (int x = 0; x < ND; x++)
                if (x == t) hb = fma(rs.ut[x], Fb[last], Fb[1 + x]);
        } else {
            hb = Fb[0];
#pragma unroll
            for (int c = 1; c < nc; c++) hb = fma(r_entry<ND, D>(rs, c, k), Fb[c], hb);
        }
        const double alpha = a.K.split ? f.ar : (k == 0 ? f.am : (k == last ? f.ap : f.a0));
        if (!UNIFORM) sums(fl[2 * k], fl[2 * k + 1]);
        double wq = l[0] * A[0], gp = l[0] * B[0];
#pragma unroll
        for (int c = 1; c < nc; c++) {
            if (shear && c != 1 + t) continue;           // zeros of a shear row
            wq = fma(l[c], A[c], wq);
            gp = fma(l[c], B[c], gp);
        }
        const double hk = fma(alpha, wq, gp), ab = hb * wq;
        double Lb[nc];
#pragma unroll
        for (int c = 0; c < nc; c++) Lb[c] = (shear && c != 0) ? 0.0 : fma(alpha, A[c], B[c]) * hb;
        if (k == 0) ab_m += ab;
        else if (k == last) ab_p += ab;
        else ab_0 += ab;
        // w_j and g_j enter h_k with weights alpha Q_j and P_j
        const double sg = half_of(hb), sw = alpha * sg;
        if (UNIFORM) {
#pragma unroll
            for (int c = 0; c < nc; c++) {
                if (shear && c != 0 && c != 1 + t) continue;
                M[c] = fma(l[c], sw, M[c]);
                N[c] = fma(l[c], sg, N[c]);
            }
        } else {
#pragma unroll
            for (int c = 0; c < nc; c++) Lk[k][c] = l[c];
            swk[k] = sw;
            sgk[k] = sg;
        }
        // R column k: Rb[c] = Fb_c h_k
        if (k == 0 || k == last) {
#pragma unroll
            for (int x = 0; x < ND; x++) {
                const double rb = Fb[1 + x] * hk;
                if (x == D) {
                    unb += rb;
                    ctb = k == 0 ? ctb - rb : ctb + rb;
                } else {
                    utb[x] += rb;
                }
            }
            const double rbE = Fb[last] * hk;
            Htb += rbE;
            unctb = k == 0 ? unctb - rbE : unctb + rbE;
        } else if (k == 1) {
#pragma unroll
            for (int x = 0; x < ND; x++) utb[x] = fma(Fb[1 + x], hk, utb[x]);
            q2b = fma(0.5 * Fb[last], hk, q2b);
        } else {
#pragma unroll
            for (int x = 0; x < ND; x++)
                if (x == t) utb[x] = fma(Fb[last], hk, utb[x]);
        }
        // L row k
        if (k == 0 || k == last) {
            const double h0 = half_of(Lb[0]);
            b2b += h0;
            uncb = k == 0 ? uncb + h0 : uncb - h0;
#pragma unroll
            for (int x = 0; x < ND; x++) {
                const double hx = half_of(Lb[1 + x]);
                if (x == D) {
                    bub -= hx;
                    cinvb = k == 0 ? cinvb - hx : cinvb + hx;
                } else {
                    b1b = fma(-rs.ut[x], hx, b1b);
                    utb[x] = fma(-b1, hx, utb[x]);
                }
            }
            b1b += half_of(Lb[last]);
        } else if (k == 1) {
            b2b -= Lb[0];
#pragma unroll
            for (int x = 0; x < ND; x++) {
                b1b = fma(rs.ut[x], Lb[1 + x], b1b);
                utb[x] = fma(b1, Lb[1 + x], utb[x]);
            }
            b1b -= Lb[last];
        } else {
#pragma unroll
            for (int x = 0; x < ND; x++)
                if (x == t) utb[x] -= Lb[0];
        }
    }

    // Chain through the Roe scalars to the two cells' velocity, enthalpy, sqrt(rho).
    unb = fma(unctb, ct, unb);
    ctb = fma(unctb, un, ctb);
    b1b = fma(bub, un, b1b);
    unb = fma(bub, b1, unb);
    unb = fma(uncb, cinv, unb);
    cinvb = fma(uncb, un, cinvb);
    q2b = fma(0.5 * b1, b2b, q2b);
    b1b = fma(0.5 * rs.q2, b2b, b1b);
    cinvb = fma(2.0 * gm1 * cinv, b1b, cinvb);
    ctb = fma(-cinv * cinv, cinvb, ctb);
    const double c2b = 0.5 * ctb * cinv;
    Htb = fma(gm1, c2b, Htb);
    q2b = fma(-0.5 * gm1, c2b, q2b);
#pragma unroll
    for (int x = 0; x < ND; x++) utb[x] = fma(2.0 * rs.ut[x], q2b, utb[x]);
    utb[D] += unb;
    // the averages are (s_l q_l + s_r q_r) inv, inv = 1 / (s_l + s_r)
    double slb, srb, ivb;
    double *row = a.rows + flin;
    {
        const double Nb = Htb * rs.inv;
        ivb = rs.Ht * Htb;                               // (s_l H_l + s_r H_r) Htb = Ht Htb / inv
        row[(R::LEFT + ND) * fs] = f.sl * Nb;
        row[(R::RIGHT + ND) * fs] = f.sr * Nb;
        slb = f.Hl * Nb;
        srb = f.Hr * Nb;
    }
#pragma unroll
    for (int x = 0; x < ND; x++) {
        const double Nb = utb[x] * rs.inv;
        ivb = fma(rs.ut[x], utb[x], ivb);
        row[(R::LEFT + x) * fs] = f.sl * Nb;
        row[(R::RIGHT + x) * fs] = f.sr * Nb;
        slb = fma(f.ul[x], Nb, slb);
        srb = fma(f.ur[x], Nb, srb);
    }
    const double Sb = -rs.inv * ivb;                     // -inv^2 (ivb / inv)
    row[(R::LEFT + ND + 1) * fs] = slb + Sb;
    row[(R::RIGHT + ND + 1) * fs] = srb + Sb;
#pragma unroll
    for (int c = 0; c < nc; c++) {                       // (zero for a mixed face)
        row[(R::M + c) * fs] = M[c];
        row[(R::N + c) * fs] = N[c];
    }
    if constexpr (!UNIFORM) {
#pragma unroll 1
        for (int j = 0; j < W; j++) {
            double Ub[nc], Fcb[nc];
#pragma unroll
            for (int c = 0; c < nc; c++) Ub[c] = Fcb[c] = 0.0;
#pragma unroll
            for (int k = 0; k < nc; k++) {
                const bool shear = (k >= 2 && k < last);
                const int t = shear ? shear_axis<ND, D>(k) : 0;
                const double cp = coef[(fl[2 * k] & 31) * W + j], cm = coef[(fl[2 * k + 1] & 31) * W + W - 1 - j];
                const double wb = swk[k] * (cp - cm), gb = sgk[k] * (cp + cm);
#pragma unroll
                for (int c = 0; c < nc; c++) {
                    if (shear && c != 0 && c != 1 + t) continue;
                    Ub[c] = fma(Lk[k][c], wb, Ub[c]);
                    Fcb[c] = fma(Lk[k][c], gb, Fcb[c]);
                }
            }
            double *out = a.slots + (size_t)j * 2 * nc * fs + flin;
#pragma unroll
            for (int c = 0; c < nc; c++) {
                out[c * fs] = Ub[c];
                out[(nc + c) * fs] = Fcb[c];
            }
        }
    }
    // Splitting-speed adjoints: |u - c| at jm, |u| at j0, |u + c| at jp; |u| + c at jr
    if (a.K.split) {
        const double s = (ab_m + ab_0) + ab_p;
        row[R::SPEED * fs] = sign_of(f.vr) * s;          // u_D
        row[(R::SPEED + 1) * fs] = s;                    // c
    } else {
        row[R::SPEED * fs] = sign_of(f.vm - f.cm) * ab_m;
        row[(R::SPEED + 1) * fs] = sign_of(f.v0) * ab_0;
        row[(R::SPEED + 2) * fs] = sign_of(f.vp + f.cp) * ab_p;
    }
    a.words[flin] = (uint16_t)(f.jm | (f.j0 << 4) | (f.jp << 8) | (f.jr << 12));
}

// Adjoint of a face's flux from the adjoint of L: face f is the right face of
// cell f-1 (-F/dx) and the left face of cell f (+F/dx).
template <int ND, int D>
__device__ __forceinline__ void flux_in(const AdjArgs &a, int64_t f, int64_t x, int64_t y, int64_t z,
                                        double (&Fb)[ND + 2])
{
    const int64_t n0 = a.g.n[0], n1 = a.g.n[1], nD = a.g.n[D];
    const int64_t st = D == 0 ? 1 : (D == 1 ? n0 : n0 * n1);
    const int64_t id = (D == 0 ? f : x) + n0 * ((D == 1 ? f : y) + n1 * (D == 2 ? f : z));
#pragma unroll
    for (int c = 0; c < ND + 2; c++) {
        const double r = f < nD ? a.lam[c * a.g.ncell + id] : 0.0;
        const double l = f > 0 ? a.lam[c * a.g.ncell + id - st] : 0.0;
        Fb[c] = (r - l) * a.inv_dx;
    }
}

// The block's table of frozen coefficients (reverse_face).
template <int H>
__device__ __forceinline__ void coef_table(double *coef)
{
    constexpr int W = 2 * H;
    for (int i = threadIdx.x; i < 32 * W; i += blockDim.x) {
        const int code = i / W, m = i - code * W;
        double v = 0.0;
#pragma unroll
        for (int k = 0; k < W; k++)
            if (k == m) v = frozen_coef<H>((uint8_t)code, k);
        coef[i] = v;
    }
    __syncthreads();
}

constexpr int kAdjWarps = 4;

template <int ND, int H, int D>
__global__ void __launch_bounds__(32 * kAdjWarps, 4) adj_face_kernel(const AdjArgs a)
{
    using SL = FaceSmem<ND, H>;
    constexpr int nc = ND + 2, W = 2 * H, NS = SL::NS;
    extern __shared__ double smem[];
    __shared__ double coef[32 * W];
    coef_table<H>(coef);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t tile = (int64_t)blockIdx.x * kAdjWarps + warp;
    if (tile >= a.tiles) return;
    double *sm = smem + (size_t)warp * SL::TOTAL;
    const double2 *UF = (const double2 *)sm;
#define TMP(q, j) sm[SL::TMP + (q) * NS + (j)]
    int64_t f0, x, y, z;
    tile_at<ND, D>(a.g.n, a.d, tile, f0, x, y, z);
    stage_cells<ND, H, D>(a.g, a.d, a.K, f0, x, y, z, sm, lane, 32);
    __syncwarp();
    const int tps = ND == 1 ? 0 : a.d.tps;
    int p, fo;
    tile_lane<D>(tps, lane, p, fo);
    const int64_t f = f0 + fo;
    const bool active = f <= a.g.n[D] && p < (D == 0 ? a.g.n[1] - y : a.g.n[0] - x);
    if (D == 0) y += p;
    else x += p;
    bool mixed = false;
    int64_t flin = 0;
    if (active) {
        const int b0 = D == 0 ? p * ((kTileFaces >> tps) + 2 * H - 1) + fo : lane, bs = D == 0 ? 1 : 1 << tps;
        flin = face_index<D>(a.g.n, f, x, y, z);
        uint8_t fl[2 * nc];
        const uint8_t *src = a.flags + flin * nc * 2;
#pragma unroll
        for (int q = 0; q < 2 * nc; q++) fl[q] = src[q];
#pragma unroll
        for (int k = 1; k < nc; k++)
            mixed = mixed || ((fl[2 * k] ^ fl[0]) & 31) || ((fl[2 * k + 1] ^ fl[1]) & 31);
        const bool large = (fl[0] & 31) == large_code(H) && (fl[1] & 31) == large_code(H);
        a.kind[flin] = (uint8_t)(mixed ? kAdjMixed : (large ? kAdjLarge : kAdjUniform));
        if (!mixed) {
            FaceSides<ND> s;
            const int bl = b0 + (H - 1) * bs, br = bl + bs;
#pragma unroll
            for (int k = 0; k < ND; k++) { s.ul[k] = TMP(SL::QV + k, bl); s.ur[k] = TMP(SL::QV + k, br); }
            s.Hl = TMP(SL::QH, bl);
            s.Hr = TMP(SL::QH, br);
            s.sl = TMP(SL::QSR, bl);
            s.sr = TMP(SL::QSR, br);
            s.am = s.a0 = s.ap = s.ar = 0.0;
            s.jm = s.j0 = s.jp = s.jr = 0;
#pragma unroll
            for (int j = 0; j < W; j++) {
                const int i = b0 + j * bs;
                const double em = TMP(SL::QLM, i), e0 = TMP(SL::QL0, i), ep = TMP(SL::QLP, i), er = TMP(SL::QLR, i);
                if (j == 0 || speed_gt(em, s.am)) { s.am = em; s.jm = j; }
                if (j == 0 || speed_gt(e0, s.a0)) { s.a0 = e0; s.j0 = j; }
                if (j == 0 || speed_gt(ep, s.ap)) { s.ap = ep; s.jp = j; }
                if (j == 0 || speed_gt(er, s.ar)) { s.ar = er; s.jr = j; }
            }
            // c = (|u| + c) - |u|, for the sign of u -+ c only; where that lies within
            // the rounding of |u| + c, the stored c
            auto sound = [&](int j, double v, double lr, double lambda) {
                if (lambda > 1.0e-15 * lr) return lr - fabs(v);
                int rule;
                const int64_t g = map_index(f - H + j, a.g.n[D], H, a.d.bc_lo, a.d.bc_hi, rule);
                const int64_t id = (D == 0 ? g : x) + a.g.n[0] * ((D == 1 ? g : y) + a.g.n[1] * (D == 2 ? g : z));
                return a.g.P[PrimRows<ND>::C * a.g.ncell + id];
            };
            const int im = b0 + s.jm * bs, ip = b0 + s.jp * bs;
            s.vm = TMP(SL::QV + D, im);
            s.cm = sound(s.jm, s.vm, TMP(SL::QLR, im), s.am);
            s.vp = TMP(SL::QV + D, ip);
            s.cp = sound(s.jp, s.vp, TMP(SL::QLR, ip), s.ap);
            s.v0 = TMP(SL::QV + D, b0 + s.j0 * bs);
            s.vr = TMP(SL::QV + D, b0 + s.jr * bs);
            double Fb[nc];
            flux_in<ND, D>(a, f, x, y, z, Fb);
            reverse_face<ND, H, D, true>(a, flin, s, Fb, fl, coef,
                                         [&](int c, int j) { return UF[c * NS + b0 + j * bs]; });
        }
    }
    const unsigned m = __ballot_sync(0xffffffffu, mixed);
    if (m) {
        unsigned at = 0;
        if (lane == 0) at = atomicAdd(a.count, (unsigned)__popc(m));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
        if (mixed) a.list[at] = (uint32_t)flin;
    }
#undef TMP
}

// The listed faces, a lane each; the stencil's halved (U, F) pairs in shared
// memory, [c][j][thread].
constexpr int kMixedThreads = 64;

template <int ND, int H, int D>
__global__ void __launch_bounds__(kMixedThreads) adj_mixed_kernel(const AdjArgs a)
{
    constexpr int nc = ND + 2, last = nc - 1, W = 2 * H;
    extern __shared__ double smem[];
    __shared__ double coef[32 * W];
    if (*a.count <= blockIdx.x * kMixedThreads) return;
    coef_table<H>(coef);
    double2 *UF = (double2 *)smem + threadIdx.x;
    const int64_t n0 = a.g.n[0], n1 = a.g.n[1], nD = a.g.n[D];
    const unsigned n = *a.count;
    for (unsigned i = blockIdx.x * kMixedThreads + threadIdx.x; i < n; i += gridDim.x * kMixedThreads) {
        const int64_t flin = a.list[i];
        int64_t x, y, z, f;
        if (D == 0) { f = flin % (n0 + 1); const int64_t r = flin / (n0 + 1); x = 0; y = r % n1; z = r / n1; }
        else if (D == 1) { x = flin % n0; const int64_t r = flin / n0; f = r % (n1 + 1); y = 0; z = r / (n1 + 1); }
        else { x = flin % n0; const int64_t r = flin / n0; y = r % n1; f = r / n1; z = 0; }
        FaceSides<ND> s;
        s.am = s.a0 = s.ap = s.ar = 0.0;
        s.jm = s.j0 = s.jp = s.jr = 0;
#pragma unroll 1
        for (int j = 0; j < W; j++) {
            int rule;
            const int64_t gi = map_index(f - H + j, nD, H, a.d.bc_lo, a.d.bc_hi, rule);
            const int64_t id = (D == 0 ? gi : x) + n0 * ((D == 1 ? gi : y) + n1 * (D == 2 ? gi : z));
            double Uc[nc];
            CellQ<ND> q;
#pragma unroll
            for (int c = 0; c < nc; c++) Uc[c] = a.g.U[c * a.g.ncell + id];
            load_prims<ND>(a.g.P, a.g.ncell, id, q);
            apply_ghost_rule<ND, D>(Uc, rule, nullptr, nullptr, 0, 0, a.K.gm1);
#pragma unroll
            for (int k = 0; k < ND; k++)
                if (rule == 2 || (rule == 1 && k == D)) q.u[k] = -q.u[k];
            const double hm = half_of(Uc[1 + D]), hp = half_of(q.p);
            UF[(0 * W + j) * kMixedThreads] = make_double2(half_of(Uc[0]), hm);
#pragma unroll
            for (int k = 0; k < ND; k++)
                UF[((1 + k) * W + j) * kMixedThreads] =
                    make_double2(half_of(Uc[1 + k]), k == D ? hm * q.u[k] + hp : hm * q.u[k]);
            const double hE = half_of(Uc[last]);
            UF[(last * W + j) * kMixedThreads] = make_double2(hE, q.u[D] * (hE + hp));
            const double v = q.u[D], c = q.c;
            const double em = fabs(v - c), e0 = fabs(v), ep = fabs(v + c), er = fabs(v) + c;
            if (j == 0 || speed_gt(em, s.am)) { s.am = em; s.jm = j; s.vm = v; s.cm = c; }
            if (j == 0 || speed_gt(e0, s.a0)) { s.a0 = e0; s.j0 = j; s.v0 = v; }
            if (j == 0 || speed_gt(ep, s.ap)) { s.ap = ep; s.jp = j; s.vp = v; s.cp = c; }
            if (j == 0 || speed_gt(er, s.ar)) { s.ar = er; s.jr = j; s.vr = v; }
            if (j == H - 1) {
#pragma unroll
                for (int k = 0; k < ND; k++) s.ul[k] = q.u[k];
                s.Hl = q.H;
                s.sl = q.sr;
            } else if (j == H) {
#pragma unroll
                for (int k = 0; k < ND; k++) s.ur[k] = q.u[k];
                s.Hr = q.H;
                s.sr = q.sr;
            }
        }
        uint8_t fl[2 * nc];
#pragma unroll
        for (int q = 0; q < 2 * nc; q++) fl[q] = a.flags[flin * nc * 2 + q];
        double Fb[nc];
        flux_in<ND, D>(a, f, x, y, z, Fb);
        reverse_face<ND, H, D, false>(a, flin, s, Fb, fl, coef,
                                      [&](int c, int j) { return UF[(c * W + j) * kMixedThreads]; });
    }
}

// One face's part in stencil position j of a cell (or of one of its ghost images);
// kind and w: the face's, loaded ahead (the products need no branch: M and N of a
// mixed face are zero).  coef: the largest stencil's c+ - c-, then c+ + c-.
template <int ND, int H, int D>
__device__ __forceinline__ void gather_face(const AdjArgs &a, int64_t flin, int j, int kind, unsigned w,
                                            const double *coef, CellBar<ND> &b)
{
    using R = AdjRows<ND>;
    constexpr int nc = ND + 2, W = 2 * H;
    const int64_t fs = a.d.nfaces;
    const double *row = a.rows + flin;
    double M[nc], N[nc];
#pragma unroll
    for (int c = 0; c < nc; c++) {
        M[c] = row[(R::M + c) * fs];
        N[c] = row[(R::N + c) * fs];
    }
    double qd = coef[j], qs = coef[W + j];
    if (kind == kAdjUniform) {
        const double cp = frozen_coef<H>(a.flags[flin * nc * 2], j);
        const double cm = frozen_coef<H>(a.flags[flin * nc * 2 + 1], W - 1 - j);
        qd = cp - cm;
        qs = cp + cm;
    }
#pragma unroll
    for (int c = 0; c < nc; c++) {
        b.U[c] = fma(qd, M[c], b.U[c]);
        b.F[c] = fma(qs, N[c], b.F[c]);
    }
    if (kind == kAdjMixed) {
        const double *sl = a.slots + (size_t)j * 2 * nc * fs + flin;
#pragma unroll
        for (int c = 0; c < nc; c++) {
            b.U[c] += sl[c * fs];
            b.F[c] += sl[(nc + c) * fs];
        }
    }
    if (j == H - 1 || j == H) {
        const int r = j == H ? R::RIGHT : R::LEFT;
#pragma unroll
        for (int k = 0; k < ND; k++) b.u[k] += row[(r + k) * fs];
        b.H += row[(r + ND) * fs];
        b.s += row[(r + ND + 1) * fs];
    }
    if (a.K.split) {
        if ((int)(w >> 12) == j) {
            b.u[D] += row[R::SPEED * fs];
            b.c += row[(R::SPEED + 1) * fs];
        }
    } else {
        if ((int)(w & 15) == j) {
            const double e = row[R::SPEED * fs];
            b.u[D] += e;
            b.c -= e;
        }
        if ((int)((w >> 4) & 15) == j) b.u[D] += row[(R::SPEED + 1) * fs];
        if ((int)((w >> 8) & 15) == j) {
            const double e = row[(R::SPEED + 2) * fs];
            b.u[D] += e;
            b.c += e;
        }
    }
}

// The parts of the faces whose stencils cover position g along D (a cell or one of
// its ghost images) at the transverse position (x, y, z): face f holds position g
// at stencil index j = g - f + H.  A position whose 2H faces all exist takes an
// unrolled loop, so that its loads are independent.
template <int ND, int H, int D>
__device__ __forceinline__ void gather_position(const AdjArgs &a, int64_t g, int64_t x, int64_t y, int64_t z,
                                                const double *coef, CellBar<ND> &b)
{
    constexpr int W = 2 * H;
    const int64_t nD = a.g.n[D];
    const int64_t fb = face_index<D>(a.g.n, 0, x, y, z);
    const int64_t fs = D == 0 ? 1 : (D == 1 ? a.g.n[0] : a.g.n[0] * a.g.n[1]);
    if (g - H + 1 >= 0 && g + H <= nD) {
        const int64_t f0 = fb + (g - H + 1) * fs;
        int kind[W];
        unsigned w[W];
#pragma unroll
        for (int t = 0; t < W; t++) {
            kind[t] = a.kind[f0 + t * fs];
            w[t] = a.words[f0 + t * fs];
        }
#pragma unroll
        for (int t = 0; t < W; t++)
            gather_face<ND, H, D>(a, f0 + t * fs, W - 1 - t, kind[t], w[t], coef, b);
    } else {
        const int64_t flo = g - H + 1 > 0 ? g - H + 1 : 0;
        const int64_t fhi = g + H < nD ? g + H : nD;
#pragma unroll 1
        for (int64_t f = flo; f <= fhi; f++)
            gather_face<ND, H, D>(a, fb + f * fs, (int)(g - f + H), a.kind[fb + f * fs],
                                  a.words[fb + f * fs], coef, b);
    }
}

// Sums of direction D added to the cells' rows; the last direction takes them to mu.
template <int ND, int H, int D>
__global__ void __launch_bounds__(128, ND == 3 ? 3 : 4) adj_gather_kernel(const AdjArgs a, double *mu)
{
    using S = AdjSums<ND>;
    constexpr int nc = ND + 2, W = 2 * H;
    __shared__ double coef[2 * W];
    if (threadIdx.x < W) {
        double cp = 0.0, cm = 0.0;
#pragma unroll
        for (int j = 0; j < W; j++)
            if (j == (int)threadIdx.x) { cp = lcoef<H>(j); cm = lcoef<H>(W - 1 - j); }
        coef[threadIdx.x] = cp - cm;
        coef[W + threadIdx.x] = cp + cm;
    }
    __syncthreads();
    const int64_t n0 = a.g.n[0], n1 = a.g.n[1], nD = a.g.n[D], nn = a.g.ncell;
    const double gamma = a.K.gamma, gm1 = a.K.gm1;
    for (int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; id < nn;
         id += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = id / n0, x = id - r * n0, z = ND < 3 ? 0 : r / n1, y = ND < 2 ? 0 : r - z * n1;
        const int64_t i = (D == 0) ? x : (D == 1 ? y : z);
        double Uc[nc];
#pragma unroll
        for (int c = 0; c < nc; c++) Uc[c] = a.g.U[c * nn + id];
        CellQ<ND> q;
        load_prims<ND>(a.g.P, nn, id, q);
        CellBar<ND> b;
        b.clear();
        gather_position<ND, H, D>(a, i, x, y, z, coef, b);
        double extra[nc];                                // of mirror images, already on U
#pragma unroll
        for (int c = 0; c < nc; c++) extra[c] = 0.0;
        if (i < H || i >= nD - H) {
            // ghost images that map to cell i, with the mirror rule of each (0 none,
            // 1 slip wall, 2 no-slip)
            int64_t gs[2 * 6 + 2];
            int ms[2 * 6 + 2];
            int ng = 0;
            if (a.d.bc_lo == 0) { gs[ng] = i - nD; ms[ng] = 0; ng++; }
            if (a.d.bc_hi == 0) { gs[ng] = i + nD; ms[ng] = 0; ng++; }
            if (a.d.bc_lo == 1 && i == 0)
                for (int k = 1; k <= H; k++) { gs[ng] = -k; ms[ng] = 0; ng++; }
            if (a.d.bc_hi == 1 && i == nD - 1)
                for (int k = 0; k < H; k++) { gs[ng] = nD + k; ms[ng] = 0; ng++; }
            if ((a.d.bc_lo == 2 || a.d.bc_lo == 3) && i < H) { gs[ng] = -i - 1; ms[ng] = a.d.bc_lo - 1; ng++; }
            if ((a.d.bc_hi == 2 || a.d.bc_hi == 3) && i >= nD - H) {
                gs[ng] = 2 * nD - 1 - i; ms[ng] = a.d.bc_hi - 1; ng++;
            }
            for (int k = 0; k < ng; k++) {
                const int64_t g = gs[k];
                if (g < -H || g > nD + H - 1) continue;
                if (!ms[k]) {
                    gather_position<ND, H, D>(a, g, x, y, z, coef, b);
                } else {
                    // the image is the mirror map M U (M diagonal, +-1): its reverse is
                    // taken at M U and M^T = M maps the adjoint back
                    CellBar<ND> e;
                    e.clear();
                    gather_position<ND, H, D>(a, g, x, y, z, coef, e);
                    double Ug[nc], ug[ND];
#pragma unroll
                    for (int c = 0; c < nc; c++) Ug[c] = Uc[c];
#pragma unroll
                    for (int c = 0; c < ND; c++) ug[c] = ms[k] == 2 || c == D ? -q.u[c] : q.u[c];
                    apply_ghost_rule<ND, D>(Ug, ms[k], nullptr, nullptr, 0, 0, gm1);
                    flux_bar<ND, D>(Ug, ug, q.p, e);
                    prim_bar<ND>(Ug, ug, q.p, q.c, q.sr, gamma, gm1, e);
                    apply_ghost_rule<ND, D>(e.U, ms[k], nullptr, nullptr, 0, 0, gm1);
#pragma unroll
                    for (int c = 0; c < nc; c++) extra[c] += e.U[c];
                }
            }
        }
        flux_bar<ND, D>(Uc, q.u, q.p, b);
#pragma unroll
        for (int c = 0; c < nc; c++) b.U[c] += extra[c];
        double *sum = a.sums + id;
        if (D > 0) {
#pragma unroll
            for (int c = 0; c < nc; c++) b.U[c] += sum[(S::U + c) * nn];
#pragma unroll
            for (int c = 0; c < ND; c++) b.u[c] += sum[(S::V + c) * nn];
            b.p += sum[S::P * nn];
            b.c += sum[S::C * nn];
            b.H += sum[S::H * nn];
            b.s += sum[S::S * nn];
        }
        if (D < ND - 1) {
#pragma unroll
            for (int c = 0; c < nc; c++) sum[(S::U + c) * nn] = b.U[c];
#pragma unroll
            for (int c = 0; c < ND; c++) sum[(S::V + c) * nn] = b.u[c];
            sum[S::P * nn] = b.p;
            sum[S::C * nn] = b.c;
            sum[S::H * nn] = b.H;
            sum[S::S * nn] = b.s;
        } else {
            prim_bar<ND>(Uc, q.u, q.p, q.c, q.sr, gamma, gm1, b);
#pragma unroll
            for (int c = 0; c < nc; c++) mu[c * nn + id] = b.U[c];
        }
    }
}

// Elementwise combinations of the SSP-RK3 reverse sweep.
__global__ void axpby_kernel(int64_t len, double a, const double *x, double b, const double *y,
                             double *out)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = a * x[i] + (y ? b * y[i] : 0.0);
}

template <int ND, int H, int D>
cudaError_t launch_adj_direction(AdjArgs &a, double *mu, cudaStream_t s)
{
    constexpr size_t smem = sizeof(double) * (size_t)FaceSmem<ND, H>::TOTAL * kAdjWarps;
    constexpr size_t mixed = sizeof(double2) * (size_t)(ND + 2) * 2 * H * kMixedThreads;
    constexpr size_t table = sizeof(double) * 32 * 2 * H;                // coef_table
    cudaError_t e;
    if ((e = allow_shared(adj_face_kernel<ND, H, D>, smem, table)) != cudaSuccess ||
        (e = allow_shared(adj_mixed_kernel<ND, H, D>, mixed, table)) != cudaSuccess)
        return e;
    const int64_t fast = D == 0 ? a.g.n[1] : a.g.n[0];
    tile_shape(a.d, a.g.n[D] + 1, fast, H);
    a.tiles = a.d.line_tiles * a.d.groups * (a.g.ncell / a.g.n[D] / fast);
    if ((e = cudaMemsetAsync(a.count, 0, sizeof(unsigned), s)) != cudaSuccess) return e;
    adj_face_kernel<ND, H, D><<<(unsigned)((a.tiles + kAdjWarps - 1) / kAdjWarps), 32 * kAdjWarps, smem, s>>>(a);
    int64_t blocks = (a.d.nfaces + kMixedThreads - 1) / kMixedThreads;
    if (blocks > 152 * 16) blocks = 152 * 16;
    adj_mixed_kernel<ND, H, D><<<(unsigned)blocks, kMixedThreads, mixed, s>>>(a);
    blocks = (a.g.ncell + 127) / 128;
    if (blocks > 152 * 64) blocks = 152 * 64;
    adj_gather_kernel<ND, H, D><<<(unsigned)blocks, 128, 0, s>>>(a, mu);
    return cudaGetLastError();
}

template <int H>
cudaError_t launch_adj(int nd, int d, AdjArgs &a, double *mu, cudaStream_t s)
{
    switch (nd * 3 + d) {
    case 3: return launch_adj_direction<1, H, 0>(a, mu, s);
    case 6: return launch_adj_direction<2, H, 0>(a, mu, s);
    case 7: return launch_adj_direction<2, H, 1>(a, mu, s);
    case 9: return launch_adj_direction<3, H, 0>(a, mu, s);
    case 10: return launch_adj_direction<3, H, 1>(a, mu, s);
    case 11: return launch_adj_direction<3, H, 2>(a, mu, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace teno

using namespace teno;

namespace {

int64_t cells_of(const teno_params *p) { return p->n[0] * p->n[1] * p->n[2]; }

int64_t faces_of(const teno_params *p, int d)
{
    int64_t s = 1;
    for (int a = 0; a < 3; a++) s *= (a == d) ? p->n[a] + 1 : p->n[a];
    return s;
}

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

struct AdjLayout {
    size_t fwd, flags, slots, rows, words, kind, list, count, prims, sums, t0, t1, t2, total;
};

AdjLayout adj_layout(const teno_params *p)
{
    AdjLayout L;
    size_t fwd = 0;
    teno_workspace_bytes(p, &fwd);
    size_t fb = 0;
    teno_flags_bytes(p, &fb);
    const int nc = p->ndim + 2, W = p->scheme;
    int64_t maxf = 0;
    for (int d = 0; d < p->ndim; d++) maxf = faces_of(p, d) > maxf ? faces_of(p, d) : maxf;
    const size_t state = sizeof(double) * (size_t)nc * cells_of(p);
    size_t off = 0;
    L.fwd = off;
    off += a256(fwd);
    L.flags = off;
    off += a256(fb);
    L.slots = off;
    off += a256(sizeof(double) * (size_t)maxf * W * 2 * nc);
    const int nd = p->ndim;
    L.rows = off;
    off += a256(sizeof(double) * (size_t)maxf * (2 * nc + 2 * (nd + 2) + 3));   // AdjRows
    L.words = off;
    off += a256(sizeof(uint16_t) * (size_t)maxf);
    L.kind = off;
    off += a256((size_t)maxf);
    L.list = off;
    off += a256(sizeof(uint32_t) * (size_t)maxf);
    L.count = off;
    off += 256;
    L.prims = off;
    off += a256(sizeof(double) * (size_t)(nd + 4) * cells_of(p));
    L.sums = off;
    off += a256(sizeof(double) * (size_t)(nc + nd + 4) * cells_of(p));          // AdjSums
    L.t0 = off;
    off += a256(state);
    L.t1 = off;
    off += a256(state);
    L.t2 = off;
    off += a256(state);
    L.total = off;
    return L;
}

Consts consts_adj(const teno_params *p)
{
    Consts K;
    K.gamma = p->gamma;
    K.gm1 = p->gamma - 1.0;
    K.alpha1 = p->ct_alpha1;
    K.alpha2 = p->ct_alpha2;
    K.cr = p->ct_cr;
    K.eps_beta = p->eps_beta;
    K.eps_eta = p->eps_eta;
    K.lim_eps = p->limiter_eps;
    K.split = p->flux_split;
    K.limiter = 0;
    return K;
}

#define CUDA_TRY(x)                                   \
    do {                                              \
        if ((x) != cudaSuccess) return TENO_ECUDA;    \
    } while (0)

int check_adj(const teno_params *p, void *ws, size_t ws_bytes)
{
    size_t b;
    int r = teno_workspace_bytes(p, &b);
    if (r) return r;
    if (p->limiter) return TENO_EINVAL;
    for (int d = 0; d < p->ndim; d++)
        if (p->bc_lo[d] >= TENO_BC_DIRICHLET || p->bc_hi[d] >= TENO_BC_DIRICHLET) return TENO_EINVAL;
    if (!ws || ((uintptr_t)ws & 255) || ws_bytes < adj_layout(p).total) return TENO_EINVAL;
    return TENO_OK;
}

void launch_axpby(int64_t len, double a, const double *x, double b, const double *y, double *out,
                  cudaStream_t s)
{
    int64_t blocks = (len + 255) / 256;
    if (blocks > 152 * 64) blocks = 152 * 64;
    axpby_kernel<<<(unsigned)blocks, 256, 0, s>>>(len, a, x, b, y, out);
}

int rhs_vjp_impl(const teno_params *p, const double *U, const double *lam, const uint8_t *flags,
                 double *mu, char *ws, cudaStream_t s)
{
    const AdjLayout L = adj_layout(p);
    const int nc = p->ndim + 2;
    if (!flags) {
        uint8_t *fl = (uint8_t *)(ws + L.flags);
        double *scratch = (double *)(ws + L.t2);
        size_t fb;
        teno_workspace_bytes(p, &fb);
        int r = teno_rhs(p, U, scratch, 0.0, fl, ws + L.fwd, fb, s);
        if (r) return r;
        flags = fl;
    }
    double *P = (double *)(ws + L.prims);
    {
        const int64_t n = cells_of(p);
        int64_t blocks = (n + 255) / 256;
        if (blocks > 152 * 64) blocks = 152 * 64;
        const Consts K = consts_adj(p);
        if (p->ndim == 1) adj_prims_kernel<1><<<(unsigned)blocks, 256, 0, s>>>(U, n, K, P);
        else if (p->ndim == 2) adj_prims_kernel<2><<<(unsigned)blocks, 256, 0, s>>>(U, n, K, P);
        else adj_prims_kernel<3><<<(unsigned)blocks, 256, 0, s>>>(U, n, K, P);
        CUDA_TRY(cudaGetLastError());
    }
    const uint8_t *fl = flags;
    for (int d = 0; d < p->ndim; d++) {
        AdjArgs a;
        memset(&a, 0, sizeof(a));
        a.g.U = U;
        a.g.P = P;
        a.g.st = (Status *)(ws + L.fwd);       // the checked build's range checks
        for (int k = 0; k < 3; k++) a.g.n[k] = p->n[k];
        a.g.ncell = cells_of(p);
        a.d.nfaces = faces_of(p, d);
        a.d.bc_lo = p->bc_lo[d];
        a.d.bc_hi = p->bc_hi[d];
        a.lam = lam;
        a.flags = fl;
        a.slots = (double *)(ws + L.slots);
        a.rows = (double *)(ws + L.rows);
        a.words = (uint16_t *)(ws + L.words);
        a.kind = (uint8_t *)(ws + L.kind);
        a.list = (uint32_t *)(ws + L.list);
        a.count = (unsigned *)(ws + L.count);
        a.sums = (double *)(ws + L.sums);
        a.inv_dx = 1.0 / p->dx[d];
        a.K = consts_adj(p);
        cudaError_t e = (p->scheme == 8)    ? launch_adj<4>(p->ndim, d, a, mu, s)
                        : (p->scheme == 10) ? launch_adj<5>(p->ndim, d, a, mu, s)
                                            : launch_adj<6>(p->ndim, d, a, mu, s);
        if (e != cudaSuccess) return TENO_ECUDA;
        fl += (size_t)faces_of(p, d) * nc * 2;
    }
    return TENO_OK;
}

}  // namespace

extern "C" {

int teno_adjoint_workspace_bytes(const teno_params *p, size_t *bytes)
{
    size_t b;
    int r = teno_workspace_bytes(p, &b);
    if (r) return r;
    if (!bytes) return TENO_EINVAL;
    *bytes = adj_layout(p).total;
    return TENO_OK;
}

int teno_rhs_vjp(const teno_params *p, const double *U, const double *lam, const uint8_t *flags,
                 double *mu, void *ws, size_t ws_bytes, void *stream)
{
    int r = check_adj(p, ws, ws_bytes);
    if (r) return r;
    if (!U || !lam || !mu || ((uintptr_t)U & 15) || ((uintptr_t)lam & 15) || ((uintptr_t)mu & 15))
        return TENO_EINVAL;
    if (mu == U || mu == lam) return TENO_EINVAL;
    return rhs_vjp_impl(p, U, lam, flags, mu, (char *)ws, (cudaStream_t)stream);
}

int teno_rk3_step_vjp(const teno_params *p, const double *Un, const double *U1, const double *U2,
                      const uint8_t *flags, double dt, double *abar, void *ws, size_t ws_bytes,
                      void *stream)
{
    int r = check_adj(p, ws, ws_bytes);
    if (r) return r;
    if (!Un || !U1 || !U2 || !abar || !flags || !(dt >= 0.0)) return TENO_EINVAL;
    const AdjLayout L = adj_layout(p);
    size_t flb;
    teno_flags_bytes(p, &flb);
    cudaStream_t s = (cudaStream_t)stream;
    char *w = (char *)ws;
    const int64_t len = (int64_t)(p->ndim + 2) * cells_of(p);
    double *t = (double *)(w + L.t0), *mu = (double *)(w + L.t1), *acc = (double *)(w + L.t2);
    // stage 3: U+ = 1/3 Un + 2/3 (U2 + dt L(U2))
    launch_axpby(len, 2.0 / 3.0, abar, 0.0, nullptr, t, s);            // t = 2/3 abar
    if ((r = rhs_vjp_impl(p, U2, t, flags + 2 * flb, mu, w, s))) return r;
    launch_axpby(len, 1.0, t, dt, mu, t, s);                             // Ubar2 = t + dt mu
    launch_axpby(len, 1.0 / 3.0, abar, 0.0, nullptr, acc, s);          // Ubar_n = 1/3 abar
    // stage 2: U2 = 3/4 Un + 1/4 (U1 + dt L(U1))
    launch_axpby(len, 0.75, t, 1.0, acc, acc, s);                        // Ubar_n += 3/4 Ubar2
    launch_axpby(len, 0.25, t, 0.0, nullptr, t, s);                      // t = 1/4 Ubar2
    if ((r = rhs_vjp_impl(p, U1, t, flags + flb, mu, w, s))) return r;
    launch_axpby(len, 1.0, t, dt, mu, t, s);                             // Ubar1 = t + dt mu
    // stage 1: U1 = Un + dt L(Un)
    if ((r = rhs_vjp_impl(p, Un, t, flags, mu, w, s))) return r;
    launch_axpby(len, 1.0, t, 1.0, acc, acc, s);                         // Ubar_n += Ubar1
    launch_axpby(len, dt, mu, 1.0, acc, abar, s);                        // abar = Ubar_n + dt mu
    CUDA_TRY(cudaGetLastError());
    return TENO_OK;
}

}  // extern "C"
