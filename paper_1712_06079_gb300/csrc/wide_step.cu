// Two-pass D2Q9 step in FP64 arithmetic for sm_103a: FP64 lattices, and FP32
// lattices that the single-pass kernel does not take (FP32 distributions, every
// operation FP64).
//
// What bounds it.  GB300 issues FP64 at 1/64 of the FP32 rate (2 operations
// per cycle and SM), so the step costs its FP64 instruction count, and small
// lattices (128^2, 1024 x 8) the number of SMs that share it.  The direct form
// of the radius-40 operator of Eq. 20 takes 320 FP64 operations per cell, three
// quarters of the step; here it takes 18:
//   The operator's kernel is geometric, c_j = -(25/12) r^j (j >= 1) plus 1/12
//   at j = 1, r = (sqrt 5 - 3)/2, so with the one-sided sums along a line
//     S_i = t_i + r S_(i-1),   T_i = t_i + r T_(i+1)
//   the derivative is D_i = (t_(i+1) - t_(i-1))/12 - (25/12) r (T_(i+1) - S_(i-1)).
//   Pass 1 (wide_potential_kernel), which holds the field of its tile on chip,
//   also writes the sums over blocks of 8 cells of each line, both directions:
//     BS = sum_i r^(last - i) t_i,  BT = sum_i r^(i - first) t_i.
//   Pass 2 (wide_collide_kernel) joins the blocks around its own into the two
//   values that enter it (5 multiply-adds for the 40 cells past which r^j is
//   below FP64 rounding, 1.9e-17) and steps S and T through the block, one
//   multiply-add per cell each.
// On a line of equal values T and S are equal up to rounding only, where the direct
// form's differences vanish.  So that such a line has no derivative bit for bit (a
// uniform lattice at rest stays at rest, a slab uniform along y stays so), pass 1 also
// writes each block's value where its cells are equal, and pass 2 drops T - S where the
// blocks around a cell all have that value: comparisons of bits, beside the FP64 work.
// No halo of 40 cells is staged and no line is walked from its start.  Lines
// whose length is no multiple of 8 end in a shorter block; with walls in y
// (Sec. 5.5) the blocks continue in mirrored order, a mirrored block's BS being
// the block's own BT.
//
// Tiles of 16 x 8 cells, 128 threads, one cell per thread: four warps reach all
// four FP64 units of an SM, and 128^2 or 1024 x 8 cells still spread over 128
// or 64 SMs.  For tau = 1 the BGK term vanishes and the equilibrium at u is
// skipped.
//
// Both passes are launched with programmatic serialization, so the next grid's
// CTAs are placed while this grid runs, on the SMs that still have room: let in
// at the top, a grid of 128 CTAs piled up on about 30 SMs (36.8 us per 128^2
// step).  Grids of up to four CTAs per SM therefore ask for shared memory that
// lets no more than their even share onto an SM, and let the next grid in at the
// top: 9.7 us, against 13.2 when it is let in after the arithmetic without that
// bound (which larger grids do, and grids of at most half the SMs, which fit
// beside each other), and 14.4 without programmatic launches.
//
// Measured, us per step (direct stencil before -> block sums): FP64 128^2 100 ->
// 9.1, FP32 1024 x 8 35 -> 9.4, FP64 1024^2 -> 244, where one at a time pass 1 takes 91
// and pass 2 159 with the FP64 units 80 and 83 % busy, which is the bound there;
// small lattices are left with the latency of two dependent grids.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "lbm_internal.h"
#include "ptx.cuh"

namespace lbm {
namespace {

constexpr int BK = 8;             // cells per block of a line
constexpr int TX = 16, TY = BK;   // tile of a CTA: two blocks along x, one along y
constexpr int NT = TX * TY;
constexpr int kReach = 40;        // cells joined on each side: r^40 is below FP64 rounding (1.9e-17)
constexpr int kJoin = 7;          // blocks joined with all loads in flight (more, in a loop, on short lines only)

// The HDM operator's constants (Eq. 20), and where the block sums live.
struct WideArgs {
    Model<double> m;
    double r, r8;            // r and r^8
    double c1, cs;           // 1/12 and -(25/12) r
    double rxl, ryl;         // r^(cells of the last block) along x, y
    int nbx, nby;            // blocks per row, per column
    int kbx, kby;            // blocks that cover kReach cells, wherever they start
    int ntx;                 // tiles per row of tiles
    // block sums BS, BT and the value of blocks of equal cells (else a NaN): y.[by * nx + x], x.[y * nbx + bx]
    double *ys, *yt, *ye, *xs, *xt, *xe;
    int early;                   // the next grid is let in at the top (see spread)
    long long nys, nxs;      // entries of each
};

// Steps through the blocks of a line of nb, from block b on in direction dir: periodic,
// or (mirror) the line continued by its mirror image, where a block's sums swap roles.
struct BlockWalk {
    int i, dir, nb;
    bool mirror, swapped = false;
    __device__ __forceinline__ void next() {
        const int k = i + dir;
        if (k >= 0 && k < nb) i = k;
        else if (!mirror) i = k < 0 ? nb - 1 : 0;
        else {
            dir = -dir;
            swapped = !swapped;
        }
    }
};

// The value of the n cells at s if they are equal and finite, else a NaN (by the bits: a
// comparison takes an FP64 slot).
__device__ __forceinline__ double value_of_equal(const double *s, int step, int n) {
    const long long v = __double_as_longlong(s[0]);
    bool same = (v & 0x7ff0000000000000LL) != 0x7ff0000000000000LL;
#pragma unroll
    for (int k = 1; k < BK; ++k) same &= k >= n || __double_as_longlong(s[k * step]) == v;
    return __longlong_as_double(same ? v : 0x7ff8000000000000LL);
}

// Block sums of a tile's fields: of `col` along its columns (warp 0), of `row`
// along its rows (warp 1), lanes 0 .. 15 BS, 16 .. 31 BT; the values of blocks of equal
// cells by warp 2 (lanes 0 .. 15 columns, 16 .. 31 rows).
__device__ __forceinline__ void write_block_sums(const WideArgs &A, const double (&col_f)[TY][TX + 1],
                                                 const double (&row_f)[TY][TX + 1], int tx, int ty) {
    const int nx = A.m.nx, ny = A.m.ny, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool fwd = lane < 16;
    if (warp == 0) {
        const int col = lane & 15, xc = tx * TX + col;
        const int h = min(TY, ny - ty * TY);
        if (xc < nx) {
            double a = 0.0;
            if (h == TY) {
#pragma unroll
                for (int k = 0; k < TY; ++k) a = fma(A.r, a, col_f[fwd ? k : TY - 1 - k][col]);
            } else {
                for (int k = 0; k < h; ++k) a = fma(A.r, a, col_f[fwd ? k : h - 1 - k][col]);
            }
            const long long o = (long long)ty * nx + xc;
            if (in_bounds(o, A.nys, A.m.chk)) (fwd ? A.ys : A.yt)[o] = a;
        }
    } else if (warp == 1) {       // 8 rows x 2 blocks
        const int row = lane & 7, b = (lane >> 3) & 1, yc = ty * TY + row, bx = 2 * tx + b;
        const int w = min(BK, nx - bx * BK);
        if (yc < ny && w > 0) {
            const double *s = row_f[row] + b * BK;
            double a = 0.0;
            if (w == BK) {
#pragma unroll
                for (int k = 0; k < BK; ++k) a = fma(A.r, a, s[fwd ? k : BK - 1 - k]);
            } else {
                for (int k = 0; k < w; ++k) a = fma(A.r, a, s[fwd ? k : w - 1 - k]);
            }
            const long long o = (long long)yc * A.nbx + bx;
            if (in_bounds(o, A.nxs, A.m.chk)) (fwd ? A.xs : A.xt)[o] = a;
        }
    } else if (warp == 2) {
        const int xc = tx * TX + (lane & 15), yc = ty * TY + (lane & 7), b = (lane >> 3) & 1, bx = 2 * tx + b;
        const int len = fwd ? min(BK, ny - ty * TY) : min(BK, nx - bx * BK);
        if (fwd ? xc < nx : yc < ny && len > 0) {
            const double v = value_of_equal(fwd ? &col_f[0][lane & 15] : &row_f[lane & 7][b * BK], fwd ? TX + 1 : 1, len);
            const long long o = fwd ? (long long)ty * nx + xc : (long long)yc * A.nbx + bx;
            if (in_bounds(o, fwd ? A.nys : A.nxs, A.m.chk)) (fwd ? A.ye : A.xe)[o] = v;
        }
    }
}

// What enters the tile's blocks, warp 0 its columns (lanes 0 .. 15 from below, 16 .. 31
// from above), warp 1 its rows (8 rows x 2 blocks): the one-sided sum of the kb blocks on
// that side (S at the cell before the block, T at the cell after it), the farthest joined
// first, returned.  Warps 2 and 3, lane by lane the same blocks: into E[0] (columns)
// and E[1] whether those of both sides have the block's own value throughout.  One code
// path for all four, without divisions: a grid this short runs most of its code once per
// SM, and waits for its fetch (128^2, a path per warp 10.8 us per step, this 9.1).
template <bool WALLS>
__device__ __forceinline__ double tile_join(const WideArgs &A, int tx, int ty, int (&E)[2][16]) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool fwd = lane < 16, cols = (warp & 1) == 0, sums = warp < 2;
    const int xc = tx * TX + (lane & 15), yc = ty * TY + (lane & 7), bx = 2 * tx + ((lane >> 3) & 1);
    const int nb = cols ? A.nby : A.nbx, kb = cols ? A.kby : A.kbx, b = cols ? ty : bx;
    const long long n = cols ? A.nys : A.nxs, o0 = cols ? xc : (long long)yc * A.nbx, stride = cols ? A.m.nx : 1;
    const double *own = cols ? (fwd ? A.ys : A.yt) : (fwd ? A.xs : A.xt);
    const double *other = fwd ? A.yt : A.ys;   // (columns only: rows are never mirrored)
    if (!sums) own = other = cols ? A.ye : A.xe;
    const double rl = cols ? A.ryl : A.rxl;
    const bool valid = cols ? xc < A.m.nx : yc < A.m.ny && bx < A.nbx;
    double acc = 0.0;
    bool same = false;
    if (valid) {
        auto at = [&](const BlockWalk &w) {
            const long long o = o0 + w.i * stride;
            return in_bounds(o, n, A.m.chk) ? (WALLS && w.swapped ? other : own)[o] : 0.0;
        };
        BlockWalk w{b, fwd ? -1 : 1, nb, WALLS && cols};
        const long long mine = __double_as_longlong(at(w));   // (of warps 2 and 3)
        same = (mine & 0x7ff0000000000000LL) != 0x7ff0000000000000LL;
        if (kb <= kJoin) {
            double v[kJoin];
            unsigned last = 0;
#pragma unroll
            for (int k = 0; k < kJoin; ++k) {
                w.next();
                v[k] = k < kb ? at(w) : 0.0;
                last |= (w.i == nb - 1 ? 1u : 0u) << k;
            }
#pragma unroll
            for (int k = kJoin - 1; k >= 0; --k) {
                if (k >= kb) continue;
                if (sums) acc = fma(last >> k & 1 ? rl : A.r8, acc, v[k]);
                else same &= __double_as_longlong(v[k]) == mine;
            }
        } else {
            // (lines so short that the cover takes more blocks: the farthest first, each found from the block)
            for (int k = kb; k >= 1; --k) {
                w = BlockWalk{b, fwd ? -1 : 1, nb, WALLS && cols};
                for (int j = 0; j < k; ++j) w.next();
                const double v = at(w);
                acc = fma(w.i == nb - 1 ? rl : A.r8, acc, v);
                same &= __double_as_longlong(v) == mine;
            }
        }
    }
    if (!sums) {
        const int both = __shfl_xor_sync(0xffffffffu, same ? 1 : 0, 16) & (same ? 1 : 0);
        if (fwd) E[warp & 1][lane] = both;
    }
    return acc;
}

// S_(i-1) and T_(i+1) of a tile's cells.
struct TileSums {
    double YS[TY][TX], YT[TY][TX];           // along the columns
    double XS[TY][TX + 1], XT[TY][TX + 1];   // along the rows
};

// Steps S (lanes 0 .. 15) and T (16 .. 31) through the tile's blocks, warp 0 the
// columns of colf, warp 1 the rows of rowf (staged with one cell around the
// tile), from the entering sums; one code path for both directions.
template <bool ABS>
__device__ __forceinline__ void tile_step(const WideArgs &A, int tx, int ty, double carry,
                                          const double (&colf)[TY + 2][TX + 2], const double (&rowf)[TY + 2][TX + 2],
                                          TileSums &M) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp >= 2) return;
    const bool fwd = lane < 16;
    const int line = warp == 0 ? lane & 15 : lane & 7, b = warp == 0 ? 0 : (lane >> 3) & 1;
    const int len = min(BK, warp == 0 ? A.m.ny - ty * TY : A.m.nx - (2 * tx + b) * BK);   // cells of the block
    const double *src = warp == 0 ? &colf[1][line + 1] : &rowf[line + 1][b * BK + 1];
    double *dst = warp == 0 ? &(fwd ? M.YS : M.YT)[0][line] : &(fwd ? M.XS : M.XT)[line][b * BK];
    const int step = warp == 0 ? TX + 2 : 1, dstep = warp == 0 ? TX : 1;
    double v = carry;
#pragma unroll
    for (int k = 0; k < BK; ++k) {
        const int i = fwd ? k : len - 1 - k;
        if (k < len) {
            dst[i * dstep] = v;
            if (k + 1 < BK) v = fma(A.r, v, ABS ? fabs(src[i * step]) : src[i * step]);
        }
    }
}

// Pass 1: rho (Eq. 3), the potential field q (Eq. 8 / 21) and, for the HDM, the
// block sums of the stencil's field (Phi = |q| for Shan-Chen, U for Zhang-Chen).
template <typename TS, bool HDM>
__global__ void __launch_bounds__(NT) wide_potential_kernel(const __grid_constant__ WideArgs A, bool sc,
                                                            const TS *f, double *q, int *err) {
    __shared__ double S[TY][TX + 1];
    const Model<double> &m = A.m;
    const int nx = m.nx, ny = m.ny;
    const long long n = (long long)nx * ny;
    const int ty = blockIdx.x / A.ntx, tx = blockIdx.x - ty * A.ntx;
    const int lx = threadIdx.x & (TX - 1), ly = threadIdx.x / TX;
    const int x = tx * TX + lx, y = ty * TY + ly;
    const bool valid = x < nx && y < ny;
    const long long c = (long long)y * nx + x;
    if (A.early) ptx::griddep_launch_dependents();
    ptx::griddep_wait();   // the previous step's pass 2 has written f
    double phi = 0.0;
    if (valid) {
        double v[kQ];
#pragma unroll
        for (int i = 0; i < kQ; ++i) v[i] = in_bounds(i * n + c, kQ * n, m.chk) ? (double)f[i * n + c] : 0.0;
        double r = v[0];
#pragma unroll
        for (int i = 1; i < kQ; ++i) r += v[i];
        // positive and finite, by the bits (a comparison takes an FP64 slot)
        const long long rb = __double_as_longlong(r);
        if (!(rb > 0 && rb < 0x7ff0000000000000LL)) atomicOr(err, kErrUnstable);
        const double U = potential_u(m, r);
        phi = sc ? sqrt(fabs(U)) : U;
        q[c] = sc ? copysign(phi, U) : U;   // s Phi (Eq. 21), s the sign of U, or U (Eq. 8)
    }
    if (!A.early) ptx::griddep_launch_dependents();
    if (!HDM) return;
    S[ly][lx] = phi;
    __syncthreads();
    write_block_sums(A, S, S, tx, ty);
}

// Pass 2: gradient of q, force (Eq. 22 / 7), exact-difference forcing with BGK
// (Eq. 1, 2, 10) and push streaming; MOM: rho and the Eq. 11 velocity instead;
// REC: also the reverse mode's record of f, planes rho, jx, jy, Dx, Dy at rho_out.
template <typename TS, bool SC, bool HDM, bool TAU1, bool WALLS, bool MOM, bool REC = false>
__global__ void __launch_bounds__(NT) wide_collide_kernel(const __grid_constant__ WideArgs A, const TS *f,
                                                          const double *q, TS *fout, TS *rho_out, TS *vx_out,
                                                          TS *vy_out) {
    constexpr int QW = TX + 2, QH = TY + 2;
    __shared__ double Q[QH][QW];                          // q over the tile and one cell around it
    __shared__ TileSums M;
    __shared__ int E[2][16];
    const Model<double> &m = A.m;
    const int nx = m.nx, ny = m.ny;
    const long long n = (long long)nx * ny;
    const int ty = blockIdx.x / A.ntx, tx = blockIdx.x - ty * A.ntx;
    const int x0 = tx * TX, y0 = ty * TY;
    const int lx = threadIdx.x & (TX - 1), ly = threadIdx.x / TX;
    const int x = x0 + lx, y = y0 + ly;
    const bool valid = x < nx && y < ny;
    const long long c = (long long)min(y, ny - 1) * nx + min(x, nx - 1);
    if (A.early) ptx::griddep_launch_dependents();
    ptx::griddep_wait();   // pass 1 has written q and the block sums

    // every load is issued before the first value is waited for; the rows and columns
    // of the tile's halo: periodic, or mirrored across a wall
    constexpr int kStage = (QH * QW + NT - 1) / NT;
    double qv[kStage];
#pragma unroll
    for (int j = 0; j < kStage; ++j) {
        const int k = threadIdx.x + j * NT, ry = k / QW, rx = k - ry * QW;
        const int gx = min(x0 - 1 + rx, nx), gy = min(y0 - 1 + ry, ny);
        const int px = gx < 0 ? nx - 1 : (gx == nx ? 0 : gx);
        const int py = gy < 0 ? (WALLS ? 0 : ny - 1) : (gy == ny ? (WALLS ? ny - 1 : 0) : gy);
        const long long g = (long long)py * nx + px;
        qv[j] = k < QH * QW && in_bounds(g, n, m.chk) ? q[g] : 0.0;
    }
    TS fv[kQ];
#pragma unroll
    for (int i = 0; i < kQ; ++i) fv[i] = in_bounds(i * n + c, kQ * n, m.chk) ? f[i * n + c] : TS(0);
    const double carry = HDM ? tile_join<WALLS>(A, tx, ty, E) : 0.0;
#pragma unroll
    for (int j = 0; j < kStage; ++j) {
        const int k = threadIdx.x + j * NT, ry = k / QW, rx = k - ry * QW;
        if (k < QH * QW) Q[ry][rx] = qv[j];
    }
    double fi[kQ];
#pragma unroll
    for (int i = 0; i < kQ; ++i) fi[i] = (double)fv[i];
    __syncthreads();
    auto mag = [](double v) { return SC ? fabs(v) : v; };
    if (HDM) tile_step<SC>(A, tx, ty, carry, Q, Q, M);
    // moments (Eq. 3) from the sums over the populations moving east, west, north, south
    const double east = fi[1] + fi[5] + fi[8], west = fi[3] + fi[6] + fi[7];
    const double r = fi[0] + fi[2] + fi[4] + east + west;
    const double jx = east - west, jy = (fi[2] + fi[5] + fi[6]) - (fi[4] + fi[7] + fi[8]);
    const double inv = 1.0 / r;
    if (HDM) __syncthreads();
    if (!A.early) ptx::griddep_launch_dependents();
    if (!valid) return;

    const double *p = &Q[ly + 1][lx + 1];
    double dx, dy;
    if (HDM) {
        const double tx_s = E[1][ly + (lx & 8)] ? 0.0 : M.XT[ly][lx] - M.XS[ly][lx];
        const double ty_s = E[0][lx] ? 0.0 : M.YT[ly][lx] - M.YS[ly][lx];
        dx = fma(A.c1, mag(p[1]) - mag(p[-1]), A.cs * tx_s);
        dy = fma(A.c1, mag(p[QW]) - mag(p[-QW]), A.cs * ty_s);
    } else {   // Eq. 15 times 1/c_s^2
        const double ne = mag(p[QW + 1]), nw = mag(p[QW - 1]), se = mag(p[-QW + 1]), sw = mag(p[-QW - 1]);
        dx = (1.0 / 3.0) * (mag(p[1]) - mag(p[-1])) + (1.0 / 12.0) * ((ne + se) - (nw + sw));
        dy = (1.0 / 3.0) * (mag(p[QW]) - mag(p[-QW])) + (1.0 / 12.0) * ((ne + nw) - (se + sw));
    }
    double Fx, Fy;
    if (SC) {   // Eq. 22: F = -2 s Phi grad Phi, p[0] = s Phi
        const double s = -2.0 * p[0];
        Fx = s * dx;
        Fy = s * dy;
    } else {    // Eq. 7
        Fx = -dx;
        Fy = -dy;
    }
    if constexpr (REC) {
        const double v[5] = {r, jx, jy, dx, dy};
#pragma unroll
        for (int k = 0; k < 5; ++k)
            if (in_bounds(k * n + c, 5 * n, m.chk)) rho_out[k * n + c] = v[k];
    }
    if (MOM) {  // Eq. 3 and Eq. 11
        if (in_bounds(c, n, m.chk)) {
            rho_out[c] = (TS)r;
            vx_out[c] = (TS)(fma(0.5, Fx, jx) * inv);
            vy_out[c] = (TS)(fma(0.5, Fy, jy) * inv);
        }
        return;
    }
    const double ux = jx * inv, uy = jy * inv;
    const double vx = fma(Fx, inv, ux), vy = fma(Fy, inv, uy);   // u + du, du = F/rho (Eq. 10)
    // f^eq_i = w_i rho (a + 4.5 (e.v)^2 + 3 e.v) with t = 3 e.v: (w_i rho / 2)(2 a + t^2) + w_i rho t,
    // 2 a = 2 - (tx^2 + ty^2) / 3
    const double tvx = 3.0 * vx, tvy = 3.0 * vy, tux = 3.0 * ux, tuy = 3.0 * uy;
    const double av = fma(-1.0 / 3.0, fma(tvx, tvx, tvy * tvy), 2.0);
    const double au = TAU1 ? 0.0 : fma(-1.0 / 3.0, fma(tux, tux, tuy * tuy), 2.0);
    const double w1 = r * (1.0 / 9.0), w2 = r * (1.0 / 36.0), h1 = r * (1.0 / 18.0), h2 = r * (1.0 / 72.0);
    const int xp = x + 1 == nx ? 0 : x + 1, xm = x == 0 ? nx - 1 : x - 1;
    const int yp = y + 1 == ny ? 0 : y + 1, ym = y == 0 ? ny - 1 : y - 1;
    // f_i* of the moving populations, direction and opposite together; the rest
    // population takes the remainder so that the collision conserves mass up to
    // rounding
    double moved = 0.0;
    auto put = [&](int i, double post) {
        const int dxs = ex(i) == 1 ? xp : (ex(i) == -1 ? xm : x);
        const int dys = ey(i) == 1 ? yp : (ey(i) == -1 ? ym : y);
        const long long k = WALLS && ((ey(i) == 1 && y == ny - 1) || (ey(i) == -1 && y == 0))
                                ? opp(i) * n + c   // half-way bounce-back off the wall
                                : i * n + (long long)dys * nx + dxs;
        moved += post;
        if (in_bounds(k, kQ * n, m.chk)) fout[k] = (TS)post;
    };
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        constexpr int kDir[4] = {1, 2, 5, 6};
        const int i = kDir[d], o = opp(i);
        const double w = d < 2 ? w1 : w2, h = d < 2 ? h1 : h2;
        const double t = d == 0 ? tvx : (d == 1 ? tvy : (d == 2 ? tvx + tvy : tvy - tvx));
        const double even = h * fma(t, t, av);
        double pi = fma(w, t, even), po = fma(-w, t, even);
        if (!TAU1) {   // (1 - omega) of the distance to f^eq(u) stays
            const double tu = d == 0 ? tux : (d == 1 ? tuy : (d == 2 ? tux + tuy : tuy - tux));
            const double eu = h * fma(tu, tu, au);
            pi = fma(1.0 - m.omega, fi[i] - fma(w, tu, eu), pi);
            po = fma(1.0 - m.omega, fi[o] - fma(-w, tu, eu), po);
        }
        put(i, pi);
        put(o, po);
    }
    if (in_bounds(c, kQ * n, m.chk)) fout[c] = (TS)(r - moved);
}

// ---- reverse step (the adjoint of the step, as adjoint.cu derives it) ----
//
// From the record of the state (rho, j, and the derivatives D the forward used)
// and its field q, kernel A does the local adjoint of the forcing and collision
// and writes D_bar with its block sums, the partial rho_bar, and kappa, theta =
// dPhi/dU (dU/drho, dU/dtheta); kernel B differentiates D_bar (the transposed
// derivative is its negative) and finishes rho_bar, T_bar and lambda(t).  Both are
// bound by FP64 instructions as the forward passes are, so the directions are
// taken in opposite pairs (sums and differences of g), Phi comes from the stored
// field instead of a square root, and kappa and theta are formed once.  16 steps
// forward and back at 256^2: 2.70 ms with the kernels that differentiate the field
// and D_bar by the direct radius-40 stencil on 32 x 16 tiles, 1.64 ms with these.
struct WideAdjArgs {
    WideArgs w;                // (its block sums: those of D_bar)
    double R, aalp;            // gas constant, a dalpha/dT
    const double *rec, *q;     // record of the state (five planes) and its field
    const double *lam;         // lambda(t+1): three planes for tau = 1, else nine
    double *lam_out;           // lambda(t)
    double *aux;               // D_bar_x, D_bar_y, rho_bar, kappa, theta[, j_bar_x, j_bar_y]
    double *Tpart;             // one FP64 slot per warp of A, then of B
};

// dU/drho and dU/dtheta (theta = T, or G for the effective mass of Eq. 4-5) times
// dPhi/dU = s / (2 Phi) (Shan-Chen, q = s Phi) or 1; U of Eq. 8 with Eq. 24, 27-29.
template <bool SC>
__device__ __forceinline__ void wide_eos(const WideAdjArgs &a, double rho, double q, double &kappa, double &theta) {
    const Model<double> &m = a.w.m;
    double dr, dt;
    if (m.eos == LBM_EOS_PSI_EXP) {
        const double e = exp(-rho * m.b), psi = 1.0 - e;
        dr = 2.0 * m.a * psi * e * m.b;
        dt = 0.5 * psi * psi;
    } else {
        double dpdr, dpdT;
        if (m.eos == LBM_EOS_CS) {
            const double e = m.b * rho * 0.25, om = 1.0 - e, inv = 1.0 / om, inv3 = inv * inv * inv;
            const double num = fma(e, fma(e, om, 1.0), 1.0);   // 1 + e + e^2 - e^3
            const double Z = num * inv3, dZ = fma(fma(e, fma(-3.0, e, 2.0), 1.0), om, 3.0 * num) * inv3 * inv;
            dpdr = fma(m.RT, fma(e, dZ, Z), -2.0 * m.a * rho);
            dpdT = a.R * rho * Z;
        } else {
            const double inv = 1.0 / (1.0 - m.b * rho), ri = rho * inv;
            dpdr = m.RT * inv * inv;
            dpdT = a.R * ri;
            if (m.eos == LBM_EOS_VDW) {
                dpdr = fma(-2.0 * m.a, rho, dpdr);
            } else if (m.eos == LBM_EOS_PR) {
                const double br = m.b * rho, id = 1.0 / fma(br, 2.0 - br, 1.0), rid = rho * id;
                dpdr -= 2.0 * m.aal * (1.0 + br) * rid * id;
                dpdT -= a.aalp * rho * rid;
            } else {   // RK, RKS
                const double br = m.b * rho, id = 1.0 / (1.0 + br), rid = rho * id;
                dpdr -= m.aal * (2.0 + br) * rid * id;
                dpdT -= a.aalp * rho * rid;
            }
        }
        dr = fma(m.k, dpdr, -1.0 / 3.0);
        dt = m.k * dpdT;
    }
    const double d = SC ? (q != 0.0 ? 0.5 / q : 0.0) : 1.0;   // s / (2 Phi) = 1 / (2 q)
    kappa = d * dr;
    theta = d * dt;
}

// Sum over the warp, added to the warp's own slot (one writer per slot and
// launch, the launches ordered: reproducible).
__device__ __forceinline__ void wide_slot_add(double v, double *part) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(part + (size_t)blockIdx.x * (NT / 32) + (threadIdx.x >> 5), v);
}

template <bool SC, bool HDM, bool TAU1>
__global__ void __launch_bounds__(NT) wide_adj_a_kernel(const __grid_constant__ WideAdjArgs a) {
    __shared__ double L[TAU1 ? 3 : 1][TY + 2][TX + 2];   // lambda with one cell around the tile
    __shared__ double SX[TY][TX + 1], SY[TY][TX + 1];    // D_bar
    const WideArgs &A = a.w;
    const Model<double> &m = A.m;
    const int nx = m.nx, ny = m.ny;
    const long long n = (long long)nx * ny;
    const int ty = blockIdx.x / A.ntx, tx = blockIdx.x - ty * A.ntx;
    const int lx = threadIdx.x & (TX - 1), ly = threadIdx.x / TX, x = tx * TX + lx, y = ty * TY + ly;
    const bool valid = x < nx && y < ny;
    const int xc = min(x, nx - 1), yc = min(y, ny - 1);
    const long long c = (long long)yc * nx + xc;
    if (A.early) ptx::griddep_launch_dependents();
    ptx::griddep_wait();
    auto rec = [&](int k) { return in_bounds(k * n + c, 5 * n, m.chk) ? a.rec[k * n + c] : 1.0; };
    const double r = rec(0), jx = rec(1), jy = rec(2), Dx = rec(3), Dy = rec(4);
    const double q = in_bounds(c, n, m.chk) ? a.q[c] : 1.0;
    double g[kQ];   // g_i = lambda_i(x + e_i)
    if (TAU1) {
        for (int k = threadIdx.x; k < 3 * (TY + 2) * (TX + 2); k += NT) {
            const int f = k / ((TY + 2) * (TX + 2)), kk = k - f * ((TY + 2) * (TX + 2));
            const int ry = kk / (TX + 2), rx = kk - ry * (TX + 2);
            const int gx = min(tx * TX - 1 + rx, nx), gy = min(ty * TY - 1 + ry, ny);
            const long long o = f * n + (long long)(gy < 0 ? ny - 1 : (gy == ny ? 0 : gy)) * nx +
                                (gx < 0 ? nx - 1 : (gx == nx ? 0 : gx));
            L[f][ry][rx] = in_bounds(o, 3 * n, m.chk) ? a.lam[o] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kQ; ++i) {   // lambda_i = rho_bar + e_i . j_bar
            double v = L[0][ly + 1 + ey(i)][lx + 1 + ex(i)];
            if (ex(i) == 1) v += L[TAU1 ? 1 : 0][ly + 1 + ey(i)][lx + 1 + ex(i)];
            if (ex(i) == -1) v -= L[TAU1 ? 1 : 0][ly + 1 + ey(i)][lx + 1 + ex(i)];
            if (ey(i) == 1) v += L[TAU1 ? 2 : 0][ly + 1 + ey(i)][lx + 1 + ex(i)];
            if (ey(i) == -1) v -= L[TAU1 ? 2 : 0][ly + 1 + ey(i)][lx + 1 + ex(i)];
            g[i] = v;
        }
    } else {
        const int xp = xc + 1 == nx ? 0 : xc + 1, xm = xc == 0 ? nx - 1 : xc - 1;
        const int yp = yc + 1 == ny ? 0 : yc + 1, ym = yc == 0 ? ny - 1 : yc - 1;
#pragma unroll
        for (int i = 0; i < kQ; ++i) {
            const long long o = i * n + (long long)(ey(i) == 1 ? yp : (ey(i) == -1 ? ym : yc)) * nx +
                                (ex(i) == 1 ? xp : (ex(i) == -1 ? xm : xc));
            g[i] = in_bounds(o, kQ * n, m.chk) ? a.lam[o] : 0.0;
        }
    }
    double kappa, theta;
    wide_eos<SC>(a, r, q, kappa, theta);
    const double inv = 1.0 / r, ux = jx * inv, uy = jy * inv;
    const double s = SC ? -2.0 * q : -1.0, Fx = s * Dx, Fy = s * Dy;   // Eq. 22 / 7
    const double vx = fma(Fx, inv, ux), vy = fma(Fy, inv, uy);
    // With f^eq_i(v) = w_i rho (a + e.v (3 + 4.5 e.v)), a = 1 - 1.5 |v|^2, the sums over
    // the directions of g_i w_i times 1, e_i (3 + 9 e.v), e.v (3 + 4.5 e.v), a direction
    // and its opposite at a time: gs, gd the sum and difference of their g.
    double G0 = (4.0 / 9.0) * g[0], Gx = 0.0, Gy = 0.0, Rv = 0.0, Hx = 0.0, Hy = 0.0, Ru = 0.0;
#pragma unroll
    for (int cl = 0; cl < 2; ++cl) {   // the axes (w = 1/9), the diagonals (1/36)
        double sg = 0.0, ax = 0.0, ay = 0.0, b = 0.0, hx = 0.0, hy = 0.0, bu = 0.0;
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            const int i = cl == 0 ? 1 + d : 5 + d, o = opp(i);
            const double gs = g[i] + g[o], g3 = 3.0 * (g[i] - g[o]);
            auto along = [&](double px, double py) { return i == 1 ? px : (i == 2 ? py : (i == 5 ? px + py : py - px)); };
            auto add = [&](double ev, double &sx, double &sy, double &sb) {
                const double t = ev * gs, A1 = fma(9.0, t, g3);
                if (ex(i) == 1) sx += A1;
                if (ex(i) == -1) sx -= A1;
                if (ey(i) == 1) sy += A1;
                sb = fma(ev, fma(4.5, t, g3), sb);
            };
            sg += gs;
            add(along(vx, vy), ax, ay, b);
            if (!TAU1) add(along(ux, uy), hx, hy, bu);
        }
        const double w = cl == 0 ? 1.0 / 9.0 : 1.0 / 36.0;
        G0 = fma(w, sg, G0);
        Gx = fma(w, ax, Gx);
        Gy = fma(w, ay, Gy);
        Rv = fma(w, b, Rv);
        if (!TAU1) {
            Hx = fma(w, hx, Hx);
            Hy = fma(w, hy, Hy);
            Ru = fma(w, bu, Ru);
        }
    }
    double rb = fma(fma(-1.5, fma(vx, vx, vy * vy), 1.0), G0, Rv);
    const double vbx = r * fma(-3.0 * vx, G0, Gx), vby = r * fma(-3.0 * vy, G0, Gy);
    double ubx = vbx, uby = vby;
    if (!TAU1) {   // the f^eq(u) terms enter with the weights -(1 - omega) g_i
        const double om1 = 1.0 - m.omega;
        rb -= om1 * fma(fma(-1.5, fma(ux, ux, uy * uy), 1.0), G0, Ru);
        ubx -= om1 * r * fma(-3.0 * ux, G0, Hx);
        uby -= om1 * r * fma(-3.0 * uy, G0, Hy);
    }
    const double Fbx = vbx * inv, Fby = vby * inv, jbx = ubx * inv, jby = uby * inv;
    rb -= fma(Fbx, Fx, Fby * Fy) * inv;
    rb -= fma(jbx, ux, jby * uy);
    const double Dbx = s * Fbx, Dby = s * Fby;
    double tacc = 0.0;
    if (SC) {   // the centre factor Phi of F = -2 s Phi D
        const double pc = (q >= 0.0 ? -2.0 : 2.0) * fma(Fbx, Dx, Fby * Dy);
        rb = fma(pc, kappa, rb);
        tacc = valid ? pc * theta : 0.0;
    }
    if (HDM) {
        SX[ly][lx] = valid ? Dbx : 0.0;
        SY[ly][lx] = valid ? Dby : 0.0;
        __syncthreads();
    }
    if (!A.early) ptx::griddep_launch_dependents();
    if (valid) {
        const double v[7] = {Dbx, Dby, rb, kappa, theta, jbx, jby};
#pragma unroll
        for (int k = 0; k < (TAU1 ? 5 : 7); ++k)
            if (in_bounds(k * n + c, 7 * n, m.chk)) a.aux[k * n + c] = v[k];
        if (TAU1 && in_bounds(2 * n + c, 3 * n, m.chk)) {
            a.lam_out[n + c] = jbx;
            a.lam_out[2 * n + c] = jby;
        }
    }
    if (HDM) write_block_sums(A, SY, SX, tx, ty);
    if (SC) wide_slot_add(tacc, a.Tpart);
}

template <bool HDM, bool TAU1>
__global__ void __launch_bounds__(NT) wide_adj_b_kernel(const __grid_constant__ WideAdjArgs a) {
    __shared__ double QX[TY + 2][TX + 2], QY[TY + 2][TX + 2];   // D_bar with one cell around the tile
    __shared__ TileSums M;
    __shared__ int E[2][16];
    const WideArgs &A = a.w;
    const Model<double> &m = A.m;
    const int nx = m.nx, ny = m.ny;
    const long long n = (long long)nx * ny;
    const int ty = blockIdx.x / A.ntx, tx = blockIdx.x - ty * A.ntx;
    const int lx = threadIdx.x & (TX - 1), ly = threadIdx.x / TX, x = tx * TX + lx, y = ty * TY + ly;
    const bool valid = x < nx && y < ny;
    const int xc = min(x, nx - 1), yc = min(y, ny - 1);
    const long long c = (long long)yc * nx + xc;
    if (A.early) ptx::griddep_launch_dependents();
    ptx::griddep_wait();   // A's output
    constexpr int kCells = (TY + 2) * (TX + 2), kStage = (kCells + NT - 1) / NT;
    double sx[kStage], sy[kStage];   // (every load before the first wait, as in pass 2)
#pragma unroll
    for (int j = 0; j < kStage; ++j) {
        const int k = threadIdx.x + j * NT, ry = k / (TX + 2), rx = k - ry * (TX + 2);
        const int gx = min(tx * TX - 1 + rx, nx), gy = min(ty * TY - 1 + ry, ny);
        const long long o = (long long)(gy < 0 ? ny - 1 : (gy == ny ? 0 : gy)) * nx + (gx < 0 ? nx - 1 : (gx == nx ? 0 : gx));
        const bool ok = k < kCells && in_bounds(o, n, m.chk);
        sx[j] = ok ? a.aux[o] : 0.0;
        sy[j] = ok ? a.aux[n + o] : 0.0;
    }
    auto aux = [&](int k) { return in_bounds(k * n + c, 7 * n, m.chk) ? a.aux[k * n + c] : 0.0; };
    const double rb0 = aux(2), kappa = aux(3), theta = aux(4);
    const double carry = HDM ? tile_join<false>(A, tx, ty, E) : 0.0;
#pragma unroll
    for (int j = 0; j < kStage; ++j) {
        const int k = threadIdx.x + j * NT, ry = k / (TX + 2), rx = k - ry * (TX + 2);
        if (k >= kCells) continue;
        QX[ry][rx] = sx[j];
        QY[ry][rx] = sy[j];
    }
    __syncthreads();
    if (HDM) {
        tile_step<false>(A, tx, ty, carry, QY, QX, M);
        __syncthreads();
    }
    if (!A.early) ptx::griddep_launch_dependents();
    const double *px = &QX[ly + 1][lx + 1], *py = &QY[ly + 1][lx + 1];
    constexpr int QW = TX + 2;
    double dd;   // Dx[D_bar_x] + Dy[D_bar_y]
    if (HDM) {
        const double tx_s = E[1][ly + (lx & 8)] ? 0.0 : M.XT[ly][lx] - M.XS[ly][lx];
        const double ty_s = E[0][lx] ? 0.0 : M.YT[ly][lx] - M.YS[ly][lx];
        dd = fma(A.c1, (px[1] - px[-1]) + (py[QW] - py[-QW]), A.cs * (tx_s + ty_s));
    } else {
        dd = (1.0 / 3.0) * ((px[1] - px[-1]) + (py[QW] - py[-QW])) +
             (1.0 / 12.0) * (((px[QW + 1] + px[-QW + 1]) - (px[QW - 1] + px[-QW - 1])) +
                             ((py[QW + 1] + py[QW - 1]) - (py[-QW + 1] + py[-QW - 1])));
    }
    const double rb = fma(-kappa, dd, rb0);
    if (valid) {
        if (TAU1) {
            if (in_bounds(c, 3 * n, m.chk)) a.lam_out[c] = rb;
        } else {
            const double jbx = aux(5), jby = aux(6), om1 = 1.0 - m.omega;
            const int xp = x + 1 == nx ? 0 : x + 1, xm = x == 0 ? nx - 1 : x - 1;
            const int yp = y + 1 == ny ? 0 : y + 1, ym = y == 0 ? ny - 1 : y - 1;
#pragma unroll
            for (int i = 0; i < kQ; ++i) {
                const long long o = i * n + (long long)(ey(i) == 1 ? yp : (ey(i) == -1 ? ym : y)) * nx +
                                    (ex(i) == 1 ? xp : (ex(i) == -1 ? xm : x));
                double li = fma(om1, in_bounds(o, kQ * n, m.chk) ? a.lam[o] : 0.0, rb);
                if (ex(i) == 1) li += jbx;
                if (ex(i) == -1) li -= jbx;
                if (ey(i) == 1) li += jby;
                if (ey(i) == -1) li -= jby;
                if (in_bounds(i * n + c, kQ * n, m.chk)) a.lam_out[i * n + c] = li;
            }
        }
    }
    wide_slot_add(valid ? -theta * dd : 0.0, a.Tpart);
}

// Blocks that cover kReach cells of the cyclic (mirror: mirrored) line of n
// cells, wherever the first of them lies.  Only starts near the short block at
// the line's end need more than kReach / BK.
int cover(int n, bool mirror) {
    const int nb = (n + BK - 1) / BK, last = n - (nb - 1) * BK, p = mirror ? 2 * nb : nb;
    int worst = 0;
    for (int s = std::max(0, nb - 2 * kReach / BK); s < (nb < 2 * kReach / BK ? p : nb); ++s) {
        int have = 0, k = 0;
        for (; have < kReach; ++k) {
            const int i = (s + k) % p;
            have += (i < nb ? i : p - 1 - i) == nb - 1 ? last : BK;
        }
        worst = std::max(worst, k);
    }
    return worst;
}

constexpr int kSpread = 4;   // CTAs per SM up to which a grid is spread (see the head of the file)

WideArgs args_of(const Model<double> &m, double *sums) {
    WideArgs a{};
    a.m = m;
    const double r = 0.5 * (sqrt(5.0) - 3.0);   // root of r^2/3 + r + 1/3 = 0 (Eq. 20's operator)
    a.r = r;
    a.r8 = pow(r, BK);
    a.c1 = 1.0 / 12.0;
    a.cs = -(25.0 / 12.0) * r;
    a.nbx = (m.nx + BK - 1) / BK;
    a.nby = (m.ny + BK - 1) / BK;
    a.rxl = pow(r, m.nx - (a.nbx - 1) * BK);
    a.ryl = pow(r, m.ny - (a.nby - 1) * BK);
    a.kbx = cover(m.nx, false);
    a.kby = cover(m.ny, m.walls != 0);
    a.ntx = (m.nx + TX - 1) / TX;
    a.nys = (long long)a.nby * m.nx;
    a.nxs = (long long)a.nbx * m.ny;
    a.ys = sums;
    a.yt = a.ys + a.nys;
    a.ye = a.yt + a.nys;
    a.xs = a.ye + a.nys;
    a.xt = a.xs + a.nxs;
    a.xe = a.xt + a.nxs;
    a.early = spread_smem((long long)a.ntx * a.nby, kSpread) > 0;
    return a;
}

template <typename K, typename... Args>
cudaError_t launch_grid(K kern, const WideArgs &w, bool pdl, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((long long)w.ntx * w.nby));
    cfg.blockDim = dim3(NT);
    cfg.stream = s;
    cfg.dynamicSmemBytes = spread_smem((long long)w.ntx * w.nby, kSpread);
    if (cfg.dynamicSmemBytes > 0) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSpreadMax);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}
template <typename K, typename... Args>
cudaError_t launch_tiles(K kern, const WideArgs &w, cudaStream_t s, Args... args) {
    return launch_grid(kern, w, true, s, w, args...);
}

template <typename TS, bool MOM>
cudaError_t pick_collide(const WideArgs &a, bool sc, bool cdm, const TS *f, const double *q, TS *fout, TS *rho, TS *vx,
                         TS *vy, cudaStream_t s) {
    const bool tau1 = MOM || a.m.omega == 1.0, walls = a.m.walls != 0;
#define LBM_WIDE(SC, HDM)                                                                                          \
    return walls ? (tau1 ? launch_tiles(wide_collide_kernel<TS, SC, HDM, true, true, MOM>, a, s, f, q, fout, rho, vx, vy) \
                         : launch_tiles(wide_collide_kernel<TS, SC, HDM, MOM, true, MOM>, a, s, f, q, fout, rho, vx, vy)) \
                 : (tau1 ? launch_tiles(wide_collide_kernel<TS, SC, HDM, true, false, MOM>, a, s, f, q, fout, rho, vx, vy) \
                         : launch_tiles(wide_collide_kernel<TS, SC, HDM, MOM, false, MOM>, a, s, f, q, fout, rho, vx, vy))
    if (sc) {
        if (cdm) LBM_WIDE(true, false);
        LBM_WIDE(true, true);
    }
    if (cdm) LBM_WIDE(false, false);
    LBM_WIDE(false, true);
#undef LBM_WIDE
}

}  // namespace

// The HDM at its default radius, and the CDM.  A radius that the caller asks for
// keeps the direct stencil (its truncation is part of the result there), and so
// does a lattice one cell wide.
bool wide_step_supported(const lbm_params &p) {
    return p.nx >= 2 && p.ny >= 2 && (p.grad == LBM_GRAD_CDM || p.hdm_radius == 0);
}

size_t wide_sums_bytes(int nx, int ny) {
    const long long nbx = (nx + BK - 1) / BK, nby = (ny + BK - 1) / BK;
    return sizeof(double) * 3 * (size_t)(nby * nx + nbx * ny);
}

template <typename TS>
cudaError_t launch_wide_potential(const Model<double> &m, bool sc, bool cdm, const TS *f, double *q, double *sums,
                                  int *err, cudaStream_t s) {
    const WideArgs a = args_of(m, sums);
    return cdm ? launch_tiles(wide_potential_kernel<TS, false>, a, s, sc, f, q, err)
               : launch_tiles(wide_potential_kernel<TS, true>, a, s, sc, f, q, err);
}

template <typename TS>
cudaError_t launch_wide_collide(const Model<double> &m, bool sc, bool cdm, const TS *f, const double *q,
                                double *sums, TS *fout, cudaStream_t s) {
    return pick_collide<TS, false>(args_of(m, sums), sc, cdm, f, q, fout, (TS *)nullptr, (TS *)nullptr, (TS *)nullptr, s);
}

template <typename TS>
cudaError_t launch_wide_moments(const Model<double> &m, bool sc, bool cdm, const TS *f, const double *q, double *sums,
                                TS *rho, TS *vx, TS *vy, cudaStream_t s) {
    return pick_collide<TS, true>(args_of(m, sums), sc, cdm, f, q, (TS *)nullptr, rho, vx, vy, s);
}

cudaError_t launch_wide_collide_rec(const Model<double> &m, bool sc, bool cdm, const double *f, const double *q,
                                    double *sums, double *fout, double *rec, cudaStream_t s) {
    const WideArgs a = args_of(m, sums);
    const bool tau1 = m.omega == 1.0;
    double *none = nullptr;
#define LBM_REC(SC, HDM)                                                                                             \
    return tau1 ? launch_tiles(wide_collide_kernel<double, SC, HDM, true, false, false, true>, a, s, f, q, fout, rec, none, none) \
                : launch_tiles(wide_collide_kernel<double, SC, HDM, false, false, false, true>, a, s, f, q, fout, rec, none, none)
    if (sc) {
        if (cdm) LBM_REC(true, false);
        LBM_REC(true, true);
    }
    if (cdm) LBM_REC(false, false);
    LBM_REC(false, true);
#undef LBM_REC
}

int wide_adjoint_slots(int nx, int ny) { return 2 * ((nx + TX - 1) / TX) * ((ny + TY - 1) / TY) * (NT / 32); }

cudaError_t launch_wide_adjoint(const Model<double> &m, double R, double aalp, bool sc, bool cdm, const double *rec,
                                const double *q, const double *lam, double *aux, double *sums, double *lam_out,
                                double *Tpart, bool overlap_prev, cudaStream_t s) {
    WideAdjArgs a{};
    a.w = args_of(m, sums);
    a.R = R;
    a.aalp = aalp;
    a.rec = rec;
    a.q = q;
    a.lam = lam;
    a.lam_out = lam_out;
    a.aux = aux;
    a.Tpart = Tpart;
    const bool tau1 = m.omega == 1.0;
    void (*ka)(const WideAdjArgs), (*kb)(const WideAdjArgs);
#define LBM_ADJ(HDM, TAU1)                                                                       \
    do {                                                                                         \
        ka = sc ? wide_adj_a_kernel<true, HDM, TAU1> : wide_adj_a_kernel<false, HDM, TAU1>;      \
        kb = wide_adj_b_kernel<HDM, TAU1>;                                                       \
    } while (0)
    if (cdm) {
        if (tau1) LBM_ADJ(false, true);
        else LBM_ADJ(false, false);
    } else {
        if (tau1) LBM_ADJ(true, true);
        else LBM_ADJ(true, false);
    }
#undef LBM_ADJ
    // (A may overlap the previous step's B, but not an event wait on the recompute's stream)
    cudaError_t e = launch_grid(ka, a.w, overlap_prev, s, a);
    if (e != cudaSuccess) return e;
    a.Tpart = Tpart + wide_adjoint_slots(m.nx, m.ny) / 2;
    return launch_grid(kb, a.w, true, s, a);
}

#define LBM_WIDE_INST(TS)                                                                                          \
    template cudaError_t launch_wide_potential<TS>(const Model<double> &, bool, bool, const TS *, double *, double *, \
                                                   int *, cudaStream_t);                                           \
    template cudaError_t launch_wide_collide<TS>(const Model<double> &, bool, bool, const TS *, const double *,     \
                                                 double *, TS *, cudaStream_t);                                    \
    template cudaError_t launch_wide_moments<TS>(const Model<double> &, bool, bool, const TS *, const double *,     \
                                                 double *, TS *, TS *, TS *, cudaStream_t);
LBM_WIDE_INST(float)
LBM_WIDE_INST(double)

}  // namespace lbm
