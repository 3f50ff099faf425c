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
// No halo of 40 cells is staged and no line is walked from its start.  Lines
// whose length is no multiple of 8 end in a shorter block; with walls in y
// (Sec. 5.5) the blocks continue in mirrored order, a mirrored block's BS being
// the block's own BT.
//
// Tiles of 16 x 8 cells, 128 threads, one cell per thread: four warps reach all
// four FP64 units of an SM, and 128^2 or 1024 x 8 cells still spread over 128
// or 64 SMs.  For tau = 1 the BGK term vanishes and the equilibrium at u is
// skipped.  Both passes are launched with programmatic serialization and let
// the next grid in after their arithmetic: let in at the top, its CTAs pile up
// on the SMs that still have room (16 of them on one SM) and a grid of 128 CTAs
// runs on 30 SMs (36.8 us per 128^2 step instead of 13.2).
//
// Measured, us per step (direct stencil before -> block sums): FP64 128^2 100 ->
// 13.2, FP32 1024 x 8 35 -> 10.6; at 1024^2 pass 1 takes 92 and pass 2 159, i.e. 53
// and 92 FP64 instructions at one per 64 cycles and unit, which is the bound
// there; small lattices are left with the latency of two dependent grids.
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
    double *ys, *yt, *xs, *xt;   // block sums: ys, yt[by * nx + x]; xs, xt[y * nbx + bx]
    long long nys, nxs;      // entries of each pair
};

// The block k of a line of nb blocks, k any integer: periodic, or (mirror) the
// line continued by its mirror image, where a block's sums swap roles.
template <bool MIRROR>
__device__ __forceinline__ int block_of(int k, int nb, bool &swapped) {
    if (MIRROR) {
        const int p = 2 * nb;
        int i = k % p;
        if (i < 0) i += p;
        swapped = i >= nb;
        return swapped ? p - 1 - i : i;
    }
    swapped = false;
    if (k >= 0 && k < nb) return k;
    k %= nb;
    return k < 0 ? k + nb : k;
}

// The one-sided sum that enters block b of a line from below (dir = -1: S at
// the cell before the block, from the blocks b - 1, b - 2, ...) or above (dir =
// 1: T at the cell after it): kb blocks joined, the farthest first.  own / other:
// the line's BS and BT for dir = -1, BT and BS for dir = 1 (stride between blocks).
template <bool MIRROR>
__device__ __forceinline__ double carry_into(const double *own, const double *other, long long stride, int b, int dir,
                                             int nb, int kb, double r8, double rl, long long n, int *err) {
    auto sum_of = [&](int k, bool &last) {
        bool sw;
        const int i = block_of<MIRROR>(b + dir * k, nb, sw);
        last = i == nb - 1;
        return in_bounds(i * stride, n, err) ? (MIRROR && sw ? other : own)[i * stride] : 0.0;
    };
    double acc = 0.0;
    if (kb <= kJoin) {
        double v[kJoin];
        bool last[kJoin];
#pragma unroll
        for (int k = 0; k < kJoin; ++k) {
            v[k] = 0.0;
            last[k] = false;
            if (k < kb) v[k] = sum_of(k + 1, last[k]);
        }
#pragma unroll
        for (int k = kJoin - 1; k >= 0; --k)
            if (k < kb) acc = fma(last[k] ? rl : r8, acc, v[k]);
    } else {
        for (int k = kb; k >= 1; --k) {
            bool last;
            const double v = sum_of(k, last);
            acc = fma(last ? rl : r8, acc, v);
        }
    }
    return acc;
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
    ptx::griddep_launch_dependents();
    if (!HDM) return;
    S[ly][lx] = phi;
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool fwd = lane < 16;   // BS, else BT
    if (warp == 0) {              // columns
        const int col = lane & 15, xc = tx * TX + col;
        const int h = min(TY, ny - ty * TY);
        if (xc < nx) {
            double a = 0.0;
            if (h == TY) {
#pragma unroll
                for (int k = 0; k < TY; ++k) a = fma(A.r, a, S[fwd ? k : TY - 1 - k][col]);
            } else {
                for (int k = 0; k < h; ++k) a = fma(A.r, a, S[fwd ? k : h - 1 - k][col]);
            }
            const long long o = (long long)ty * nx + xc;
            if (in_bounds(o, A.nys, m.chk)) (fwd ? A.ys : A.yt)[o] = a;
        }
    } else if (warp == 1) {       // rows: 8 rows x 2 blocks
        const int row = lane & 7, b = (lane >> 3) & 1, yc = ty * TY + row, bx = 2 * tx + b;
        const int w = min(BK, nx - bx * BK);
        if (yc < ny && w > 0) {
            const double *s = S[row] + b * BK;
            double a = 0.0;
            if (w == BK) {
#pragma unroll
                for (int k = 0; k < BK; ++k) a = fma(A.r, a, s[fwd ? k : BK - 1 - k]);
            } else {
                for (int k = 0; k < w; ++k) a = fma(A.r, a, s[fwd ? k : w - 1 - k]);
            }
            const long long o = (long long)yc * A.nbx + bx;
            if (in_bounds(o, A.nxs, m.chk)) (fwd ? A.xs : A.xt)[o] = a;
        }
    }
}

// Pass 2: gradient of q, force (Eq. 22 / 7), exact-difference forcing with BGK
// (Eq. 1, 2, 10) and push streaming; MOM: rho and the Eq. 11 velocity instead.
template <typename TS, bool SC, bool HDM, bool TAU1, bool WALLS, bool MOM>
__global__ void __launch_bounds__(NT) wide_collide_kernel(const __grid_constant__ WideArgs A, const TS *f,
                                                          const double *q, TS *fout, TS *rho_out, TS *vx_out,
                                                          TS *vy_out) {
    constexpr int QW = TX + 2, QH = TY + 2;
    __shared__ double Q[QH][QW];                          // q over the tile and one cell around it
    __shared__ double YS[TY][TX], YT[TY][TX];             // S_(y-1), T_(y+1) along the column
    __shared__ double XS[TY][TX + 1], XT[TY][TX + 1];     // S_(x-1), T_(x+1) along the row
    const Model<double> &m = A.m;
    const int nx = m.nx, ny = m.ny;
    const long long n = (long long)nx * ny;
    const int ty = blockIdx.x / A.ntx, tx = blockIdx.x - ty * A.ntx;
    const int x0 = tx * TX, y0 = ty * TY;
    const int lx = threadIdx.x & (TX - 1), ly = threadIdx.x / TX;
    const int x = x0 + lx, y = y0 + ly;
    const bool valid = x < nx && y < ny;
    const long long c = (long long)min(y, ny - 1) * nx + min(x, nx - 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    ptx::griddep_wait();   // pass 1 has written q and the block sums

    // the rows and columns of the tile's halo: periodic, or mirrored across a wall
    for (int k = threadIdx.x; k < QH * QW; k += NT) {
        const int ry = k / QW, rx = k - ry * QW;
        const int gx = min(x0 - 1 + rx, nx), gy = min(y0 - 1 + ry, ny);
        const int px = gx < 0 ? nx - 1 : (gx == nx ? 0 : gx);
        const int py = gy < 0 ? (WALLS ? 0 : ny - 1) : (gy == ny ? (WALLS ? ny - 1 : 0) : gy);
        const long long g = (long long)py * nx + px;
        Q[ry][rx] = in_bounds(g, n, m.chk) ? q[g] : 0.0;
    }
    // warps 0 and 1: the sums that enter the tile's blocks (columns; rows)
    const bool fwd = lane < 16;
    double carry = 0.0;
    if (HDM && warp == 0) {
        const int xc = x0 + (lane & 15);
        if (xc < nx)
            carry = carry_into<WALLS>((fwd ? A.ys : A.yt) + xc, (fwd ? A.yt : A.ys) + xc, nx, ty, fwd ? -1 : 1, A.nby,
                                      A.kby, A.r8, A.ryl, A.nys - xc, m.chk);
    } else if (HDM && warp == 1) {
        const int yc = y0 + (lane & 7), bx = 2 * tx + ((lane >> 3) & 1);
        if (yc < ny && bx < A.nbx) {
            const long long o = (long long)yc * A.nbx;
            carry = carry_into<false>((fwd ? A.xs : A.xt) + o, (fwd ? A.xt : A.xs) + o, 1, bx, fwd ? -1 : 1, A.nbx,
                                      A.kbx, A.r8, A.rxl, A.nxs - o, m.chk);
        }
    }
    double fi[kQ];
#pragma unroll
    for (int i = 0; i < kQ; ++i) fi[i] = in_bounds(i * n + c, kQ * n, m.chk) ? (double)f[i * n + c] : 0.0;
    __syncthreads();
    auto mag = [](double v) { return SC ? fabs(v) : v; };
    if (HDM && warp < 2) {   // S upwards (lanes 0 .. 15), T downwards, one code path for both
        const int line = warp == 0 ? lane & 15 : lane & 7, b = warp == 0 ? 0 : (lane >> 3) & 1;
        const int len = min(BK, warp == 0 ? ny - y0 : nx - (2 * tx + b) * BK);   // cells of the block
        const double *src = warp == 0 ? &Q[1][line + 1] : &Q[line + 1][b * BK + 1];
        double *dst = warp == 0 ? &(fwd ? YS : YT)[0][line] : &(fwd ? XS : XT)[line][b * BK];
        const int step = warp == 0 ? QW : 1, dstep = warp == 0 ? TX : 1;
        double v = carry;
#pragma unroll
        for (int k = 0; k < BK; ++k) {
            const int i = fwd ? k : len - 1 - k;
            if (k < len) {
                dst[i * dstep] = v;
                if (k + 1 < BK) v = fma(A.r, v, mag(src[i * step]));
            }
        }
    }
    // moments (Eq. 3) from the sums over the populations moving east, west, north, south
    const double east = fi[1] + fi[5] + fi[8], west = fi[3] + fi[6] + fi[7];
    const double r = fi[0] + fi[2] + fi[4] + east + west;
    const double jx = east - west, jy = (fi[2] + fi[5] + fi[6]) - (fi[4] + fi[7] + fi[8]);
    const double inv = 1.0 / r;
    if (HDM) __syncthreads();
    ptx::griddep_launch_dependents();
    if (!valid) return;

    const double *p = &Q[ly + 1][lx + 1];
    double dx, dy;
    if (HDM) {
        dx = fma(A.c1, mag(p[1]) - mag(p[-1]), A.cs * (XT[ly][lx] - XS[ly][lx]));
        dy = fma(A.c1, mag(p[QW]) - mag(p[-QW]), A.cs * (YT[ly][lx] - YS[ly][lx]));
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
    a.xs = a.yt + a.nys;
    a.xt = a.xs + a.nxs;
    return a;
}

template <typename K, typename... Args>
cudaError_t launch_tiles(K kern, const WideArgs &a, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((long long)a.ntx * a.nby));
    cfg.blockDim = dim3(NT);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a, args...);
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
    return sizeof(double) * 2 * (size_t)(nby * nx + nbx * ny);
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
