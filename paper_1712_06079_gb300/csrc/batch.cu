// Batched sweep: many independent periodic lattices of uneven size, each with
// its own equation of state, temperature and relaxation time, advanced by one
// persistent cooperative launch (captured in a CUDA graph) instead of two
// launches per instance per step.
//
// One step = phase A (rho = sum f, potential field of Eq. 8/21 for every cell)
// + grid barrier + phase B (HDM/CDM gradient of the potential, force Eq. 22 /
// Eq. 7, exact-difference forcing + BGK of Eq. 1, 2, 10, periodic push
// streaming within the instance) + grid barrier.  The grid barrier is a counter
// in global memory that only grows within a launch (an arrival needs no answer,
// a wait is a poll); every wait is bounded by %globaltimer and sets
// LBM_E_TIMEOUT and an abort flag that all blocks check, so no block can spin
// forever.
//
// A batch of FP32 HDM lattices at the default radius with rows of at least 53
// cells takes the vector path: a thread holds four consecutive cells of a row (16-byte loads and
// stores; rows are pitched to four cells, the field's rows carry 32 ghost columns
// on each side), a group of 128 threads a tile of 64 x 8 cells (lattices of at
// most 8 rows) or 32 x 16.  The tile's populations are copied into shared memory
// once per step (cp.async, at the step's start) and serve both phases when every
// group has one tile; with several, phase B starts with the one that phase A ended
// with.  Phase B stages the field with its halo, takes d/dx of the four cells from
// one 60-value window in recurrence form on packed pairs (hdm_window4_paired, as the
// single-pass kernel does), d/dy likewise from windows of the columns or, on short
// columns, from the folded weights, and collides the four cells as two packed pairs.  Every other batch (FP64, or with a CDM lattice,
// another radius or a narrower row in it) takes the form this replaced: one cell a
// thread, 26 + 26 (40 + 40) taps loaded one by one.  us per step, per-cell form ->
// vector path: twenty 200^2 lattices in the grid form 86.9 -> 28.4 (waiting per
// lattice and per group instead of for the whole grid was no faster, and neither was
// starting the next tile's copy as soon as this one's populations are in registers; 1850
// instructions per thread and step); the 64-lattice sweep (616,000 cells) 41.5 -> 23 in the
// grid form, 31.8 -> 20.3 with one cluster size, 27.6 -> 17.0 as tuned (grouped).
//
// A cell's operations depend on its absolute position only (the groups of four
// start at multiples of four), packed pairs round as single operations do, and
// products that feed a sum are rounded on their own, so the grid form, the
// cluster form and the grouped form give the same bits.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <string>
#include <vector>

#include "lbm.h"
#include "lbm_internal.h"
#include "ptx.cuh"

namespace lbm {
namespace {

constexpr int kAlign = 512;       // instance offsets (in the caller's order of cells) are multiples of this many cells
constexpr int kTableGrain = 128;  // cells per entry of the cell group -> instance table
constexpr int NT = 128;           // threads of a group: one tile, or 128 cells of the per-cell path
constexpr int FK = 26;            // HDM radius of the vector path
constexpr int QG = 32;            // ghost columns on each side of the field's rows there
constexpr int XH = 28;            // staged columns on each side of a tile (the window of a group of four)

template <typename T>
struct Inst {
    Model<T> m;
    int off;  // first cell of the instance in the caller's order of cells
    int sc;   // Shan-Chen (Eq. 22) or Zhang-Chen (Eq. 7) form
    int cdm;  // CDM (Eq. 15) instead of HDM (Eq. 20)
    int vec;  // vector path (all of a batch or none)
    // on the device cell (x, y) is entry fo + y P + x of a population's plane and
    // entry qo + y QP + qx + x of the field
    int P, QP, qx;
    long long fo, qo;
};

struct BarrierState {
    unsigned int count;   // arrivals since the launch began
    int abort;
};

template <typename T>
struct BatchArgs {
    const Inst<T> *inst;
    const int4 *tiles;     // work items: instance, and first column and row of a tile or first cell (per-cell path)
    int ntiles;
    T *f[2];               // the two distribution buffers (ping-pong by step parity)
    T *q;                  // potential field
    float r, r5, r25;      // r = (sqrt 5 - 3)/2 of Eq. 20's operator and its powers (vector path)
    long long nplane, nq;  // entries of a population's plane, of the field
    int nsteps;
    int parity0;           // buffer holding the state at the first step
    int *err;
    BarrierState *bar;
    unsigned long long limit_ns;
    int skip_block;        // test hook: this block never arrives at the first barrier (-1: none)
};

__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Grid-wide barrier with a wall-time bound: the arrivals of all barriers of the
// launch are counted in one word, so an arrival needs no answer and a wait polls
// for `target` arrivals.  The CTA's barrier orders its threads' writes before thread
// 0's release, and that release before another CTA's acquire and barrier: there is no
// further fence.  Returns false if the batch was aborted
// (by a timeout here or elsewhere).
__device__ bool grid_sync(BarrierState *b, unsigned int target, int *err, unsigned long long limit_ns) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&b->count) : "memory");
        auto arrived = [&] {
            unsigned int v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&b->count) : "memory");
            return v;
        };
        volatile int *vabort = &b->abort;
        const unsigned long long t0 = gtimer();
        for (unsigned int it = 1; (int)(arrived() - target) < 0; ++it) {
            if ((it & 63) != 0) continue;
            if (*vabort) break;
            if (gtimer() - t0 > limit_ns) {
                atomicOr(err, kErrTimeout);
                atomicExch(&b->abort, 1);
                break;
            }
        }
        ok = !*vabort;
    }
    __syncthreads();
    return ok;
}

template <typename T>
__device__ __forceinline__ T qabs(T v, bool sc) {
    return sc ? fabs(v) : v;
}

// Arithmetic of one cell (float, double) or of two as a packed FP32 pair, every
// operation rounded on its own.
struct F2 {
    float2 v;
};
__device__ __forceinline__ float add_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float rcp_(float a) { return __frcp_rn(a); }
__device__ __forceinline__ double add_(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double rcp_(double a) { return __drcp_rn(a); }
__device__ __forceinline__ F2 add_(F2 a, F2 b) { return {__fadd2_rn(a.v, b.v)}; }
__device__ __forceinline__ F2 mul_(F2 a, F2 b) { return {__fmul2_rn(a.v, b.v)}; }
__device__ __forceinline__ F2 fma_(F2 a, F2 b, F2 c) { return {__ffma2_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ F2 rcp_(F2 a) { return {make_float2(__frcp_rn(a.v.x), __frcp_rn(a.v.y))}; }
template <typename V>
struct Const {
    static __device__ __forceinline__ V of(double c) { return V(c); }
};
template <>
struct Const<F2> {
    static __device__ __forceinline__ F2 of(double c) { return {make_float2((float)c, (float)c)}; }
};
template <typename V>
__device__ __forceinline__ V sub_(V a, V b) { return fma_(b, Const<V>::of(-1.0), a); }

// rho and j (Eq. 3)
template <typename V>
__device__ __forceinline__ V cell_density(const V (&f)[kQ]) {
    return add_(add_(add_(f[0], f[2]), f[4]), add_(add_(add_(f[1], f[5]), f[8]), add_(add_(f[3], f[6]), f[7])));
}
template <typename V>
__device__ __forceinline__ void cell_momentum(const V (&f)[kQ], V &jx, V &jy) {
    jx = sub_(add_(add_(f[1], f[5]), f[8]), add_(add_(f[3], f[6]), f[7]));
    jy = sub_(add_(add_(f[2], f[5]), f[6]), add_(add_(f[4], f[7]), f[8]));
}

__device__ __forceinline__ float div_(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ double div_(double a, double b) { return __ddiv_rn(a, b); }
__device__ __forceinline__ float sqrt_(float a) { return __fsqrt_rn(a); }
__device__ __forceinline__ double sqrt_(double a) { return __dsqrt_rn(a); }

// The field of the stencils at density rho: s sqrt|U| (Eq. 21, s the sign of U) or
// U (Eq. 8; equations of state Eq. 24, 27-29, or the effective mass of Eq. 4-5), as
// potential_field gives it, each operation rounded on its own.
template <typename T>
__device__ __forceinline__ T field_at(const Model<T> &m, T rho, bool sc) {
    T U;
    const T one = T(1);
    if (m.eos == LBM_EOS_PSI_EXP) {
        const T psi = sub_(one, exp(mul_(-rho, m.b)));
        U = mul_(mul_(m.a, psi), psi);
    } else {
        const T br = mul_(m.b, rho), rt = mul_(rho, m.RT);
        T p;
        if (m.eos == LBM_EOS_CS) {
            const T e = mul_(br, T(0.25)), om = sub_(one, e);
            const T num = mul_(rt, fma_(e, fma_(e, om, one), one));
            p = fma_(mul_(-m.a, rho), rho, div_(num, mul_(mul_(om, om), om)));
        } else {
            const T rep = div_(rt, sub_(one, br));
            if (m.eos == LBM_EOS_VDW) p = fma_(mul_(-m.a, rho), rho, rep);
            else p = sub_(rep, div_(mul_(mul_(m.aal, rho), rho),
                                    m.eos == LBM_EOS_PR ? fma_(br, sub_(T(2), br), one) : add_(one, br)));
        }
        U = fma_(m.k, p, mul_(rho, T(-1.0 / 3.0)));
    }
    if (!sc) return U;
    const T phi = sqrt_(U >= T(0) ? U : -U);
    return U >= T(0) ? phi : -phi;
}

// Moments (Eq. 3), exact-difference forcing (Eq. 10) and BGK (Eq. 1) with
// interaction force (Fx, Fy): f becomes the post-collision populations; the rest
// population takes rho minus the other eight.  With t = 3 e.v,
// f^eq_i = (w_i rho / 2)(2 a + t^2) + w_i rho t, 2 a = 2 - 3 |v|^2, direction and
// opposite together; for tau = 1 (om1 = 1 - omega = 0) the BGK term vanishes.
template <typename V, bool TAU1>
__device__ __forceinline__ void collide_with(V om1, V Fx, V Fy, V (&f)[kQ]) {
    const V r = cell_density(f);
    V jx, jy;
    cell_momentum(f, jx, jy);
    const V inv = rcp_(r), three = Const<V>::of(3.0), third = Const<V>::of(-1.0 / 3.0), two = Const<V>::of(2.0);
    const V ux = mul_(jx, inv), uy = mul_(jy, inv);
    const V vx = mul_(three, fma_(Fx, inv, ux)), vy = mul_(three, fma_(Fy, inv, uy));
    const V av = fma_(third, fma_(vx, vx, mul_(vy, vy)), two);
    V tx = vx, ty = vy, au = av;
    if (!TAU1) {
        tx = mul_(three, ux);
        ty = mul_(three, uy);
        au = fma_(third, fma_(tx, tx, mul_(ty, ty)), two);
    }
    V moved = Const<V>::of(0.0);
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        constexpr int kDir[4] = {1, 2, 5, 6};
        const int i = kDir[d], o = opp(i);
        const V w = mul_(r, Const<V>::of(d < 2 ? 1.0 / 9.0 : 1.0 / 36.0)), h = mul_(r, Const<V>::of(d < 2 ? 1.0 / 18.0 : 1.0 / 72.0));
        auto along = [&](V x, V y) { return d == 0 ? x : (d == 1 ? y : (d == 2 ? add_(x, y) : sub_(y, x))); };
        const V t = along(vx, vy), even = mul_(h, fma_(t, t, av)), odd = mul_(w, t);
        V pi = add_(even, odd), po = sub_(even, odd);
        if (!TAU1) {   // (1 - omega) of the distance to f^eq(u) stays
            const V tu = along(tx, ty), eu = mul_(h, fma_(tu, tu, au)), ou = mul_(w, tu);
            pi = fma_(om1, sub_(f[i], add_(eu, ou)), pi);
            po = fma_(om1, sub_(f[o], sub_(eu, ou)), po);
        }
        f[i] = pi;
        f[o] = po;
        moved = add_(moved, add_(pi, po));
    }
    f[0] = sub_(r, moved);
}
template <typename V, typename T>
__device__ __forceinline__ void collide(const Model<T> &m, V Fx, V Fy, V (&f)[kQ]) {
    const V om1 = Const<V>::of((double)(T(1) - m.omega));
    if (m.omega == T(1)) collide_with<V, true>(om1, Fx, Fy, f);
    else collide_with<V, false>(om1, Fx, Fy, f);
}

template <typename V>
__device__ __forceinline__ void force_of(bool sc, V qc, V dx, V dy, V &Fx, V &Fy) {
    const V s = sc ? mul_(Const<V>::of(-2.0), qc) : Const<V>::of(-1.0);   // Eq. 22 (q = s Phi) or Eq. 7
    Fx = mul_(s, dx);
    Fy = mul_(s, dy);
}

// Eq. 15 times 1/c_s^2; at(ox, oy): the field at an offset from the cell.
template <typename T, typename F>
__device__ __forceinline__ void cdm_gradient(F at, T &dx, T &dy) {
    const T ne = at(1, 1), nw = at(-1, 1), se = at(1, -1), sw = at(-1, -1);
    dx = fma_(T(1.0 / 3.0), sub_(at(1, 0), at(-1, 0)), mul_(T(1.0 / 12.0), sub_(add_(ne, se), add_(nw, sw))));
    dy = fma_(T(1.0 / 3.0), sub_(at(0, 1), at(0, -1)), mul_(T(1.0 / 12.0), sub_(add_(ne, nw), add_(se, sw))));
}
// One direction of the explicit periodic form of Eq. 20 (folded weights for
// short lines); at(j): the field j cells along the line.
template <typename T, typename F>
__device__ __forceinline__ T direct_derivative(const T *w, int k, F at) {
    T d = T(0);
    for (int j = 1; j <= k; ++j) d = fma_(w[j], sub_(at(j), at(-j)), d);
    return d;
}
// The derivative at four consecutive cells from the field at window positions p
// = 2 .. 57 (the cells at 28 .. 31), each value entering as its deviation from
// ref, the second cell's: hdm_window4_paired's operations, fed from the window's
// two ends inwards, pair j the positions 2 + j and 57 - j, so that a thread holds a
// few values at a time instead of the whole window (the batch kernels run at 64
// registers).
struct WindowSum {
    float2 r2, r52, mr25, S0, G, head[3], tail[4];
    __device__ WindowSum(float r, float r5, float r25)
        : r2(make_float2(r, r)), r52(make_float2(r5, r5)), mr25(make_float2(-r25, -r25)) {}
    __device__ __forceinline__ void feed(int j, float lo, float hi, float ref) {   // j = 0, 1, .., 27 in turn (a constant)
        const float2 v = make_float2(add_(lo, -ref), add_(hi, -ref));
        if (j < 3) head[j] = v;
        if (j >= 24) tail[j - 24] = v;
        if (j >= 25) return;
        G = j % 5 == 0 ? v : __ffma2_rn(r2, G, v);             // groups of five
        if (j == 4) S0 = G;
        else if (j % 5 == 4) S0 = __ffma2_rn(r52, S0, G);      // joined by r^5
    }
    __device__ __forceinline__ void finish(float w1, float w2, float (&d)[4]) {
        float2 S[4];   // S_c = (P_c, Q_(3-c))
        S[0] = S0;
#pragma unroll
        for (int c = 1; c < 4; ++c) S[c] = __ffma2_rn(mr25, head[c - 1], __ffma2_rn(r2, S[c - 1], tail[c]));
        auto at = [&](int p) { return p <= 29 ? tail[p - 26].x : tail[31 - (p - 2)].y; };   // t_p, p = 27 .. 32
#pragma unroll
        for (int c = 0; c < 4; ++c) d[c] = fma_(w1, add_(at(29 + c), -at(27 + c)), mul_(w2, add_(S[3 - c].y, -S[c].x)));
    }
};
// (a fence for the compiler: keeps it from loading the whole window ahead)
__device__ __forceinline__ void in_order() { asm volatile("" ::: "memory"); }
template <typename F>
__device__ __forceinline__ void window_derivative(F at, const float *w, float r, float r5, float r25, float (&d)[4]) {
    const float ref = at(29);
    WindowSum s(r, r5, r25);
#pragma unroll
    for (int j = 0; j < 28; ++j) {
        if (j % 8 == 0) in_order();
        s.feed(j, at(2 + j), at(57 - j), ref);
    }
    s.finish(w[1], w[2], d);
}

// Barrier of a group of 128 threads (named barrier 1 + group; 0 is the CTA's).
__device__ __forceinline__ void group_sync(int g) {
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(NT) : "memory");
}

// ---- vector path ----

// (LBM_CHECKED builds) the entries [o, o + n) lie in an array of `size` entries, shared
// memory here: a rank's own or another's, which is laid out alike.
__device__ __forceinline__ bool span_ok(long long o, int n, long long size, int *err) {
    return in_bounds(o, size, err) && in_bounds(o + n - 1, size, err);
}

// A tile, four cells a thread: 64 x 8 on lattices of at most 8 rows (THIN), else
// 32 x 16.
template <bool THIN>
struct Tile {
    static constexpr int TW = THIN ? 64 : 32, TH = THIN ? 8 : 16, GPR = TW / 4;   // GPR: groups of four per row
    static constexpr int XW = TW + 2 * XH;   // staged row: the tile and the windows' reach
};
// Shared memory of a group (floats): the populations [9][th][tw], the field's
// rows with the x halo [th][tw + 56], its columns with the y halo
// [th + 2 ky][tw] and d/dy [th][tw] where it comes from windows.
constexpr int kTileF = kQ * 4 * NT;
constexpr int tile_floats(int ny) {
    return kTileF + (ny <= 8 ? 8 * Tile<true>::XW + (8 + 6) * 64 : 16 * Tile<false>::XW + (16 + 2 * FK) * 32 + 16 * 32);
}

// Populations of the tile into shared memory.
template <bool THIN>
__device__ __forceinline__ void tile_load(const BatchArgs<float> &a, const float *f, const Inst<float> &I, const int4 &tile,
                                          float *S, int t) {
    const int row = t / Tile<THIN>::GPR, gx = t % Tile<THIN>::GPR, x = tile.y + 4 * gx, y = tile.z + row;
    if (x < I.m.nx && y < I.m.ny) {
        const long long o = I.fo + (long long)y * I.P + x;
        const float *src = f + o;
#pragma unroll
        for (int i = 0; i < kQ; ++i, src += a.nplane)
            if (in_bounds(i * a.nplane + o + 3, kQ * a.nplane, I.m.chk)) ptx::cp_async16_l2(S + (i * NT + t) * 4, src);
    }
    ptx::cp_async_wait_all();   // (each thread reads what it copied itself)
}

__device__ __forceinline__ float comp(const float4 &v, int c) { return c == 0 ? v.x : (c == 1 ? v.y : (c == 2 ? v.z : v.w)); }

// The field at the four cells whose populations are v; flags the first nc of
// them where the density is not positive and finite.
__device__ __forceinline__ void four_potentials(const Model<float> &m, bool sc, const float4 (&v)[kQ], int nc, float (&q)[4],
                                                int *err) {
    bool bad = false;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float fc[kQ];
#pragma unroll
        for (int i = 0; i < kQ; ++i) fc[i] = comp(v[i], c);
        const float r = cell_density(fc);
        bad |= c < nc && (!(r > 0.f) || !isfinite(r));
        q[c] = field_at(m, r, sc);
    }
    if (bad) atomicOr(err, kErrUnstable);
}

// Phase A of a tile: density and potential field, with the field's ghost columns.
template <bool SC, bool THIN>
__device__ __forceinline__ void tile_potential(const BatchArgs<float> &a, const Inst<float> &I, const int4 &tile,
                                               const float *S, int t) {
    const int nx = I.m.nx, row = t / Tile<THIN>::GPR, gx = t % Tile<THIN>::GPR, x = tile.y + 4 * gx, y = tile.z + row;
    if (x >= nx || y >= I.m.ny) return;
    float4 v[kQ];
#pragma unroll
    for (int i = 0; i < kQ; ++i) v[i] = *reinterpret_cast<const float4 *>(S + (i * NT + t) * 4);
    const int nc = min(4, nx - x);
    float q[4];
    four_potentials(I.m, SC, v, nc, q, a.err);
    float *qr = a.q + I.qo + (long long)y * I.QP + QG;
    auto put = [&](int xx, float val) {
        if (in_bounds(qr + xx - a.q, a.nq, I.m.chk)) qr[xx] = val;
    };
    if (nc == 4 && in_bounds(qr + x + 3 - a.q, a.nq, I.m.chk))
        *reinterpret_cast<float4 *>(qr + x) = make_float4(q[0], q[1], q[2], q[3]);
    if (nc == 4 && x >= QG && x + 3 < nx - QG) return;   // (no image in the ghost columns)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        if (c >= nc) break;
        if (nc < 4) put(x + c, q[c]);
        if (x + c < QG) put(x + c + nx, q[c]);
        if (x + c >= nx - QG) put(x + c - nx, q[c]);
    }
}

// d/dy of four cells of a row from the folded weights; c0: the first cell, pitch W.
template <bool SC>
__device__ __forceinline__ void folded_tap(float w, const float *up, const float *down, float (&dy)[4]) {
    auto mag = [](float v) { return SC ? fabsf(v) : v; };
    const float4 u = *reinterpret_cast<const float4 *>(up), d = *reinterpret_cast<const float4 *>(down);
#pragma unroll
    for (int c = 0; c < 4; ++c) dy[c] = fma_(w, sub_(mag(comp(u, c)), mag(comp(d, c))), dy[c]);
}
// (THIN: at most three taps)
template <bool SC, bool THIN>
__device__ __forceinline__ void folded_dy(const float *c0, int W, const Model<float> &m, float (&dy)[4]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) dy[c] = 0.f;
    if constexpr (THIN) {
#pragma unroll
        for (int j = 1; j <= 3; ++j)
            if (j <= m.ky) folded_tap<SC>(m.wy[j], c0 + j * W, c0 - j * W, dy);
    } else {
        for (int j = 1; j <= m.ky; ++j) folded_tap<SC>(m.wy[j], c0 + j * W, c0 - j * W, dy);
    }
}
// d/dx of four cells of a row from the staged row, w: window position 0 (28
// columns before the first cell, 16-byte aligned); the cells' field into qc.
template <bool SC>
__device__ __forceinline__ void window_dx(const float *w, const Model<float> &m, float r, float r5, float r25,
                                          float (&dx)[4], float (&qc)[4]) {
    auto mag = [](float v) { return SC ? fabsf(v) : v; };
    const float4 mid = *reinterpret_cast<const float4 *>(w + 28);
    const float ref = mag(mid.y);
    WindowSum s(r, r5, r25);
#pragma unroll
    for (int k = 0; k < 7; ++k) {   // positions 4k .. 4k+3 and 56-4k .. 59-4k
        if (k % 2 == 0) in_order();
        const float4 lo = *reinterpret_cast<const float4 *>(w + 4 * k), hi = *reinterpret_cast<const float4 *>(w + 56 - 4 * k);
        if (k > 0) {
            s.feed(4 * k - 2, mag(lo.x), mag(hi.w), ref);
            s.feed(4 * k - 1, mag(lo.y), mag(hi.z), ref);
        }
        s.feed(4 * k, mag(lo.z), mag(hi.y), ref);
        s.feed(4 * k + 1, mag(lo.w), mag(hi.x), ref);
    }
    s.feed(26, mag(mid.x), mag(mid.w), ref);
    s.feed(27, mag(mid.y), mag(mid.z), ref);
    s.finish(m.wx[1], m.wx[2], dx);
#pragma unroll
    for (int c = 0; c < 4; ++c) qc[c] = comp(mid, c);
}

// Phase B of a tile up to the forces: stages the field and leaves d/dx, d/dy
// and the field of the thread's four cells.
template <bool SC, bool THIN>
__device__ __forceinline__ void tile_gradient(const BatchArgs<float> &a, const Inst<float> &I, const int4 &tile,
                                              float *S, int t, int g, float (&dx)[4], float (&dy)[4], float (&qc)[4]) {
    constexpr int TW = Tile<THIN>::TW, TH = Tile<THIN>::TH, GPR = Tile<THIN>::GPR, XW = Tile<THIN>::XW;
    const Model<float> &m = I.m;
    const int ny = m.ny, ky = m.ky, yrows = TH + 2 * ky;
    float *X = S + kTileF, *Y = X + TH * XW, *D = Y + yrows * TW;
    const int xq = min(XW, I.QP - (QG - XH) - tile.y) / 4;   // 16-byte pieces of a row that the field has
    const int yq = min(TW, (m.nx + 3) / 4 * 4 - tile.y) / 4;
    const float *q0 = a.q + I.qo + QG + tile.y;
    for (int k = t; k < TH * (XW / 4); k += NT) {
        const int row = k / (XW / 4), c = k % (XW / 4);
        const float *src = q0 + (long long)wrap_index(tile.z + row, ny) * I.QP - XH + 4 * c;
        if (c < xq && in_bounds(src + 3 - a.q, a.nq, m.chk)) ptx::cp_async16_l2(X + row * XW + 4 * c, src);
    }
    for (int k = t; k < yrows * GPR; k += NT) {
        const int row = k / GPR, c = k % GPR;
        const float *src = q0 + (long long)wrap_index(tile.z - ky + row, ny) * I.QP + 4 * c;
        if (c < yq && in_bounds(src + 3 - a.q, a.nq, m.chk)) ptx::cp_async16_l2(Y + row * TW + 4 * c, src);
    }
    ptx::cp_async_wait_all();
    group_sync(g);
    const int row = t / GPR, gx = t % GPR;
    const long long nY = (long long)yrows * TW;
    // (the group's region holds the tile, and the window of d/dx lies in the staged row)
    if (!in_bounds(kTileF + TH * XW + nY + (!THIN && ky == FK ? TH * TW : 0) - 1, tile_floats(ny), m.chk) ||
        !span_ok(row * XW + 4 * gx, 60, TH * XW, m.chk)) {
#pragma unroll
        for (int c = 0; c < 4; ++c) dx[c] = dy[c] = qc[c] = 0.f;
        return;
    }
    bool folded = true;
    if constexpr (!THIN) {
        folded = ky != FK;
        if (!folded) {   // rows 4 rg .. 4 rg + 3 of a column each
            const int col = t & 31, rg = t >> 5, w0 = (4 * rg - 2) * TW + col;
            const float *w = Y + w0;
            float d[4];
            window_derivative([&](int p) {
                const float u = in_bounds(w0 + p * TW, nY, m.chk) ? w[p * TW] : 0.f;
                return SC ? fabsf(u) : u;
            }, m.wy, a.r, a.r5, a.r25, d);
#pragma unroll
            for (int c = 0; c < 4; ++c) D[(4 * rg + c) * TW + col] = d[c];
            group_sync(g);
            const float4 v = *reinterpret_cast<const float4 *>(D + 4 * t);
            dy[0] = v.x; dy[1] = v.y; dy[2] = v.z; dy[3] = v.w;
        }
    }
    if (folded) {
        if (span_ok(row * TW + 4 * gx, 2 * ky * TW + 4, nY, m.chk)) folded_dy<SC, THIN>(Y + (row + ky) * TW + 4 * gx, TW, m, dy);
        else
#pragma unroll
            for (int c = 0; c < 4; ++c) dy[c] = 0.f;
    }
    window_dx<SC>(X + row * XW + 4 * gx, m, a.r, a.r5, a.r25, dx, qc);
}

__device__ __forceinline__ F2 pair_of(const float4 &v, int h) {
    return {h ? make_float2(v.z, v.w) : make_float2(v.x, v.y)};
}

// Collision of four cells as two pairs, one after the other (the second pair's
// force is made to wait for the first pair's last result: interleaved, the two need
// more registers than there are).
template <bool SC>
__device__ __forceinline__ void four_collide(const Model<float> &m, float (&dx)[4], float (&dy)[4], const float (&qc)[4],
                                             F2 (&post)[2][kQ]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        F2 Fx, Fy;
        force_of(SC, F2{make_float2(qc[2 * h], qc[2 * h + 1])}, F2{make_float2(dx[2 * h], dx[2 * h + 1])},
                 F2{make_float2(dy[2 * h], dy[2 * h + 1])}, Fx, Fy);
        collide(m, Fx, Fy, post[h]);
        if (h == 0)
            asm volatile("" : "+f"(dx[2]), "+f"(dx[3]), "+f"(dy[2]), "+f"(dy[3]) : "f"(post[0][0].v.x), "f"(post[0][0].v.y));
    }
}

// Push of four cells' populations.  Those moving along x change groups by one
// cell: a group stores its own four columns with the value its neighbouring lane
// hands over; the first and last group of a run of lanes (first, last) and a
// row's shorter last group (nc < 4) store cell by cell what leaves the run.
// row(i): the row that receives population i, put(i, p, xx, v): the entry of
// column xx in it (the caller wraps).
template <typename Row, typename Put>
__device__ __forceinline__ void push_four(const F2 (&post)[2][kQ], bool valid, int nc, bool first, bool last, int x, Row row,
                                          Put put) {
    const bool full = nc == 4;
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
        const float p[4] = {post[0][i].v.x, post[0][i].v.y, post[1][i].v.x, post[1][i].v.y};
        float in = 0.f;
        if (ex(i) == 1) in = __shfl_up_sync(0xffffffffu, p[3], 1);     // the left group's last cell
        if (ex(i) == -1) in = __shfl_down_sync(0xffffffffu, p[0], 1);  // the right group's first cell
        if (!valid) continue;
        float *d = row(i);
        auto put4 = [&](float v0, float v1, float v2, float v3) {
            if (d) *reinterpret_cast<float4 *>(d + x) = make_float4(v0, v1, v2, v3);
        };
        if (ex(i) == 0) {
            if (full) put4(p[0], p[1], p[2], p[3]);
            else
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    if (c < nc) put(i, d, x + c, p[c]);
        } else if (ex(i) == 1) {
            if (!first && full) put4(in, p[0], p[1], p[2]);
            else {
                if (!first) put(i, d, x, in);
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    if (c < nc) put(i, d, x + c + 1, p[c]);
            }
            if (last && full) put(i, d, x + 4, p[3]);
        } else {
            if (!last) put4(p[1], p[2], p[3], in);
            else
#pragma unroll
                for (int c = 1; c < 4; ++c)
                    if (c < nc) put(i, d, x + c - 1, p[c]);
            if (first) put(i, d, x - 1, p[0]);
        }
    }
}

// Phase B of a tile.
template <bool SC, bool THIN>
__device__ __forceinline__ void tile_collide(const BatchArgs<float> &a, const Inst<float> &I, const int4 &tile,
                                             float *S, int t, int g, float *fo) {
    const Model<float> &m = I.m;
    float dx[4], dy[4], qc[4];
    tile_gradient<SC, THIN>(a, I, tile, S, t, g, dx, dy, qc);
    constexpr int GPR = Tile<THIN>::GPR;
    const int nx = m.nx, ny = m.ny, gx = t % GPR, x = tile.y + 4 * gx, y = tile.z + t / GPR;
    F2 post[2][kQ];
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
        const float4 v = *reinterpret_cast<const float4 *>(S + (i * NT + t) * 4);
        post[0][i] = pair_of(v, 0);
        post[1][i] = pair_of(v, 1);
    }
    four_collide<SC>(m, dx, dy, qc, post);
    float *base = fo + I.fo;
    const long long up = (long long)(y + 1 >= ny ? 0 : y + 1) * I.P, here = (long long)y * I.P,
                    down = (long long)(y == 0 ? ny - 1 : y - 1) * I.P;
    push_four(post, x < nx && y < ny, min(4, nx - x), gx == 0, gx == GPR - 1 || x + 4 >= nx, x,
              [&](int i) {
                  float *d = base + i * a.nplane + (ey(i) == 1 ? up : (ey(i) == -1 ? down : here));
                  return in_bounds(d + (min(x, nx - 1) | 3) - fo, kQ * a.nplane, m.chk) ? d : nullptr;
              },
              [&](int, float *d, int xx, float v) {
                  if (d) d[xx < 0 ? nx - 1 : (xx >= nx ? 0 : xx)] = v;
              });
}

// ---- per-cell path ----

// Density and potential field of one cell.
template <typename T>
__device__ __forceinline__ void cell_potential(const BatchArgs<T> &a, const T *f, const Inst<T> &I, int local) {
    const Model<T> &m = I.m;
    if (local >= m.nx * m.ny) return;
    const int y = local / m.nx, x = local - y * m.nx;
    const long long o = I.fo + (long long)y * I.P + x, k = I.qo + (long long)y * I.QP + I.qx + x;
    T fi[kQ];
#pragma unroll
    for (int i = 0; i < kQ; ++i) fi[i] = in_bounds(i * a.nplane + o, kQ * a.nplane, m.chk) ? __ldcg(f + i * a.nplane + o) : T(0);
    const T r = cell_density(fi);
    if (!(r > T(0)) || !isfinite(r)) atomicOr(a.err, kErrUnstable);
    if (in_bounds(k, a.nq, m.chk)) a.q[k] = field_at(m, r, I.sc != 0);
}

// Populations and interaction force of the cell at (x, y).
template <typename T>
__device__ __forceinline__ void cell_force(const BatchArgs<T> &a, const T *f, const Inst<T> &I, int x, int y,
                                           T (&fi)[kQ], T &Fx, T &Fy) {
    const Model<T> &m = I.m;
    const bool sc = I.sc != 0;
    const T *q = a.q + I.qo + I.qx;
    // (written by other SMs before the barrier, whose acquire orders plain loads too: the taps
    // of neighbouring cells overlap, and L1 serves them)
    auto q_at = [&](int xx, int yy) { return q[(long long)yy * I.QP + xx]; };
    auto phi = [&](int xx, int yy) { return qabs(q_at(xx, yy), sc); };
    auto wrap1 = [](int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); };
    T dx, dy;
    if (I.cdm) {
        cdm_gradient<T>([&](int ox, int oy) { return phi(wrap1(x + ox, m.nx), wrap1(y + oy, m.ny)); }, dx, dy);
    } else {
        dx = direct_derivative(m.wx, m.kx, [&](int j) { return phi(wrap1(x + j, m.nx), y); });
        dy = direct_derivative(m.wy, m.ky, [&](int j) { return phi(x, wrap1(y + j, m.ny)); });
    }
    force_of(sc, q_at(x, y), dx, dy, Fx, Fy);
    const long long o = I.fo + (long long)y * I.P + x;
#pragma unroll
    for (int i = 0; i < kQ; ++i) fi[i] = in_bounds(i * a.nplane + o, kQ * a.nplane, m.chk) ? __ldcg(f + i * a.nplane + o) : T(0);
}

template <typename T>
__device__ __forceinline__ void cell_collide(const BatchArgs<T> &a, const T *f, const Inst<T> &I, int local, T *fo) {
    const Model<T> &m = I.m;
    if (local >= m.nx * m.ny) return;
    const int y = local / m.nx, x = local - y * m.nx;
    T fi[kQ], Fx, Fy;
    cell_force(a, f, I, x, y, fi, Fx, Fy);
    collide(m, Fx, Fy, fi);
    const int xp = x + 1 == m.nx ? 0 : x + 1, xm = x == 0 ? m.nx - 1 : x - 1;
    const int yp = y + 1 == m.ny ? 0 : y + 1, ym = y == 0 ? m.ny - 1 : y - 1;
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
        const int dxs = ex(i) == 1 ? xp : (ex(i) == -1 ? xm : x);
        const int dys = ey(i) == 1 ? yp : (ey(i) == -1 ? ym : y);
        const long long k = i * a.nplane + I.fo + (long long)dys * I.P + dxs;
        if (in_bounds(k, kQ * a.nplane, m.chk)) fo[k] = fi[i];
    }
}

// Persistent kernel of the grid form; VEC: a batch on the vector path.
// Registers: shared memory lets three blocks of 256 threads of the vector path onto an
// SM, so they may take 80 (at 64 it spilled 450 bytes: twenty 200^2 lattices 31.6 -> 28.4
// us per step, the 64-lattice sweep 25.9 -> 23); the per-cell path keeps 1280 (FP32) or
// 1152 (FP64) threads resident.
template <typename T, bool VEC>
__global__ void __maxnreg__(VEC ? 80 : (sizeof(T) == 4 ? 48 : 56)) batch_kernel(const BatchArgs<T> a, int floats) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int g = threadIdx.x / NT, t = threadIdx.x & (NT - 1);
    float *S = reinterpret_cast<float *>(smem_raw) + (size_t)g * floats;
    const unsigned int nblocks = gridDim.x;
    const int first = g * (int)nblocks + (int)blockIdx.x, stride = (int)nblocks * (blockDim.x / NT);
    const int last = first + (a.ntiles - 1 - first) / stride * stride;   // its populations stay for phase B, which goes backwards
    unsigned int target = 0;
    for (int step = 0; step < a.nsteps; ++step) {
        const bool odd = ((a.parity0 + step) & 1) != 0;  // (a select, not a dynamic index into the parameters)
        const T *f = odd ? a.f[1] : a.f[0];
        T *fo = odd ? a.f[0] : a.f[1];
        for (int k = first; k < a.ntiles; k += stride) {
            const int4 tile = a.tiles[k];
            const Inst<T> &I = a.inst[tile.x];
            if constexpr (VEC) {
                const bool thin = I.m.ny <= 8;
                if (thin) tile_load<true>(a, f, I, tile, S, t);
                else tile_load<false>(a, f, I, tile, S, t);
                if (thin) I.sc ? tile_potential<true, true>(a, I, tile, S, t) : tile_potential<false, true>(a, I, tile, S, t);
                else I.sc ? tile_potential<true, false>(a, I, tile, S, t) : tile_potential<false, false>(a, I, tile, S, t);
            } else {
                cell_potential(a, f, I, tile.y + t);
            }
        }
        if (step == 0 && (int)blockIdx.x == a.skip_block) return;  // test hook: never arrive
        if (!grid_sync(a.bar, target += nblocks, a.err, a.limit_ns)) return;
        for (int k = first < a.ntiles ? last : -1; k >= 0; k -= stride) {
            const int4 tile = a.tiles[k];
            const Inst<T> &I = a.inst[tile.x];
            if constexpr (VEC) {
                const bool thin = I.m.ny <= 8;
                if (k != last) {
                    if (thin) tile_load<true>(a, f, I, tile, S, t);
                    else tile_load<false>(a, f, I, tile, S, t);
                }
                if (thin) I.sc ? tile_collide<true, true>(a, I, tile, S, t, g, fo)
                                      : tile_collide<false, true>(a, I, tile, S, t, g, fo);
                else I.sc ? tile_collide<true, false>(a, I, tile, S, t, g, fo)
                          : tile_collide<false, false>(a, I, tile, S, t, g, fo);
                group_sync(g);   // (the next tile overwrites the shared field)
            } else {
                cell_collide(a, f, I, tile.y + t, fo);
            }
        }
        if (!grid_sync(a.bar, target += nblocks, a.err, a.limit_ns)) return;
    }
}

// Cluster form: one thread-block cluster of C CTAs per instance, with the
// instance's state on chip for the whole launch.  On the per-cell path CTA rank k
// owns the columns [k nx / C, (k + 1) nx / C) of every row (widths differ by one at most); its two distribution buffers and
// its potential field (with hx halo columns on each side) live in shared
// memory.  One step: phase A (rho and the potential field of the owned cells),
// a cluster barrier, the halo columns copied from the neighbouring ranks'
// shared memory (ranks k - 1 and k + 1 modulo C: x is periodic), phase B
// (gradient, force, forcing + BGK, push streaming: a population that leaves
// the owned columns is stored into the neighbour's buffer), a cluster barrier.
// Global f is read before the first step and written after the last.  The
// only waits are the cluster barriers, reached the same number of times by
// every thread, and no CTA exits before the last barrier, so no access reaches
// the shared memory of a CTA that has left.  The per-cell arithmetic is the
// grid form's, term for term.
template <typename T>
struct ClusterArgs {
    const Inst<T> *inst;
    const int *order;  // instance of each cluster: largest first, so no large one starts last
    const T *fin;    // state at the first step
    T *fout;         // receives the state after nsteps (may be fin)
    float r, r5, r25;   // as in BatchArgs
    long long nplane;
    int nsteps;
    int *err;
};

template <typename T>
__global__ void __launch_bounds__(1024) cluster_batch_kernel(const ClusterArgs<T> a) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int C = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();
    const Inst<T> &I = a.inst[a.order[blockIdx.x / C]];   // clusters lie along x, one per instance
    const Model<T> &m = I.m;
    const bool sc = I.sc != 0, cdm = I.cdm != 0;
    const int nx = m.nx, ny = m.ny;
    // rank k owns columns [k nx / C, (k + 1) nx / C): widths differ by one at
    // most; every rank lays its slice out with the pitch of the widest, so a
    // neighbour's element sits at the same offset in every CTA
    const int x0 = (int)((long long)rank * nx / C), w = (int)((long long)(rank + 1) * nx / C) - x0;
    const int wmax = (nx + C - 1) / C;
    const int hx = cdm ? 1 : m.kx;
    const int W = wmax + 2 * hx;                // potential row pitch
    const int ncell = w * ny;                   // owned cells
    const int plane = wmax * ny;                // distribution plane stride
    T *fa = reinterpret_cast<T *>(smem_raw);   // [kQ][ny][wmax]
    T *fb = fa + (size_t)kQ * plane;
    T *ph = fb + (size_t)kQ * plane;           // [ny][W], owned column xl at hx + xl
    const int left = rank == 0 ? C - 1 : rank - 1, right = rank == C - 1 ? 0 : rank + 1;
    const int wl = (int)((long long)(left + 1) * nx / C) - (int)((long long)left * nx / C);   // the left rank's width

    for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
        const int y = c / w, xl = c - y * w;
        const long long g = I.fo + (long long)y * I.P + x0 + xl;
#pragma unroll
        for (int i = 0; i < kQ; ++i)
            if (in_bounds(i * a.nplane + g, kQ * a.nplane, m.chk)) fa[i * plane + y * wmax + xl] = a.fin[i * a.nplane + g];
    }
    __syncthreads();
    for (int step = 0; step < a.nsteps; ++step) {
        // ---- phase A: density and potential field of the owned cells ----
        for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
            const int y = c / w, xl = c - y * w;
            T fi[kQ];
#pragma unroll
            for (int i = 0; i < kQ; ++i) fi[i] = fa[i * plane + y * wmax + xl];
            const T r = cell_density(fi);
            if (!(r > T(0)) || !isfinite(r)) atomicOr(a.err, kErrUnstable);
            ph[y * W + hx + xl] = field_at(m, r, sc);
        }
        cluster.sync();
        // ---- halo: the left neighbour's columns wl - hx .. wl - 1, the right one's 0 .. hx - 1 ----
        {
            const T *pl = cluster.map_shared_rank(ph, left);
            const T *pr = cluster.map_shared_rank(ph, right);
            const int nh = hx * ny;
            for (int c = threadIdx.x; c < 2 * nh; c += blockDim.x) {
                const int side = c < nh ? 0 : 1, k = c - side * nh;
                const int y = k / hx, j = k - y * hx;
                if (side == 0) ph[y * W + j] = pl[y * W + wl + j];
                else ph[y * W + hx + w + j] = pr[y * W + hx + j];
            }
        }
        __syncthreads();
        // ---- phase B: gradient, force, forcing + BGK, push streaming ----
        T *fbl = cluster.map_shared_rank(fb, left);
        T *fbr = cluster.map_shared_rank(fb, right);
        for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
            const int y = c / w, xl = c - y * w;
            const T *row = ph + y * W + hx + xl;   // row[j]: the field at column xl + j
            auto wrapy = [&](int i) { return i < 0 ? i + ny : (i >= ny ? i - ny : i); };
            auto column = [&](int j) { return qabs(ph[wrapy(y + j) * W + hx + xl], sc); };
            T dx, dy, Fx, Fy;
            if (cdm) {
                cdm_gradient<T>([&](int ox, int oy) { return qabs(ph[wrapy(y + oy) * W + hx + xl + ox], sc); }, dx, dy);
            } else {
                dx = direct_derivative(m.wx, m.kx, [&](int j) { return qabs(row[j], sc); });
                dy = direct_derivative(m.wy, m.ky, column);
            }
            force_of(sc, row[0], dx, dy, Fx, Fy);
            T post[kQ];
#pragma unroll
            for (int i = 0; i < kQ; ++i) post[i] = fa[i * plane + y * wmax + xl];
            collide(m, Fx, Fy, post);
            const int yp = y + 1 == ny ? 0 : y + 1, ym = y == 0 ? ny - 1 : y - 1;
#pragma unroll
            for (int i = 1; i < kQ; ++i) {
                const int dys = ey(i) == 1 ? yp : (ey(i) == -1 ? ym : y);
                const int xd = xl + ex(i);
                T *dst = xd < 0 ? fbl : (xd >= w ? fbr : fb);
                const int xc = xd < 0 ? wl - 1 : (xd >= w ? 0 : xd);
                if (in_bounds(i * plane + dys * wmax + xc, (long long)kQ * plane, m.chk))
                    dst[i * plane + dys * wmax + xc] = post[i];   // own buffer or a neighbour's (same layout)
            }
            fb[y * wmax + xl] = post[0];
        }
        cluster.sync();
        T *t = fa;
        fa = fb;
        fb = t;
    }
    for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
        const int y = c / w, xl = c - y * w;
        const long long g = I.fo + (long long)y * I.P + x0 + xl;
#pragma unroll
        for (int i = 0; i < kQ; ++i)
            if (in_bounds(i * a.nplane + g, kQ * a.nplane, m.chk)) a.fout[i * a.nplane + g] = fa[i * plane + y * wmax + xl];
    }
}

// Cluster form of the vector path: a thread per group of four cells of a row, for
// the whole launch (as many threads as a CTA's slice has groups).  The slices are
// whole groups, CTA rank k owns the groups [k ng / C, (k + 1) ng / C).  The
// populations lie in shared memory as the collision leaves them, unstreamed, and a
// step begins by pulling f(t) from the neighbouring cells (for the slice's first and
// last groups from the neighbouring ranks); once every rank has pulled, a thread
// writes only its own cells.  So one buffer is enough, which halves the shared
// memory of a CTA, so that twice the clusters are resident, and no store crosses a
// slice's edge.  One step: f(t) pulled, rho and the field of the own cells; cluster
// barrier; f(t) kept in the own cells' entries, 28 field columns read from the ranks
// on each side; d/dx from a window of the staged row, d/dy from the folded weights
// or from windows of the columns; collision as two packed pairs into the own
// entries; cluster barrier.
constexpr int kPieces = 2 * XH / 4 + 1;   // pieces of the field's halo per row (cluster_vec_steps)
struct SliceShape {   // shared memory of a CTA (floats), for the widest slice of ngm groups
    int ngm, wf, wp;  // groups; row pitch of a population, of the field
    __host__ __device__ SliceShape(int nx, int C) : ngm(((nx + 3) / 4 + C - 1) / C), wf(4 * ngm), wp(4 * ngm + 2 * XH) {}
    __host__ __device__ size_t floats(int ny, bool windows_y) const {
        return (size_t)ny * (kQ * wf + wp + (windows_y ? wf : 0));
    }
};

// A CTA's slice of an instance.
struct Slice {
    int C, rank, ng, nx, x0, w, ngw;
    __device__ int group0(int k) const { return k * ng / C; }   // first group of rank k (a slice fits a CTA: no overflow)
    __device__ Slice(int nx_, int C_, int rank_) : C(C_), rank(rank_), ng((nx_ + 3) / 4), nx(nx_) {
        x0 = 4 * group0(rank);
        ngw = group0(rank + 1) - group0(rank);
        w = min(nx - x0, 4 * ngw);
    }
    __device__ int owner(int x) const { return ((x / 4 + 1) * C - 1) / ng; }   // rank of column x
};

// The field's halo, 28 columns to each side, in pieces of four columns: of each row 7 on
// the left and 7 on the right, from the end of the last group, and the columns that a
// shorter last group lacks (its window, laid out for four cells, reads what the grid
// form's ghost columns hold there).  A piece lies in a run of some rank's columns, or ends
// in the next rank's; in row 0 that of piece j:
struct Piece {
    const float *src, *src2;   // its first column, and column 0 of the next rank less `have`
    int col, n, have;          // first column in this rank's rows, length, columns of the first run
    int whole;                 // four columns on 16 bytes
};
__device__ __forceinline__ Piece piece_of(float *ph, const Slice &sl, int j, int wp, int *err) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int nx = sl.nx;
    Piece p;
    p.col = j < XH / 4 ? 4 * j - XH : (j < XH / 2 ? 4 * (sl.ngw + j) - XH : sl.w);
    p.n = j < XH / 2 ? 4 : 4 * sl.ngw - sl.w;
    const int xx = sl.x0 + p.col, xg = xx < 0 ? xx + nx : (xx >= nx ? xx - nx : xx), rk = sl.owner(xg);
    const int next = rk + 1 == sl.C ? 0 : rk + 1;
    p.have = min(p.n, (next == 0 ? nx : 4 * sl.group0(next)) - xg);
    p.whole = p.n == 4 && p.have == 4 && (xg & 3) == 0;
    p.src = cluster.map_shared_rank(ph + XH + (xg - 4 * sl.group0(rk)), rk);
    p.src2 = cluster.map_shared_rank(ph + XH, next) - p.have;
    // (within the rows, here and there, whose pitch every rank shares; a row is one of ny)
    if (p.n > 0 && !(span_ok(XH + p.col, p.n, wp, err) && span_ok(XH + xg - 4 * sl.group0(rk), p.have, wp, err) &&
                     span_ok(XH, max(1, p.n - p.have), wp, err)))
        p.n = p.whole = 0;
    return p;
}
// The copies of a step, every row by the pieces of row 0.  Column by column, with the
// place of all but a thread's first found again in every step, short slices took seven rounds;
// and a call of its own, so that its few values do not spill those of the step (bytes of
// spills in the four variants of 64 registers 1148 -> 520).  us per step: 16 x (128 x 8)
// 5.0 -> 4.0, 64 x (250 x 8) 5.8 -> 5.1, the 64-lattice sweep (grouped) 18.7 -> 17.0.
__device__ __noinline__ void copy_halo(float *ph, int wp, int ny, const Piece *pieces) {
    for (int k = threadIdx.x; k < ny * kPieces; k += blockDim.x) {
        const int ry = k / kPieces;
        const Piece &p = pieces[k - ry * kPieces];
        float *dst = ph + ry * wp + XH + p.col;
        const float *src = p.src + ry * wp;
        if (p.whole) {
            *reinterpret_cast<float4 *>(dst) = *reinterpret_cast<const float4 *>(src);
            continue;
        }
        const float *src2 = p.src2 + ry * wp;
        const int n = p.n, have = p.have;
        float v[4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (c < n) v[c] = (c < have ? src : src2)[c];
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (c < n) dst[c] = v[c];
    }
}

template <bool SC, bool THIN>
__device__ __forceinline__ void cluster_vec_steps(const ClusterArgs<float> &a, const Inst<float> &I, float *F, Piece *pieces) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const Model<float> &m = I.m;
    const int ny = m.ny;
    const Slice sl(m.nx, (int)cluster.num_blocks(), (int)cluster.block_rank());
    const SliceShape sh(m.nx, sl.C);
    const int plane = ny * sh.wf, nx = sl.nx, x0 = sl.x0, w = sl.w;
    float *ph = F + kQ * plane, *D = ph + ny * sh.wp;
    const int nF = kQ * plane, nP = ny * sh.wp, nD = ny * sh.wf;   // entries of each (checked build)
    const int left = sl.rank == 0 ? sl.C - 1 : sl.rank - 1, right = sl.rank == sl.C - 1 ? 0 : sl.rank + 1;
    const int t = threadIdx.x, row = t / sl.ngw, gx = t - row * sl.ngw, lane = t & 31;
    const bool valid = row < ny;
    const int y = min(row, ny - 1), xs = 4 * gx, nc = min(4, w - xs);   // xs: column within the slice
    const int wl = (left == sl.C - 1 ? nx : 4 * sl.group0(left + 1)) - 4 * sl.group0(left);   // the left rank's width
    // the cells beside the group's first and last, where another lane of the warp does not hold them
    const bool first = gx == 0 || lane == 0, last = gx == sl.ngw - 1 || lane == 31;
    const float *Le = gx == 0 ? cluster.map_shared_rank(F, left) + wl - 1 : F + xs - 1;
    const float *Re = gx == sl.ngw - 1 ? cluster.map_shared_rank(F, right) : F + xs + 4;
    const int up = (y + 1 >= ny ? 0 : y + 1) * sh.wf, here = y * sh.wf, down = (y == 0 ? ny - 1 : y - 1) * sh.wf;
    float *pr = ph + y * sh.wp + XH + xs;
    if (t < kPieces) pieces[t] = piece_of(ph, sl, t, sh.wp, m.chk);   // (read after the first step's cluster barrier)

    for (int step = 0; step < a.nsteps; ++step) {
        float4 f4[kQ];
#pragma unroll
        for (int i = 0; i < kQ; ++i) {   // f_i(x) = post_i(x - e_i)
            const int o = i * plane + (ey(i) == 1 ? down : (ey(i) == -1 ? up : here));
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (span_ok(o + xs, 4, nF, m.chk)) v = *reinterpret_cast<const float4 *>(F + o + xs);
            if (ex(i) == 1) {
                float l = __shfl_up_sync(0xffffffffu, v.w, 1);
                if (first && in_bounds(o + (gx == 0 ? wl : xs) - 1, nF, m.chk)) l = Le[o];
                v = make_float4(l, v.x, v.y, v.z);
            } else if (ex(i) == -1) {
                float r = __shfl_down_sync(0xffffffffu, v.x, 1);
                if (last && in_bounds(o + (gx == sl.ngw - 1 ? 0 : xs + 4), nF, m.chk)) r = Re[o];
                v = make_float4(v.y, v.z, v.w, r);
                if (nc == 1) v.x = r;   // (a row's shorter last group)
                if (nc == 2) v.y = r;
                if (nc == 3) v.z = r;
            }
            f4[i] = v;
        }
        float q[4];
        four_potentials(m, SC, f4, valid ? nc : 0, q, a.err);
        if (valid && span_ok(pr - ph, nc, nP, m.chk)) {
            if (nc == 4) *reinterpret_cast<float4 *>(pr) = make_float4(q[0], q[1], q[2], q[3]);
            else
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    if (c < nc) pr[c] = q[c];
        }
        cluster.sync();   // every rank has pulled, and formed its field
        if (valid)
#pragma unroll
            for (int i = 0; i < kQ; ++i)
                if (span_ok(i * plane + here + xs, 4, nF, m.chk)) *reinterpret_cast<float4 *>(F + i * plane + here + xs) = f4[i];
        copy_halo(ph, sh.wp, ny, pieces);
        __syncthreads();
        float dx[4], dy[4], qc[4];
        if (THIN || m.ky != FK) {
#pragma unroll
            for (int c = 0; c < 4; ++c) dy[c] = 0.f;
            int yp = y, ym = y;
            auto tap = [&](float wj) {   // (folded_dy on the wrapped rows)
                yp = yp + 1 == ny ? 0 : yp + 1;
                ym = ym == 0 ? ny - 1 : ym - 1;
                if (span_ok(yp * sh.wp + XH + xs, 4, nP, m.chk) && span_ok(ym * sh.wp + XH + xs, 4, nP, m.chk))
                    folded_tap<SC>(wj, ph + yp * sh.wp + XH + xs, ph + ym * sh.wp + XH + xs, dy);
            };
            if constexpr (THIN) {
#pragma unroll
                for (int j = 1; j <= 3; ++j)
                    if (j <= m.ky) tap(m.wy[j]);
            } else {
                for (int j = 1; j <= m.ky; ++j) tap(m.wy[j]);
            }
        } else {
            for (int k = t; k < w * ((ny + 3) / 4); k += blockDim.x) {
                const int rg = k / w, xl = k - rg * w;
                float d[4];
                window_derivative([&](int p) {
                    const int o = wrap_index(4 * rg - 28 + p, ny) * sh.wp + XH + xl;
                    const float u = in_bounds(o, nP, m.chk) ? ph[o] : 0.f;
                    return SC ? fabsf(u) : u;
                }, m.wy, a.r, a.r5, a.r25, d);
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (4 * rg + c < ny && in_bounds((4 * rg + c) * sh.wf + xl, nD, m.chk)) D[(4 * rg + c) * sh.wf + xl] = d[c];
            }
            __syncthreads();
            float4 d4 = make_float4(0.f, 0.f, 0.f, 0.f);
            if (span_ok(here + xs, 4, nD, m.chk)) d4 = *reinterpret_cast<const float4 *>(D + here + xs);
            dy[0] = d4.x; dy[1] = d4.y; dy[2] = d4.z; dy[3] = d4.w;
        }
        if (span_ok(pr - XH - ph, 60, nP, m.chk)) window_dx<SC>(pr - XH, m, a.r, a.r5, a.r25, dx, qc);
        else
#pragma unroll
            for (int c = 0; c < 4; ++c) dx[c] = qc[c] = 0.f;
        F2 post[2][kQ];
#pragma unroll
        for (int i = 0; i < kQ; ++i) {
            float4 v4 = make_float4(0.f, 0.f, 0.f, 0.f);
            if (span_ok(i * plane + here + xs, 4, nF, m.chk)) v4 = *reinterpret_cast<const float4 *>(F + i * plane + here + xs);
            post[0][i] = pair_of(v4, 0);
            post[1][i] = pair_of(v4, 1);
        }
        four_collide<SC>(m, dx, dy, qc, post);
        if (valid)
#pragma unroll
            for (int i = 0; i < kQ; ++i)
                if (span_ok(i * plane + here + xs, 4, nF, m.chk))
                    *reinterpret_cast<float4 *>(F + i * plane + here + xs) =
                        make_float4(post[0][i].v.x, post[0][i].v.y, post[1][i].v.x, post[1][i].v.y);
        cluster.sync();
    }
}

template <int MAXT, int PER>
__global__ void __launch_bounds__(MAXT, PER) cluster_vec_kernel(const ClusterArgs<float> a) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Piece pieces[kPieces];
    float *F = reinterpret_cast<float *>(smem_raw);
    const Inst<float> &I = a.inst[a.order[blockIdx.x / cluster.num_blocks()]];
    const int nx = I.m.nx, ny = I.m.ny;
    const Slice sl(nx, (int)cluster.num_blocks(), (int)cluster.block_rank());
    const SliceShape sh(nx, sl.C);
    const int plane = ny * sh.wf;
    // the entry of post_i at the cell that population i of cell (x, y) came from
    // is where f_i is kept between launches' steps: x - e_i, on whatever rank
    auto source = [&](int i, int xl, int y) {
        const int yy = y - ey(i) < 0 ? ny - 1 : (y - ey(i) >= ny ? 0 : y - ey(i)), xx = sl.x0 + xl - ex(i);
        const int xg = xx < 0 ? nx - 1 : (xx >= nx ? 0 : xx), rk = sl.owner(xg);
        const int e = i * plane + yy * sh.wf + (xg - 4 * sl.group0(rk));
        float *o = F + (in_bounds(e, (long long)kQ * plane, I.m.chk) ? e : 0);
        return rk == sl.rank ? o : cluster.map_shared_rank(o, rk);
    };
    for (int c = threadIdx.x; c < kQ * plane; c += blockDim.x) F[c] = 1.f;   // (columns past a shorter slice: computed on, dropped)
    cluster.sync();
    for (int c = threadIdx.x; c < ny * sl.w; c += blockDim.x) {
        const int y = c / sl.w, xl = c - y * sl.w;
        const long long g = I.fo + (long long)y * I.P + sl.x0 + xl;
#pragma unroll
        for (int i = 0; i < kQ; ++i)
            if (in_bounds(i * a.nplane + g, kQ * a.nplane, I.m.chk)) *source(i, xl, y) = a.fin[i * a.nplane + g];
    }
    cluster.sync();
    if (ny <= 8) I.sc ? cluster_vec_steps<true, true>(a, I, F, pieces) : cluster_vec_steps<false, true>(a, I, F, pieces);
    else I.sc ? cluster_vec_steps<true, false>(a, I, F, pieces) : cluster_vec_steps<false, false>(a, I, F, pieces);
    for (int c = threadIdx.x; c < ny * sl.w; c += blockDim.x) {
        const int y = c / sl.w, xl = c - y * sl.w;
        const long long g = I.fo + (long long)y * I.P + sl.x0 + xl;
#pragma unroll
        for (int i = 0; i < kQ; ++i)
            if (in_bounds(i * a.nplane + g, kQ * a.nplane, I.m.chk)) a.fout[i * a.nplane + g] = *source(i, xl, y);
    }
    cluster.sync();   // (no rank leaves while another reads its memory)
}

// The cell of the caller's order at a padded index: its instance and its entry of
// a population's plane; false for padding.
template <typename T>
__device__ __forceinline__ bool find_cell(const Inst<T> *inst, const int *table, long long cell, long long &entry) {
    const int ii = table[cell / kTableGrain];
    if (ii < 0) return false;
    const Inst<T> &I = inst[ii];
    const int local = (int)(cell - I.off);   // (an instance has at most 2^30 cells and its padding)
    if (local >= I.m.nx * I.m.ny) return false;
    entry = I.fo + local;
    if (I.P != I.m.nx) entry += (long long)(local / I.m.nx) * (I.P - I.m.nx);   // padded rows
    return true;
}

template <typename T>
__global__ void batch_init_kernel(const Inst<T> *inst, const int *table, const T *rho, T *f, long long ntot,
                                  long long nplane) {
    for (long long cell = blockIdx.x * (long long)blockDim.x + threadIdx.x; cell < ntot;
         cell += (long long)gridDim.x * blockDim.x) {
        long long k;
        if (!find_cell(inst, table, cell, k)) continue;
#pragma unroll
        for (int i = 0; i < kQ; ++i) f[i * nplane + k] = rho[cell] * wq<T>(i);  // f^eq(rho, 0), Eq. 2
    }
}

template <typename T>
__global__ void batch_density_kernel(const Inst<T> *inst, const int *table, const T *f, T *rho, long long ntot,
                                     long long nplane) {
    for (long long cell = blockIdx.x * (long long)blockDim.x + threadIdx.x; cell < ntot;
         cell += (long long)gridDim.x * blockDim.x) {
        long long k;
        if (!find_cell(inst, table, cell, k)) continue;
        T fi[kQ];
#pragma unroll
        for (int i = 0; i < kQ; ++i) fi[i] = f[i * nplane + k];
        rho[cell] = cell_density(fi);
    }
}

// Phase A of the step as a launch of its own (for lbm_batch_moments), one work
// item per block.
template <typename T>
__global__ void __launch_bounds__(NT) batch_potential_kernel(const BatchArgs<T> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int4 tile = a.tiles[blockIdx.x];
    const Inst<T> &I = a.inst[tile.x];
    const T *f = a.parity0 ? a.f[1] : a.f[0];
    if constexpr (sizeof(T) == 4) {
        if (I.vec) {
            float *S = reinterpret_cast<float *>(smem_raw);
            const bool thin = I.m.ny <= 8;
            const int t = threadIdx.x;
            if (thin) tile_load<true>(a, f, I, tile, S, t);
            else tile_load<false>(a, f, I, tile, S, t);
            if (thin) I.sc ? tile_potential<true, true>(a, I, tile, S, t) : tile_potential<false, true>(a, I, tile, S, t);
            else I.sc ? tile_potential<true, false>(a, I, tile, S, t) : tile_potential<false, false>(a, I, tile, S, t);
            return;
        }
    }
    cell_potential(a, f, I, tile.y + threadIdx.x);
}

// rho (Eq. 3) and the half-step velocity v = (sum_i e_i f_i + F/2) / rho of
// Eq. 11, with F the step's interaction force from the potential field, in the
// caller's order of cells.
template <typename T>
__global__ void __launch_bounds__(NT) batch_moments_kernel(const BatchArgs<T> a, T *rho, T *vx, T *vy) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int4 tile = a.tiles[blockIdx.x];
    const Inst<T> &I = a.inst[tile.x];
    const T *f = a.parity0 ? a.f[1] : a.f[0];
    const int nx = I.m.nx, ny = I.m.ny, t = threadIdx.x;
    auto put = [&](long long cell, const T (&fi)[kQ], T Fx, T Fy) {
        const T r = cell_density(fi);
        T jx, jy;
        cell_momentum(fi, jx, jy);
        rho[cell] = r;
        vx[cell] = fma_(T(0.5), Fx, jx) / r;
        vy[cell] = fma_(T(0.5), Fy, jy) / r;
    };
    if constexpr (sizeof(T) == 4) {
        if (I.vec) {
            float *S = reinterpret_cast<float *>(smem_raw), dx[4], dy[4], qc[4];
            if (ny <= 8) tile_load<true>(a, f, I, tile, S, t);
            else tile_load<false>(a, f, I, tile, S, t);
            if (ny <= 8) I.sc ? tile_gradient<true, true>(a, I, tile, S, t, 0, dx, dy, qc)
                              : tile_gradient<false, true>(a, I, tile, S, t, 0, dx, dy, qc);
            else I.sc ? tile_gradient<true, false>(a, I, tile, S, t, 0, dx, dy, qc)
                      : tile_gradient<false, false>(a, I, tile, S, t, 0, dx, dy, qc);
            const int gpr = ny <= 8 ? Tile<true>::GPR : Tile<false>::GPR;
            const int row = t / gpr, x = tile.y + 4 * (t - row * gpr), y = tile.z + row;
            if (y >= ny) return;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (x + c >= nx) break;
                float fi[kQ], Fx, Fy;
#pragma unroll
                for (int i = 0; i < kQ; ++i) fi[i] = S[(i * NT + t) * 4 + c];
                force_of(I.sc != 0, qc[c], dx[c], dy[c], Fx, Fy);
                put(I.off + (long long)y * nx + x + c, fi, Fx, Fy);
            }
            return;
        }
    }
    const int local = tile.y + t;
    if (local >= nx * ny) return;
    T fi[kQ], Fx, Fy;
    cell_force(a, f, I, local % nx, local / nx, fi, Fx, Fy);
    put(I.off + local, fi, Fx, Fy);
}

}  // namespace
}  // namespace lbm

using namespace lbm;

struct lbm_batch {
    int n = 0;
    int prec = LBM_F32;
    size_t esz = 4;
    long long ntot = 0;
    std::vector<lbm_params> params;
    std::vector<long long> off;
    void *inst_dev = nullptr;
    int *table_dev = nullptr;
    int4 *tiles_dev = nullptr;     // work items of the grid form
    int ntiles = 0;
    bool vec = false;              // the batch takes the vector path
    int tile_floats = 0;           // shared memory of a group's tile (floats)
    long long nplane = 0, nq = 0;  // entries of a population's plane and of the field on the device
    std::vector<int> pitch;        // row pitch of each instance's populations
    std::vector<long long> fo;     // its first entry of a plane
    int *order_dev = nullptr;      // instances by decreasing cell count (cluster form)
    void *f[2] = {nullptr, nullptr};
    void *q = nullptr;
    void *stage_dev = nullptr;   // rho staging (ntot values of the precision)
    void *stage_host = nullptr;  // pinned host staging
    void *mom_dev = nullptr;     // rho, vx, vy of lbm_batch_moments (3 ntot values, allocated on first use)
    void *mom_host = nullptr;    // their pinned host copy
    int *err = nullptr;
    BarrierState *bar = nullptr;
    int cur = 0;
    cudaStream_t stream = nullptr;
    int block_threads = 256;
    int grid_blocks = 0;
    int cluster = 0;               // CTAs per instance in the cluster form (0: grid form, -1: grouped)
    int cluster_threads = 256;
    size_t cluster_smem = 0;       // dynamic shared memory per CTA of the cluster form
    // grouped cluster form: one cluster launch per cluster size, each on its own
    // stream (forked from and joined to the batch's stream), instances of group
    // g at gorder_dev[first .. first + count) by decreasing cell count
    struct Group {
        int cluster, first, count;
        size_t smem;
    };
    std::vector<Group> groups;
    std::vector<int> group_cluster;   // cluster size of each instance in the grouped form
    int *gorder_dev = nullptr;
    cudaStream_t gstream[3] = {nullptr, nullptr, nullptr};
    cudaEvent_t gfork = nullptr, gjoin[3] = {nullptr, nullptr, nullptr};
    int groups_gen = 0;            // changes with every grouping (graph cache key)
    std::vector<int> halo;         // x halo of each instance (kx for HDM, 1 for CDM)
    unsigned long long limit_ns = 2000000000ull;  // 2 s per barrier wait
    int skip_block = -1;
    bool initialized = false;
    bool unstable = false;
    // graphs of the last step count, one per starting buffer parity
    cudaGraph_t graph[2] = {nullptr, nullptr};
    cudaGraphExec_t graph_exec[2] = {nullptr, nullptr};
    int graph_steps[2] = {-1, -1}, graph_block[2] = {-1, -1}, graph_grid[2] = {-1, -1};
    int graph_cluster[2] = {-1, -1}, graph_gen[2] = {-1, -1};
    bool use_graph = true;
    int graph_launches = 0;  // persistent launches issued through a graph
    std::string msg;
};

namespace {

lbm_status bfail(lbm_batch *b, lbm_status st, const std::string &m) {
    if (b) b->msg = m;
    return st;
}

#define BCK(b, expr, what)                                                                         \
    do {                                                                                           \
        cudaError_t e_ = (expr);                                                                   \
        if (e_ != cudaSuccess)                                                                     \
            return bfail(b, e_ == cudaErrorMemoryAllocation ? LBM_E_NOMEM : LBM_E_CUDA,            \
                         std::string(what) + ": " + cudaGetErrorString(e_));                       \
    } while (0)

template <typename T>
lbm_status build_instances(lbm_batch *b, std::vector<Inst<T>> &out) {
    out.resize(b->n);
    b->halo.assign(b->n, 0);
    for (int i = 0; i < b->n; ++i) {
        const lbm_params &p = b->params[i];
        Inst<T> &I = out[i];
        I = Inst<T>{};
        ModelScalars ms;
        if (model_scalars(p, &ms) != LBM_OK)
            return bfail(b, LBM_E_INVALID, "no critical point for instance " + std::to_string(i));
        I.m.nx = p.nx;
        I.m.ny = p.ny;
        I.m.eos = p.eos;
        I.m.RT = (T)ms.RT;
        I.m.a = (T)ms.a;
        I.m.b = (T)ms.b;
        I.m.aal = (T)ms.aal;
        I.m.k = (T)ms.k;
        I.m.omega = (T)(1.0 / p.tau);
        const int radius = p.hdm_radius ? p.hdm_radius : (b->prec == LBM_F64 ? 40 : 26);
        double wx[kMaxRadius + 1] = {}, wy[kMaxRadius + 1] = {};
        lbm_hdm_weights(p.nx, radius, wx, &I.m.kx);
        lbm_hdm_weights(p.ny, radius, wy, &I.m.ky);
        for (int j = 0; j <= kMaxRadius; ++j) {
            I.m.wx[j] = (T)wx[j];
            I.m.wy[j] = (T)wy[j];
        }
        I.off = (int)b->off[i];
        I.sc = p.force == LBM_FORCE_SC;
        I.cdm = p.grad == LBM_GRAD_CDM;
        b->halo[i] = I.cdm ? 1 : I.m.kx;
    }
    // the vector path: the whole batch or none of it (the windows' weights are the
    // unfolded ones: radius 26 on lines of at least 53 cells)
    b->vec = b->prec == LBM_F32;
    for (int i = 0; i < b->n; ++i) b->vec = b->vec && !out[i].cdm && b->params[i].hdm_radius == 0 && out[i].m.kx == FK;
    for (int i = 0; i < b->n; ++i) {
        const lbm_params &p = b->params[i];
        Inst<T> &I = out[i];
        I.vec = b->vec;
        I.P = I.vec ? (p.nx + 3) / 4 * 4 : p.nx;
        I.QP = I.vec ? I.P + 2 * QG : p.nx;
        I.qx = I.vec ? QG : 0;
        b->nplane = (b->nplane + 3) / 4 * 4;   // (16-byte rows on the vector path)
        b->nq = (b->nq + 3) / 4 * 4;
        I.fo = b->nplane;
        I.qo = b->nq;
        b->nplane += (long long)I.P * p.ny;
        b->nq += (long long)I.QP * p.ny;
        b->pitch.push_back(I.P);
        b->fo.push_back(I.fo);
        if (I.vec) b->tile_floats = std::max(b->tile_floats, tile_floats(p.ny));
    }
    b->nplane = (b->nplane + 3) / 4 * 4;
    b->nq = (b->nq + 3) / 4 * 4;
    return LBM_OK;
}

// Work items of the grid form: tiles of the vector path, else runs of 128 cells.
template <typename T>
std::vector<int4> work_items(const std::vector<Inst<T>> &v) {
    std::vector<int4> out;
    for (int i = 0; i < (int)v.size(); ++i) {
        const int nx = v[i].m.nx, ny = v[i].m.ny;
        if (v[i].vec) {
            const int tw = ny <= 8 ? 64 : 32, th = ny <= 8 ? 8 : 16;
            for (int y = 0; y < ny; y += th)
                for (int x = 0; x < nx; x += tw) out.push_back(make_int4(i, x, y, 0));
        } else {
            for (long long c = 0; c < (long long)nx * ny; c += NT) out.push_back(make_int4(i, (int)c, 0, 0));
        }
    }
    return out;
}

template <typename A>
void set_powers(A &a) {
    const double r = 0.5 * (std::sqrt(5.0) - 3.0);   // root of r^2/3 + r + 1/3 = 0 (Eq. 20's operator)
    a.r = (float)r;
    a.r5 = (float)std::pow(r, 5);
    a.r25 = (float)std::pow(r, 25);
}

template <typename T>
BatchArgs<T> make_args(lbm_batch *b, int nsteps) {
    BatchArgs<T> a{};
    a.inst = (const Inst<T> *)b->inst_dev;
    a.tiles = b->tiles_dev;
    a.ntiles = b->ntiles;
    a.f[0] = (T *)b->f[0];
    a.f[1] = (T *)b->f[1];
    a.q = (T *)b->q;
    a.nplane = b->nplane;
    a.nq = b->nq;
    set_powers(a);
    a.nsteps = nsteps;
    a.parity0 = b->cur;
    a.err = b->err;
    a.bar = b->bar;
    a.limit_ns = b->limit_ns;
    a.skip_block = b->skip_block;
    return a;
}

// The grid form's kernel for this batch, and its dynamic shared memory.
template <typename T>
auto grid_kernel(const lbm_batch *b) -> void (*)(const BatchArgs<T>, int) {
    if constexpr (sizeof(T) == 4)
        if (b->vec) return batch_kernel<T, true>;
    return batch_kernel<T, false>;
}
size_t grid_smem(const lbm_batch *b, int threads) { return (size_t)(threads / NT) * b->tile_floats * sizeof(float); }

// (The limit of shared memory belongs to the function: it is always set to the largest
// any batch takes, so that another batch, or another thread's, never lowers it.)
template <typename T>
int max_blocks_per_sm(const lbm_batch *b, int threads) {
    const size_t smem = grid_smem(b, threads);
    int nb = 0;
    const int limit = b->vec ? (int)((512 / NT) * tile_floats(9) * sizeof(float)) : 0;
    if (cudaFuncSetAttribute(grid_kernel<T>(b), cudaFuncAttributeMaxDynamicSharedMemorySize, limit) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, grid_kernel<T>(b), threads, smem) != cudaSuccess)
        return 0;
    return nb;
}
int max_blocks_per_sm(const lbm_batch *b, int threads) {
    return b->prec == LBM_F64 ? max_blocks_per_sm<double>(b, threads) : max_blocks_per_sm<float>(b, threads);
}

int sm_count() {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n;
}

// Shared memory per CTA of the cluster form with `cluster` CTAs per instance on
// the per-cell path (both distribution buffers and the haloed potential field of
// the widest slice), or 0 when some instance does not split: a slice narrower than
// the instance's x halo, or more than the opt-in shared memory of a block.  The
// vector path takes less, and splits where this does.
size_t cluster_smem_bytes(const lbm_batch *b, int cluster) {
    size_t need = 0;
    for (int i = 0; i < b->n; ++i) {
        const int nx = b->params[i].nx, ny = b->params[i].ny;
        const int wmin = nx / cluster, wmax = (nx + cluster - 1) / cluster;   // slice widths
        if (b->halo[i] > wmin) return 0;
        const size_t bytes = ((size_t)2 * kQ * wmax * ny + (size_t)ny * (wmax + 2 * b->halo[i])) * b->esz;
        need = std::max(need, bytes);
    }
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return need <= (size_t)optin ? need : 0;
}

// Launch of the cluster form over the instances picked by `in`: kernel, threads
// per CTA and shared memory.  The vector path's kernel takes a thread per group of
// four cells of its widest slice whatever `threads` asks, and one per piece of the halo
// up to 128 (each further round of copies from other ranks takes 0.35 us) (a slice that
// cluster_smem_bytes admits has at most 768 of them, and never more shared memory than
// that).  Up to 512 threads two CTAs share an SM, which with 64 registers and 650 bytes
// of spills (520 since the halo's copies are a call) measured 18.8 us per step of the 64-lattice sweep (one cluster size) against
// 21.1 with one CTA of 118 registers.  Above that there is one CTA per SM in any case and
// it may take 80 registers: as tuned, 34 + 12 of the 64 lattices in CTAs of 744 threads,
// 18.2 us with the 64 registers of 1024 threads, 16.9 with 80.
template <typename T>
struct ClusterLaunch {
    void (*kern)(const ClusterArgs<T>);
    int threads;
    size_t smem;
};
template <typename T, typename In>
ClusterLaunch<T> cluster_launch(const lbm_batch *b, int cluster, int threads, size_t smem, In in) {
    if constexpr (sizeof(T) == 4) {
        if (b->vec) {
            int groups = 0, pieces = 0;
            size_t need = 0;
            for (int i = 0; i < b->n; ++i) {
                const int nx = b->params[i].nx, ny = b->params[i].ny;
                if (!in(i)) continue;
                const SliceShape sh(nx, cluster);
                groups = std::max(groups, sh.ngm * ny);
                pieces = std::max(pieces, kPieces * ny);
                need = std::max(need, sizeof(float) * sh.floats(ny, ny > 2 * FK));
            }
            const int t = (std::max(groups, std::min(pieces, 128)) + 31) / 32 * 32;
            return {t <= 512 ? cluster_vec_kernel<512, 2> : cluster_vec_kernel<768, 1>, t, need};
        }
    }
    return {cluster_batch_kernel<T>, threads, smem};
}
const auto every = [](int) { return true; };

template <typename T>
cudaLaunchConfig_t cluster_config(const lbm_batch *b, int cluster, int threads, size_t smem,
                                  cudaLaunchAttribute *attr) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(cluster * b->n));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = b->stream;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// Prepare a cluster launch and check that at least one cluster of it can be
// resident.  Returns 0 or an error message.  The kernel's limit of shared memory belongs
// to the function, not to the batch: every batch sets it to all that a block may take, so
// that none, on whatever thread, lowers it before another's launch.
template <typename T>
const char *configure_cluster(const lbm_batch *b, const ClusterLaunch<T> &L, int cluster) {
    int dev = 0, optin = 0;
    cudaFuncAttributes fa{};
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaFuncGetAttributes(&fa, L.kern) != cudaSuccess || L.smem + fa.sharedSizeBytes > (size_t)optin ||
        cudaFuncSetAttribute(L.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes) !=
            cudaSuccess)
        return "shared memory of the cluster form not available";
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = cluster_config<T>(b, cluster, L.threads, L.smem, attr);
    int nc = 0;
    if (cudaOccupancyMaxActiveClusters(&nc, L.kern, &cfg) != cudaSuccess || nc < 1) {
        cudaGetLastError();
        return "no cluster of this shape fits on the device";
    }
    return nullptr;
}

// The instances of group g of the grouped form (pick: group's cluster size per instance).
auto in_group(const lbm_batch *b, int cluster) {
    return [b, cluster](int i) { return b->group_cluster[i] == cluster; };
}

// Queue one launch running nsteps steps: the cluster form when one is set
// (and no barrier test hook is armed), else the persistent cooperative grid form.
template <typename T>
cudaError_t enqueue(lbm_batch *b, int nsteps) {
    if (b->cluster < 0 && b->skip_block < 0) {   // grouped: fork, one launch per group, join
        cudaError_t e = cudaEventRecord(b->gfork, b->stream);
        for (size_t g = 0; g < b->groups.size() && e == cudaSuccess; ++g) {
            const lbm_batch::Group &G = b->groups[g];
            ClusterArgs<T> ca{};
            ca.inst = (const Inst<T> *)b->inst_dev;
            ca.order = b->gorder_dev + G.first;
            ca.fin = (const T *)b->f[b->cur];
            ca.fout = (T *)b->f[(b->cur + nsteps) & 1];
            ca.nplane = b->nplane;
            set_powers(ca);
            ca.nsteps = nsteps;
            ca.err = b->err;
            const auto L = cluster_launch<T>(b, G.cluster, b->cluster_threads, G.smem, in_group(b, G.cluster));
            cudaLaunchAttribute attr[1];
            cudaLaunchConfig_t cfg = cluster_config<T>(b, G.cluster, L.threads, L.smem, attr);
            cfg.gridDim = dim3((unsigned)(G.cluster * G.count));
            cfg.stream = b->gstream[g];
            e = cudaStreamWaitEvent(b->gstream[g], b->gfork, 0);
            if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, L.kern, ca);
            if (e == cudaSuccess) e = cudaEventRecord(b->gjoin[g], b->gstream[g]);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(b->stream, b->gjoin[g], 0);
        }
        return e;
    }
    if (b->cluster > 0 && b->skip_block < 0) {
        ClusterArgs<T> ca{};
        ca.inst = (const Inst<T> *)b->inst_dev;
        ca.order = b->order_dev;
        ca.fin = (const T *)b->f[b->cur];
        ca.fout = (T *)b->f[(b->cur + nsteps) & 1];
        ca.nplane = b->nplane;
        set_powers(ca);
        ca.nsteps = nsteps;
        ca.err = b->err;
        const auto L = cluster_launch<T>(b, b->cluster, b->cluster_threads, b->cluster_smem, every);
        cudaLaunchAttribute attr[1];
        cudaLaunchConfig_t cfg = cluster_config<T>(b, b->cluster, L.threads, L.smem, attr);
        return cudaLaunchKernelEx(&cfg, L.kern, ca);
    }
    cudaError_t e = cudaMemsetAsync(b->bar, 0, sizeof(BarrierState), b->stream);
    if (e != cudaSuccess) return e;
    BatchArgs<T> a = make_args<T>(b, nsteps);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(b->grid_blocks);   // (a cooperative launch: never more than is resident at once)
    cfg.blockDim = dim3(b->block_threads);
    cfg.dynamicSmemBytes = grid_smem(b, b->block_threads);
    cfg.stream = b->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, grid_kernel<T>(b), a, b->tile_floats);
}

void drop_graph(lbm_batch *b, int k) {
    if (b->graph_exec[k]) cudaGraphExecDestroy(b->graph_exec[k]);
    if (b->graph[k]) cudaGraphDestroy(b->graph[k]);
    b->graph_exec[k] = nullptr;
    b->graph[k] = nullptr;
    b->graph_steps[k] = -1;
}

// nsteps steps as one persistent launch, replayed from a CUDA graph captured
// for this (step count, starting buffer, launch shape).
template <typename T>
lbm_status run_steps(lbm_batch *b, int nsteps) {
    if (nsteps == 0) return LBM_OK;
    const int k = b->cur;
    if (b->use_graph && b->skip_block < 0) {
        const int shape_block = b->cluster != 0 ? b->cluster_threads : b->block_threads;
        if (!b->graph_exec[k] || b->graph_steps[k] != nsteps || b->graph_block[k] != shape_block ||
            b->graph_grid[k] != b->grid_blocks || b->graph_cluster[k] != b->cluster ||
            b->graph_gen[k] != b->groups_gen) {
            drop_graph(b, k);
            bool ok = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
            if (ok) {
                cudaError_t e1 = enqueue<T>(b, nsteps);
                cudaError_t e2 = cudaStreamEndCapture(b->stream, &b->graph[k]);
                ok = e1 == cudaSuccess && e2 == cudaSuccess &&
                     cudaGraphInstantiate(&b->graph_exec[k], b->graph[k], 0) == cudaSuccess;
            }
            if (!ok) {  // graphs unavailable for this launch: plain launches from now on
                cudaGetLastError();
                drop_graph(b, k);
                b->use_graph = false;
            } else {
                b->graph_steps[k] = nsteps;
                b->graph_block[k] = shape_block;
                b->graph_grid[k] = b->grid_blocks;
                b->graph_cluster[k] = b->cluster;
                b->graph_gen[k] = b->groups_gen;
            }
        }
        if (b->graph_exec[k]) {
            BCK(b, cudaGraphLaunch(b->graph_exec[k], b->stream), "cudaGraphLaunch");
            b->graph_launches += 1;
            b->cur = (b->cur + nsteps) & 1;
            return LBM_OK;
        }
    }
    BCK(b, enqueue<T>(b, nsteps), "batch launch");
    b->cur = (b->cur + nsteps) & 1;
    return LBM_OK;
}

// The populations between the device's layout (d: rows at the batch's pitch) and the
// caller's, instance after instance, each 9 x ny x nx; row by row: a division per value
// took four times as long (the 64-lattice sweep, 5.3 M values: 2.8 and 12 ms).
template <typename T, typename F, typename Row>
void for_each_row(const lbm_batch *b, T *d, F *f, Row row) {
    for (int i = 0; i < b->n; ++i) {
        const int nx = b->params[i].nx, ny = b->params[i].ny;
        for (int k = 0; k < kQ; ++k) {
            T *p = d + (size_t)k * b->nplane + b->fo[i];
            for (int y = 0; y < ny; ++y, p += b->pitch[i], f += nx) row(p, f, nx);
        }
    }
}
template <typename T>
void unpack_f(const lbm_batch *b, T *d, double *f) {
    for_each_row(b, d, f, [](const T *p, double *o, int nx) {
        for (int x = 0; x < nx; ++x) o[x] = (double)p[x];
    });
}
template <typename T>
void pack_f(const lbm_batch *b, T *d, const double *f) {
    for_each_row(b, d, f, [](T *p, const double *o, int nx) {
        for (int x = 0; x < nx; ++x) p[x] = (T)o[x];
    });
}

// The caller's concatenated FP64 field into the staging layout of T (instances at
// multiples of 512 cells, zeros between); false if a value is not a positive finite
// number.  Plain loops over one type, no exit in the middle: the compiler turns
// them into vector code (590,000 cells: 0.45 -> 0.15 ms).
template <typename T>
bool stage_density(const lbm_batch *b, const double *rho, T *h) {
    bool good = true;
    for (int i = 0; i < b->n; ++i) {
        const long long cells = (long long)b->params[i].nx * b->params[i].ny;
        const long long end = i + 1 < b->n ? b->off[i + 1] : b->ntot;
        T *d = h + b->off[i];
        int ok = 1;
        for (long long c = 0; c < cells; ++c) {
            const double v = rho[c];
            ok &= (int)(v > 0.0) & (int)(v <= 1.7976931348623157e308);
            d[c] = (T)v;
        }
        good = good && ok;
        std::fill(d + cells, h + end, T(0));
        rho += cells;
    }
    return good;
}
// ... and a staged field back into the caller's concatenated FP64 array.
template <typename T>
void unstage_field(const lbm_batch *b, const T *h, double *out) {
    for (int i = 0; i < b->n; ++i) {
        const long long cells = (long long)b->params[i].nx * b->params[i].ny;
        const T *d = h + b->off[i];
        for (long long c = 0; c < cells; ++c) out[c] = (double)d[c];
        out += cells;
    }
}

lbm_status batch_sync(lbm_batch *b) {
    int h = 0;
    BCK(b, cudaMemcpyAsync(&h, b->err, sizeof(int), cudaMemcpyDeviceToHost, b->stream), "read error word");
    BCK(b, cudaStreamSynchronize(b->stream), "cudaStreamSynchronize");
    if (h & kErrTimeout) return bfail(b, LBM_E_TIMEOUT, "a grid barrier wait timed out");
    if (h & kErrUnstable) {
        b->unstable = true;
        return bfail(b, LBM_E_UNSTABLE, "unstable: NaN or non-positive density");
    }
    return LBM_OK;
}

}  // namespace

extern "C" {

lbm_status lbm_batch_create(const lbm_params *p, int n, lbm_batch **out) {
    if (!out) return LBM_E_INVALID;
    *out = nullptr;
    if (!p || n < 1) return LBM_E_INVALID;
    const int prec = p[0].prec;
    if (prec != LBM_F32 && prec != LBM_F64) return LBM_E_INVALID;
    long long padded = 0;
    for (int i = 0; i < n; ++i) {
        const lbm_params &q = p[i];
        const char *why = "";
        if (q.prec != prec || check_params(q, &why) != LBM_OK || (long long)q.nx * q.ny > (1LL << 30) ||
            (q.flags & LBM_FLAG_WALLS_Y))   // the batch steps periodic lattices only
            return LBM_E_INVALID;
        padded += ((long long)q.nx * q.ny + kAlign - 1) / kAlign * kAlign;
    }
    // instance offsets are int cell indices on the device: the padded total
    // must stay below 2^31 cells
    if (padded >= (1LL << 31)) return LBM_E_INVALID;
    lbm_batch *b = new (std::nothrow) lbm_batch();
    if (!b) return LBM_E_NOMEM;
    b->n = n;
    b->prec = prec;
    b->esz = prec == LBM_F64 ? sizeof(double) : sizeof(float);
    b->params.assign(p, p + n);
    b->stream = (cudaStream_t)p[0].stream;
    long long o = 0;
    for (int i = 0; i < n; ++i) {
        b->off.push_back(o);
        long long cells = (long long)p[i].nx * p[i].ny;
        o += (cells + kAlign - 1) / kAlign * kAlign;
    }
    b->ntot = o;
    auto bail = [&](lbm_status st) {
        lbm_batch_destroy(b);
        return st;
    };

    std::vector<int> table(b->ntot / kTableGrain, -1);
    for (int i = 0; i < n; ++i) {
        long long cells = (long long)p[i].nx * p[i].ny;
        for (long long g = b->off[i] / kTableGrain; g < (b->off[i] + cells + kTableGrain - 1) / kTableGrain; ++g)
            table[g] = i;
    }
    std::vector<int> order(n);
    for (int i = 0; i < n; ++i) order[i] = i;
    std::stable_sort(order.begin(), order.end(), [&](int u, int v) {
        return (long long)p[u].nx * p[u].ny > (long long)p[v].nx * p[v].ny;
    });
    size_t inst_bytes;
    std::vector<unsigned char> inst_host;
    std::vector<int4> tiles;
    if (prec == LBM_F64) {
        std::vector<Inst<double>> v;
        if (build_instances<double>(b, v) != LBM_OK) return bail(LBM_E_INVALID);
        tiles = work_items(v);
        inst_bytes = v.size() * sizeof(Inst<double>);
        inst_host.assign((unsigned char *)v.data(), (unsigned char *)v.data() + inst_bytes);
    } else {
        std::vector<Inst<float>> v;
        if (build_instances<float>(b, v) != LBM_OK) return bail(LBM_E_INVALID);
        tiles = work_items(v);
        inst_bytes = v.size() * sizeof(Inst<float>);
        inst_host.assign((unsigned char *)v.data(), (unsigned char *)v.data() + inst_bytes);
    }
    b->ntiles = (int)tiles.size();
    const size_t fbytes = (size_t)kQ * b->nplane * b->esz;
    if (dev_alloc((void **)&b->tiles_dev, tiles.size() * sizeof(int4)) != cudaSuccess ||
        dev_alloc(&b->inst_dev, inst_bytes) != cudaSuccess || dev_alloc((void **)&b->table_dev, table.size() * sizeof(int)) != cudaSuccess ||
        dev_alloc(&b->f[0], fbytes) != cudaSuccess || dev_alloc(&b->f[1], fbytes) != cudaSuccess ||
        dev_alloc(&b->q, b->nq * b->esz) != cudaSuccess || dev_alloc(&b->stage_dev, b->ntot * b->esz) != cudaSuccess ||
        dev_alloc((void **)&b->err, sizeof(int)) != cudaSuccess || dev_alloc((void **)&b->bar, sizeof(BarrierState)) != cudaSuccess ||
        dev_alloc((void **)&b->order_dev, n * sizeof(int)) != cudaSuccess ||
        host_alloc(&b->stage_host, b->ntot * sizeof(double)) != cudaSuccess)
        return bail(LBM_E_NOMEM);
    // the instances' bounds-check error word (LBM_CHECKED builds) is the batch's
    for (int i = 0; i < n; ++i) {
        if (prec == LBM_F64) reinterpret_cast<Inst<double> *>(inst_host.data())[i].m.chk = b->err;
        else reinterpret_cast<Inst<float> *>(inst_host.data())[i].m.chk = b->err;
    }
    if (cudaMemcpy(b->inst_dev, inst_host.data(), inst_bytes, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(b->tiles_dev, tiles.data(), tiles.size() * sizeof(int4), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(b->table_dev, table.data(), table.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(b->order_dev, order.data(), n * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(b->f[0], 0, fbytes) != cudaSuccess || cudaMemset(b->f[1], 0, fbytes) != cudaSuccess ||
        cudaMemset(b->err, 0, sizeof(int)) != cudaSuccess)
        return bail(LBM_E_CUDA);
    // default launch shape: 256 threads, as many co-resident blocks as occupancy allows
    const int per_sm = max_blocks_per_sm(b, 256);
    if (per_sm < 1) return bail(LBM_E_CUDA);
    b->block_threads = 256;
    b->grid_blocks = per_sm * sm_count();
    *out = b;
    return LBM_OK;
}

lbm_status lbm_batch_set_launch(lbm_batch *b, int block_threads, int blocks_per_sm) {
    if (!b) return LBM_E_INVALID;
    if (block_threads != 128 && block_threads != 256 && block_threads != 512)
        return bfail(b, LBM_E_INVALID, "block_threads must be 128, 256 or 512");
    // A shape is accepted up to the threads per SM that the per-cell kernels can keep
    // resident; the vector path's tiles allow fewer, and a larger shape runs with those.
    const int maxb = (b->prec == LBM_F64 ? 1152 : 1280) / block_threads;
    if (blocks_per_sm < 1 || blocks_per_sm > maxb)
        return bfail(b, LBM_E_INVALID, "blocks_per_sm must be in [1, " + std::to_string(maxb) + "]");
    const int resident = max_blocks_per_sm(b, block_threads);
    if (resident < 1) return bfail(b, LBM_E_CUDA, "no block of this shape is resident");
    b->block_threads = block_threads;
    b->grid_blocks = std::min(blocks_per_sm, resident) * sm_count();
    b->cluster = 0;   // an explicit grid shape selects the grid form
    return LBM_OK;
}

lbm_status lbm_batch_get_launch(lbm_batch *b, int *block_threads, int *grid_blocks) {
    if (!b || !block_threads || !grid_blocks) return LBM_E_INVALID;
    *block_threads = b->cluster != 0 ? b->cluster_threads : b->block_threads;
    int blocks = b->grid_blocks;
    if (b->cluster > 0) blocks = b->cluster * b->n;
    if (b->cluster < 0) {
        blocks = 0;
        for (const auto &G : b->groups) blocks += G.cluster * G.count;
    }
    *grid_blocks = blocks;
    return LBM_OK;
}

lbm_status lbm_batch_set_cluster(lbm_batch *b, int cluster, int block_threads) {
    if (!b) return LBM_E_INVALID;
    if (cluster == 0) {
        b->cluster = 0;
        return LBM_OK;
    }
    if (cluster != 2 && cluster != 4 && cluster != 8)
        return bfail(b, LBM_E_INVALID, "cluster must be 0, 2, 4 or 8");
    if (block_threads != 128 && block_threads != 256 && block_threads != 512 && block_threads != 1024)
        return bfail(b, LBM_E_INVALID, "block_threads must be 128, 256, 512 or 1024");
    size_t smem = cluster_smem_bytes(b, cluster);
    if (smem == 0) return bfail(b, LBM_E_INVALID, "an instance does not split over a cluster of this size");
    const char *why = nullptr;
    if (b->prec == LBM_F64) {
        why = configure_cluster(b, cluster_launch<double>(b, cluster, block_threads, smem, every), cluster);
    } else {
        const auto L = cluster_launch<float>(b, cluster, block_threads, smem, every);
        why = configure_cluster(b, L, cluster);
        smem = L.smem;
    }
    if (why) return bfail(b, LBM_E_INVALID, why);
    b->cluster = cluster;
    b->cluster_threads = block_threads;
    b->cluster_smem = smem;
    return LBM_OK;
}

lbm_status lbm_batch_set_groups(lbm_batch *b, int max_smem_bytes, int block_threads) {
    if (!b) return LBM_E_INVALID;
    if (block_threads != 256 && block_threads != 512 && block_threads != 1024)
        return bfail(b, LBM_E_INVALID, "block_threads must be 256, 512 or 1024");
    if (max_smem_bytes < LBM_GROUPS_BALANCED) return bfail(b, LBM_E_INVALID, "max_smem_bytes must be >= -1");
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return bfail(b, LBM_E_CUDA, "device attributes");
    auto slice_bytes = [&](int i, int C) {   // both buffers and the haloed field of instance i's widest slice
        const int nx = b->params[i].nx, ny = b->params[i].ny, wmax = (nx + C - 1) / C;
        return ((size_t)2 * kQ * wmax * ny + (size_t)ny * (wmax + 2 * b->halo[i])) * b->esz;
    };
    size_t cap = max_smem_bytes > 0 ? std::min<size_t>(max_smem_bytes, optin) : (size_t)optin;
    if (max_smem_bytes == LBM_GROUPS_BALANCED) {   // no CTA holds more than the largest 8-CTA slice
        cap = 0;
        for (int i = 0; i < b->n; ++i) cap = std::max(cap, slice_bytes(i, 8));
        cap = std::min(cap, (size_t)optin);
    }
    // each instance: the smallest cluster whose slices split it (no slice
    // narrower than the x halo) within `cap`, else within the opt-in maximum
    const int sizes[3] = {2, 4, 8};
    std::vector<int> pick(b->n, -1);
    std::vector<size_t> need(b->n, 0);
    for (int i = 0; i < b->n; ++i) {
        const int nx = b->params[i].nx;
        for (size_t limit : {cap, (size_t)optin}) {
            for (int g = 0; g < 3 && pick[i] < 0; ++g) {
                const int C = sizes[g], wmin = nx / C;
                const size_t bytes = slice_bytes(i, C);
                if (b->halo[i] <= wmin && bytes <= limit) {
                    pick[i] = g;
                    need[i] = bytes;
                }
            }
            if (pick[i] >= 0) break;
        }
        if (pick[i] < 0)
            return bfail(b, LBM_E_INVALID, "instance " + std::to_string(i) + " does not split over a cluster of 8");
    }
    std::vector<int> order(b->n);
    for (int i = 0; i < b->n; ++i) order[i] = i;
    std::stable_sort(order.begin(), order.end(), [&](int u, int v) {   // by group, then largest first
        if (pick[u] != pick[v]) return pick[u] > pick[v];
        return (long long)b->params[u].nx * b->params[u].ny > (long long)b->params[v].nx * b->params[v].ny;
    });
    std::vector<lbm_batch::Group> groups;
    for (int k = 0; k < b->n; ++k) {
        const int i = order[k];
        if (groups.empty() || groups.back().cluster != sizes[pick[i]])
            groups.push_back({sizes[pick[i]], k, 0, 0});
        groups.back().count += 1;
        groups.back().smem = std::max(groups.back().smem, need[i]);
    }
    // every group must place at least one cluster
    const bool f64 = b->prec == LBM_F64;
    std::vector<int> group_cluster(b->n);
    for (int i = 0; i < b->n; ++i) group_cluster[i] = sizes[pick[i]];
    for (auto &G : groups) {
        auto in = [&](int i) { return group_cluster[i] == G.cluster; };
        const char *why = nullptr;
        if (f64) {
            why = configure_cluster(b, cluster_launch<double>(b, G.cluster, block_threads, G.smem, in), G.cluster);
        } else {
            const auto L = cluster_launch<float>(b, G.cluster, block_threads, G.smem, in);
            why = configure_cluster(b, L, G.cluster);
            G.smem = L.smem;
        }
        if (why) return bfail(b, LBM_E_INVALID, why);
    }
    if (!b->gorder_dev) BCK(b, dev_alloc((void **)&b->gorder_dev, b->n * sizeof(int)), "cudaMalloc(group order)");
    for (int g = 0; g < 3; ++g) {
        if (!b->gstream[g]) BCK(b, cudaStreamCreateWithFlags(&b->gstream[g], cudaStreamNonBlocking), "stream");
        if (!b->gjoin[g]) BCK(b, cudaEventCreateWithFlags(&b->gjoin[g], cudaEventDisableTiming), "event");
    }
    if (!b->gfork) BCK(b, cudaEventCreateWithFlags(&b->gfork, cudaEventDisableTiming), "event");
    BCK(b, cudaMemcpyAsync(b->gorder_dev, order.data(), b->n * sizeof(int), cudaMemcpyHostToDevice, b->stream),
        "group order upload");
    BCK(b, cudaStreamSynchronize(b->stream), "group order upload");
    b->groups = groups;
    b->group_cluster = group_cluster;
    b->cluster = -1;
    b->cluster_threads = block_threads;
    b->groups_gen += 1;
    return LBM_OK;
}

lbm_status lbm_batch_get_groups(lbm_batch *b, int *ngroups, int *cluster, int *count, int *smem_bytes) {
    if (!b || !ngroups) return LBM_E_INVALID;
    *ngroups = b->cluster < 0 ? (int)b->groups.size() : 0;
    for (int g = 0; g < *ngroups; ++g) {
        if (cluster) cluster[g] = b->groups[g].cluster;
        if (count) count[g] = b->groups[g].count;
        if (smem_bytes) smem_bytes[g] = (int)b->groups[g].smem;
    }
    return LBM_OK;
}

lbm_status lbm_batch_get_cluster(lbm_batch *b, int *cluster) {
    if (!b || !cluster) return LBM_E_INVALID;
    *cluster = b->cluster;
    return LBM_OK;
}

lbm_status lbm_batch_init_density(lbm_batch *b, const double *rho) {
    if (!b || !rho) return LBM_E_INVALID;
    const size_t esz = b->esz;
    void *h = b->stage_host;
    BCK(b, cudaStreamSynchronize(b->stream), "sync before staging");
    if (!(b->prec == LBM_F64 ? stage_density(b, rho, (double *)h) : stage_density(b, rho, (float *)h)))
        return bfail(b, LBM_E_INVALID, "rho must be positive and finite");
    BCK(b, cudaMemcpyAsync(b->stage_dev, h, b->ntot * esz, cudaMemcpyHostToDevice, b->stream), "copy rho");
    b->cur = 0;
    const int blocks = (int)std::min<long long>((b->ntot + 255) / 256, 152 * 16);
    if (b->prec == LBM_F64)
        batch_init_kernel<double><<<blocks, 256, 0, b->stream>>>((const Inst<double> *)b->inst_dev, b->table_dev,
                                                                 (const double *)b->stage_dev, (double *)b->f[0], b->ntot, b->nplane);
    else
        batch_init_kernel<float><<<blocks, 256, 0, b->stream>>>((const Inst<float> *)b->inst_dev, b->table_dev,
                                                                (const float *)b->stage_dev, (float *)b->f[0], b->ntot, b->nplane);
    BCK(b, cudaGetLastError(), "init kernel");
    BCK(b, cudaMemsetAsync(b->err, 0, sizeof(int), b->stream), "clear error word");
    b->initialized = true;
    b->unstable = false;
    return LBM_OK;
}

lbm_status lbm_batch_step(lbm_batch *b, int nsteps) {
    NvtxRange nvtx("lbm_batch_step");
    if (!b) return LBM_E_INVALID;
    if (!b->initialized) return bfail(b, LBM_E_STATE, "batch not initialised");
    if (b->unstable) return bfail(b, LBM_E_UNSTABLE, "batch is in the error state");
    if (nsteps < 0) return bfail(b, LBM_E_INVALID, "nsteps must be >= 0");
    return b->prec == LBM_F64 ? run_steps<double>(b, nsteps) : run_steps<float>(b, nsteps);
}

lbm_status lbm_batch_sync(lbm_batch *b) {
    if (!b) return LBM_E_INVALID;
    return batch_sync(b);
}

lbm_status lbm_batch_density(lbm_batch *b, double *rho) {
    if (!b || !rho) return LBM_E_INVALID;
    if (!b->initialized) return bfail(b, LBM_E_STATE, "batch not initialised");
    const int blocks = (int)std::min<long long>((b->ntot + 255) / 256, 152 * 16);
    if (b->prec == LBM_F64)
        batch_density_kernel<double><<<blocks, 256, 0, b->stream>>>((const Inst<double> *)b->inst_dev, b->table_dev,
                                                                    (const double *)b->f[b->cur], (double *)b->stage_dev, b->ntot, b->nplane);
    else
        batch_density_kernel<float><<<blocks, 256, 0, b->stream>>>((const Inst<float> *)b->inst_dev, b->table_dev,
                                                                   (const float *)b->f[b->cur], (float *)b->stage_dev, b->ntot, b->nplane);
    BCK(b, cudaGetLastError(), "density kernel");
    BCK(b, cudaMemcpyAsync(b->stage_host, b->stage_dev, b->ntot * b->esz, cudaMemcpyDeviceToHost, b->stream), "copy rho");
    lbm_status st = batch_sync(b);
    if (st != LBM_OK && st != LBM_E_UNSTABLE) return st;
    if (b->prec == LBM_F64) unstage_field(b, (const double *)b->stage_host, rho);
    else unstage_field(b, (const float *)b->stage_host, rho);
    return st;
}

lbm_status lbm_batch_moments(lbm_batch *b, double *rho, double *vx, double *vy) {
    if (!b || !rho) return LBM_E_INVALID;
    if (!b->initialized) return bfail(b, LBM_E_STATE, "batch not initialised");
    const size_t fb = b->ntot * b->esz;
    if (!b->mom_dev && dev_alloc(&b->mom_dev, 3 * fb) != cudaSuccess)
        return bfail(b, LBM_E_NOMEM, "moment buffers");
    if (!b->mom_host && host_alloc(&b->mom_host, 3 * fb) != cudaSuccess)
        return bfail(b, LBM_E_NOMEM, "pinned moment staging");
    unsigned char *md = (unsigned char *)b->mom_dev;
    const size_t smem = grid_smem(b, NT);   // (at most 35 KB: no attribute needed)
    if (b->prec == LBM_F64) {
        const BatchArgs<double> a = make_args<double>(b, 0);
        batch_potential_kernel<double><<<b->ntiles, NT, smem, b->stream>>>(a);
        batch_moments_kernel<double><<<b->ntiles, NT, smem, b->stream>>>(a, (double *)md, (double *)(md + fb),
                                                                         (double *)(md + 2 * fb));
    } else {
        const BatchArgs<float> a = make_args<float>(b, 0);
        batch_potential_kernel<float><<<b->ntiles, NT, smem, b->stream>>>(a);
        batch_moments_kernel<float><<<b->ntiles, NT, smem, b->stream>>>(a, (float *)md, (float *)(md + fb),
                                                                        (float *)(md + 2 * fb));
    }
    BCK(b, cudaGetLastError(), "moments kernels");
    BCK(b, cudaMemcpyAsync(b->mom_host, b->mom_dev, 3 * fb, cudaMemcpyDeviceToHost, b->stream), "copy moments");
    lbm_status st = batch_sync(b);
    if (st != LBM_OK && st != LBM_E_UNSTABLE) return st;
    double *out[3] = {rho, vx, vy};
    for (int k = 0; k < 3; ++k) {
        if (!out[k]) continue;
        const unsigned char *h = (const unsigned char *)b->mom_host + k * fb;
        if (b->prec == LBM_F64) unstage_field(b, (const double *)h, out[k]);
        else unstage_field(b, (const float *)h, out[k]);
    }
    return st;
}

lbm_status lbm_batch_get_f(lbm_batch *b, double *f) {
    if (!b || !f) return LBM_E_INVALID;
    if (!b->initialized) return bfail(b, LBM_E_STATE, "batch not initialised");
    std::vector<unsigned char> all((size_t)kQ * b->nplane * b->esz);
    BCK(b, cudaMemcpyAsync(all.data(), b->f[b->cur], all.size(), cudaMemcpyDeviceToHost, b->stream), "copy f");
    lbm_status st = batch_sync(b);
    if (st != LBM_OK && st != LBM_E_UNSTABLE) return st;
    if (b->prec == LBM_F64) unpack_f(b, (double *)all.data(), f);
    else unpack_f(b, (float *)all.data(), f);
    return st;
}

lbm_status lbm_batch_set_f(lbm_batch *b, const double *f) {
    if (!b || !f) return LBM_E_INVALID;
    std::vector<unsigned char> all((size_t)kQ * b->nplane * b->esz, 0);
    if (b->prec == LBM_F64) pack_f(b, (double *)all.data(), f);
    else pack_f(b, (float *)all.data(), f);
    BCK(b, cudaMemcpyAsync(b->f[0], all.data(), all.size(), cudaMemcpyHostToDevice, b->stream), "copy f");
    BCK(b, cudaStreamSynchronize(b->stream), "sync f copy");
    BCK(b, cudaMemsetAsync(b->err, 0, sizeof(int), b->stream), "clear error word");
    b->cur = 0;
    b->initialized = true;
    b->unstable = false;
    return LBM_OK;
}

lbm_status lbm_batch_tune(lbm_batch *b, int trial_steps, int *block_threads, int *grid_blocks) {
    NvtxRange nvtx("lbm_batch_tune");
    if (!b || trial_steps < 2) return LBM_E_INVALID;
    if (!b->initialized) return bfail(b, LBM_E_STATE, "batch not initialised");
    // work on a copy of the state: the trials advance it
    const size_t fbytes = (size_t)kQ * b->nplane * b->esz;
    void *save = nullptr;
    BCK(b, dev_alloc(&save, fbytes), "cudaMalloc(tune state)");
    const int cur0 = b->cur;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    int best_t = b->block_threads, best_g = b->grid_blocks;
    int best_c = b->cluster, best_ct = b->cluster_threads;
    const int threads[3] = {128, 256, 512};
    lbm_status st = LBM_OK;
    if (cudaMemcpyAsync(save, b->f[cur0], fbytes, cudaMemcpyDeviceToDevice, b->stream) != cudaSuccess) st = LBM_E_CUDA;
    // a warm-up launch, then a timed one (plain launches: no graph per trial)
    auto trial = [&](float *ms) -> bool {
        const bool g = b->use_graph;
        b->use_graph = false;
        lbm_status s1 = b->prec == LBM_F64 ? run_steps<double>(b, 2) : run_steps<float>(b, 2);
        cudaEventRecord(e0, b->stream);
        lbm_status s2 = b->prec == LBM_F64 ? run_steps<double>(b, trial_steps) : run_steps<float>(b, trial_steps);
        cudaEventRecord(e1, b->stream);
        b->use_graph = g;
        if (s1 != LBM_OK || s2 != LBM_OK || cudaEventSynchronize(e1) != cudaSuccess) return false;
        return cudaEventElapsedTime(ms, e0, e1) == cudaSuccess;
    };
    // grid form: block sizes x co-resident blocks per SM
    b->cluster = 0;
    for (int ti = 0; ti < 3 && st == LBM_OK; ++ti) {
        const int maxb = max_blocks_per_sm(b, threads[ti]);
        for (int per = 1; per <= maxb && st == LBM_OK; per = per < maxb && per * 2 > maxb ? maxb : per * 2) {
            b->block_threads = threads[ti];
            b->grid_blocks = per * sm_count();
            float ms = 0;
            if (!trial(&ms)) { st = LBM_E_CUDA; break; }
            if (ms < best) { best = ms; best_t = b->block_threads; best_g = b->grid_blocks; best_c = 0; }
            if (per == maxb) break;
        }
    }
    // cluster form: CTAs per instance x threads per CTA, where the instances split
    const int grid_t = best_t, grid_g = best_g;
    const int cthreads[3] = {256, 512, 1024};
    const int tfirst = b->vec ? 1 : 0, tlast = b->vec ? 1 : 2;   // (the vector path picks its own thread count)
    for (int c = 2; c <= 8 && st == LBM_OK; c *= 2) {
        for (int ti = tfirst; ti <= tlast && st == LBM_OK; ++ti) {
            if (lbm_batch_set_cluster(b, c, cthreads[ti]) != LBM_OK) continue;
            float ms = 0;
            if (!trial(&ms)) { st = LBM_E_CUDA; break; }
            if (ms < best) {
                best = ms;
                best_c = c;
                best_ct = cthreads[ti];
            }
        }
    }
    // grouped cluster form: each instance on the smallest cluster whose slices
    // fit a shared-memory cap (balanced against the largest 8-CTA slice, the
    // whole opt-in size, or 72 KB), one launch per cluster size
    const int caps[3] = {LBM_GROUPS_BALANCED, 0, 72 * 1024};
    int best_cap = -1;
    for (int ci = 0; ci < 3 && st == LBM_OK; ++ci) {
        for (int ti = tfirst; ti <= tlast && st == LBM_OK; ++ti) {
            if (lbm_batch_set_groups(b, caps[ci], cthreads[ti]) != LBM_OK) continue;
            float ms = 0;
            if (!trial(&ms)) { st = LBM_E_CUDA; break; }
            if (ms < best) {
                best = ms;
                best_c = -1;
                best_ct = cthreads[ti];
                best_cap = caps[ci];
            }
        }
    }
    b->block_threads = grid_t;
    b->grid_blocks = grid_g;
    b->cluster = 0;
    if (best_c > 0 && st == LBM_OK && lbm_batch_set_cluster(b, best_c, best_ct) != LBM_OK)
        st = LBM_E_CUDA;   // re-applies the kernel attributes of the winning shape
    if (best_c < 0 && st == LBM_OK && lbm_batch_set_groups(b, best_cap, best_ct) != LBM_OK) st = LBM_E_CUDA;
    // restore the state and the error word
    if (cudaMemcpyAsync(b->f[cur0], save, fbytes, cudaMemcpyDeviceToDevice, b->stream) != cudaSuccess) st = LBM_E_CUDA;
    b->cur = cur0;
    cudaMemsetAsync(b->err, 0, sizeof(int), b->stream);
    cudaStreamSynchronize(b->stream);
    dev_free(save);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    int t_out = 0, g_out = 0;
    lbm_batch_get_launch(b, &t_out, &g_out);
    if (block_threads) *block_threads = t_out;
    if (grid_blocks) *grid_blocks = g_out;
    return st == LBM_OK ? LBM_OK : bfail(b, st, "autotuning failed");
}

lbm_status lbm_batch_debug_skip_barrier(lbm_batch *b, int block, double limit_seconds) {
    if (!b || !(limit_seconds > 0) || limit_seconds > 60) return LBM_E_INVALID;
    b->skip_block = block;
    b->limit_ns = (unsigned long long)(limit_seconds * 1e9);
    return LBM_OK;
}

const char *lbm_batch_last_error(const lbm_batch *b) { return b ? b->msg.c_str() : "null batch"; }

void lbm_batch_destroy(lbm_batch *b) {
    if (!b) return;
    if (b->stream) cudaStreamSynchronize(b->stream);
    else cudaDeviceSynchronize();
    drop_graph(b, 0);
    drop_graph(b, 1);
    dev_free(b->inst_dev);
    dev_free(b->table_dev);
    dev_free(b->tiles_dev);
    dev_free(b->order_dev);
    dev_free(b->gorder_dev);
    for (int g = 0; g < 3; ++g) {
        if (b->gstream[g]) cudaStreamDestroy(b->gstream[g]);
        if (b->gjoin[g]) cudaEventDestroy(b->gjoin[g]);
    }
    if (b->gfork) cudaEventDestroy(b->gfork);
    dev_free(b->f[0]);
    dev_free(b->f[1]);
    dev_free(b->q);
    dev_free(b->stage_dev);
    dev_free(b->mom_dev);
    if (b->mom_host) host_free(b->mom_host);
    dev_free(b->err);
    dev_free(b->bar);
    if (b->stage_host) host_free(b->stage_host);
    delete b;
}

}  // extern "C"
