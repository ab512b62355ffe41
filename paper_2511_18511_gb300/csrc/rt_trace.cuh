// rt_trace.cuh — device-side ray tracer for the two-point ray-tracing library.
//
// One ray per thread. The sound-speed field is packed per node as
// (c, h*dc/dx, h*dc/dy, s=1/c) (float4 or 32-byte double4), L2-resident, and
// sampled bilinearly (paper Sec. 3.3.1: field and gradient are interpolated
// from the four vertices of the enclosing cell). Positions are kept
// cell-local: an integer cell (ci, cj) plus a fraction in [0, 1) per axis,
// so FP32 keeps ~1e-8 of a cell of resolution anywhere on a 1024^2 grid. The
// current cell's bilinear coefficients are cached in registers and reloaded
// only when a sample falls in another cell (about once per 8 steps at
// ds = h/10), which turns the march from L2-gather-bound into FMA-bound.
//
// Ray equations (paper Sec. 3.2.3: x and unit d evolve from the sound speed
// and its gradient), written in cell units s~ = s/h:
//     dX/ds~ = d,    dd/ds~ = -(g - (g.d) d) / c,    g = h grad c,
// marched with classic RK4 at a fixed step and d renormalised after each step.
// A trace ends at the first step (after the first) that ends on or outside the
// ring |x| = R; the last point is replaced by the boundary interception, reached
// by a shortened RK4 step ds' (paper Sec. 4.2), found from the chord-circle
// root plus two Newton corrections in FP64. The travel time is the trapezoid
// rule over the points with the interpolated slowness plus the first-order
// endpoint correction s(x_M) d_M.(x_r - x_M) (Appendix: grad T.grad T = c^-2,
// so grad T = s d along the ray).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace rt {

struct __align__(32) D4 {
    double x, y, z, w;
};

template <typename T> struct Vec4T;
template <> struct Vec4T<float> { using type = float4; };
template <> struct Vec4T<double> { using type = D4; };

// Bilinear coefficients of one grid cell for the four sampled fields
// (c, h dc/dx, h dc/dy, s): f(tx, ty) = a + tx bx + ty (by + tx bxy), each field
// one vector (a, bx, by, bxy). Cell (i, j) spans nodes i..i+1, j..j+1 and is
// stored at j*(nx-1) + i. A cell reload is four contiguous vector loads.
template <typename T>
struct CellCoef {
    typename Vec4T<T>::type c, gx, gy, s;
};

template <typename T> struct NodeT { using type = CellCoef<T>; };

// Per-launch geometry (kernel parameter).
struct Geom {
    int nx, ny;
    double h, x0, y0, R;
    double inv_R2;          // 1 / R^2
    int heun;               // 1: Heun's second-order Runge-Kutta, 0: classic RK4
    int interp;             // enum rt_interpolator of the packed field
    double ds;              // mm
    int Ox, Oy;             // floor of the ring centre in cell coordinates (-x0/h, -y0/h)
    double oxf, oyf;        // fractional parts of the ring centre
    long long Q;            // floor((R/h)^2)
    double q;               // (R/h)^2 - Q
    long long max_steps;    // ceil(8 R / ds)
    int max_steps_i;
    const double* tx;       // [2 n_tx]
    int n_tx;
    const int* pairs;       // [2 n_pairs] or null
    int n_pairs;
    const int* bad_field;   // device flag set by the pack kernel (c <= 0 or NaN)
    const double* tx_phi;   // [n_tx] polar angle of each transducer, NaN if off the ring; null = compute
    // FP32 copies of the per-step constants, so the FP32 march issues no FP64
    float Hf, dsf, Rcf, oxff, oyff, qf;
    double Hd, Rcd;         // ds / h and R / h
    int ilast, jlast, row;  // nx - 2, ny - 2: the last cell of an axis; nx - 1: cells per row
    int Qi;                 // Q as 32-bit (grids up to 32k cells per side)
};

// Per-step constants in the marching precision.
template <typename T> struct StepK;
template <> struct StepK<float> {
    __device__ __forceinline__ static float H(const Geom& G) { return G.Hf; }
    __device__ __forceinline__ static float ds(const Geom& G) { return G.dsf; }
    __device__ __forceinline__ static float Rc(const Geom& G) { return G.Rcf; }
    __device__ __forceinline__ static float oxf(const Geom& G) { return G.oxff; }
    __device__ __forceinline__ static float oyf(const Geom& G) { return G.oyff; }
    __device__ __forceinline__ static float q(const Geom& G) { return G.qf; }
};
template <> struct StepK<double> {
    __device__ __forceinline__ static double H(const Geom& G) { return G.Hd; }
    __device__ __forceinline__ static double ds(const Geom& G) { return G.ds; }
    __device__ __forceinline__ static double Rc(const Geom& G) { return G.Rcd; }
    __device__ __forceinline__ static double oxf(const Geom& G) { return G.oxf; }
    __device__ __forceinline__ static double oyf(const Geom& G) { return G.oyf; }
    __device__ __forceinline__ static double q(const Geom& G) { return G.q; }
};

__device__ __forceinline__ void pair_of(const Geom& G, int k, int& e, int& r) {
    if (G.pairs) {
        e = G.pairs[2 * k];
        r = G.pairs[2 * k + 1];
    } else {
        int n1 = G.n_tx - 1;
        e = k / n1;
        int rr = k - e * n1;
        r = rr + (rr >= e);
    }
}

// 1/c for the ray equations: the hardware approximation (about 1 ulp) in FP32.
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// In FP64 the hardware's approximation refined by two Newton steps, each of
// which squares the error: 4 FP64 operations against a division's 8 or more, on
// a part whose FP64 rate is 1/64 of FP32. The sound speed is a normal number.
__device__ __forceinline__ double rcp_approx(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}

// 0 <= u, v < 1 without a branch between the tests. In FP64 on the high words,
// which keeps the test off the FP64 pipe: those of a non-negative number below 1
// are below 1's, those of a negative one (-0 too) or NaN are not. The same form on
// FP32 bits was slower in the bicubic march: a cold link of 16,256 pairs and its
// gradient at 384^2 10.3 ms, 9.5 by comparisons, 65,280 warm links 7.9 and 7.2,
// ray-Born maps of 8 transducers at 128^2 3.10 and 2.87.
__device__ __forceinline__ bool in_unit(float u, float v) {
    return (u >= 0.0f) & (u < 1.0f) & (v >= 0.0f) & (v < 1.0f);
}
__device__ __forceinline__ bool in_unit(double u, double v) {
    return max((unsigned)__double2hiint(u), (unsigned)__double2hiint(v)) < 0x3ff00000u;
}

// Two FP32 values in one 64-bit register pair. Each operation below is one
// instruction that rounds both halves exactly as its scalar form does, so the
// march's (x, y) pairs cost half the issue slots of scalar code.
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 pk2(float x, float y) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ F2 dup2(float x) { return pk2(x, x); }
__device__ __forceinline__ void unpk2(F2 a, float& x, float& y) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 sub2(F2 a, F2 b) {
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

// ---------------------------------------------------------------- field cache

// The cell (i, j) and in-cell fractions (tx, ty) of a point given by fractions
// (u, v) relative to cell (ci, cj); returns whether (i, j) differs from the
// cached cell (pi, pj). Stage points lie within one cell of the current one
// when ds <= h, so the offsets come from comparisons (no conversion
// instructions, which are slow on this part); larger offsets take the floor path.
template <typename T>
__device__ __forceinline__ bool cell_locate(int ci, int cj, T u, T v, int pi, int pj, int& i, int& j, T& tx,
                                            T& ty) {
    const bool in = in_unit(u, v);
    if (ci == pi && cj == pj && in) {
        tx = u;
        ty = v;
        return false;
    }
    if (u >= (T)-1 && u < (T)2 && v >= (T)-1 && v < (T)2) {
        const bool ul = u < (T)0, uh = u >= (T)1, vl = v < (T)0, vh = v >= (T)1;
        tx = ul ? u + (T)1 : (uh ? u - (T)1 : u);
        ty = vl ? v + (T)1 : (vh ? v - (T)1 : v);
        i = ci + (ul ? -1 : (uh ? 1 : 0));
        j = cj + (vl ? -1 : (vh ? 1 : 0));
    } else {
        const T fu = floor(u), fv = floor(v);
        i = ci + (int)fu;
        j = cj + (int)fv;
        tx = u - fu;
        ty = v - fv;
    }
    return i != pi || j != pj;
}

template <typename T>
struct Cell {
    using V = CellCoef<T>;
    const V* __restrict__ F;
    int nx, ny;
    int pi, pj;                       // cached cell
    T ca, cbx, cby, cbxy;             // c      = ca + tx cbx + ty (cby + tx cbxy)
    T xa, xbx, xby, xbxy;             // h dc/dx
    T ya, ybx, yby, ybxy;             // h dc/dy
    T sa, sbx, sby, sbxy;             // s

    __device__ __forceinline__ void grid(const Geom& G) { nx = G.nx; ny = G.ny; }

    __device__ __forceinline__ void load(int i, int j) {
        pi = i;
        pj = j;
        // clamp for memory safety; rays stay inside by the ring/grid check
        i = min(max(i, 0), nx - 2);
        j = min(max(j, 0), ny - 2);
        const V* p = F + (size_t)j * (nx - 1) + i;
        const auto c = p->c, x = p->gx, y = p->gy, w = p->s;
        ca = c.x; cbx = c.y; cby = c.z; cbxy = c.w;
        xa = x.x; xbx = x.y; xby = x.z; xbxy = x.w;
        ya = y.x; ybx = y.y; yby = y.z; ybxy = y.w;
        sa = w.x; sbx = w.y; sby = w.z; sbxy = w.w;
    }

    // (u, v): fractions relative to cell (ci, cj), possibly outside [0, 1)
    __device__ __forceinline__ void at(int ci, int cj, T u, T v, T& c, T& gx, T& gy, T& tx, T& ty) {
        int i, j;
        if (cell_locate(ci, cj, u, v, pi, pj, i, j, tx, ty)) load(i, j);
        c = ca + tx * cbx + ty * (cby + tx * cbxy);
        gx = xa + tx * xbx + ty * (xby + tx * xbxy);
        gy = ya + tx * ybx + ty * (yby + tx * ybxy);
    }

    // slowness at fractions (tx, ty) of the cached cell
    __device__ __forceinline__ T slow(T tx, T ty) const { return sa + tx * sbx + ty * (sby + tx * sbxy); }
};

// The FP32 cell: the same bilinear coefficients as two pairs of fields, (c, s)
// and (h dc/dx, h dc/dy), so that a sample is packed arithmetic. o = (ci - pi,
// cj - pj) of a step carries fractions of the step's own cell to the cached
// one, which makes the in-cell test of a stage three instructions.
struct __align__(32) CellPairs {
    float4 v[4];   // (a_c, a_s, bx_c, bx_s), (by_c, by_s, bxy_c, bxy_s), then the same of (gx, gy)
};

template <>
struct CellCoef<float> {
    CellPairs p;
};

// The cell i of fraction u in [-1, 2) of cell c, and the offset c - i.
__device__ __forceinline__ void axis_move(float u, int c, int& i, float& o) {
    const bool lo = u < 0.0f, hi = u >= 1.0f;
    o = lo ? 1.0f : (hi ? -1.0f : 0.0f);
    i = c + (lo ? -1 : (hi ? 1 : 0));
}

template <>
struct Cell<float> {
    using V = CellCoef<float>;
    const V* __restrict__ F;
    int ilast, jlast, row;            // Geom's
    int pi, pj;                       // cached cell
    F2 sa, sx, sy, sxy;               // (c, s) = sa + tx sx + ty (sy + tx sxy)
    F2 ga, gx, gy, gxy;               // (h dc/dx, h dc/dy)

    __device__ __forceinline__ void grid(const Geom& G) { ilast = G.ilast; jlast = G.jlast; row = G.row; }

    __device__ __forceinline__ void load(int i, int j) {
        pi = i;
        pj = j;
        // to the edge cell on each axis, as in FP64, one instruction each:
        // max(min(i, nx - 2), 0). The ring check leaves a step and a cell around
        // the ring; stages of steps of several cells in a steep field go beyond.
        // The bounds come from the kernel's parameter: formed here from nx and ny
        // they cost registers (all travel times of 261,632 pairs at 1024^2 16.7 ms
        // against 15.1, 65,280 adjoints 5.03 against 4.95). One clamp of the linear
        // index, which took another row's cell out there, measures the same (0.1 % on
        // the mean of fifty calls, links, travel times, adjoints and batches).
        i = __vimin_s32_relu(i, ilast);
        j = __vimin_s32_relu(j, jlast);
        const V* p = F + ((unsigned)j * (unsigned)row + (unsigned)i);
        asm("ld.global.nc.v4.b64 {%0, %1, %2, %3}, [%4];" : "=l"(sa.v), "=l"(sx.v), "=l"(sy.v), "=l"(sxy.v) : "l"(p));
        asm("ld.global.nc.v4.b64 {%0, %1, %2, %3}, [%4 + 32];" : "=l"(ga.v), "=l"(gx.v), "=l"(gy.v), "=l"(gxy.v) : "l"(p));
    }

    // Moves the cache to the cell of a point outside it: its fractions and the
    // offset of the step's cell (ci, cj) from it.
    __device__ __forceinline__ void move(int ci, int cj, float u, float v, float& ox, float& oy, float& tx, float& ty) {
        int i, j;
        axis_move(u, ci, i, ox);
        axis_move(v, cj, j, oy);
        if (!(u >= -1.0f && u < 2.0f && v >= -1.0f && v < 2.0f)) {   // steps longer than a cell
            const float fu = floorf(u), fv = floorf(v);
            i = ci + (int)fu;
            j = cj + (int)fv;
            ox = -fu;
            oy = -fv;
        }
        tx = u + ox;
        ty = v + oy;
        load(i, j);
    }

    // First point of a step, (u, v) relative to cell (ci, cj).
    __device__ __forceinline__ void seek(int ci, int cj, float u, float v, float& ox, float& oy, float& tx, float& ty) {
        // opaque zeros: known ones would let the compiler clone the rest of the
        // step for the unmoved case, which keeps the lanes of a warp apart
        asm("mov.f32 %0, 0f00000000;" : "=f"(ox));
        asm("mov.f32 %0, 0f00000000;" : "=f"(oy));
        tx = u;
        ty = v;
        if (!(ci == pi && cj == pj && max(__float_as_uint(u), __float_as_uint(v)) < 0x3f800000u))
            move(ci, cj, u, v, ox, oy, tx, ty);
    }
    // A later point of the step. Bits below those of 1.0f are the fractions in
    // [0, 1): u + ox is then the fraction cell_locate gives for that cell.
    __device__ __forceinline__ void next(int ci, int cj, F2 p, float& ox, float& oy, float& tx, float& ty) {
        unpk2(add2(p, pk2(ox, oy)), tx, ty);
        if (max(__float_as_uint(tx), __float_as_uint(ty)) >= 0x3f800000u) {
            float u, v;
            unpk2(p, u, v);
            move(ci, cj, u, v, ox, oy, tx, ty);
        }
    }
    __device__ __forceinline__ F2 cs(float tx, float ty) const {
        const F2 x = dup2(tx);
        return fma2(dup2(ty), fma2(x, sxy, sy), fma2(x, sx, sa));
    }
    __device__ __forceinline__ float c(float tx, float ty) const {
        float a, b, d, e, t;
        unpk2(sa, a, t);
        unpk2(sx, b, t);
        unpk2(sy, d, t);
        unpk2(sxy, e, t);
        return fmaf(ty, fmaf(tx, e, d), fmaf(tx, b, a));
    }
    __device__ __forceinline__ F2 grad(float tx, float ty) const {
        const F2 x = dup2(tx);
        return fma2(dup2(ty), fma2(x, gxy, gy), fma2(x, gx, ga));
    }

    __device__ __forceinline__ void at(int ci, int cj, float u, float v, float& c_, float& gx_, float& gy_, float& tx,
                                       float& ty) {
        float ox, oy;
        seek(ci, cj, u, v, ox, oy, tx, ty);
        c_ = c(tx, ty);
        unpk2(grad(tx, ty), gx_, gy_);
    }
    __device__ __forceinline__ float slow(float tx, float ty) const {
        float a, b, d, e, t;
        unpk2(sa, t, a);
        unpk2(sx, t, b);
        unpk2(sy, t, d);
        unpk2(sxy, t, e);
        return fmaf(ty, fmaf(tx, e, d), fmaf(tx, b, a));
    }
};

// ---------------------------------------------------------------- direction

template <typename T> struct Dir;

// FP64: plain unit vector
template <> struct Dir<double> {
    double x, y;
    __device__ __forceinline__ void set(double th) { sincos(th, &y, &x); }
    __device__ __forceinline__ void set_cs(double c, double s) { x = c; y = s; }
    __device__ __forceinline__ double hx() const { return x; }
    __device__ __forceinline__ double hy() const { return y; }
    __device__ __forceinline__ double lx() const { return 0.0; }
    __device__ __forceinline__ double ly() const { return 0.0; }
    __device__ __forceinline__ void add_normalize(double ix, double iy) {
        x += ix;
        y += iy;
        // |d|^2 = 1 + e: 1/sqrt(1 + e) by its series, whose next term is below
        // 3e-17 here, in place of a root and two divisions
        const double e = fma(x, x, fma(y, y, -1.0));
        if (fabsf((float)e) < 1e-4f) {
            const double k = e * fma(e, fma(e, -0.3125, 0.375), -0.5);
            x = fma(x, k, x);
            y = fma(y, k, y);
        } else {
            const double n = sqrt(x * x + y * y);
            x /= n;
            y /= n;
        }
    }
    __device__ __forceinline__ double dx() const { return x; }
    __device__ __forceinline__ double dy() const { return y; }
};

// FP32-compensated: double-float unit vector (hi + lo), so that thousands of
// small RK4 increments do not random-walk the ray angle by FP32 rounding.
template <> struct Dir<float> {
    float x, y, ex, ey;   // value = (x + ex, y + ey)
    __device__ __forceinline__ void set(double th) {
        double c, s;
        sincos(th, &s, &c);
        set_cs(c, s);
    }
    __device__ __forceinline__ void set_cs(double c, double s) {
        x = (float)c; ex = (float)(c - (double)x);
        y = (float)s; ey = (float)(s - (double)y);
    }
    __device__ __forceinline__ float hx() const { return x; }
    __device__ __forceinline__ float hy() const { return y; }
    __device__ __forceinline__ float lx() const { return ex; }
    __device__ __forceinline__ float ly() const { return ey; }
    __device__ __forceinline__ void add_normalize(float ix, float iy) {
        // two-sum of hi + increment, error into lo
        float s = x + ix, bb = s - x;
        ex += (x - (s - bb)) + (ix - bb);
        x = s;
        s = y + iy; bb = s - y;
        ey += (y - (s - bb)) + (iy - bb);
        y = s;
        // |d|^2 - 1 to first order in lo, then d *= 1/sqrt(1+e) = 1 + delta
        float e = fmaf(x, x, fmaf(y, y, -1.0f)) + 2.0f * (x * ex + y * ey);
        float delta = e * fmaf(0.375f, e, -0.5f);
        ex = fmaf(x + ex, delta, ex);
        ey = fmaf(y + ey, delta, ey);
        // renormalise the hi/lo split (fast two-sum, |hi| >= |lo|)
        s = x + ex; ex -= s - x; x = s;
        s = y + ey; ey -= s - y; y = s;
    }
    __device__ __forceinline__ double dx() const { return (double)x + (double)ex; }
    __device__ __forceinline__ double dy() const { return (double)y + (double)ey; }
};

// ---------------------------------------------------------------- RK4 in cell units

template <typename T>
struct RayState {
    int ci, cj;
    T fx, fy;      // fraction of the cell
    T lx, ly;      // FP32: rounding residual of the fraction (two-sum), FP64: 0
    Dir<T> d;
};

// fraction += inc, keeping the rounding error in the residual (FP32 only)
__device__ __forceinline__ void add_frac(float& f, float& lo, float inc) {
    const float s = f + inc, bb = s - f;
    lo += (f - (s - bb)) + (inc - bb);
    const float s2 = s + lo;
    lo -= s2 - s;
    f = s2;
}
__device__ __forceinline__ void add_frac(double& f, double&, double inc) { f += inc; }

// (g.e) e - g over c for stage direction e
template <typename T>
__device__ __forceinline__ void ray_rhs(T c, T gx, T gy, T ex, T ey, T& kx, T& ky) {
    T ic = rcp_approx(c);
    T gd = gx * ex + gy * ey;
    kx = (gd * ex - gx) * ic;
    ky = (gd * ey - gy) * ic;
}

// One RK4 step of length H (cell units) from S into N. s_here receives the
// slowness at S's position (stage-1 sample) for the trapezoid rule.
template <typename T, typename CellT>
__device__ __forceinline__ void rk4_step(CellT& C, const RayState<T>& S, T H, RayState<T>& N, T& s_here,
                                         T& tx1, T& ty1, int& i1, int& j1) {
    const T Hh = (T)0.5 * H, H6 = H / (T)6;
    const T dx = S.d.hx(), dy = S.d.hy();
    T c, gx, gy, tx, ty, k1x, k1y, k2x, k2y, k3x, k3y, k4x, k4y;
    C.at(S.ci, S.cj, S.fx, S.fy, c, gx, gy, tx1, ty1);
    i1 = C.pi;
    j1 = C.pj;
    s_here = C.slow(tx1, ty1);
    ray_rhs(c, gx, gy, dx, dy, k1x, k1y);
    T e2x = dx + Hh * k1x, e2y = dy + Hh * k1y;
    C.at(S.ci, S.cj, S.fx + Hh * dx, S.fy + Hh * dy, c, gx, gy, tx, ty);
    ray_rhs(c, gx, gy, e2x, e2y, k2x, k2y);
    T e3x = dx + Hh * k2x, e3y = dy + Hh * k2y;
    C.at(S.ci, S.cj, S.fx + Hh * e2x, S.fy + Hh * e2y, c, gx, gy, tx, ty);
    ray_rhs(c, gx, gy, e3x, e3y, k3x, k3y);
    T e4x = dx + H * k3x, e4y = dy + H * k3y;
    C.at(S.ci, S.cj, S.fx + H * e3x, S.fy + H * e3y, c, gx, gy, tx, ty);
    ray_rhs(c, gx, gy, e4x, e4y, k4x, k4y);
    // every stage direction carries the low part of d, so the position
    // increment gets it in full: H d_lo (zero in FP64); the fraction is
    // accumulated with its rounding residual in FP32
    T nfx = S.fx, nfy = S.fy;
    N.lx = S.lx;
    N.ly = S.ly;
    if constexpr (sizeof(T) == 8) {
        nfx += H6 * (dx + (T)2 * (e2x + e3x) + e4x);
        nfy += H6 * (dy + (T)2 * (e2y + e3y) + e4y);
    } else {
        add_frac(nfx, N.lx, H6 * (dx + (T)2 * (e2x + e3x) + e4x) + H * S.d.lx());
        add_frac(nfy, N.ly, H6 * (dy + (T)2 * (e2y + e3y) + e4y) + H * S.d.ly());
    }
    N.d = S.d;
    N.d.add_normalize(H6 * (k1x + (T)2 * (k2x + k3x) + k4x), H6 * (k1y + (T)2 * (k2y + k3y) + k4y));
    N.ci = S.ci;
    N.cj = S.cj;
    // f - 1 is exact for f in [1, 2); f + 1 for f in [-1, 0) rounds, so it goes
    // through the residual too
    if (sizeof(T) == 4 || !in_unit(nfx, nfy)) {
        if (nfx >= (T)1) { N.ci += 1; nfx -= (T)1; } else if (nfx < (T)0) { N.ci -= 1; add_frac(nfx, N.lx, (T)1); }
        if (nfy >= (T)1) { N.cj += 1; nfy -= (T)1; } else if (nfy < (T)0) { N.cj -= 1; add_frac(nfy, N.ly, (T)1); }
    }
    N.fx = nfx;
    N.fy = nfy;
}

// One step of Heun's second-order Runge-Kutta method (the slopes at S and at
// the Euler end point S + H (d, k1), averaged), in the same cell-unit,
// compensated form as rk4_step.
template <typename T, typename CellT>
__device__ __forceinline__ void heun_step(CellT& C, const RayState<T>& S, T H, RayState<T>& N, T& s_here,
                                          T& tx1, T& ty1, int& i1, int& j1) {
    const T Hh = (T)0.5 * H;
    const T dx = S.d.hx(), dy = S.d.hy();
    T c, gx, gy, tx, ty, k1x, k1y, k2x, k2y;
    C.at(S.ci, S.cj, S.fx, S.fy, c, gx, gy, tx1, ty1);
    i1 = C.pi;
    j1 = C.pj;
    s_here = C.slow(tx1, ty1);
    ray_rhs(c, gx, gy, dx, dy, k1x, k1y);
    const T e2x = dx + H * k1x, e2y = dy + H * k1y;
    C.at(S.ci, S.cj, S.fx + H * dx, S.fy + H * dy, c, gx, gy, tx, ty);
    ray_rhs(c, gx, gy, e2x, e2y, k2x, k2y);
    T nfx = S.fx, nfy = S.fy;
    N.lx = S.lx;
    N.ly = S.ly;
    if constexpr (sizeof(T) == 8) {
        nfx += Hh * (dx + e2x);
        nfy += Hh * (dy + e2y);
    } else {
        add_frac(nfx, N.lx, Hh * (dx + e2x) + H * S.d.lx());
        add_frac(nfy, N.ly, Hh * (dy + e2y) + H * S.d.ly());
    }
    N.d = S.d;
    N.d.add_normalize(Hh * (k1x + k2x), Hh * (k1y + k2y));
    N.ci = S.ci;
    N.cj = S.cj;
    if (sizeof(T) == 4 || !in_unit(nfx, nfy)) {
        if (nfx >= (T)1) { N.ci += 1; nfx -= (T)1; } else if (nfx < (T)0) { N.ci -= 1; add_frac(nfx, N.lx, (T)1); }
        if (nfy >= (T)1) { N.cj += 1; nfy -= (T)1; } else if (nfy < (T)0) { N.cj -= 1; add_frac(nfy, N.ly, (T)1); }
    }
    N.fx = nfx;
    N.fy = nfy;
}

// ((g.e) e - g) / c of the FP32 march, in the operation order of ray_rhs with
// the signs of both factors flipped (exact).
__device__ __forceinline__ F2 ray_rhs2(float c, F2 g, F2 e) {
    float gx, gy, ex, ey;
    unpk2(g, gx, gy);
    unpk2(e, ex, ey);
    const float nic = rcp_approx(-c);
    const float ngd = fmaf(-gy, ey, -__fmul_rn(gx, ex));
    return mul2(fma2(dup2(ngd), e, g), dup2(nic));
}
// a + the same, the product with 1/c rounded once with the sum
__device__ __forceinline__ F2 add_rhs2(F2 a, float c, F2 g, F2 e) {
    float gx, gy, ex, ey;
    unpk2(g, gx, gy);
    unpk2(e, ex, ey);
    const float nic = rcp_approx(-c);
    const float ngd = fmaf(-gy, ey, -__fmul_rn(gx, ex));
    return fma2(fma2(dup2(ngd), e, g), dup2(nic), a);
}

// Position and direction of a step from its increments: position by sum Hp
// E + H d_lo, direction by Hp K, both as rk4_step forms them.
__device__ __forceinline__ void commit2(const RayState<float>& S, float H, float Hp, F2 E, F2 K, RayState<float>& N) {
    const F2 dl = pk2(S.d.ex, S.d.ey), hp = dup2(Hp), h1 = dup2(H);
    // compensated position
    const F2 f = pk2(S.fx, S.fy), l = pk2(S.lx, S.ly);
    const F2 inc = fma2(h1, dl, mul2(hp, E));
    const F2 s = add2(f, inc), b = sub2(s, f);
    F2 lo = add2(l, add2(sub2(f, sub2(s, b)), sub2(inc, b)));
    const F2 nf = add2(s, lo);
    lo = sub2(lo, sub2(nf, s));
    unpk2(lo, N.lx, N.ly);
    // compensated direction, renormalised
    const F2 d = pk2(S.d.x, S.d.y);
    const F2 x = fma2(hp, K, d), nb = sub2(d, x);
    F2 e = add2(dl, add2(sub2(d, add2(x, nb)), fma2(hp, K, nb)));
    float dx, dy, ex, ey;
    unpk2(x, dx, dy);
    unpk2(e, ex, ey);
    const float q = fmaf(dx, ex, __fmul_rn(dy, ey));
    const float er = fmaf(2.0f, q, fmaf(dx, dx, fmaf(dy, dy, -1.0f)));
    const F2 delta = dup2(__fmul_rn(er, fmaf(0.375f, er, -0.5f)));
    e = fma2(add2(x, e), delta, e);
    const F2 xs = add2(x, e);
    e = sub2(e, sub2(xs, x));
    unpk2(xs, N.d.x, N.d.y);
    unpk2(e, N.d.ex, N.d.ey);
    float nfx, nfy;
    unpk2(nf, nfx, nfy);
    N.ci = S.ci;
    N.cj = S.cj;
    // into the next cell: f - 1 is exact for f in [1, 2); f + 1 for f < 0 rounds,
    // so it goes through the residual (both axes at once, add_frac's operations)
    if (max(__float_as_uint(nfx), __float_as_uint(nfy)) >= 0x3f800000u) {
        const bool xl = nfx < 0.0f, xh = nfx >= 1.0f, yl = nfy < 0.0f, yh = nfy >= 1.0f;
        const F2 a = pk2(xl ? 1.0f : (xh ? -1.0f : 0.0f), yl ? 1.0f : (yh ? -1.0f : 0.0f));
        const F2 t = add2(nf, a), tb = sub2(t, nf);
        F2 r = add2(lo, add2(sub2(nf, sub2(t, tb)), sub2(a, tb)));
        const F2 t2 = add2(t, r);
        r = sub2(r, sub2(t2, t));
        float x1, y1, x2, y2, rx, ry;
        unpk2(t, x1, y1);
        unpk2(t2, x2, y2);
        unpk2(r, rx, ry);
        nfx = xl ? x2 : x1;
        nfy = yl ? y2 : y1;
        if (xl) N.lx = rx;
        if (yl) N.ly = ry;
        N.ci += xl ? -1 : (xh ? 1 : 0);
        N.cj += yl ? -1 : (yh ? 1 : 0);
    }
    N.fx = nfx;
    N.fy = nfy;
}

// rk4_step of the FP32 bilinear march: the same operations on packed pairs,
// bit for bit. The march issues instructions (a full GPU) or waits for its own
// dependent chain (few rays); it moves almost no memory. Packing takes a lone
// ray from 258 to 186 instructions a step; a packed operation has a longer
// latency, so that alone saved 4 % of a full launch and nothing of a lone ray.
// The rest came from what surrounds the arithmetic: a cell move of 20
// instructions in place of 45 (every lane that leaves its cell costs the whole
// warp one), two 32-byte loads a cell, one branch for the wrap of both axes,
// one for all rare ends of a step. Each stage's cell lookup comes before the
// slopes of the stage before it, so that those slopes and the new sample are
// one block of independent work. Together, on the breast medium (1024^2, 512
// transducers): recording link 56 -> 45.5 ms cold, 25.3 -> 22.2 ms warm; plain
// link 50 -> 40.4 and 19.3 -> 15.9 ms; adjoint 24.1 -> 20.8 ms; one ray 345 ->
// 266 ns a step. Loading the next cell ahead of its use (L1 prefetch, cp.async
// or a plain load at the entry of a cell) and scalar slopes were no faster.
__device__ __forceinline__ void rk4_slopes(Cell<float>& C, const RayState<float>& S, float H, F2& E, F2& K,
                                           float& s_here, float& tx1, float& ty1, int& i1, int& j1) {
    const F2 hh = dup2(0.5f * H), h1 = dup2(H), f = pk2(S.fx, S.fy), d = pk2(S.d.x, S.d.y), two = dup2(2.0f);
    float ox, oy, tx, ty, c;
    C.seek(S.ci, S.cj, S.fx, S.fy, ox, oy, tx1, ty1);
    i1 = C.pi;
    j1 = C.pj;
    unpk2(C.cs(tx1, ty1), c, s_here);
    F2 g = C.grad(tx1, ty1);
    C.next(S.ci, S.cj, fma2(hh, d, f), ox, oy, tx, ty);
    const F2 k1 = ray_rhs2(c, g, d);
    c = C.c(tx, ty);
    g = C.grad(tx, ty);
    const F2 e2 = fma2(hh, k1, d);
    C.next(S.ci, S.cj, fma2(hh, e2, f), ox, oy, tx, ty);
    const F2 k2 = ray_rhs2(c, g, e2);
    c = C.c(tx, ty);
    g = C.grad(tx, ty);
    const F2 e3 = fma2(hh, k2, d);
    C.next(S.ci, S.cj, fma2(h1, e3, f), ox, oy, tx, ty);
    const F2 k3 = ray_rhs2(c, g, e3);
    const F2 e4 = fma2(h1, k3, d);
    c = C.c(tx, ty);
    g = C.grad(tx, ty);
    E = add2(fma2(two, add2(e2, e3), d), e4);
    K = add_rhs2(fma2(two, add2(k2, k3), k1), c, g, e4);
}

// The same for a step whose four samples all lie in the cached cell, assumed
// first and tested last: one branch a step, and the samples' arithmetic
// overlaps. Returns whether they did; if not, the outputs mean nothing.
__device__ __forceinline__ bool rk4_slopes_inside(const Cell<float>& C, const RayState<float>& S, float H, F2& E, F2& K,
                                                  float& s_here) {
    const F2 hh = dup2(0.5f * H), h1 = dup2(H), f = pk2(S.fx, S.fy), d = pk2(S.d.x, S.d.y), two = dup2(2.0f);
    float x, y, c;
    unsigned m = max(__float_as_uint(S.fx), __float_as_uint(S.fy));
    unpk2(fma2(hh, d, f), x, y);
    m = max(m, max(__float_as_uint(x), __float_as_uint(y)));
    const float c2 = C.c(x, y);
    const F2 g2 = C.grad(x, y);
    unpk2(C.cs(S.fx, S.fy), c, s_here);
    const F2 k1 = ray_rhs2(c, C.grad(S.fx, S.fy), d);
    const F2 e2 = fma2(hh, k1, d);
    unpk2(fma2(hh, e2, f), x, y);
    m = max(m, max(__float_as_uint(x), __float_as_uint(y)));
    const F2 k2 = ray_rhs2(c2, g2, e2);
    const F2 e3 = fma2(hh, k2, d);
    const F2 k3 = ray_rhs2(C.c(x, y), C.grad(x, y), e3);
    unpk2(fma2(h1, e3, f), x, y);
    m = max(m, max(__float_as_uint(x), __float_as_uint(y)));
    const F2 e4 = fma2(h1, k3, d);
    E = add2(fma2(two, add2(e2, e3), d), e4);
    K = add_rhs2(fma2(two, add2(k2, k3), k1), C.c(x, y), C.grad(x, y), e4);
    return S.ci == C.pi && S.cj == C.pj && m < 0x3f800000u;
}

__device__ __forceinline__ void rk4_step(Cell<float>& C, const RayState<float>& S, float H, RayState<float>& N,
                                         float& s_here, float& tx1, float& ty1, int& i1, int& j1, bool sparse) {
    F2 E, K;
    bool inside = false;
    if (sparse) {
        tx1 = S.fx;
        ty1 = S.fy;
        i1 = S.ci;
        j1 = S.cj;
        inside = rk4_slopes_inside(C, S, H, E, K, s_here);
    }
    if (!inside) rk4_slopes(C, S, H, E, K, s_here, tx1, ty1, i1, j1);
    commit2(S, H, H / 6.0f, E, K, N);
}

// heun_step of the FP32 bilinear march, packed likewise.
__device__ __forceinline__ void heun_step(Cell<float>& C, const RayState<float>& S, float H, RayState<float>& N,
                                          float& s_here, float& tx1, float& ty1, int& i1, int& j1) {
    const float Hh = 0.5f * H;
    const F2 h1 = dup2(H), f = pk2(S.fx, S.fy), d = pk2(S.d.x, S.d.y);
    float ox, oy, tx, ty, c;
    C.seek(S.ci, S.cj, S.fx, S.fy, ox, oy, tx1, ty1);
    i1 = C.pi;
    j1 = C.pj;
    unpk2(C.cs(tx1, ty1), c, s_here);
    F2 g = C.grad(tx1, ty1);
    C.next(S.ci, S.cj, fma2(h1, d, f), ox, oy, tx, ty);
    const F2 k1 = ray_rhs2(c, g, d);
    const F2 e2 = fma2(h1, k1, d);
    c = C.c(tx, ty);
    g = C.grad(tx, ty);
    const F2 K = add_rhs2(k1, c, g, e2);
    commit2(S, H, Hh, add2(d, e2), K, N);
}

// Lanes of a warp up to which a step is first tried inside the cached cell.
// Each ray leaves its cell about every eighth step, and the warp then pays for
// both forms of the step: worth it for one to three lanes (one ray 300 ns a
// step against 348 without at the time; 1 or 6 lanes in place of 3 change the
// cold link of 261,632 pairs by less than its runs differ, which is where the line
// was tried; launches of 4 or 5 lanes a warp were not measured). One-trace kernels of wide warps
// leave the form out: it made the adjoint 10 % slower through its registers.
constexpr int kSparseLanes = 3;
__device__ __forceinline__ bool sparse_warp() { return __popc(__activemask()) <= kSparseLanes; }

// The step of the configured integrator (uniform over a launch).
template <typename T, typename CellT>
__device__ __forceinline__ void ray_step(CellT& C, const Geom& G, const RayState<T>& S, T H, RayState<T>& N,
                                         T& s_here, T& tx1, T& ty1, int& i1, int& j1, bool) {
    if (G.heun) heun_step(C, S, H, N, s_here, tx1, ty1, i1, j1);
    else rk4_step(C, S, H, N, s_here, tx1, ty1, i1, j1);
}
__device__ __forceinline__ void ray_step(Cell<float>& C, const Geom& G, const RayState<float>& S, float H,
                                         RayState<float>& N, float& s_here, float& tx1, float& ty1, int& i1, int& j1,
                                         bool sparse) {
    if (G.heun) heun_step(C, S, H, N, s_here, tx1, ty1, i1, j1);
    else rk4_step(C, S, H, N, s_here, tx1, ty1, i1, j1, sparse);
}

// |x|^2 - (R/h)^2 in cell^2 units, exact integer part plus a small fractional
// part, so the sign is reliable to ~1e-7 cell even in FP32.
template <typename T>
__device__ __forceinline__ T ring_excess(const Geom& G, const RayState<T>& S) {
    const int Ix = S.ci - G.Ox, Iy = S.cj - G.Oy;
    const T px = S.fx - StepK<T>::oxf(G), py = S.fy - StepK<T>::oyf(G);
    const int I2 = Ix * Ix + Iy * Iy - G.Qi;
    const T d0 = (T)I2 - StepK<T>::q(G);
    return d0 + (T)2 * ((T)Ix * px + (T)Iy * py) + px * px + py * py;
}

template <typename T>
__device__ __forceinline__ void abs_pos(const Geom& G, const RayState<T>& S, double& X, double& Y) {
    X = G.x0 + G.h * ((double)S.ci + ((double)S.fx + (double)S.lx));
    Y = G.y0 + G.h * ((double)S.cj + ((double)S.fy + (double)S.ly));
}

// ---------------------------------------------------------------- scatter (adjoint / matrix rows)

// Exact float -> double by integer bit operations (normal numbers; zeros and
// subnormals give +-0), avoiding a conversion instruction.
__device__ __forceinline__ double f2d_bits(float f) {
    const unsigned u = __float_as_uint(f);
    const unsigned ex = (u >> 23) & 0xffu;
    const unsigned long long sign = (unsigned long long)(u & 0x80000000u) << 32;
    if (ex == 0) return __longlong_as_double((long long)sign);
    if (ex == 0xffu)   // inf / NaN keep their class
        return __longlong_as_double((long long)(sign | (0x7ffull << 52) | ((unsigned long long)(u & 0x7fffffu) << 29)));
    const unsigned long long bits = sign | ((unsigned long long)(ex + 896u) << 52) |
                                    ((unsigned long long)(u & 0x7fffffu) << 29);
    return __longlong_as_double((long long)bits);
}

__device__ __forceinline__ double to_double(float f) { return f2d_bits(f); }
__device__ __forceinline__ double to_double(double d) { return d; }

// Accumulates the trapezoid-weighted bilinear weights of consecutive points
// that fall in one cell, as (sum w, sum w tx, sum w ty, sum w tx ty).
template <typename T>
struct CellAcc {
    int ai, aj;
    T W, Wx, Wy, Wxy;
    __device__ __forceinline__ void reset() { ai = INT_MIN; aj = INT_MIN; W = Wx = Wy = Wxy = (T)0; }
    __device__ __forceinline__ void node_weights(double& w00, double& w10, double& w01, double& w11) const {
        w11 = (double)Wxy;
        w10 = (double)Wx - w11;
        w01 = (double)Wy - w11;
        w00 = (double)W - (double)Wx - (double)Wy + w11;
    }
};

// Trace outcome.
struct TraceOut {
    double T;          // travel time (us) incl. endpoint correction
    double hx, hy;     // interception
    int flags;         // bit0: step cap, bit1: left outward at once
    long long steps;   // RK4 steps taken (incl. landing)
};

// Sink interface used by trace(): add(ci, cj, tx, ty, w) for each point.
struct NoSink {
    template <typename T>
    __device__ __forceinline__ void add(int, int, T, T, T) {}
    __device__ __forceinline__ void finish() {}
};

// Resumable trace: begin / step (until it reports the end) / end. The
// persistent linking kernel interleaves traces of different pairs per lane.
template <typename T>
struct TraceState {
    RayState<T> S;
    T s_first, s_cur;
    T Ssum, Scomp;            // Kahan sum of s at points 1..M-1
    int m;                    // index of the current point
    int safe;                 // steps that cannot reach the ring (exit test skipped)
    int flags;                // bit0 step cap, bit1 left outward at once
    int iL, jL;               // cell and fractions of the last full-step point
    T txL, tyL;
};

// Starts a trace at (xe, ye) with unit launch direction (c, s).
template <typename T>
__device__ __forceinline__ void trace_begin_cs(TraceState<T>& ts, const Geom& G, double xe, double ye, double c,
                                               double s) {
    const double u = (xe - G.x0) / G.h, v = (ye - G.y0) / G.h;
    const double fu = floor(u), fv = floor(v);
    ts.S.ci = (int)fu;
    ts.S.cj = (int)fv;
    ts.S.fx = (T)(u - fu);
    ts.S.fy = (T)(v - fv);
    ts.S.lx = (T)((u - fu) - (double)ts.S.fx);
    ts.S.ly = (T)((v - fv) - (double)ts.S.fy);
    ts.S.d.set_cs(c, s);
    ts.s_first = ts.s_cur = (T)0;
    ts.Ssum = ts.Scomp = (T)0;
    ts.m = 0;
    ts.safe = 0;
    ts.flags = 0;
    ts.iL = ts.jL = 0;
    ts.txL = ts.tyL = (T)0;
}

template <typename T>
__device__ __forceinline__ void trace_begin(TraceState<T>& ts, const Geom& G, double xe, double ye, double theta) {
    double c, s;
    sincos(theta, &s, &c);
    trace_begin_cs(ts, G, xe, ye, c, s);
}

// One RK4 step. Returns true when the trace has ended: the step ended on or
// outside the ring (flags bit1 if that was the very first step) or the step
// cap was reached (flags bit0). On exit ts.S is still the last inside point.
template <typename T, typename CellT, typename Sink>
__device__ __forceinline__ bool trace_step(CellT& C, const Geom& G, TraceState<T>& ts, Sink& sink, bool sparse) {
    const T H = StepK<T>::H(G);
    T w = StepK<T>::ds(G);
    RayState<T> N;
    T tx1, ty1;
    int i1, j1;
    ray_step(C, G, ts.S, H, N, ts.s_cur, tx1, ty1, i1, j1, sparse);
    int end = 0;   // 1: the step ended on or outside the ring, 2: as the first step, 3: the step cap
    // Everything that can only happen on a step that may reach the ring, on the
    // first step (safe starts at 0) or at the step cap is behind this one test.
    if (--ts.safe < 0) {
        const T ex = ring_excess(G, N);
        if (ex >= (T)0) end = ts.m == 0 ? 2 : 1;
        if (ts.m == 0) {
            ts.s_first = ts.s_cur;
            ts.Scomp = ts.s_cur;   // the sum below stays 0 on this step
            w *= (T)0.5;
        }
        if (!end) {
            // distance to the ring in cells, -ex / (R + r); no step moves farther than ~H
            const T Rc = StepK<T>::Rc(G);
            const T r = sqrt(Rc * Rc + ex);
            const T dist = -ex / (Rc + r);
            const int left = G.max_steps_i - 2 - ts.m;   // free steps before the last one allowed
            ts.safe = min((int)(dist * (T)0.98 / H) - 1, left);
            if (left < 0) end = 3;
        }
    }
    // opaque: with the end codes known per path the compiler clones the rest of
    // the step, and the lanes of a warp that took this branch stay apart
    asm volatile("" : "+r"(end));
    if (end == 2) {   // left outward: no path, no weights
        ts.s_first = (T)0;
        ts.flags |= 2;
        return true;
    }
    const T y = ts.s_cur - ts.Scomp;
    const T t = ts.Ssum + y;
    ts.Scomp = (t - ts.Ssum) - y;
    ts.Ssum = t;
    sink.add(i1, j1, tx1, ty1, w);
    if (end == 1) {
        ts.iL = i1; ts.jL = j1; ts.txL = tx1; ts.tyL = ty1;
        return true;
    }
    ts.S = N;
    ++ts.m;
    if (end == 3) ts.flags |= 1;
    return end != 0;
}

// Landing, travel time and final weights of an ended trace. The endpoint
// correction is taken toward (xr, yr).
template <typename T, typename CellT, typename Sink>
__device__ TraceOut trace_end(CellT& C, const Geom& G, TraceState<T>& ts, double xe, double ye, double xr,
                              double yr, Sink& sink) {
    TraceOut out;
    out.flags = ts.flags;
    if (ts.flags & 1) {
        // step cap: no interception; report the current point
        abs_pos(G, ts.S, out.hx, out.hy);
        out.T = G.ds * (0.5 * (double)ts.s_first + ((double)ts.Ssum - (double)ts.Scomp));
        out.steps = ts.m;
        sink.finish();
        return out;
    }
    if (ts.flags & 2) {
        out.T = 0.0;
        out.hx = xe;
        out.hy = ye;
        out.steps = 1;
        sink.finish();
        return out;
    }
    const RayState<T>& S = ts.S;
    RayState<T> N;
    double X, Y;
    abs_pos(G, S, X, Y);
    double b = X * S.d.dx() + Y * S.d.dy();
    double qq = X * X + Y * Y - G.R * G.R;
    double disc = b * b - qq;
    if (disc < 0) disc = 0;
    double sq = sqrt(disc);
    double t = (b >= 0) ? (-qq) / (b + sq) : (sq - b);
    if (!(t >= 0)) t = 0;
    if (t > G.ds) t = G.ds;
    T s_dummy, txd, tyd;
    int id, jd;
    for (int it = 0; it < 2; ++it) {
        ray_step(C, G, S, (T)(t / G.h), N, s_dummy, txd, tyd, id, jd, false);
        double NX, NY;
        abs_pos(G, N, NX, NY);
        double r = sqrt(NX * NX + NY * NY);
        double drdt = (NX * N.d.dx() + NY * N.d.dy()) / r;
        if (drdt > 0) t -= (r - G.R) / drdt;
        if (!(t >= 0)) t = 0;
        if (t > G.ds) t = G.ds;
    }
    ray_step(C, G, S, (T)(t / G.h), N, s_dummy, txd, tyd, id, jd, false);
    double MX, MY;
    abs_pos(G, N, MX, MY);
    T c_, gx_, gy_, txM, tyM;
    C.at(N.ci, N.cj, N.fx, N.fy, c_, gx_, gy_, txM, tyM);
    const int iM = C.pi, jM = C.pj;
    const double sM = (double)C.slow(txM, tyM);
    const double sL = (double)ts.s_cur;   // slowness at x_{M-1}
    const double corr = N.d.dx() * (xr - MX) + N.d.dy() * (yr - MY);
    const double S_int = (double)ts.Ssum - (double)ts.Scomp;   // s_1 + ... + s_{M-1}
    out.T = G.ds * (0.5 * (double)ts.s_first + S_int - 0.5 * sL) + 0.5 * t * (sL + sM) + sM * corr;
    out.hx = MX;
    out.hy = MY;
    out.steps = ts.m + 4;   // the full steps inside, the one that crossed, three to land
    // alpha_{M-1} = (ds + ds')/2 (ds was given by trace_step), alpha_M = ds'/2 + corr
    sink.add(ts.iL, ts.jL, ts.txL, ts.tyL, (T)(0.5 * (t - G.ds)));
    sink.add(iM, jM, txM, tyM, (T)(0.5 * t + corr));
    sink.finish();
    return out;
}

// Traces one ray from (xe, ye) at angle theta (begin + steps + end). With a
// sink, every sample point m reports its trapezoid weight alpha_m (and the
// endpoint weight) with its cell and fractions.
template <typename T, typename CellT, typename Sink>
__device__ TraceOut trace_ray(CellT& C, const Geom& G, double xe, double ye, double theta, double xr,
                              double yr, Sink& sink, bool sparse = false) {
    TraceState<T> ts;
    trace_begin(ts, G, xe, ye, theta);
    while (!trace_step(C, G, ts, sink, sparse)) {
    }
    return trace_end(C, G, ts, xe, ye, xr, yr, sink);
}

}  // namespace rt
