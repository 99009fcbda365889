// Fluid stages for 2D FP32 grids (part of the unit flux.cu, whose flags flush
// subnormals): the discretisation of flux.cu (MUSCL/van Leer + Rusanov +
// central viscous/heat fluxes, SSP-RK2 stages) as a march in y by independent
// warps.
//
// One warp owns a strip of 60 columns and walks up a chunk of rows; lane l
// holds the two neighbouring columns ox - 2 + 2l and ox - 1 + 2l, so lanes 0
// and 31 are the strip's two-column halo.  What a face needs along y - the
// primitives of three rows, the limited y-slope and the flux below - stays in
// the lane's registers from row to row; what it needs along x comes from the
// neighbouring lanes by shuffles.  There is no shared memory and no barrier:
// every cell of the strip is loaded and converted once per chunk, every
// limited slope is evaluated once, and every face once (the halo lanes and
// the first row of a chunk repeat their neighbours' work: 64/60 of the
// columns, and about 0.7 row per chunk).
//
// Bound: instruction issue and latency (348 / 430 thread instructions per
// cell and stage at 50 % issue with three to four warps per scheduler, against
// 32 or 48 bytes of memory traffic).  The form this replaces - one cell per
// thread of a 16 x 16 tile, primitives and face fluxes in shared memory, both
// slopes of every face - took ~750.  64-case batch (7.45 M cells): stage 1
// 227 -> 140 us, stage 2 274 -> 171 us; 1024 x 512: 17.7 -> 14.3 and 22.6 ->
// 17.6 us.  Unrolling the row loop (no register moves) overflows the
// instruction cache: 209 and 291 us.
//
// A row's arithmetic does not depend on where its strip or chunk begins, and
// every operation is an explicit rounding (packed FP32x2 intrinsics, no
// contraction left to the compiler), so single grids and batches, whatever
// their chunk height, give the same bits.
#pragma once

#include <float.h>
#include <stdint.h>

#include "flux_pair.cuh"
#include "internal.h"

namespace ibmk {
namespace {

constexpr int YM_W = 60;                  // columns a warp writes
constexpr int YM_ROW_W = 28;              // the same of the single-row form
constexpr int YM_WARPS = 4;               // warps (work items) per CTA
constexpr int YM_T = 32 * YM_WARPS;
constexpr int NC = 4;

using FC = FloatConsts;

__device__ __forceinline__ float from_left(float v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float from_right(float v) { return __shfl_down_sync(0xffffffffu, v, 1); }

// What a strip needs of a grid, in registers: a batch reads it per item from
// the case table, where a reference would reload it after every store.
struct YK {
    int nx, ny;
    long long N;
    int bc0, bc1, bc2, bc3;
    float E_inf;
    // The fluxes are evaluated doubled (mass, momentum) and four-fold
    // (energy), so that no half remains in them; T stands for p / rho.
    float gamma, gm1;
    float e1, h1;          // 2/(gamma-1), 2 + 2/(gamma-1): 2 rho E and 2 rho H less rho |u|^2
    float s2;              // 2 S r
    float km;              // 2 mu / h less T^2 rsqrt(T (T + 2 S r)^2), T the two cells' sum
    float kl;              // 2 c_p / (Pr r)
    float ih2, ih4;        // 1/(2h), 1/(4h)
    float p2;              // 2 p_inf: see less_p
    float ih, kr;          // 1/h and FloatConsts::kr, for the step-size rate
    bool viscous;
};

__device__ __forceinline__ YK make_yk(const GridParams &g) {
    const FC &c = g.f;
    YK k;
    k.nx = g.n[0];
    k.ny = g.n[1];
    k.N = g.N;
    k.bc0 = g.bc[0];
    k.bc1 = g.bc[1];
    k.bc2 = g.bc[2];
    k.bc3 = g.bc[3];
    k.E_inf = c.E_inf;
    k.gamma = c.gamma;
    k.gm1 = c.gm1;
    k.e1 = c.e1;
    k.h1 = c.h1;
    k.s2 = c.s2;
    k.km = c.km;
    k.kl = c.kl;
    k.ih2 = 0.5f * c.inv_h;
    k.ih4 = c.qinv_h;
    k.ih = c.inv_h;
    k.kr = c.kr;
    k.p2 = c.p2;
    k.viscous = c.viscous != 0;
    return k;
}

__device__ __forceinline__ RateK rate_k(const YK &k) {
    return RateK{k.gamma, k.gm1, k.s2, k.km, k.kr, k.ih};
}

// primitives (rho, u, v, p) and p / rho of one row
template <typename V>
struct RowT {
    V w[NC];
    V T;
};
using Row = RowT<float2>;   // the lane's two cells

// Flux of a face, or two, in the face frame: wl, wr the states
// (rho, u_n, u_t, p) on the two sides; dn, dt, dT the differences and sn, st,
// sT the sums over the two cells (upper - lower, upper + lower) of the normal
// and tangential velocity and p / rho; d1n, d1t the sums over the two cells
// of the central differences (w[+1] - w[-1]) of u_n and u_t along the tangent.
// F = 2 (mass, normal momentum, tangential momentum), 4 energy.  The speed of
// sound is gamma p rsqrt(gamma p rho), the viscosity's T^(3/2) / (T + S) is
// T^2 rsqrt(T (T + S)^2): one special-function operation each.
template <typename V>
__device__ __forceinline__ void flux_of(const YK &c, const V (&wl)[NC], const V (&wr)[NC],
                                          V dn, V dt, V dT, V sn, V st,
                                          V sT, V d1n, V d1t, V (&F)[NC]) {
    const V unL = wl[1], unR = wr[1];
    const V mLn = wl[0] * unL, mRn = wr[0] * unR;
    const V mLt = wl[0] * wl[2], mRt = wr[0] * wr[2];
    const V rkL = fma2(mLn, unL, mLt * wl[2]), rkR = fma2(mRn, unR, mRt * wr[2]);
    const V gpL = cmul(c.gamma, wl[3]), gpR = cmul(c.gamma, wr[3]);
    const V sL = fabs_fma(gpL, rsqrt2(gpL * wl[0]), unL);
    const V sR = fabs_fma(gpR, rsqrt2(gpR * wr[0]), unR);
    const V s = max2(sL, sR);
    F[0] = fma2(s, wl[0] - wr[0], mLn + mRn);
    F[1] = fma2(s, mLn - mRn, fma2(mLn, unL, wl[3]) + fma2(mRn, unR, wr[3]));
    F[2] = fma2(s, mLt - mRt, fma2(mLt, unL, mRt * unR));
    const V HL = cfma(c.h1, wl[3], rkL), HR = cfma(c.h1, wr[3], rkR);
    const V EL = cfma(c.e1, wl[3], rkL), ER = cfma(c.e1, wr[3], rkR);
    F[3] = fma2(s, EL - ER, fma2(HL, unL, HR * unR));
    if (!c.viscous) return;
    const V y = cadd(c.s2, sT);
    const V m = cmul(c.km, sT) * (sT * rsqrt2(sT * y * y));
    const V tNN = m * cfma(4.0f / 3.0f, dn, cmul(-1.0f / 6.0f, d1t));
    const V tNT = m * cfma(0.25f, d1n, dt);
    F[1] = F[1] - tNN;
    F[2] = F[2] - tNT;
    F[3] = F[3] - fma2(sn, tNN, fma2(st, tNT, cmul(c.kl, m) * dT));
}

// The lane's columns of a strip.  On an even nx with 8-byte aligned arrays
// (PAIRED) every lane loads the aligned pair that holds its two source columns
// - a ghost pair's sources are the first or last two columns - and, in a warp
// with ghosts, picks and flips its values; otherwise the two columns are
// loaded one by one.
struct Cols {
    int s0, s1;       // source columns; PAIRED: s0 the pair's first column
    unsigned flags;
};
constexpr unsigned FLIP0 = 1, FLIP1 = 2, FREE0 = 4, FREE1 = 8, HI0 = 16, HI1 = 32, GHOSTS = 64,
                   PAIRED = 128;

__device__ __forceinline__ Cols strip_cols(const YK &k, int x, bool aligned) {
    Cols c{x, x + 1, 0u};
    const bool inside = x >= 0 && x + 1 < k.nx;
    if (!inside) {
        int flip = 0, fs = 0;
        c.s0 = map_axis(x, k.nx, k.bc0, k.bc1, 0, flip, fs);
        c.flags = (flip ? FLIP0 : 0u) | (fs ? FREE0 : 0u);
        flip = fs = 0;
        c.s1 = map_axis(x + 1, k.nx, k.bc0, k.bc1, 0, flip, fs);
        c.flags |= (flip ? FLIP1 : 0u) | (fs ? FREE1 : 0u);
    }
    if (!__all_sync(0xffffffffu, inside)) c.flags |= GHOSTS;
    if (aligned && (k.nx & 1) == 0) {
        // (columns past the two ghosts feed no output: any pair serves)
        c.flags |= PAIRED | (c.s0 & 1 ? HI0 : 0u) | (c.s1 & 1 ? HI1 : 0u);
        c.s0 &= ~1;
    }
    return c;
}

__device__ __forceinline__ float2 ldg2(const float *p) {
    return __ldg(reinterpret_cast<const float2 *>(p));
}

// conserved values of the lane's two cells in row gy (a ghost row through the
// boundary conditions).  INNER: a warp without ghost columns that loads pairs
template <bool INNER>
__device__ __forceinline__ void load_row(const YK &k, const float *__restrict__ U, const Cols &c,
                                         int gy, float2 (&u)[NC], int *err) {
    int flip = 0, fs = 0;
    if ((unsigned)gy >= (unsigned)k.ny) gy = map_axis(gy, k.ny, k.bc2, k.bc3, 1, flip, fs);
    const long long row = (long long)k.nx * gy;
    if (INNER || (c.flags & PAIRED)) {
        const bool ok = in_bounds(row + c.s0 + 1, k.N, err);
        const float *p = U + row + c.s0;
#pragma unroll
        for (int m = 0; m < NC; ++m)
            u[m] = ok ? ldg2(p + m * k.N) : sp(0.0f);
    } else {
        const bool ok = in_bounds(row + c.s0, k.N, err) && in_bounds(row + c.s1, k.N, err);
#pragma unroll
        for (int m = 0; m < NC; ++m) {
            const float *p = U + m * k.N + row;
            u[m] = ok ? make_float2(__ldg(p + c.s0), __ldg(p + c.s1)) : sp(0.0f);
        }
    }
    if (!INNER && (c.flags & GHOSTS)) {
        if (c.flags & PAIRED) {
#pragma unroll
            for (int m = 0; m < NC; ++m)
                u[m] = make_float2(c.flags & HI0 ? u[m].y : u[m].x, c.flags & HI1 ? u[m].y : u[m].x);
        }
        if (c.flags & FLIP0) u[1].x = -u[1].x;
        if (c.flags & FLIP1) u[1].y = -u[1].y;
        if (c.flags & FREE0) { u[0].x = 1.0f; u[1].x = 1.0f; u[2].x = 0.0f; u[3].x = k.E_inf; }
        if (c.flags & FREE1) { u[0].y = 1.0f; u[1].y = 1.0f; u[2].y = 0.0f; u[3].y = k.E_inf; }
    }
    if (flip) u[2] = make_float2(-u[2].x, -u[2].y);
    if (fs) {
        u[0] = u[1] = sp(1.0f);
        u[2] = sp(0.0f);
        u[3] = sp(k.E_inf);
    }
}

template <typename V>
__device__ __forceinline__ void to_primitive(const YK &c, const V (&u)[NC], RowT<V> &r) {
    const V inv = rcp2(u[0]);
    r.w[0] = u[0];
    r.w[1] = u[1] * inv;
    r.w[2] = u[2] * inv;
    const V rk = fma2(u[1], r.w[1], u[2] * r.w[2]);   // rho |u|^2
    r.w[3] = cmul(c.gm1, cfma(-0.5f, rk, u[3]));
    r.T = r.w[3] * inv;
}

// x-neighbours of the lane's pair: column 2t - 1 (lane below) and 2t + 2
struct Side {
    float l, r;
};
__device__ __forceinline__ Side sides(float2 w) { return Side{from_left(w.y), from_right(w.x)}; }
// unscaled central differences along x of the two cells
__device__ __forceinline__ float2 cdx(float2 w) {
    const Side s = sides(w);
    return make_float2(__fsub_rn(w.y, s.l), __fsub_rn(s.r, w.x));
}

// x-faces of row P0 (P1 the row above; dpu, dpv: u and v of P0 less those of
// the row below) and acc = Fyl + their differences, Fyl the flux through the
// row's lower side
__device__ __forceinline__ void x_faces(const YK &k, const Row &P0, const Row &P1, float2 dpu,
                                        float2 dpv, const float2 (&Fyl)[NC], float2 (&acc)[NC]) {
    // x-faces at 2t - 1/2 and 2t + 1/2; what is shifted by one cell is
    // formed lane by lane (its pairs do not line up with the
    // registers' pairs)
    float2 wl[NC], wr[NC], dn, dt2, sn, st;
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        const float2 w = P0.w[m];
        const Side s = sides(w);
        const float d0 = __fsub_rn(w.x, s.l), d1 = __fsub_rn(w.y, w.x),
                    d2 = __fsub_rn(s.r, w.y);
        const float2 h = make_float2(vlh1(d0, d1), vlh1(d1, d2));
        wl[m] = make_float2(__fadd_rn(s.l, from_left(h.y)), __fadd_rn(w.x, h.x));
        wr[m] = w - h;
        if (m == 1) {
            dn = make_float2(d0, d1);
            sn = make_float2(__fadd_rn(s.l, w.x), __fadd_rn(w.x, w.y));
        }
        if (m == 2) {
            dt2 = make_float2(d0, d1);
            st = make_float2(__fadd_rn(s.l, w.x), __fadd_rn(w.x, w.y));
        }
    }
    const float tl = from_left(P0.T.y);
    const float2 dT = make_float2(__fsub_rn(P0.T.x, tl), __fsub_rn(P0.T.y, P0.T.x));
    const float2 sT = make_float2(__fadd_rn(tl, P0.T.x), __fadd_rn(P0.T.x, P0.T.y));
    // along y: the central differences of rows y+1 and y-1
    const float2 dyu = dpu + (P1.w[1] - P0.w[1]), dyv = dpv + (P1.w[2] - P0.w[2]);
    const float2 dun = make_float2(__fadd_rn(from_left(dyu.y), dyu.x), __fadd_rn(dyu.x, dyu.y));
    const float2 dvt = make_float2(__fadd_rn(from_left(dyv.y), dyv.x), __fadd_rn(dyv.x, dyv.y));
    float2 F[NC];
    flux_of(k, wl, wr, dn, dt2, dT, sn, st, sT, dun, dvt, F);
#pragma unroll
    for (int m = 0; m < NC; ++m)
        acc[m] = Fyl[m] + make_float2(__fsub_rn(F[m].x, F[m].y),
                                      __fsub_rn(F[m].y, from_right(F[m].x)));
}

// The flux of normal momentum through a y-face less its free-stream pressure.
// A row's sum starts from the flux below it, and rounded at the size of p (1 /
// (gamma Ma^2): 18 at Ma 0.2) it made the momentum part of L 2.4 % less
// accurate than differences summed; the pressure off, exactly where p varies
// by less than a factor of two, it is as accurate.  (Holding the flux below
// until the one above is known takes eight registers more: 1 % of a batch's
// time, 7 % of 4095 x 2047.)
template <typename V> __device__ __forceinline__ V less_p(const YK &k, V F) { return cadd(-k.p2, F); }

// y-faces between rows P0 and P1 with their halved limited slopes, in the
// cells' frame
__device__ __forceinline__ void y_faces(const YK &k, const Row &P0, const Row &P1,
                                        const float2 (&wl)[NC], const float2 (&wr)[NC],
                                        float2 (&Fy)[NC]) {
    float2 F[NC];
    const float2 cxu = cdx(P0.w[1]) + cdx(P1.w[1]), cxv = cdx(P0.w[2]) + cdx(P1.w[2]);
    flux_of(k, wl, wr, P1.w[2] - P0.w[2], P1.w[1] - P0.w[1], P1.T - P0.T, P0.w[2] + P1.w[2],
              P0.w[1] + P1.w[1], P0.T + P1.T, cxv, cxu, F);
    Fy[0] = F[0];
    Fy[1] = F[2];
    Fy[2] = less_p(k, F[1]);
    Fy[3] = F[3];
}

// The stage's output of the lane's cells from acc and the flux through the
// row's upper side; o1, o2: the operands Uin and Un of a PAIRED lane
template <int MODE>
__device__ __forceinline__ void row_out(const YK &k, bool paired, bool in1, long long j,
                                        const float2 (&acc)[NC], const float2 (&Fyu)[NC],
                                        const float2 (&o1)[NC], const float2 (&o2)[NC],
                                        const float *__restrict__ Uin, const float *__restrict__ Un,
                                        float *__restrict__ out, float dt,
                                        const unsigned *__restrict__ band_bits, float &smax, bool &ok) {
    float2 r[NC];
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        const float2 L = cmul(m == NC - 1 ? k.ih4 : k.ih2, acc[m] - Fyu[m]);
        const long long jm = m * k.N + j;
        if (paired) {
            float2 o = L;
            if (MODE != 0) o = cfma(dt, L, o1[m]);
            if (MODE == 2) o = cfma(0.5f, o2[m], cmul(0.5f, o));
            *reinterpret_cast<float2 *>(out + jm) = o;
            r[m] = o;
        } else {
            // the same roundings cell by cell (a missing second cell: 1,
            // whose rate is not looked at)
            float o[2] = {L.x, in1 ? L.y : 1.0f};
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                if (i == 1 && !in1) break;
                if (MODE != 0) o[i] = __fmaf_rn(dt, o[i], __ldg(Uin + jm + i));
                if (MODE == 2) o[i] = __fmaf_rn(0.5f, __ldg(Un + jm + i), __fmul_rn(0.5f, o[i]));
                out[jm + i] = o[i];
            }
            r[m] = make_float2(o[0], o[1]);
        }
    }
    if (MODE == 2) {
        float2 p;
        const float2 sr = rate_2d(rate_k(k), r, p);
        if (!band_bit(band_bits, j)) {
            smax = fmaxf(smax, sr.x);
            ok = ok && rate_ok(r[0].x, p.x, sr.x);
        }
        if (in1 && !band_bit(band_bits, j + 1)) {
            smax = fmaxf(smax, sr.y);
            ok = ok && rate_ok(r[0].y, p.y, sr.y);
        }
    }
}

// One strip chunk of one stage by one warp: columns ox .. ox + 59, rows y0 ..
// y1 - 1.  MODE 0: out = L(Uin).  MODE 1: out = U1 = Uin + dt L(Uin).  MODE 2:
// out = U* = Un/2 + (Uin + dt L(Uin))/2 with Uin = U1; smax collects s_j(U*)
// over the cells outside the band, ok is cleared by an invalid one.
template <int MODE, bool INNER, bool LATE>
__device__ __forceinline__ void march(const YK &k, const Cols &c, int x, int y0, int y1,
                                            const float *__restrict__ Uin,
                                            const float *__restrict__ Un, float *__restrict__ out,
                                            float dt, const unsigned *__restrict__ band_bits,
                                            float &smax, bool &ok, int *err) {
    const int lane = threadIdx.x & 31;
    const bool in0 = lane >= 1 && lane <= 30 && x < k.nx, in1 = in0 && x + 1 < k.nx;
    const bool paired = INNER || (c.flags & PAIRED);   // (then in1 = in0)
    constexpr int fy[NC] = {0, 2, 1, 3};   // face frame of a y-face (rho, v, u, p)
    // P0, P1: rows y and y+1; raw: row y+2 on its way; sig: halved limited
    // y-slopes of row y; dpu, dpv: u and v of row y less those of row y-1;
    // Fyl: the flux through y - 1/2.  The march starts one row early, for the
    // flux below the chunk's first row.
    Row P0, P1;
    float2 raw[NC], sig[NC], Fyl[NC], dpu, dpv;
    {
        Row A;
        float2 ra[NC], rb[NC], rc[NC];
        load_row<INNER>(k, Uin, c, y0 - 2, ra, err);
        load_row<INNER>(k, Uin, c, y0 - 1, rb, err);
        load_row<INNER>(k, Uin, c, y0, rc, err);
        load_row<INNER>(k, Uin, c, y0 + 1, raw, err);
        to_primitive(k, ra, A);
        to_primitive(k, rb, P0);
        to_primitive(k, rc, P1);
#pragma unroll
        for (int m = 0; m < NC; ++m) {
            sig[m] = vlh2(P0.w[m] - A.w[m], P1.w[m] - P0.w[m]);
            Fyl[m] = sp(0.0f);
        }
        dpu = P0.w[1] - A.w[1];
        dpv = P0.w[2] - A.w[2];
    }
#pragma unroll 1
    for (int y = y0 - 1; y < y1; ++y) {
        const long long j = x + (long long)k.nx * y;
        float2 acc[NC], o1[NC], o2[NC];
        // the output's operands: loaded ahead of the faces, or (LATE, eight to
        // sixteen registers fewer) where they are used
        auto operands = [&]() {
            if (!in_bounds(j + 1, k.N, err)) return;
#pragma unroll
            for (int m = 0; m < NC; ++m) {
                o1[m] = ldg2(Uin + m * k.N + j);
                if (MODE == 2) o2[m] = ldg2(Un + m * k.N + j);
            }
        };
        // toward L2: the rows three iterations ahead (a first touch of DRAM
        // takes longer than one row of a dozen warps)
        if (in0 && y + 5 < k.ny && y + 3 < y1) {
            const long long jp = j + 5 * (long long)k.nx;
#pragma unroll
            for (int m = 0; m < NC; ++m) {
                asm volatile("prefetch.global.L2 [%0];" ::"l"(Uin + m * k.N + jp));
                if (MODE == 2)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(Un + m * k.N + jp - 2 * (long long)k.nx));
            }
        }
        if (y >= y0) {
            if (MODE != 0 && !LATE && paired && in0) operands();
            x_faces(k, P0, P1, dpu, dpv, Fyl, acc);
        }
        // y-faces at y + 1/2
        Row P2;
        to_primitive(k, raw, P2);
        if (y + 1 < y1) load_row<INNER>(k, Uin, c, y + 3, raw, err);
        {
            float2 wl[NC], wr[NC];
#pragma unroll
            for (int m = 0; m < NC; ++m) wl[m] = P0.w[fy[m]] + sig[fy[m]];
#pragma unroll
            for (int m = 0; m < NC; ++m) sig[m] = vlh2(P1.w[m] - P0.w[m], P2.w[m] - P1.w[m]);
#pragma unroll
            for (int m = 0; m < NC; ++m) wr[m] = P1.w[fy[m]] - sig[fy[m]];
            y_faces(k, P0, P1, wl, wr, Fyl);
            dpu = P1.w[1] - P0.w[1];
            dpv = P1.w[2] - P0.w[2];
            P0 = P1;
            P1 = P2;
        }
        if (y < y0 || !in0 || !in_bounds(j + (in1 ? 1 : 0), k.N, err)) continue;
        if (MODE != 0 && LATE && paired) operands();
        row_out<MODE>(k, paired, in1, j, acc, Fyl, o1, o2, Uin, Un, out, dt, band_bits, smax, ok);
    }
}

// A single row of 28 columns, without the march and with one column per lane:
// the form for grids that leave most of the GPU idle, where a step takes as
// long as one warp's chain of instructions.  Every load and face waits for
// nothing but its own operands, and a warp issues 700 (stage 2: 820)
// instructions against 1070 (1230) with two columns per lane.  The operations are those of the march, one
// face or cell at a time.
__device__ __forceinline__ F1 left1(F1 v) { return {from_left(v.x)}; }
__device__ __forceinline__ F1 right1(F1 v) { return {from_right(v.x)}; }

template <int MODE>
__device__ __forceinline__ void one_row(const YK &k, int x, int y, const float *__restrict__ Uin,
                                        const float *__restrict__ Un, float *__restrict__ out,
                                        float dt, const unsigned *__restrict__ band_bits,
                                        float &smax, bool &ok, int *err) {
    const int lane = threadIdx.x & 31;
    const long long j = x + (long long)k.nx * y;
    const bool in = lane >= 2 && lane <= 29 && x < k.nx && in_bounds(j, k.N, err);
    int xs = x, flip = 0, fs = 0;
    if ((unsigned)x >= (unsigned)k.nx) xs = map_axis(x, k.nx, k.bc0, k.bc1, 0, flip, fs);
    F1 u[5][NC], o1[NC], o2[NC];
    int yflip[5], yfs[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        int ys = y - 2 + i;
        yflip[i] = yfs[i] = 0;
        if ((unsigned)ys >= (unsigned)k.ny) ys = map_axis(ys, k.ny, k.bc2, k.bc3, 1, yflip[i], yfs[i]);
        const long long js = xs + (long long)k.nx * ys;
        const bool inside = in_bounds(js, k.N, err);
#pragma unroll
        for (int m = 0; m < NC; ++m) u[i][m].x = inside ? __ldg(Uin + m * k.N + js) : 0.0f;
    }
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        o1[m] = u[2][m];
        o2[m].x = MODE == 2 && in ? __ldg(Un + m * k.N + j) : 0.0f;
    }
    RowT<F1> P[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        if (flip) u[i][1].x = -u[i][1].x;
        if (yflip[i]) u[i][2].x = -u[i][2].x;
        if (fs || yfs[i]) {
            u[i][0].x = u[i][1].x = 1.0f;
            u[i][2].x = 0.0f;
            u[i][3].x = k.E_inf;
        }
        to_primitive(k, u[i], P[i]);
    }
    // y-faces below (0) and above (1) the row
    F1 Fy[2][NC], sg[3][NC];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int m = 0; m < NC; ++m)
            sg[i][m] = vlh2(P[i + 1].w[m] - P[i].w[m], P[i + 2].w[m] - P[i + 1].w[m]);
    F1 cu[3], cv[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        cu[i] = right1(P[i + 1].w[1]) - left1(P[i + 1].w[1]);
        cv[i] = right1(P[i + 1].w[2]) - left1(P[i + 1].w[2]);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        constexpr int fy[NC] = {0, 2, 1, 3};
        const RowT<F1> &A = P[i + 1], &B = P[i + 2];
        F1 wl[NC], wr[NC], F[NC];
#pragma unroll
        for (int m = 0; m < NC; ++m) {
            wl[m] = A.w[fy[m]] + sg[i][fy[m]];
            wr[m] = B.w[fy[m]] - sg[i + 1][fy[m]];
        }
        flux_of(k, wl, wr, B.w[2] - A.w[2], B.w[1] - A.w[1], B.T - A.T, A.w[2] + B.w[2],
                A.w[1] + B.w[1], A.T + B.T, cv[i] + cv[i + 1], cu[i] + cu[i + 1], F);
        Fy[i][0] = F[0];
        Fy[i][1] = F[2];
        Fy[i][2] = less_p(k, F[1]);
        Fy[i][3] = F[3];
    }
    // the x-face at x - 1/2
    F1 acc[NC];
    {
        F1 wl[NC], wr[NC], l[NC], d[NC], F[NC];
#pragma unroll
        for (int m = 0; m < NC; ++m) {
            const F1 w = P[2].w[m];
            l[m] = left1(w);
            d[m] = w - l[m];
            const F1 h = vlh2(d[m], right1(w) - w);
            wl[m] = l[m] + left1(h);
            wr[m] = w - h;
        }
        const F1 tl = left1(P[2].T);
        const F1 dyu = (P[2].w[1] - P[1].w[1]) + (P[3].w[1] - P[2].w[1]);
        const F1 dyv = (P[2].w[2] - P[1].w[2]) + (P[3].w[2] - P[2].w[2]);
        flux_of(k, wl, wr, d[1], d[2], P[2].T - tl, l[1] + P[2].w[1], l[2] + P[2].w[2], tl + P[2].T,
                left1(dyu) + dyu, left1(dyv) + dyv, F);
#pragma unroll
        for (int m = 0; m < NC; ++m) acc[m] = Fy[0][m] + (F[m] - right1(F[m]));
    }
    if (!in) return;
    F1 r[NC];
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        F1 o = cmul(m == NC - 1 ? k.ih4 : k.ih2, acc[m] - Fy[1][m]);
        if (MODE != 0) o = cfma(dt, o, o1[m]);
        if (MODE == 2) o = cfma(0.5f, o2[m], cmul(0.5f, o));
        out[m * k.N + j] = o.x;
        r[m] = o;
    }
    if (MODE == 2 && !band_bit(band_bits, j)) {
        F1 p;
        const F1 sr = rate_2d(rate_k(k), r, p);
        smax = fmaxf(smax, sr.x);
        ok = ok && rate_ok(r[0].x, p.x, sr.x);
    }
}

template <int MODE, bool LATE, bool ROW1>
__device__ __forceinline__ void strip_chunk(const YK &k, int strip, int y0, int y1,
                                            const float *__restrict__ Uin,
                                            const float *__restrict__ Un, float *__restrict__ out,
                                            float dt, const unsigned *__restrict__ band_bits,
                                            float &smax, bool &ok, int *err) {
    if constexpr (ROW1) {
        const int x = strip * YM_ROW_W - 2 + (int)(threadIdx.x & 31);
        one_row<MODE>(k, x, y0, Uin, Un, out, dt, band_bits, smax, ok, err);
        return;
    }
    const int x = strip * YM_W - 2 + 2 * (threadIdx.x & 31);
    const bool aligned = (((uintptr_t)Uin | (uintptr_t)Un | (uintptr_t)out) & 7) == 0;
    const Cols c = strip_cols(k, x, aligned);
    if ((c.flags & (PAIRED | GHOSTS)) == PAIRED)
        march<MODE, true, LATE>(k, c, x, y0, y1, Uin, Un, out, dt, band_bits, smax, ok, err);
    else
        march<MODE, false, LATE>(k, c, x, y0, y1, Uin, Un, out, dt, band_bits, smax, ok, err);
}

// Four CTAs per SM (128 registers; a few spills and the operands loaded late
// pay for the fourth: 30.1 us for both stages of 1024 x 512 against 33.8 with
// three); the batch form, whose constants take registers too, spills more and
// runs better with three (313 us for both stages of the 64 cases against 343).
constexpr int YM_CTAS = 4, YM_BATCH_CTAS = 3, YM_ROW_CTAS = 5;
template <int MODE, bool ROW1>
__global__ void __launch_bounds__(YM_T, ROW1 ? YM_ROW_CTAS : YM_CTAS)
ymarch_kernel(const GridParams g, int rows, int strips, int items, const float *__restrict__ Uin,
              const float *__restrict__ Un, float *__restrict__ out, double *__restrict__ blockmax,
              const double *__restrict__ dt_ptr, int *__restrict__ err,
              const unsigned *__restrict__ band_bits, double dt_fixed) {
    const int it = blockIdx.x * YM_WARPS + (threadIdx.x >> 5);
    const float dt = MODE == 0 ? 0.0f : (float)(dt_fixed > 0.0 ? dt_fixed : *dt_ptr);
    float smax = 0.0f;
    bool ok = true;
    if (it < items) {
        const int y0 = it / strips * rows;
        strip_chunk<MODE, true, ROW1>(make_yk(g), it % strips, y0, min(y0 + rows, g.n[1]), Uin,
                                      Un, out, dt, band_bits, smax, ok, err);
    }
    if (MODE == 2) {
        __shared__ float s_red[YM_WARPS];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) smax = fmaxf(smax, __shfl_xor_sync(0xffffffffu, smax, o));
        const int bad = __syncthreads_or(!ok);
        if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = smax;
        __syncthreads();
        if (threadIdx.x == 0) {
            float m = s_red[0];
            for (int w = 1; w < YM_WARPS; ++w) m = fmaxf(m, s_red[w]);
            blockmax[blockIdx.x] = (double)m;
            if (bad) record_error(err, ERR_NONFINITE);
        }
    }
}

// The same over a batch: one warp per (case, strip chunk) item; MODE 2 writes
// one maximum per item.
template <int MODE, bool ROW1>
__global__ void __launch_bounds__(YM_T, ROW1 ? YM_ROW_CTAS : YM_BATCH_CTAS)
batch_ymarch_kernel(const BatchCase *__restrict__ cases, const int2 *__restrict__ items, int n_items,
                    int rows, double *__restrict__ item_max, double dt_fixed) {
    const int it = blockIdx.x * YM_WARPS + (threadIdx.x >> 5);
    if (it >= n_items) return;
    const int2 w = items[it];
    const BatchCase &bc = cases[w.x];
    const GridParams &g = bc.g;
    const YK k = make_yk(g);
    constexpr int W = ROW1 ? YM_ROW_W : YM_W;
    const int strips = (k.nx + W - 1) / W;
    const int y0 = w.y / strips * rows;
    const float dt = (float)(dt_fixed > 0.0 ? dt_fixed : *bc.dt);
    float smax = 0.0f;
    bool ok = true;
    strip_chunk<MODE, false, ROW1>(k, w.y % strips, y0, min(y0 + rows, k.ny),
                                   (const float *)(MODE == 2 ? bc.U1 : bc.Un), (const float *)bc.Un,
                                   (float *)(MODE == 2 ? bc.Us : bc.U1), dt, bc.band_bits, smax, ok,
                                   bc.err);
    if (MODE == 2) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) smax = fmaxf(smax, __shfl_xor_sync(0xffffffffu, smax, o));
        const bool bad = __any_sync(0xffffffffu, !ok);
        if ((threadIdx.x & 31) == 0) {
            item_max[it] = (double)smax;
            if (bad) record_error(bc.err, ERR_NONFINITE);
        }
    }
}

// Work of a grid: strips and rows per chunk.  As few rows as let every warp be
// resident at once: a second wave of few warps takes as long as the first, and
// a march takes ~1.4 us per row however few warps there are (one wave of 8 / 4 /
// 2 / 1 rows of 219 x 103: 41 / 26 / 20 / 16.5 us a step).  Where single rows
// of 28 columns are one wave, those: 11.6 us, and 13.1 / 14.7 us at 300 x 150 /
// 350 x 200 against 18.1 and 19 by the march; the 16 x 16 tiles these forms
// replace took 13.8, 15.9 and 16.1.  Larger, with the step's finish: 468 x 428
// 28.8 (30.9 by tiles), 640 x 480 28.9 (34.8), 2048 x 1024 86 (136).  Odd nx,
// whose pairs are loaded and stored one by one, gains less: 467 x 428 30.9
// (30.9), 641 x 481 33.5 (35.4), 1025 x 513 43.2 (48), 2047 x 1023 107 (135),
// 4095 x 2047 361 (500); batches of 32 cases of 101 to 105, 201 to 205 and 401
// to 405 columns 35 (39), 81 (102) and 338 (381).  At most 64 rows.
struct YmPlan {
    int width, rows;
};
constexpr int YM_SLOTS = 152 * YM_CTAS * YM_WARPS;
constexpr int YM_ROW_SLOTS = 152 * YM_ROW_CTAS * YM_WARPS;
constexpr int YM_BATCH_SLOTS = 152 * YM_BATCH_CTAS * YM_WARPS;

long long ym_items(int nx, int ny, YmPlan p) {
    return (long long)((nx + p.width - 1) / p.width) * ((ny + p.rows - 1) / p.rows);
}
YmPlan ym_plan(const GridParams &g) {
    YmPlan p{YM_ROW_W, 1};
    if (ym_items(g.n[0], g.n[1], p) <= YM_ROW_SLOTS) return p;
    const int cap = YM_SLOTS / ((g.n[0] + YM_W - 1) / YM_W);   // chunks per strip in one wave
    const int r = cap > 0 ? (g.n[1] + cap - 1) / cap : 64;
    return YmPlan{YM_W, r < 1 ? 1 : r > 64 ? 64 : r};
}

template <int MODE>
cudaError_t ym_launch(const GridParams &g, const void *Uin, const void *Un, void *out,
                      const FluidBuffers &fb, double dt_fixed, cudaStream_t s) {
    const YmPlan p = ym_plan(g);
    const long long items = ym_items(g.n[0], g.n[1], p);
    const auto kernel = p.width == YM_ROW_W ? ymarch_kernel<MODE, true> : ymarch_kernel<MODE, false>;
    kernel<<<(unsigned)((items + YM_WARPS - 1) / YM_WARPS), YM_T, 0, s>>>(
        g, p.rows, (g.n[0] + p.width - 1) / p.width, (int)items, (const float *)Uin,
        (const float *)Un, (float *)out, fb.blockmax, fb.dt, fb.err, fb.band_bits, dt_fixed);
    return cudaGetLastError();
}

}  // namespace

size_t ymarch_blocks(const GridParams &g) {
    return (size_t)((ym_items(g.n[0], g.n[1], ym_plan(g)) + YM_WARPS - 1) / YM_WARPS);
}

cudaError_t launch_ymarch(int mode, const GridParams &g, const void *Uin, const void *Un, void *out,
                          const FluidBuffers &fb, double dt_fixed, cudaStream_t s) {
    if (mode == 1) return ym_launch<1>(g, Uin, Un, out, fb, dt_fixed, s);
    if (mode == 2) return ym_launch<2>(g, Uin, Un, out, fb, dt_fixed, s);
    return ym_launch<0>(g, Uin, Un, out, fb, dt_fixed, s);
}

// A batch's rows per chunk: 16, 8, 32 or 64 by the tuned shape, fewer where
// the cases' rows then still fit one wave; 0 stands for single rows of 28
// columns.
int ymarch_batch_rows(int shape, int ncases, const ibm_grid_desc *descs) {
    static const int H[kBatchShapes] = {16, 8, 32, 64};
    for (int r = 0; r < H[shape]; ++r) {
        const long long slots = r == 0 ? YM_ROW_SLOTS : YM_BATCH_SLOTS;
        long long items = 0;
        for (int c = 0; c < ncases && items <= slots; ++c) items += ymarch_batch_items(descs[c], r);
        if (items <= slots) return r;
    }
    return H[shape];
}

long long ymarch_batch_items(const ibm_grid_desc &d, int rows) {
    return ym_items(d.n[0], d.n[1], rows == 0 ? YmPlan{YM_ROW_W, 1} : YmPlan{YM_W, rows});
}

template <int MODE>
static cudaError_t batch_ym_launch(int rows, const BatchCase *cases, const int2 *items, int n_items,
                                   double *item_max, double dt_fixed, cudaStream_t s) {
    const unsigned nb = (unsigned)((n_items + YM_WARPS - 1) / YM_WARPS);
    const auto kernel = rows == 0 ? batch_ymarch_kernel<MODE, true> : batch_ymarch_kernel<MODE, false>;
    kernel<<<nb, YM_T, 0, s>>>(cases, items, n_items, rows == 0 ? 1 : rows, item_max, dt_fixed);
    return cudaGetLastError();
}

cudaError_t launch_batch_ymarch(int mode, int rows, const BatchCase *cases, const int2 *items,
                                int n_items, double *item_max, double dt_fixed, cudaStream_t s) {
    if (mode == 1) return batch_ym_launch<1>(rows, cases, items, n_items, item_max, dt_fixed, s);
    if (mode == 2) return batch_ym_launch<2>(rows, cases, items, n_items, item_max, dt_fixed, s);
    return cudaErrorInvalidValue;
}

}  // namespace ibmk
