// Fluid stages for 3D FP32 grids: the same discretisation as flux.cu
// (MUSCL/van Leer + Rusanov + central viscous/heat fluxes, SSP-RK2 stages),
// organised as a z-march for GB300.
//
// A CTA of 256 threads owns a 32 x 16 column of cells and walks up a chunk of
// z-planes; each thread owns two neighbouring cells of one row, (2t, r) and
// (2t+1, r).  Shared memory holds a ring of five primitive planes (z-1 ..
// z+3) with a two-cell halo in x and y, so every cell is loaded from memory
// and converted to primitives once per chunk.  Per plane and thread:
//   - the x-faces 2t-1/2 and 2t+1/2 of its row as one packed FP32x2 pair:
//     the five cells 2t-2 .. 2t+2 give the three limited slopes of cells
//     2t-1, 2t, 2t+1 (the middle one serves both faces);
//   - the y-faces below its two cells (row r-1/2) as a pair;
//   - the z-faces above its two cells (z+1/2) as a pair; the limited z-slope
//     of plane z+1 and the z-face fluxes are carried in registers to the
//     next plane, where they are the lower plane's;
//   - warp 7 also evaluates the tile's upper x- and y-edge faces;
//   - plane z+3 is converted into the ring slot of plane z-2;
// one barrier, then each thread forms the flux divergence of its two cells
// from its own faces (registers), the x-face of its right neighbour (a warp
// shuffle), the y-faces of the row above (a shuffle within a warp's two rows,
// shared memory between warps), and writes both cells with 8-byte accesses.
// The five ring slots and two sets of exchanged faces make that barrier the
// only one: what a thread ahead of the others overwrites was last read before
// the barrier it has passed.  Neighbouring cells sit in adjacent
// 32-bit words of the ring, so most stencil loads are 8-byte (two cells).
// All constants are single precision: the kernel issues no FP64 work except
// the per-CTA step-size maximum.
//
// Bound: instruction issue and latency (16 warps per SM at 62 % issue in stage
// 1, 57 % in stage 2, 636 and 729 thread instructions per cell; fixed-latency
// waits, the barrier and the FMA pipe's throttle are the rest).  What was
// gained, both stages of 256^3 (192^3): 1151 us (561) at two barriers per plane; 1067 (511) with the halves and 1/h folded out of the
// fluxes, one special-function operation for the sound speed and one for
// Sutherland's law, plain reciprocals, and scalar arithmetic where a one-cell
// shift breaks the register pairs; 1026 (462) with one barrier per plane,
// ghosts found once per chunk and taken from the staged plane, and the rates
// of stage 2 as pairs; 979 (443) with chunks of full waves, the columns at the
// domain's edge first.  Measured and not kept: converting pairs of cells
// (18 x 20 of them do not divide among 256 threads: 532 us for stage 1), and
// per-pair source tables with asynchronous copies in place of the mapped loads
// (510 and 679 us, stage 2 spilling).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <float.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>

#include "flux_pair.cuh"
#include "internal.h"

namespace ibmk {
namespace {

constexpr int TX = 32, TY = 16, NTH = 256;               // tile cells; 16 threads per row
constexpr int PX = TX + 4, PY = TY + 4, PP = PX * PY;    // plane with a 2-cell halo
constexpr int NW = 6;                                     // rho, u, v, w, p, T
constexpr int NC = 5;
constexpr int RING = 5;
constexpr int SLOT = NW * PP;
// TMA staging box of one plane: x from ox-4 (16-byte aligned) over 40 cells,
// y from oy-2 over 20 rows, the five conserved components
constexpr int SBX = TX + 8, SBY = TY + 4;
constexpr int STAGE = NC * SBX * SBY;                     // floats
constexpr int FYR = TY / 2 + 1;                           // y-faces below the even rows and the edge
constexpr int FYN = NC * FYR * TX;
constexpr int FXE = NC * TY;                              // x-face fluxes of the upper x edge
constexpr size_t SMEM_BASE = sizeof(float) * (size_t)(RING * SLOT + 2 * (FYN + FXE));
constexpr size_t SMEM_TMA_OFF = (SMEM_BASE + 127) / 128 * 128;
constexpr size_t SMEM = SMEM_TMA_OFF + sizeof(float) * STAGE + 16;   // + mbarrier
constexpr long long TMA_WAIT_LIMIT = 1ll << 20;           // bounded mbarrier waits
static_assert(PX % 2 == 0 && PP % 2 == 0 && SLOT % 2 == 0, "8-byte ring loads need even strides");

using FC = FloatConsts;

// step-size rates of two cells, or one, from their conserved states, single
// precision throughout (step_rate's formula); p the pressure
template <typename V>
__device__ __forceinline__ V rate_of(const FC &c, const V (&u)[NC], V &p) {
    const V inv = rcp2(u[0]);
    const V vx = u[1] * inv, vy = u[2] * inv, vz = u[3] * inv;
    const V rk = fma2(u[1], vx, fma2(u[2], vy, u[3] * vz));   // rho |u|^2
    p = cmul(c.gm1, cfma(-0.5f, rk, u[4]));
    const V T = p * inv, c2 = cmul(c.gamma, T), Tf = T + T;
    const V y = cadd(c.s2, Tf);
    const V m = cmul(c.km, Tf) * (Tf * rsqrt2(Tf * y * y));   // 2 mu / h
    const V snd = c2 * rsqrt2(c2);
    return cfma(c.inv_h, cfma(3.0f, snd, abs2(vx) + abs2(vy) + abs2(vz)),
                cmul(3.0f * c.kvisc * c.inv_h, m) * inv);
}

FC make_fc(const GridParams &g) { return float_consts(g); }

// two neighbouring ring cells (the first at an even index)
__device__ __forceinline__ float2 ld2(const float *p) { return *reinterpret_cast<const float2 *>(p); }
__device__ __forceinline__ void st2(float *p, float2 v) { *reinterpret_cast<float2 *>(p) = v; }

// Fluxes are evaluated doubled (mass, momentum) and four-fold (energy), so no
// half remains in them: the output scales by 1/(2h) and 1/(4h).

// Rusanov flux of two faces from their reconstructed states in the face
// frame (rho, u_n, u_t1, u_t2, p): F = 2 (mass, normal momentum, t1 momentum,
// t2 momentum), 4 energy.  The speed of sound is gamma p rsqrt(gamma p rho):
// one special-function operation per side.
__device__ __forceinline__ void euler_pair(const FC &c, const float2 (&wl)[NC],
                                           const float2 (&wr)[NC], float2 (&F)[NC]) {
    const float2 unL = wl[1], unR = wr[1];
    const float2 mLn = wl[0] * unL, mRn = wr[0] * unR;
    const float2 mL1 = wl[0] * wl[2], mR1 = wr[0] * wr[2];
    const float2 mL2 = wl[0] * wl[3], mR2 = wr[0] * wr[3];
    const float2 rkL = fma2(mLn, unL, fma2(mL1, wl[2], mL2 * wl[3]));   // rho |u|^2
    const float2 rkR = fma2(mRn, unR, fma2(mR1, wr[2], mR2 * wr[3]));
    const float2 gpL = cmul(c.gamma, wl[4]), gpR = cmul(c.gamma, wr[4]);
    const float2 sL = fabs_fma(gpL, rsqrt2(gpL * wl[0]), unL);
    const float2 sR = fabs_fma(gpR, rsqrt2(gpR * wr[0]), unR);
    const float2 sm = max2(sL, sR);
    F[0] = fma2(sm, wl[0] - wr[0], mLn + mRn);
    F[1] = fma2(sm, mLn - mRn, fma2(mLn, unL, wl[4]) + fma2(mRn, unR, wr[4]));
    F[2] = fma2(sm, mL1 - mR1, fma2(mL1, unL, mR1 * unR));
    F[3] = fma2(sm, mL2 - mR2, fma2(mL2, unL, mR2 * unR));
    const float2 HL = cfma(c.h1, wl[4], rkL), HR = cfma(c.h1, wr[4], rkR);   // 2 rho H
    const float2 EL = cfma(c.e1, wl[4], rkL), ER = cfma(c.e1, wr[4], rkR);   // 2 rho E
    F[4] = fma2(sm, EL - ER, fma2(HL, unL, HR * unR));
}

// Viscous stress and heat flux of two faces, subtracted from F (face frame).
// dn, d1, d2, dT: differences (upper - lower cell) and sn, s1, s2, sT sums of
// u_n, u_t1, u_t2 and T = p / rho over the two cells; d1n, d11: the sums over
// the two cells of the central differences (w[+1] - w[-1], unscaled) of u_n
// and u_t1 along t1; d2n, d22: of u_n and u_t2 along t2.  Tangential
// derivatives are those sums / (4h) (reading 11).  T^(3/2) / (T + S) is
// T^2 rsqrt(T (T + S)^2).
__device__ __forceinline__ void visc_pair(const FC &c, float2 dn, float2 d1, float2 d2, float2 dT,
                                          float2 sn, float2 s1, float2 s2, float2 sT, float2 d1n,
                                          float2 d11, float2 d2n, float2 d22, float2 (&F)[NC]) {
    const float2 y = make_float2(__fadd_rn(sT.x, c.s2), __fadd_rn(sT.y, c.s2));
    const float2 m = cmul(c.km, sT) * (sT * rsqrt2(sT * y * y));   // 2 mu / h
    const float2 tNN = m * cfma(4.0f / 3.0f, dn, cmul(-1.0f / 6.0f, d11 + d22));
    const float2 tN1 = m * cfma(0.25f, d1n, d1);
    const float2 tN2 = m * cfma(0.25f, d2n, d2);
    F[1] = F[1] - tNN;
    F[2] = F[2] - tN1;
    F[3] = F[3] - tN2;
    F[4] = F[4] - fma2(sn, tNN, fma2(s1, tN1, fma2(s2, tN2, cmul(c.kl, m) * dT)));
}
// from the cell values a (lower) and b (upper) of (n, t1, t2) and T
__device__ __forceinline__ void visc_cells(const FC &c, const float2 (&ca)[NC],
                                           const float2 (&cb)[NC], float2 Ta, float2 Tb, float2 d1n,
                                           float2 d11, float2 d2n, float2 d22, float2 (&F)[NC]) {
    visc_pair(c, cb[1] - ca[1], cb[2] - ca[2], cb[3] - ca[3], Tb - Ta, ca[1] + cb[1], ca[2] + cb[2],
              ca[3] + cb[3], Ta + Tb, d1n, d11, d2n, d22, F);
}

// central differences (unscaled) along x of a field at cells 2t, 2t+1 of one
// row: w[x+1] - w[x-1] from the pair (given) and its neighbours
__device__ __forceinline__ float2 cdx2(const float *f, float2 mid) {
    return make_float2(__fsub_rn(mid.y, f[-1]), __fsub_rn(f[2], mid.x));
}

// x-faces 2t-1/2 (.x) and 2t+1/2 (.y) of one row; b: ring index of cell 2t
// in the plane slot R points at; up, dn: offsets to the planes above and
// below.  Output in (rho, rho u, rho v, rho w, rho E) order.
__device__ __forceinline__ void x_pair(const FC &c, const float *__restrict__ R, int b, int up,
                                       int dn, float2 (&F)[NC]) {
    float2 wl[NC], wr[NC];
    float2 df[3], sm[3];     // differences and sums of u, v, w over each face's cells
    // The five cells 2t-2 .. 2t+2 and their three slopes; formed lane by lane,
    // since values shifted by one cell do not line up with register pairs
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        const float *f = R + m * PP + b;
        const float2 lo = ld2(f - 2), mid = ld2(f);
        const float w2 = f[2];
        const float d0 = __fsub_rn(lo.y, lo.x), d1 = __fsub_rn(mid.x, lo.y),
                    d2 = __fsub_rn(mid.y, mid.x), d3 = __fsub_rn(w2, mid.y);
        const float sa = vlh1(d0, d1), sb = vlh1(d1, d2), sc = vlh1(d2, d3);
        wl[m] = make_float2(__fadd_rn(lo.y, sa), __fadd_rn(mid.x, sb));
        wr[m] = make_float2(__fsub_rn(mid.x, sb), __fsub_rn(mid.y, sc));
        if (m >= 1 && m <= 3) {
            df[m - 1] = make_float2(d1, d2);
            sm[m - 1] = make_float2(__fadd_rn(lo.y, mid.x), __fadd_rn(mid.x, mid.y));
        }
    }
    euler_pair(c, wl, wr, F);
    if (!c.viscous) return;
    const float *T = R + 5 * PP + b;
    const float2 Tm = ld2(T);
    const float tl = T[-1];
    const float2 dT = make_float2(__fsub_rn(Tm.x, tl), __fsub_rn(Tm.y, Tm.x));
    const float2 sT = make_float2(__fadd_rn(tl, Tm.x), __fadd_rn(Tm.x, Tm.y));
    // central differences of cells 2t-1, 2t, 2t+1 between the offsets hi and
    // lo, summed pairwise per face
    auto cd = [&](const float *f, int hi, int lo) {
        const float cm = __fsub_rn(f[hi - 1], f[lo - 1]);
        const float2 c01 = ld2(f + hi) - ld2(f + lo);
        return make_float2(__fadd_rn(cm, c01.x), __fadd_rn(c01.x, c01.y));
    };
    const float *U = R + PP + b, *V = R + 2 * PP + b, *W = R + 3 * PP + b;
    // along y: u (normal), v (t1); along z: u (normal) and w (t2)
    const float2 d1n = cd(U, PX, -PX), d11 = cd(V, PX, -PX);
    const float2 d2n = cd(U, up, dn), d22 = cd(W, up, dn);
    visc_pair(c, df[0], df[1], df[2], dT, sm[0], sm[1], sm[2], sT, d1n, d11, d2n, d22, F);
}

// y-faces at row r-1/2 of cells 2t (.x) and 2t+1 (.y); b: ring index of cell
// (2t, r).  Output in (rho, rho u, rho v, rho w, rho E) order.
__device__ __forceinline__ void y_pair(const FC &c, const float *__restrict__ R, int b, int up,
                                       int dn, float2 (&Fo)[NC]) {
    constexpr int fy[NC] = {0, 2, 1, 3, 4};   // face frame (rho, v, u, w, p)
    float2 wl[NC], wr[NC], ca[NC], cb[NC];
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        const float *f = R + fy[m] * PP + b;
        const float2 x0 = ld2(f - 2 * PX), x1 = ld2(f - PX), x2 = ld2(f), x3 = ld2(f + PX);
        const float2 d0 = x1 - x0, d1 = x2 - x1, d2 = x3 - x2;
        wl[m] = x1 + vlh2(d0, d1);
        wr[m] = x2 - vlh2(d1, d2);
        ca[m] = x1;
        cb[m] = x2;
    }
    float2 F[NC];
    euler_pair(c, wl, wr, F);
    if (c.viscous) {
        const float *T = R + 5 * PP + b;
        const float2 Ta = ld2(T - PX), Tb = ld2(T);
        const float *U = R + PP + b, *V = R + 2 * PP + b, *W = R + 3 * PP + b;
        // along x: v (normal) and u (t1) at rows r-1 and r
        const float2 d1n = cdx2(V - PX, ca[1]) + cdx2(V, cb[1]);
        const float2 d11 = cdx2(U - PX, ca[2]) + cdx2(U, cb[2]);
        // along z: v (normal) and w (t2)
        const float2 d2n = (ld2(V - PX + up) - ld2(V - PX + dn)) + (ld2(V + up) - ld2(V + dn));
        const float2 d22 = (ld2(W - PX + up) - ld2(W - PX + dn)) + (ld2(W + up) - ld2(W + dn));
        visc_cells(c, ca, cb, Ta, Tb, d1n, d11, d2n, d22, F);
    }
    Fo[0] = F[0]; Fo[1] = F[2]; Fo[2] = F[1]; Fo[3] = F[3]; Fo[4] = F[4];
}

// halved limited z-slopes of cells 2t, 2t+1 at the plane of slot sm, from the
// planes below (sl) and above (sh); b: ring index of cell (2t, r)
__device__ __forceinline__ void z_slopes(const float *__restrict__ ring, int sl, int sm, int sh,
                                         int b, float2 (&sig)[NC]) {
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        const float *f = ring + m * PP + b;
        const float2 lo = ld2(f + sl), mid = ld2(f + sm), hi = ld2(f + sh);
        sig[m] = vlh2(mid - lo, hi - mid);
    }
}

// z-faces between the planes of slots sa (below) and sb (above) for cells
// 2t (.x) and 2t+1 (.y): siga, sigb are the halved limited z-slopes of the
// two planes (lab field order).  Output in (rho, rho u, rho v, rho w, rho E)
// order.
__device__ __forceinline__ void z_pair(const FC &c, const float *__restrict__ ring, int sa, int sb,
                                       int b, const float2 (&siga)[NC], const float2 (&sigb)[NC],
                                       float2 (&Fo)[NC]) {
    constexpr int fz[NC] = {0, 3, 1, 2, 4};   // face frame (rho, w, u, v, p)
    float2 wl[NC], wr[NC], ca[NC], cb[NC];
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        const int f = fz[m];
        ca[m] = ld2(ring + sa + f * PP + b);
        cb[m] = ld2(ring + sb + f * PP + b);
        wl[m] = ca[m] + siga[f];
        wr[m] = cb[m] - sigb[f];
    }
    float2 F[NC];
    euler_pair(c, wl, wr, F);
    if (c.viscous) {
        const float *A = ring + sa + b, *B = ring + sb + b;
        const float2 Ta = ld2(A + 5 * PP), Tb = ld2(B + 5 * PP);
        // along x: w (normal) and u (t1); along y: w (normal) and v (t2)
        const float2 d1n = cdx2(A + 3 * PP, ca[1]) + cdx2(B + 3 * PP, cb[1]);
        const float2 d11 = cdx2(A + PP, ca[2]) + cdx2(B + PP, cb[2]);
        const float2 d2n = (ld2(A + 3 * PP + PX) - ld2(A + 3 * PP - PX)) +
                           (ld2(B + 3 * PP + PX) - ld2(B + 3 * PP - PX));
        const float2 d22 = (ld2(A + 2 * PP + PX) - ld2(A + 2 * PP - PX)) +
                           (ld2(B + 2 * PP + PX) - ld2(B + 2 * PP - PX));
        visc_cells(c, ca, cb, Ta, Tb, d1n, d11, d2n, d22, F);
    }
    Fo[0] = F[0]; Fo[1] = F[2]; Fo[2] = F[3]; Fo[3] = F[1]; Fo[4] = F[4];
}

// Two faces of the tile's upper edges (warp 7), one per pair lane: the x-face
// between cells 31 and 32 of a row or the y-face between rows 15 and 16 of a
// column.  aA, aB: ring index of each face's lower cell; sn: the cell stride
// along the face normal (1 for x, PX for y), st the stride along the other
// in-plane axis; nf: the normal velocity field (1 = u, 2 = v).  Output in
// (rho, rho u, rho v, rho w, rho E) order.
__device__ __forceinline__ void edge_pair(const FC &c, const float *__restrict__ R, int aA, int aB,
                                          int sn, int st, int nf, int up, int dn,
                                          float2 (&Fo)[NC]) {
    // face frame (rho, normal, in-plane tangent, w, p)
    const int f[NC] = {0, nf, 3 - nf, 3, 4};
    float2 wl[NC], wr[NC], ca[NC], cb[NC];
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        const float *X = R + f[m] * PP + aA, *Y = R + f[m] * PP + aB;
        const float2 x0 = make_float2(X[-sn], Y[-sn]);
        const float2 x1 = make_float2(X[0], Y[0]);
        const float2 x2 = make_float2(X[sn], Y[sn]);
        const float2 x3 = make_float2(X[2 * sn], Y[2 * sn]);
        const float2 d0 = x1 - x0, d1 = x2 - x1, d2 = x3 - x2;
        wl[m] = x1 + vlh2(d0, d1);
        wr[m] = x2 - vlh2(d1, d2);
        ca[m] = x1;
        cb[m] = x2;
    }
    float2 F[NC];
    euler_pair(c, wl, wr, F);
    if (c.viscous) {
        const float *TA = R + 5 * PP + aA, *TB = R + 5 * PP + aB;
        const float2 Ta = make_float2(TA[0], TB[0]), Tb = make_float2(TA[sn], TB[sn]);
        const float *NA = R + f[1] * PP + aA, *NB = R + f[1] * PP + aB;   // normal velocity
        const float *PA = R + f[2] * PP + aA, *PB = R + f[2] * PP + aB;   // in-plane tangent
        const float *WA = R + 3 * PP + aA, *WB = R + 3 * PP + aB;
        auto cd = [&](const float *A, const float *B, int o, int mo) {   // both cells of each face
            return make_float2(A[o] - A[mo], B[o] - B[mo]) +
                   make_float2(A[sn + o] - A[sn + mo], B[sn + o] - B[sn + mo]);
        };
        const float2 d1n = cd(NA, NB, st, -st), d11 = cd(PA, PB, st, -st);
        const float2 d2n = cd(NA, NB, up, dn), d22 = cd(WA, WB, up, dn);
        visc_cells(c, ca, cb, Ta, Tb, d1n, d11, d2n, d22, F);
    }
    // back to lab order: the normal momentum goes to u (x-face) or v (y-face)
    const bool xf = nf == 1;
    Fo[0] = F[0];
    Fo[1] = xf ? F[1] : F[2];
    Fo[2] = xf ? F[2] : F[1];
    Fo[3] = F[3];
    Fo[4] = F[4];
}

// ---- TMA: one bulk tensor copy per plane into the staging box -------------
__device__ __forceinline__ unsigned smem_u32(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned mbar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// issue the copy of plane gz (thread 0 only)
__device__ __forceinline__ void tma_issue(const CUtensorMap *tmap, unsigned dst, unsigned mbar,
                                          int x0, int y0, int gz) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                 ::"r"(mbar), "r"((unsigned)(sizeof(float) * STAGE)) : "memory");
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(dst), "l"((unsigned long long)tmap), "r"(x0), "r"(y0), "r"(gz), "r"(0), "r"(mbar)
        : "memory");
}
// wait for the phase with the given parity; bounded: after TMA_WAIT_LIMIT
// polls it gives up, sets the error flag and returns false
__device__ __forceinline__ bool tma_wait(unsigned mbar, unsigned parity, int *err) {
    for (long long it = 0; it < TMA_WAIT_LIMIT; ++it) {
        unsigned done;
        asm volatile(
            "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;"
            " selp.u32 %0, 1, 0, p; }"
            : "=r"(done) : "r"(mbar), "r"(parity) : "memory");
        if (done) return true;
    }
    record_error(err, ERR_TIMEOUT);
    return false;
}

// primitives (rho, u, v, w, p, T = p / rho) of one conserved cell into ring cell q
__device__ __forceinline__ void to_primitive(const FC &c, const float (&u)[NC],
                                             float *__restrict__ slot, int q) {
    const float rho = u[0];
    const float inv = rcp_ftz(rho);
    const float vx = u[1] * inv, vy = u[2] * inv, vz = u[3] * inv;
    const float p = c.gm1 * (u[4] - 0.5f * rho * (vx * vx + vy * vy + vz * vz));
    slot[q] = rho;
    slot[PP + q] = vx;
    slot[2 * PP + q] = vy;
    slot[3 * PP + q] = vz;
    slot[4 * PP + q] = p;
    slot[5 * PP + q] = p * inv;
}

// conserved state of a ghost or interior cell through the boundary maps
__device__ __forceinline__ void mapped_cell(const GridParams &g, const FC &c,
                                            const float *__restrict__ U, int gx, int gy, int gz,
                                            float (&u)[NC], int *err) {
    int flip = 0, fs = 0;
    const int sx = map_axis(gx, g.n[0], g.bc[0], g.bc[1], 0, flip, fs);
    const int sy = map_axis(gy, g.n[1], g.bc[2], g.bc[3], 1, flip, fs);
    const int sz = map_axis(gz, g.n[2], g.bc[4], g.bc[5], 2, flip, fs);
    if (fs) {
        u[0] = 1.0f;
        u[1] = 1.0f;
        u[2] = 0.0f;
        u[3] = 0.0f;
        u[4] = c.E_inf;
        return;
    }
    const long long N = g.N;
    const long long j = sx + (long long)g.n[0] * (sy + (long long)g.n[1] * sz);
    const bool okj = in_bounds(j, N, err);
#pragma unroll
    for (int m = 0; m < NC; ++m) u[m] = okj ? __ldg(U + m * N + j) : 0.0f;
#pragma unroll
    for (int d = 0; d < 3; ++d)
        if ((flip >> d) & 1) u[1 + d] = -u[1 + d];
}

// The thread's cells of a plane (ring cells tid, tid + 256, tid + 512), their
// source cells through the x and y boundary conditions, found once per chunk:
// the tiles at the domain's edge, a third of 256^3 and most of 96^3, otherwise
// map every ghost again in every plane, in all lanes of their warps.
// off: in-plane index of the source; flags, four bits a cell: slip flips of u
// and v, free stream.
constexpr int NQ = (PP + NTH - 1) / NTH;
constexpr unsigned SRC_FREE = 4, SRC_FAR = 8;
constexpr int SRC_BITS = 14;
struct Sources {
    int off[NQ];
    unsigned flags;
};
__device__ __forceinline__ Sources plane_sources(const GridParams &g, int ox, int oy) {
    Sources s;
    s.flags = 0u;
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
        const int q = min((int)threadIdx.x + i * NTH, PP - 1);
        int flip = 0, fs = 0;
        const int sx = map_axis(ox + q % PX - 2, g.n[0], g.bc[0], g.bc[1], 0, flip, fs);
        const int sy = map_axis(oy + q / PX - 2, g.n[1], g.bc[2], g.bc[3], 1, flip, fs);
        s.off[i] = sx + g.n[0] * sy;
        s.flags |= ((unsigned)flip | (fs ? SRC_FREE : 0u)) << (4 * i);
    }
    return s;
}
// the same for a staged plane, 14 bits a cell: stage index, with the flags
// from bit 10; FAR: the source is not in the staging box (a periodic image)
static_assert(SBX * SBY <= 1024 && NQ * SRC_BITS <= 64, "packed stage sources");
__device__ __forceinline__ unsigned long long stage_sources(const GridParams &g, const Sources &p,
                                                            int ox, int oy) {
    unsigned long long st = 0;
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
        const int x = p.off[i] % g.n[0] - (ox - 4), y = p.off[i] / g.n[0] - (oy - 2);
        const bool in = x >= 0 && x < SBX && y >= 0 && y < SBY;
        const unsigned f = ((p.flags >> (4 * i)) & 7u) | (in ? 0u : SRC_FAR);
        st |= (unsigned long long)((in ? y * SBX + x : 0) | (int)(f << 10)) << (SRC_BITS * i);
    }
    return st;
}

__device__ __forceinline__ void apply_source(const FC &c, unsigned f, float (&u)[NC]) {
    if (f & 1u) u[1] = -u[1];
    if (f & 2u) u[2] = -u[2];
    if (f & SRC_FREE) {
        u[0] = 1.0f;
        u[1] = 1.0f;
        u[2] = 0.0f;
        u[3] = 0.0f;
        u[4] = c.E_inf;
    }
}

// Convert the staged plane gz into one ring slot.  (One cell after the other:
// three at once do not fit the registers.)
__device__ __forceinline__ void convert_staged(const GridParams &g, const FC &c,
                                               const float *__restrict__ U,
                                               const float *__restrict__ st,
                                               float *__restrict__ slot, unsigned long long src,
                                               int ox, int oy, int gz, int *err) {
#pragma unroll 1
    for (int q = threadIdx.x; q < PP; q += NTH) {
        const unsigned e = (unsigned)src & ((1u << SRC_BITS) - 1u);
        src >>= SRC_BITS;
        const float *p = st + (e & 1023u);
        float u[NC];
#pragma unroll
        for (int m = 0; m < NC; ++m) u[m] = p[m * (SBX * SBY)];
        if (e >> 10) {
            if (e >> 10 & SRC_FAR)
                mapped_cell(g, c, U, ox + q % PX - 2, oy + q / PX - 2, gz, u, err);
            else
                apply_source(c, e >> 10, u);
        }
        to_primitive(c, u, slot, q);
    }
}

// Load plane gz (ghosts through the boundary conditions) and convert it to
// primitives into one ring slot.
__device__ __forceinline__ void load_plane(const GridParams &g, const FC &c,
                                           const float *__restrict__ U, float *__restrict__ slot,
                                           const Sources &s, int gz, int *err) {
    const long long N = g.N;
    int flip = 0, fs = 0;
    const int sz = map_axis(gz, g.n[2], g.bc[4], g.bc[5], 2, flip, fs);
    const float *P = U + (long long)g.n[0] * g.n[1] * sz;
    int o = s.off[0], o1 = s.off[1], o2 = s.off[2];
    unsigned fl = s.flags;
#pragma unroll 1
    for (int q = threadIdx.x; q < PP; q += NTH) {
        const bool okj = in_bounds((P - U) + o, N, err);
        float u[NC];
#pragma unroll
        for (int m = 0; m < NC; ++m) u[m] = okj ? __ldg(P + m * N + o) : 0.0f;
        if (flip) u[3] = -u[3];
        const unsigned f = (fl & 7u) | (fs ? SRC_FREE : 0u);
        if (f) apply_source(c, f, u);
        to_primitive(c, u, slot, q);
        o = o1;
        o1 = o2;
        fl >>= 4;
    }
}
static_assert(NQ == 3, "load_plane's sources");

__device__ __forceinline__ double warp_max_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

#ifndef IBM_ZM_MIN_BLOCKS
#define IBM_ZM_MIN_BLOCKS 2
#endif
#ifndef IBM_ZM_PREFETCH
#define IBM_ZM_PREFETCH 1
#endif

// The chunk of this CTA (column x, y and z), CTAs taken in launch order: with
// more than one wave of them the columns at the domain's edge come first,
// since they take longer and what starts last should be short (256^3, both
// stages: 992 -> 977 us, 192^3 450 -> 438; grids whose planes arrive by thread
// loads lose more of their neighbours' cached lines than that: 837 -> 887 us
// at 255 x 201 x 190).
constexpr int ZM_SLOTS = 2 * 152;
__device__ __forceinline__ int3 chunk_order() {
    const int nbx = gridDim.x, nby = gridDim.y;
    const int inner = max(nbx - 2, 0) * max(nby - 2, 0);
    if (inner == 0 || nbx * nby * (int)gridDim.z <= ZM_SLOTS)
        return make_int3(blockIdx.x, blockIdx.y, blockIdx.z);
    const int edges = nbx * nby - inner;
    const int L = blockIdx.x + nbx * (blockIdx.y + nby * blockIdx.z), first = edges * gridDim.z;
    if (L >= first) {
        const int e = (L - first) % inner;
        return make_int3(1 + e % (nbx - 2), 1 + e / (nbx - 2), (L - first) / inner);
    }
    int e = L % edges;
    if (e < nbx) return make_int3(e, 0, L / edges);
    if (e < 2 * nbx) return make_int3(e - nbx, nby - 1, L / edges);
    e -= 2 * nbx;
    return make_int3(e & 1 ? nbx - 1 : 0, 1 + (e >> 1), L / edges);
}

// MODE 0: out = L(Uin).  MODE 1: out = U1 = Uin + dt L(Uin).
// MODE 2: out = U* = Un/2 + (Uin + dt L(Uin))/2 with Uin = U1, plus the
// per-CTA maximum of s_j(U*) over the cells outside the band.
// TMA: the planes of Uin inside the domain arrive by bulk tensor copies,
// each prefetched one plane ahead while the faces of the current plane are
// evaluated (needs nx % 4 == 0); otherwise every plane is loaded by threads.
template <int MODE, bool TMA>
__global__ void __launch_bounds__(NTH, IBM_ZM_MIN_BLOCKS)
zmarch_kernel(const __grid_constant__ CUtensorMap tmap, const GridParams g, const FC c, int zc,
              const float *__restrict__ Uin, const float *__restrict__ Un,
              float *__restrict__ out, double *__restrict__ blockmax,
              const double *__restrict__ dt_ptr, int *__restrict__ err,
              const unsigned *__restrict__ band_bits, double dt_fixed) {
    extern __shared__ __align__(128) float smem_zm[];
    float *ring = smem_zm;
    // exchanged faces, two sets (even and odd planes): y-faces below the even
    // rows and above row 15 ([NC][FYR][TX]), x-faces between cells 31 and 32
    // ([NC][TY])
    float *FYs = ring + RING * SLOT;
    __shared__ double s_red[NTH / 32];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int r = tid >> 4, t = tid & 15;     // row of the thread, its cells 2t and 2t+1
    const int3 blk = TMA ? chunk_order() : make_int3(blockIdx.x, blockIdx.y, blockIdx.z);
    const int ox = blk.x * TX, oy = blk.y * TY;
    const int z0 = blk.z * zc, z1 = min(z0 + zc, g.n[2]);
    const long long N = g.N;
    const float dt = MODE == 0 ? 0.0f : (float)(dt_fixed > 0.0 ? dt_fixed : *dt_ptr);
    const Sources src = plane_sources(g, ox, oy);
    const unsigned long long ssrc = TMA ? stage_sources(g, src, ox, oy) : 0ull;
    const int b = (2 * t + 2) + PX * (r + 2);   // ring index of cell (2t, r)

    float *stage = reinterpret_cast<float *>(reinterpret_cast<char *>(smem_zm) + SMEM_TMA_OFF);
    const unsigned st_addr = smem_u32(stage);
    const unsigned mbar = smem_u32(stage + STAGE);
    unsigned parity = 0;
    const int nz = g.n[2];
    // A copy that does not complete within the bounded wait switches the CTA
    // to thread loads.  Each thread decides for the cells it converts: a
    // thread whose wait gave up loads its own cells of the plane from global
    // memory, one whose wait completed converts the staged copy; both give
    // the same values, so threads may decide differently within one plane.
    // The shared flag only stops further copies; thread 0 reads it after the
    // plane's barrier.  Thread 0 tracks the copy it issued last and, if it
    // never saw that copy complete, drains it (bounded) before the CTA exits.
    __shared__ int s_tma_dead;
    volatile int *tma_dead = &s_tma_dead;
    bool outstanding = false;   // thread 0 only
    if (TMA) {
        if (tid == 0) {
            *tma_dead = 0;
            mbar_init(mbar);
            if (z0 + 2 < nz) {
                tma_issue(&tmap, st_addr, mbar, ox - 4, oy - 2, z0 + 2);
                outstanding = true;
            }

        }
        __syncthreads();
    }
    // planes z0-2 .. z0+1 by threads; z0+2 comes from the copy just issued.
    // Ring slots of planes z-2 (the next to be overwritten) .. z+2 at plane z:
    int sm2 = 0, sm1 = SLOT, s0 = 2 * SLOT, s1 = 3 * SLOT, s2 = 4 * SLOT;
    for (int i = 0; i < 4; ++i)
        load_plane(g, c, Uin, ring + i * SLOT, src, z0 - 2 + i, err);
    {
        bool use_stage = TMA && z0 + 2 < nz;
        if (use_stage && !tma_wait(mbar, parity, err)) {
            use_stage = false;
            *tma_dead = 1;
        }
        if (use_stage) {
            parity ^= 1u;
            if (tid == 0) outstanding = false;
            convert_staged(g, c, Uin, stage, ring + s2, ssrc, ox, oy, z0 + 2, err);
        } else {
            load_plane(g, c, Uin, ring + s2, src, z0 + 2, err);
        }
    }
    __syncthreads();
    if (TMA && tid == 0 && !*tma_dead && z0 + 1 < z1 && z0 + 3 < nz) {
        tma_issue(&tmap, st_addr, mbar, ox - 4, oy - 2, z0 + 3);
        outstanding = true;
    }

    // carried from plane to plane: the halved limited z-slopes of the current
    // plane and the z-face fluxes below it
    float2 sig[NC], Fzl[NC];
    {
        float2 sgm[NC];
        z_slopes(ring, sm2, sm1, s0, b, sgm);
        z_slopes(ring, sm1, s0, s1, b, sig);
        z_pair(c, ring, sm1, s0, b, sgm, sig, Fzl);
    }
    __syncthreads();   // plane z0-2's slot is about to take plane z0+3

    // the edge lanes of warp 7: 0-15 the y-faces above row 15 (columns 2l,
    // 2l+1), 16-23 the x-faces right of column 31 (rows q and q + 8)
    const bool edge = warp == 7 && lane < 24;
    int eA = 0, eB = 0, esn = 1, est = PX, enf = 1;
    if (warp == 7) {
        if (lane < 16) {
            eA = (2 * lane + 2) + PX * (TY - 1 + 2);
            eB = eA + 1;
            esn = PX;
            est = 1;
            enf = 2;
        } else if (lane < 24) {
            const int q = lane - 16;
            eA = (TX - 1 + 2) + PX * (q + 2);
            eB = eA + 8 * PX;
        }
    }

    const int gx = ox + 2 * t, gy = oy + r;
    const bool row_in = gy < g.n[1];
    const bool in0 = row_in && gx < g.n[0], in1 = row_in && gx + 1 < g.n[0];
    // both cells at once, 8-byte aligned (a caller's L may be 4-byte aligned only)
    const bool vec = in1 && g.n[0] % 2 == 0 && (MODE != 0 || ((uintptr_t)out & 7) == 0);
    float smaxf = 0.0f;
    bool ok = true;
    for (int z = z0; z < z1; ++z) {
        const int up = s1 - s0, dn = sm1 - s0;
        float *FY = FYs + (z & 1) * (FYN + FXE), *FXe = FY + FYN;
#if IBM_ZM_PREFETCH
        // stage 2 reads U^n at its output cells, which nothing has touched:
        // start those lines toward L2 two planes ahead
        if (MODE == 2 && z + 2 < z1 && in0) {
            const long long jp = gx + (long long)g.n[0] * (gy + (long long)g.n[1] * (z + 2));
#pragma unroll
            for (int m = 0; m < NC; ++m)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(Un + m * N + jp));
        }
#endif
        // faces of plane z: x pair, y pair (an even row's stored for the row
        // below, which the warp below holds), z pair
        float2 Fx[NC], Fy[NC], acc[NC];
        x_pair(c, ring + s0, b, up, dn, Fx);
        y_pair(c, ring + s0, b, up, dn, Fy);
        if (!(r & 1)) {
#pragma unroll
            for (int m = 0; m < NC; ++m) st2(FY + (m * FYR + (r >> 1)) * TX + 2 * t, Fy[m]);
        }
        {
            float2 sgh[NC], Fzh[NC];
            z_slopes(ring, s0, s1, s2, b, sgh);
            z_pair(c, ring, s0, s1, b, sig, sgh, Fzh);
#pragma unroll
            for (int m = 0; m < NC; ++m) {
                sig[m] = sgh[m];
                acc[m] = Fzl[m] - Fzh[m];
                Fzl[m] = Fzh[m];
            }
        }
        if (edge) {
            float2 Fe[NC];
            edge_pair(c, ring + s0, eA, eB, esn, est, enf, up, dn, Fe);
            if (lane < 16) {
#pragma unroll
                for (int m = 0; m < NC; ++m) st2(FY + (m * FYR + FYR - 1) * TX + 2 * lane, Fe[m]);
            } else {
                const int q = lane - 16;
#pragma unroll
                for (int m = 0; m < NC; ++m) {
                    FXe[m * TY + q] = Fe[m].x;
                    FXe[m * TY + q + 8] = Fe[m].y;
                }
            }
        }
        // output operands of the two cells: U^n (stage 2) is issued now and
        // used after the next plane's conversion, so its latency overlaps it;
        // the input state at the cells is rebuilt from the ring at the output
        const long long j = gx + (long long)g.n[0] * (gy + (long long)g.n[1] * z);
        float2 o1[NC], o2[NC];
        unsigned bits = 0u;   // the band word of the two cells (vec: one word holds both)
        if (MODE == 2 && vec && in_bounds(j + 1, N, err)) {
#pragma unroll
            for (int m = 0; m < NC; ++m) o2[m] = ld2(Un + m * N + j);
            if (band_bits) bits = __ldg(band_bits + (j >> 5)) >> (j & 31);
        }

        // plane z+3 into the slot of z-2 (last read before the last barrier)
        if (z + 1 < z1) {
            bool use_stage = TMA && z + 3 < nz && !*tma_dead;
            if (use_stage && !tma_wait(mbar, parity, err)) {
                use_stage = false;
                *tma_dead = 1;
            }
            if (use_stage) {
                parity ^= 1u;
                if (tid == 0) outstanding = false;
                convert_staged(g, c, Uin, stage, ring + sm2, ssrc, ox, oy, z + 3, err);
            } else {
                load_plane(g, c, Uin, ring + sm2, TMA ? plane_sources(g, ox, oy) : src, z + 3, err);
            }
        }
        __syncthreads();
        if (TMA && tid == 0 && !*tma_dead && z + 2 < z1 && z + 4 < nz) {
            tma_issue(&tmap, st_addr, mbar, ox - 4, oy - 2, z + 4);
            outstanding = true;
        }

        // flux divergence of the two cells
#pragma unroll
        for (int m = 0; m < NC; ++m) {
            // x-face right of cell 2t+1: the neighbour's first face, or the edge
            float fr = __shfl_down_sync(0xffffffffu, Fx[m].x, 1);
            if (t == 15) fr = FXe[m * TY + r];
            const float2 dx = make_float2(__fsub_rn(Fx[m].x, Fx[m].y), __fsub_rn(Fx[m].y, fr));
            // y-face above: the warp's other row holds it, or the next warp
            float2 Fyu = make_float2(__shfl_down_sync(0xffffffffu, Fy[m].x, 16),
                                     __shfl_down_sync(0xffffffffu, Fy[m].y, 16));
            if (r & 1) Fyu = ld2(FY + (m * FYR + (r >> 1) + 1) * TX + 2 * t);
            acc[m] = cmul(m == NC - 1 ? c.qinv_h : c.hinv_h, (dx + (Fy[m] - Fyu)) + acc[m]);
        }

        if (in0 && in_bounds(j + (vec ? 1 : 0), N, err)) {
            // the input state at the two cells, rebuilt from the primitives
            // of plane z in the ring (a few FP32 roundings from the stored
            // values; saves holding them in registers across the conversion).
            // Cells of a ragged tile edge or an odd nx load it instead.
            auto u_from_ring = [&](float2 (&u)[NC]) {
                const float *P = ring + s0 + b;
                const float2 rh = ld2(P), vu = ld2(P + PP), vv = ld2(P + 2 * PP),
                             vw = ld2(P + 3 * PP), pr = ld2(P + 4 * PP);
                const float2 ke = fma2(vu, vu, fma2(vv, vv, vw * vw));
                u[0] = rh;
                u[1] = rh * vu;
                u[2] = rh * vv;
                u[3] = rh * vw;
                u[4] = cfma(c.inv_gm1, pr, cmul(0.5f, rh) * ke);
            };
            if (vec) {
                if (MODE != 0) u_from_ring(o1);
                if (MODE == 0) {
#pragma unroll
                    for (int m = 0; m < NC; ++m) st2(out + m * N + j, acc[m]);
                } else if (MODE == 1) {
#pragma unroll
                    for (int m = 0; m < NC; ++m) st2(out + m * N + j, cfma(dt, acc[m], o1[m]));
                } else {
                    float2 us[NC], p;
#pragma unroll
                    for (int m = 0; m < NC; ++m) {
                        us[m] = cfma(0.5f, o2[m], cmul(0.5f, cfma(dt, acc[m], o1[m])));
                        st2(out + m * N + j, us[m]);
                    }
                    const float2 sr = rate_of(c, us, p);
                    if (!(bits & 1u)) {
                        smaxf = fmaxf(smaxf, sr.x);
                        ok = ok && rate_ok(us[0].x, p.x, sr.x);
                    }
                    if (!(bits & 2u)) {
                        smaxf = fmaxf(smaxf, sr.y);
                        ok = ok && rate_ok(us[0].y, p.y, sr.y);
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    if (k == 1 && !in1) break;
                    const long long jk = j + k;
                    float us[NC];
#pragma unroll
                    for (int m = 0; m < NC; ++m) {
                        const float a = k == 0 ? acc[m].x : acc[m].y;
                        if (MODE == 0) {
                            out[m * N + jk] = a;
                        } else if (MODE == 1) {
                            out[m * N + jk] = fmaf(dt, a, __ldg(Uin + m * N + jk));
                        } else {
                            const float un = __ldg(Un + m * N + jk);
                            const float u1 = __ldg(Uin + m * N + jk);
                            us[m] = 0.5f * un + 0.5f * fmaf(dt, a, u1);
                            out[m * N + jk] = us[m];
                        }
                    }
                    if (MODE == 2 && !band_bit(band_bits, jk)) {
                        F1 v[NC], p;
#pragma unroll
                        for (int m = 0; m < NC; ++m) v[m].x = us[m];
                        const float sr = rate_of(c, v, p).x;
                        smaxf = fmaxf(smaxf, sr);
                        ok = ok && rate_ok(us[0], p.x, sr);
                    }
                }
            }
        }
        const int sn = sm2;
        sm2 = sm1;
        sm1 = s0;
        s0 = s1;
        s1 = s2;
        s2 = sn;
    }

    // thread 0 flips its parity only on copies it saw complete, so `parity`
    // is the phase of a copy still outstanding
    if (TMA && tid == 0 && outstanding) tma_wait(mbar, parity, err);


    if (MODE == 2) {
        const double smax = warp_max_d((double)smaxf);
        const int bad = __syncthreads_or(!ok);
        if (lane == 0) s_red[warp] = smax;
        __syncthreads();
        if (tid == 0) {
            double m = s_red[0];
            for (int w = 1; w < NTH / 32; ++w) m = fmax(m, s_red[w]);
            blockmax[blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)] = m;
            if (bad) record_error(err, ERR_NONFINITE);
        }
    }
}

}  // namespace

// Planes per CTA.  A chunk of zc planes costs about zc + 1 plane times (its
// prologue of five planes, whose loads overlap, and the z-faces below it), and
// the grid runs in waves of two CTAs per SM, so the chunk count k is the one
// with the least waves(k) * (zc + 1); a grid of at most one CTA per SM runs
// each of them in ~0.7 of the time.  Both stages, with 2.5 and 0.6 in their
// place, of which the prologue once took its share -> now: 48^3 32.5 -> 30.4,
// 64^3 44.9 -> 39.1, 150 x 90 x 74 124.8 -> 96.8 us.  At most ZM_CHUNK_MAX
// planes (24: 192^3 462, 256^3 1026 us; 48: 450, 992; 96: 448, 992).
constexpr int ZM_CHUNK_MAX = 96;
int zmarch_chunk(const GridParams &g) {
    const long long cols = (long long)((g.n[0] + TX - 1) / TX) * ((g.n[1] + TY - 1) / TY);
    const long long slots = ZM_SLOTS;
    const int kmin = (g.n[2] + ZM_CHUNK_MAX - 1) / ZM_CHUNK_MAX;
    const long long most = std::max<long long>(kmin, 8 * slots / cols + 1);
    const int kmax = (int)std::min<long long>(most, g.n[2]);
    int best = 1;
    double cost = 1e300;
    for (int k = kmin; k <= kmax; ++k) {
        const int zc = (g.n[2] + k - 1) / k;
        const long long ctas = cols * ((g.n[2] + zc - 1) / zc);
        const double c = (double)((ctas + slots - 1) / slots) * (zc + 1.0) * (2 * ctas <= slots ? 0.7 : 1.0);
        if (c < cost) {
            cost = c;
            best = zc;
        }
    }
    return best;
}

size_t zmarch_blocks(const GridParams &g) {
    const int zc = zmarch_chunk(g);
    return (size_t)((g.n[0] + TX - 1) / TX) * ((g.n[1] + TY - 1) / TY) * ((g.n[2] + zc - 1) / zc);
}

// cuTensorMapEncodeTiled through the runtime's driver entry point
// (a driver function, the same for every device; resolved once, thread-safe)
static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static const PFN_cuTensorMapEncodeTiled_v12000 fn = []() {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return (PFN_cuTensorMapEncodeTiled_v12000)p;
        return (PFN_cuTensorMapEncodeTiled_v12000) nullptr;
    }();
    return fn;
}

// 4D map over a conserved state: (x, y, z, component), box 40 x 20 x 1 x 5
static bool make_state_map(const GridParams &g, const void *U, CUtensorMap *map) {
    if (g.n[0] % 4 != 0 || ((uintptr_t)U) % 16 != 0) return false;
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc) return false;
    const cuuint64_t dims[4] = {(cuuint64_t)g.n[0], (cuuint64_t)g.n[1], (cuuint64_t)g.n[2], NC};
    const cuuint64_t strides[3] = {(cuuint64_t)g.n[0] * 4, (cuuint64_t)g.n[0] * g.n[1] * 4,
                                   (cuuint64_t)g.N * 4};
    const cuuint32_t box[4] = {SBX, SBY, 1, NC};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void *>(U), dims, strides, box,
               estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int MODE, bool TMA>
static cudaError_t zm_launch_t(const GridParams &g, const CUtensorMap &map, const void *Uin,
                               const void *Un, void *out, const FluidBuffers &fb, double dt_fixed,
                               cudaStream_t s) {
    cudaError_t e = func_smem_attr((const void *)zmarch_kernel<MODE, TMA>, SMEM, 100);
    if (e != cudaSuccess) return e;
    const int zc = zmarch_chunk(g);
    dim3 grid((g.n[0] + TX - 1) / TX, (g.n[1] + TY - 1) / TY, (g.n[2] + zc - 1) / zc);
    zmarch_kernel<MODE, TMA><<<grid, NTH, SMEM, s>>>(map, g, make_fc(g), zc,
                                                     (const float *)Uin,
                                                     (const float *)Un, (float *)out, fb.blockmax,
                                                     fb.dt, fb.err, fb.band_bits, dt_fixed);
    return cudaGetLastError();
}

template <int MODE>
static cudaError_t zm_launch(const GridParams &g, const void *Uin, const void *Un, void *out,
                             const FluidBuffers &fb, double dt_fixed, cudaStream_t s) {
    CUtensorMap map;
    memset(&map, 0, sizeof(map));
    if (make_state_map(g, Uin, &map))
        return zm_launch_t<MODE, true>(g, map, Uin, Un, out, fb, dt_fixed, s);
    return zm_launch_t<MODE, false>(g, map, Uin, Un, out, fb, dt_fixed, s);
}

cudaError_t launch_zmarch(int mode, const GridParams &g, const void *Uin, const void *Un,
                          void *out, const FluidBuffers &fb, double dt_fixed, cudaStream_t s) {
    if (mode == 1) return zm_launch<1>(g, Uin, Un, out, fb, dt_fixed, s);
    if (mode == 2) return zm_launch<2>(g, Uin, Un, out, fb, dt_fixed, s);
    return zm_launch<0>(g, Uin, Un, out, fb, dt_fixed, s);
}

}  // namespace ibmk
