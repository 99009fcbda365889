// Fluid stages of the IBM step: the explicit finite-volume discretisation of
// the compressible Navier-Stokes equations of Sec. 2.1 on a uniform grid.
//
//   L(U) = -(1/h) sum_d (Fhat_{i+1/2} - Fhat_{i-1/2}),
//   Fhat = Rusanov(MUSCL/van Leer states of (rho, u, p)) - viscous/heat flux,
//
// advanced by SSP-RK2 as the source-free predictor of App. B (step 1):
//   stage 1:  U^1 = U^n + dt L(U^n)
//   stage 2:  U* = U^n/2 + (U^1 + dt L(U^1))/2
// with dt = cfl / max_j s_j(U^n), formed at the end of the previous step (or
// by dt_init after a new state) so that stage 1 can write U^1 directly.
//
// Here: FP64 grids (FP32 grids march: flux_zm.cu, flux_ym.cuh).  Each CTA owns
// a BX x BY x BZ tile of cells.  It loads the tile plus a two-cell halo once
// (ghost cells mapped through the boundary conditions on the fly), converts
// to primitives in shared memory, then per direction evaluates every limited
// slope once and every face of the tile once into shared buffers and
// accumulates the flux differences in registers.
//
// Bound: the FP64 pipe (two operations per SM cycle).  What is kept small is
// their number: no division or IEEE square root (drcp, drsqrt), slopes once
// per cell, constants folded on the host, signs and maxima by integer
// instructions.  Stages 1 / 2: 128 x 64 24.0 -> 13.1 and 29.0 -> 15.2 us, 64^3
// 629 -> 346 and 710 -> 373 us.
#include <atomic>
#include <float.h>

#include <type_traits>

#include "internal.h"

namespace ibmk {
namespace {

constexpr int NT = 256;

constexpr int cmax(int a, int b) { return a > b ? a : b; }

// A BX x BY x BZ tile of cells with its two-cell halo, 256 threads.
template <int DIM_, int BX_, int BY_, int BZ_>
struct BoxT {
    static constexpr int DIM = DIM_;
    static constexpr int BX = BX_, BY = BY_, BZ = DIM_ == 3 ? BZ_ : 1;
    static constexpr int PX = BX + 4, PY = BY + 4, PZ = DIM == 3 ? BZ + 4 : 1;
    static constexpr int PN = PX * PY * PZ;          // cells in tile + halo
    static constexpr int NC = DIM + 2;               // conserved components
    static constexpr int NW = DIM + 3;               // rho, u.., p, T = p / rho
    static constexpr int SX = 1, SY = PX, SZ = PX * PY;
    static constexpr int NCELL = BX * BY * BZ;
    static constexpr int CPT = (NCELL + NT - 1) / NT;
    static constexpr int NF0 = (BX + 1) * BY * BZ;
    static constexpr int NF1 = BX * (BY + 1) * BZ;
    static constexpr int NF2 = DIM == 3 ? BX * BY * (BZ + 1) : 0;
    static constexpr int NFMAX = cmax(NF0, cmax(NF1, NF2));
    // cells whose slope along an axis is needed: one more at either end
    static constexpr int NS0 = (BX + 2) * BY * BZ;
    static constexpr int NS1 = BX * (BY + 2) * BZ;
    static constexpr int NS2 = DIM == 3 ? BX * BY * (BZ + 2) : 0;
    static constexpr int NSMAX = cmax(NS0, cmax(NS1, NS2));
    static constexpr size_t SMEM = sizeof(double) * (size_t)(NW * PN + NC * (NFMAX + NSMAX));
};

// Tile of the single-grid kernels.
template <int DIM> struct DefaultBox;
template <> struct DefaultBox<3> { using type = BoxT<3, 8, 8, 4>; };
template <> struct DefaultBox<2> { using type = BoxT<2, 16, 16, 1>; };

// Small 2D FP64 grids: FP64 arithmetic runs at a small fraction of the FP32
// rate on this GPU, so the stage time of a grid with few 16 x 16 tiles is set
// by how many SMs take part; 8 x 8 tiles spread it over four times as many.
using SmallBox2D = BoxT<2, 8, 8, 1>;
inline bool small_2d_fp64(const GridParams &g) {
    return g.dim == 2 && (long long)((g.n[0] + 15) / 16) * ((g.n[1] + 15) / 16) < 256;
}
template <int DIM, bool SMALL>
using StageBox = typename std::conditional<SMALL, SmallBox2D, typename DefaultBox<DIM>::type>::type;

// 2D tile shapes of the batched kernel (all 256 cells): the autotuner's
// choices.  Every face is evaluated by the same arithmetic whatever the
// tile, so the shape changes the speed, never the result.
template <int S> struct Shape2;
template <> struct Shape2<0> { using type = BoxT<2, 16, 16, 1>; };
template <> struct Shape2<1> { using type = BoxT<2, 32, 8, 1>; };
template <> struct Shape2<2> { using type = BoxT<2, 64, 4, 1>; };
template <> struct Shape2<3> { using type = BoxT<2, 8, 32, 1>; };

// explicit roundings: no kernel's bits depend on what the compiler contracts
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }

// Half the limited slopes along axis D, ab / (a + b) where ab > 0 (the states
// are w +- psi/2, psi = 2ab/(a+b)), of (rho, u.., p) of the tile's cells and
// one more at either end: one work item per value, so that even a small tile
// keeps every scheduler's FP64 pipe busy.  Each slope serves the two faces of
// its cell.
template <typename B, int D>
__device__ __forceinline__ void slope_pass(const double *__restrict__ sW, double *__restrict__ sS) {
    constexpr int DIM = B::DIM;
    constexpr int EX = B::BX + 2 * (D == 0), EY = B::BY + 2 * (D == 1),
                  EZ = B::BZ + 2 * (D == 2 && DIM == 3);
    constexpr int NS = EX * EY * EZ;
    constexpr int s = D == 0 ? B::SX : (D == 1 ? B::SY : B::SZ);
    for (int i = threadIdx.x; i < NS * B::NC; i += NT) {
        const int m = i / NS, q = i - m * NS;
        const int x = q % EX, r = q / EX, y = r % EY, z = r / EY;
        const int a = (x + 2 - (D == 0)) + B::PX * (y + 2 - (D == 1)) +
                      (DIM == 3 ? B::PX * B::PY * (z + 2 - (D == 2)) : 0);
        const double *w = sW + m * B::PN + a;
        const double d0 = sub(w[0], w[-s]), d1 = sub(w[s], w[0]);
        const double ab = mul(d0, d1);
        const double h = mul(ab, drcp(add(d0, d1)));
        sS[i] = dpos(ab) ? h : 0.0;
    }
}

// Numerical flux through the face between box cells a and a + s_D, doubled
// (mass, momentum) and four-fold (energy); h0, h1: its cells' entries in the
// slope buffer.  ~110 FP64 operations in 3D where the form with divisions,
// both slopes per face and IEEE square roots took ~340.
template <typename B, int D>
__device__ __forceinline__ void face_flux(const GridParams &g, const double *__restrict__ sW, int a,
                                          const double *__restrict__ h, int hs, int ns,
                                          double (&F)[B::DIM + 2]) {
    constexpr int DIM = B::DIM;
    constexpr int NC = DIM + 2;
    constexpr int s = D == 0 ? B::SX : (D == 1 ? B::SY : B::SZ);
    const DoubleConsts &k = g.d;
    const int b = a + s;
    double wl[NC], wr[NC];
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        wl[m] = add(sW[m * B::PN + a], h[m * ns]);
        wr[m] = sub(sW[m * B::PN + b], h[m * ns + hs]);
    }
    // Rusanov; the speed of sound is gamma p / sqrt(gamma p rho)
    const double unL = wl[1 + D], unR = wr[1 + D], pL = wl[NC - 1], pR = wr[NC - 1];
    double mL[DIM], mR[DIM], rkL = 0.0, rkR = 0.0;
#pragma unroll
    for (int m = 0; m < DIM; ++m) {
        mL[m] = mul(wl[0], wl[1 + m]);
        mR[m] = mul(wr[0], wr[1 + m]);
        rkL = fma(mL[m], wl[1 + m], rkL);
        rkR = fma(mR[m], wr[1 + m], rkR);
    }
    const double gpL = mul(g.gamma, pL), gpR = mul(g.gamma, pR);
    const double sL = fma(gpL, drsqrt(mul(gpL, wl[0])), fabs(unL));
    const double sR = fma(gpR, drsqrt(mul(gpR, wr[0])), fabs(unR));
    const double sm = dmax_nonneg(sL, sR);
    F[0] = fma(sm, sub(wl[0], wr[0]), add(mL[D], mR[D]));
#pragma unroll
    for (int m = 0; m < DIM; ++m) {
        const double f = m == D ? add(fma(mL[m], unL, pL), fma(mR[m], unR, pR))
                                : fma(mL[m], unL, mul(mR[m], unR));
        F[1 + m] = fma(sm, sub(mL[m], mR[m]), f);
    }
    const double HL = fma(pL, k.h1, rkL), HR = fma(pR, k.h1, rkR);   // 2 rho H
    const double EL = fma(pL, k.e1, rkL), ER = fma(pR, k.e1, rkR);   // 2 rho E
    F[NC - 1] = fma(sm, sub(EL, ER), fma(HL, unL, mul(HR, unR)));
    if (!(g.mu_inf > 0.0)) return;

    // viscous stress and heat flux; face values from the two adjacent cells,
    // tangential derivatives from the average of the two cells' central
    // differences; T^(3/2) / (T + S) is T^2 / sqrt(T (T + S)^2)
    const double *T = sW + (DIM + 2) * B::PN;
    const double sT = add(T[a], T[b]), y = add(sT, k.s2);
    const double mm = mul(mul(k.km, sT), mul(sT, drsqrt(mul(mul(sT, y), y))));   // 2 mu / h
    const double *un = sW + (1 + D) * B::PN;
    double dt = 0.0, work = 0.0;     // tangential part of the divergence; 2 u . tau
#pragma unroll
    for (int m = 0; m < DIM; ++m) {
        if (m == D) continue;
        const int t = m == 0 ? B::SX : (m == 1 ? B::SY : B::SZ);
        const double *um = sW + (1 + m) * B::PN;
        // along axis m: the normal and the m-th velocity
        const double d1n = add(sub(un[a + t], un[a - t]), sub(un[b + t], un[b - t]));
        const double d1m = add(sub(um[a + t], um[a - t]), sub(um[b + t], um[b - t]));
        dt = add(dt, d1m);
        const double tau = mul(mm, fma(0.25, d1n, sub(um[b], um[a])));
        F[1 + m] = sub(F[1 + m], tau);
        work = fma(add(um[a], um[b]), tau, work);
    }
    const double tnn = mul(mm, fma(4.0 / 3.0, sub(un[b], un[a]), mul(-1.0 / 6.0, dt)));
    F[1 + D] = sub(F[1 + D], tnn);
    work = fma(add(un[a], un[b]), tnn, work);
    F[NC - 1] = sub(F[NC - 1], fma(mul(k.kl, mm), sub(T[b], T[a]), work));
}

// One direction: the limited slopes, all faces of the tile normal to axis D,
// then each cell's flux difference added to its accumulator.
template <typename B, int D>
__device__ __forceinline__ void direction_pass(const GridParams &g, const double *__restrict__ sW,
                                               double *__restrict__ sF, double *__restrict__ sS,
                                               double (&acc)[B::CPT][B::DIM + 2]) {
    constexpr int DIM = B::DIM;
    constexpr int NC = DIM + 2;
    constexpr int dx = D == 0, dy = D == 1, dz = (D == 2 && DIM == 3);
    constexpr int FX = B::BX + dx, FY = B::BY + dy, FZ = B::BZ + dz;
    constexpr int NF = FX * FY * FZ;
    // the slope buffer's extents and its stride along D
    constexpr int EX = B::BX + 2 * dx, EY = B::BY + 2 * dy, EZ = B::BZ + 2 * dz, NS = EX * EY * EZ;
    constexpr int HS = D == 0 ? 1 : (D == 1 ? EX : EX * EY);
    slope_pass<B, D>(sW, sS);
    __syncthreads();
    for (int f = threadIdx.x; f < NF; f += NT) {
        const int fx = f % FX;
        const int r = f / FX;
        const int fy = r % FY;
        const int fz = r / FY;
        const int a = (fx - dx + 2) + B::PX * (fy - dy + 2) +
                      (DIM == 3 ? B::PX * B::PY * (fz - dz + 2) : 0);
        double F[NC];
        face_flux<B, D>(g, sW, a, sS + fx + EX * (fy + EY * fz), HS, NS, F);
#pragma unroll
        for (int c = 0; c < NC; ++c) sF[c * B::NFMAX + f] = F[c];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < B::CPT; ++i) {
        const int cell = threadIdx.x + i * NT;
        if (cell < B::NCELL) {
            const int cx = cell % B::BX;
            const int cy = (cell / B::BX) % B::BY;
            const int cz = cell / (B::BX * B::BY);
            const int flo = cx + FX * (cy + FY * cz);
            const int fhi = (cx + dx) + FX * ((cy + dy) + FY * (cz + dz));
#pragma unroll
            for (int c = 0; c < NC; ++c)
                acc[i][c] = add(acc[i][c], sub(sF[c * B::NFMAX + flo], sF[c * B::NFMAX + fhi]));
        }
    }
    // (no barrier: the next pass writes the slopes, read before the barrier
    // above, and its faces only after its own)
}

// One tile of one stage.  MODE 0: out = L(Uin).  MODE 1: out = U1 = Uin +
// dt L(Uin).  MODE 2: out = U* = Un/2 + (Uin + dt L(Uin))/2 with Uin = U1,
// and the maximum of s_j(U*) over the tile's cells outside the band is
// returned to thread 0 (every thread must call; the function synchronises;
// a later call may reuse s_red only after its own first barrier).
template <typename B, int MODE>
__device__ __forceinline__ double stage_tile(const GridParams &g, int ox, int oy, int oz,
                                             const double *__restrict__ Uin,
                                             const double *__restrict__ Un,
                                             double *__restrict__ out, const double dt,
                                             const unsigned *__restrict__ band_bits,
                                             unsigned char *smem_raw, double *s_red, bool &bad,
                                             int *err) {
    constexpr int DIM = B::DIM;
    constexpr int NC = DIM + 2;
    double *sW = reinterpret_cast<double *>(smem_raw);
    double *sF = sW + B::NW * B::PN;
    double *sS = sF + NC * B::NFMAX;

    const int tid = threadIdx.x;
    const long long N = g.N;
    const double gm1 = g.gamma - 1.0;

    // ---- load tile + halo, to primitives
    // Tiles whose halo lies inside the domain index directly; the others map
    // every halo index through the boundary conditions.  The halo's corners
    // (outside the tile along two axes, by two cells along one of them, or
    // along three) are read by no face.
    const bool interior = ox >= 2 && oy >= 2 && ox + B::BX + 2 <= g.n[0] &&
                          oy + B::BY + 2 <= g.n[1] &&
                          (DIM == 2 || (oz >= 2 && oz + B::BZ + 2 <= g.n[2]));
    for (int q = tid; q < B::PN; q += NT) {
        const int lx = q % B::PX;
        const int r = q / B::PX;
        const int ly = r % B::PY;
        const int lz = r / B::PY;
        auto outside = [](int l, int n) { return l < 2 ? 2 - l : l > n + 1 ? l - n - 1 : 0; };
        const int ex = outside(lx, B::BX), ey = outside(ly, B::BY),
                  ez = DIM == 3 ? outside(lz, B::BZ) : 0;
        if (ex + ey + ez > 2 || (ex && ey && ez)) continue;
        double u[NC];
        if (interior) {
            const long long j = (ox + lx - 2) +
                                (long long)g.n[0] * ((oy + ly - 2) + (long long)g.n[1] * (oz + lz - 2 * (DIM == 3)));
            const bool okj = in_bounds(j, N, err);
#pragma unroll
            for (int c = 0; c < NC; ++c) u[c] = okj ? __ldg(Uin + c * N + j) : 0.0;
        } else {
            int flip = 0, fs = 0;
            const int sx = map_axis(ox + lx - 2, g.n[0], g.bc[0], g.bc[1], 0, flip, fs);
            const int sy = map_axis(oy + ly - 2, g.n[1], g.bc[2], g.bc[3], 1, flip, fs);
            const int sz = DIM == 3 ? map_axis(oz + lz - 2, g.n[2], g.bc[4], g.bc[5], 2, flip, fs) : 0;
            if (fs) {
                u[0] = 1.0;
                u[1] = 1.0;
#pragma unroll
                for (int d = 1; d < DIM; ++d) u[1 + d] = 0.0;
                u[NC - 1] = g.d.E_inf;
            } else {
                const long long j = sx + (long long)g.n[0] * (sy + (long long)g.n[1] * sz);
                const bool okj = in_bounds(j, N, err);
#pragma unroll
                for (int c = 0; c < NC; ++c) u[c] = okj ? __ldg(Uin + c * N + j) : 0.0;
#pragma unroll
                for (int d = 0; d < DIM; ++d)
                    if ((flip >> d) & 1) u[1 + d] = -u[1 + d];
            }
        }
        const double inv = drcp(u[0]);
        double rk = 0.0;
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            const double v = mul(u[1 + d], inv);
            sW[(1 + d) * B::PN + q] = v;
            rk = fma(u[1 + d], v, rk);
        }
        const double p = mul(gm1, fma(-0.5, rk, u[NC - 1]));
        sW[q] = u[0];
        sW[(DIM + 1) * B::PN + q] = p;
        sW[(DIM + 2) * B::PN + q] = mul(p, inv);
    }
    __syncthreads();

    // ---- faces, one direction at a time
    double acc[B::CPT][NC];
#pragma unroll
    for (int i = 0; i < B::CPT; ++i)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[i][c] = 0.0;
    direction_pass<B, 0>(g, sW, sF, sS, acc);
    direction_pass<B, 1>(g, sW, sF, sS, acc);
    if constexpr (DIM == 3) direction_pass<B, 2>(g, sW, sF, sS, acc);

    // ---- outputs
    double smax_t = 0.0;
    bool ok = true;
#pragma unroll
    for (int i = 0; i < B::CPT; ++i) {
        const int cell = tid + i * NT;
        if (cell >= B::NCELL) continue;
        const int cx = cell % B::BX;
        const int cy = (cell / B::BX) % B::BY;
        const int cz = cell / (B::BX * B::BY);
        const int gx = ox + cx, gy = oy + cy, gz = oz + cz;
        if (gx >= g.n[0] || gy >= g.n[1] || (DIM == 3 && gz >= g.n[2])) continue;
        const long long j = gx + (long long)g.n[0] * (gy + (long long)g.n[1] * gz);
        if (!in_bounds(j, N, err)) continue;
        double us[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const double L = mul(c == NC - 1 ? g.d.qinv_h : g.d.hinv_h, acc[i][c]);
            if (MODE == 0) us[c] = L;
            else us[c] = fma(dt, L, __ldg(Uin + c * N + j));
            if (MODE == 2) us[c] = fma(0.5, __ldg(Un + c * N + j), mul(0.5, us[c]));
            out[c * N + j] = us[c];
        }
        if (MODE == 2 && !band_bit(band_bits, j))
            smax_t = fmax(smax_t, step_rate<DIM, double>(g, us, ok));
    }

    if (MODE == 2) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            smax_t = dmax_nonneg(smax_t, __shfl_xor_sync(0xffffffffu, smax_t, o));
        bad = __syncthreads_or(!ok) != 0;
        if ((tid & 31) == 0) s_red[tid >> 5] = smax_t;
        __syncthreads();
        if (tid != 0) return 0.0;
        double m = s_red[0];
        for (int w = 1; w < NT / 32; ++w) m = dmax_nonneg(m, s_red[w]);
        return m;
    }
    return 0.0;
}

template <int DIM, int MODE, bool SMALL>
__global__ void __launch_bounds__(NT, 2)
stage_kernel(const GridParams g, const double *__restrict__ Uin, const double *__restrict__ Un,
             double *__restrict__ out, double *__restrict__ blockmax,
             const double *__restrict__ dt_ptr, int *__restrict__ err,
             const unsigned *__restrict__ band_bits, double dt_fixed) {
    using B = StageBox<DIM, SMALL>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double s_red[NT / 32];
    const int ox = blockIdx.x * B::BX, oy = blockIdx.y * B::BY;
    const int oz = DIM == 3 ? blockIdx.z * B::BZ : 0;
    const double dt = MODE == 0 ? 0.0 : (dt_fixed > 0.0 ? dt_fixed : *dt_ptr);
    bool bad = false;
    const double m = stage_tile<B, MODE>(g, ox, oy, oz, Uin, Un, out, dt, band_bits, smem_raw, s_red,
                                         bad, err);
    if (MODE == 2 && threadIdx.x == 0) {
        blockmax[blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)] = m;
        if (bad) record_error(err, ERR_NONFINITE);
    }
}

// The same stages over a batch of 2D grids: one persistent launch walks a
// list of (case, tile) work items; every case keeps its own parameters,
// state, step size and error word.  MODE 2 writes one maximum per item.
template <int S, int MODE>
__global__ void __launch_bounds__(NT, 2)
batch_stage_kernel(const BatchCase *__restrict__ cases, const int2 *__restrict__ items,
                   int n_items, double *__restrict__ item_max, double dt_fixed) {
    using B = typename Shape2<S>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double s_red[NT / 32];
    for (int it = blockIdx.x; it < n_items; it += gridDim.x) {
        const int2 w = items[it];
        const BatchCase &bc = cases[w.x];
        const GridParams g = bc.g;
        const int ntx = (g.n[0] + B::BX - 1) / B::BX;
        const int ox = (w.y % ntx) * B::BX, oy = (w.y / ntx) * B::BY;
        const double dt = dt_fixed > 0.0 ? dt_fixed : *bc.dt;
        const double *Uin = (const double *)(MODE == 2 ? bc.U1 : bc.Un);
        double *out = (double *)(MODE == 2 ? bc.Us : bc.U1);
        bool bad = false;
        const double m = stage_tile<B, MODE>(g, ox, oy, 0, Uin, (const double *)bc.Un, out, dt,
                                             bc.band_bits, smem_raw, s_red, bad, bc.err);
        if (MODE == 2 && threadIdx.x == 0) {
            item_max[it] = m;
            if (bad) record_error(bc.err, ERR_NONFINITE);
        }
        __syncthreads();   // the next item rewrites the tile's shared memory
    }
}

// First step size of a new state, *dt = cfl / max_j s_j(U) over every cell, and
// its time and step count (where given): per-CTA maxima, which the last CTA to
// finish reduces.  Bound by memory on large grids; the cells' and a warp's maxima
// stay in the grid's type, and those of warps and CTAs are integer work: on FP32
// grids a conversion and an FP64 maximum per cell kept the FP64 pipe busy for
// most of 103 us at 256^3 (now 56, 50 for its bytes; 1024 x 512 17.0 -> 10.8).
template <int DIM, typename T>
__global__ void __launch_bounds__(NT)
dt_init_kernel(const GridParams g, const T *__restrict__ U, double *__restrict__ blockmax,
               unsigned *__restrict__ counter, double *__restrict__ dt, int *__restrict__ err,
               int cells, double *__restrict__ t, long long *__restrict__ steps) {
    constexpr int NC = DIM + 2;
    __shared__ double s_red[NT / 32];
    __shared__ int s_last;
    const long long N = g.N;
    const long long j0 = (long long)blockIdx.x * cells;
    const long long j1 = j0 + cells < N ? j0 + cells : N;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T smax = T(0);
    bool ok = true;
    constexpr int B = sizeof(T) == 4 ? 4 : 1;   // cells whose loads are issued together
    for (long long jb = j0 + threadIdx.x; jb < j1; jb += B * NT) {
        T u[B][NC];
#pragma unroll
        for (int i = 0; i < B; ++i)
#pragma unroll
            for (int c = 0; c < NC; ++c) u[i][c] = jb + i * NT < j1 ? U[c * N + jb + i * NT] : T(0);
#pragma unroll
        for (int i = 0; i < B; ++i)
            if (jb + i * NT < j1) smax = fmax(smax, step_rate<DIM, T>(g, u[i], ok));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) smax = fmax(smax, __shfl_xor_sync(0xffffffffu, smax, o));
    const int bad = __syncthreads_or(!ok);
    if (lane == 0) s_red[warp] = (double)smax;
    __syncthreads();
    if (threadIdx.x == 0) {
        double m = s_red[0];
        for (int w = 1; w < NT / 32; ++w) m = dmax_nonneg(m, s_red[w]);
        blockmax[blockIdx.x] = m;
        if (bad) record_error(err, ERR_NONFINITE);
        __threadfence();
        s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double m = 0.0;
    for (unsigned b = threadIdx.x; b < gridDim.x; b += NT) m = dmax_nonneg(m, __ldcg(blockmax + b));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = dmax_nonneg(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) s_red[warp] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        double mm = s_red[0];
        for (int w = 1; w < NT / 32; ++w) mm = dmax_nonneg(mm, s_red[w]);
        const bool good = mm > 0.0 && mm <= DBL_MAX && !(__ldcg(err) & ERR_NONFINITE);
        if (!good) record_error(err, ERR_NONFINITE);
        *dt = good ? g.cfl / mm : 0.0;
        *counter = 0u;
        if (t) {
            *t = 0.0;
            *steps = 0;
        }
    }
}

template <int DIM, bool SMALL = false>
dim3 stage_grid(const GridParams &g) {
    using B = StageBox<DIM, SMALL>;
    return dim3((g.n[0] + B::BX - 1) / B::BX, (g.n[1] + B::BY - 1) / B::BY,
                DIM == 3 ? (g.n[2] + B::BZ - 1) / B::BZ : 1);
}

template <int DIM, int MODE, bool SMALL>
cudaError_t launch_box(const GridParams &g, const void *Uin, const void *Un, void *out,
                       const FluidBuffers &fb, double dt_fixed, cudaStream_t s) {
    using B = StageBox<DIM, SMALL>;
    cudaError_t e = func_smem_attr((const void *)stage_kernel<DIM, MODE, SMALL>, B::SMEM);
    if (e != cudaSuccess) return e;
    stage_kernel<DIM, MODE, SMALL><<<stage_grid<DIM, SMALL>(g), NT, B::SMEM, s>>>(
        g, (const double *)Uin, (const double *)Un, (double *)out, fb.blockmax, fb.dt, fb.err,
        fb.band_bits, dt_fixed);
    return cudaGetLastError();
}

template <int MODE>
cudaError_t dispatch(const GridParams &g, int fp_bytes, const void *Uin, const void *Un, void *out,
                     const FluidBuffers &fb, double dt_fixed, cudaStream_t s) {
    if (fp_bytes == 4)
        return g.dim == 3 ? launch_zmarch(MODE, g, Uin, Un, out, fb, dt_fixed, s)
                          : launch_ymarch(MODE, g, Uin, Un, out, fb, dt_fixed, s);
    if (g.dim == 3) return launch_box<3, MODE, false>(g, Uin, Un, out, fb, dt_fixed, s);
    return small_2d_fp64(g) ? launch_box<2, MODE, true>(g, Uin, Un, out, fb, dt_fixed, s)
                            : launch_box<2, MODE, false>(g, Uin, Un, out, fb, dt_fixed, s);
}

template <int S, int MODE>
cudaError_t batch_stage_t(const BatchCase *cases, const int2 *items, int n_items,
                          double *item_max, double dt_fixed, int n_sm, cudaStream_t s) {
    using B = typename Shape2<S>::type;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = func_smem_attr((const void *)batch_stage_kernel<S, MODE>, B::SMEM);
    if (e != cudaSuccess) return e;
    // resident blocks per SM, per device ordinal (0: not yet asked)
    static std::atomic<int> per_sm_of[64];
    int per_sm = dev < 64 ? per_sm_of[dev].load() : 0;
    if (per_sm == 0) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_stage_kernel<S, MODE>, NT,
                                                          B::SMEM);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
        if (dev < 64) per_sm_of[dev].store(per_sm);
    }
    long long ctas = (long long)per_sm * (n_sm > 0 ? n_sm : 1);
    if (ctas > n_items) ctas = n_items;
    if (ctas < 1) return cudaSuccess;
    batch_stage_kernel<S, MODE><<<(unsigned)ctas, NT, B::SMEM, s>>>(cases, items, n_items, item_max,
                                                                     dt_fixed);
    return cudaGetLastError();
}

template <int MODE>
cudaError_t batch_stage_shape(int shape, const BatchCase *cases, const int2 *items, int n_items,
                              double *item_max, double dt_fixed, int n_sm, cudaStream_t s) {
    switch (shape) {
    case 0: return batch_stage_t<0, MODE>(cases, items, n_items, item_max, dt_fixed, n_sm, s);
    case 1: return batch_stage_t<1, MODE>(cases, items, n_items, item_max, dt_fixed, n_sm, s);
    case 2: return batch_stage_t<2, MODE>(cases, items, n_items, item_max, dt_fixed, n_sm, s);
    case 3: return batch_stage_t<3, MODE>(cases, items, n_items, item_max, dt_fixed, n_sm, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

void batch_tile_shape(int shape, int *bx, int *by) {
    static const int X[kBatchShapes] = {16, 32, 64, 8}, Y[kBatchShapes] = {16, 8, 4, 32};
    *bx = X[shape];
    *by = Y[shape];
}

cudaError_t launch_batch_stage(int mode, int shape, int rows, int fp_bytes, const BatchCase *cases,
                               const int2 *items, int n_items, double *item_max, double dt_fixed,
                               int n_sm, cudaStream_t s) {
    if (n_items <= 0) return cudaSuccess;
    if (fp_bytes == 4)
        return launch_batch_ymarch(mode, rows, cases, items, n_items, item_max, dt_fixed, s);
    if (mode == 1)
        return batch_stage_shape<1>(shape, cases, items, n_items, item_max, dt_fixed, n_sm, s);
    if (mode == 2)
        return batch_stage_shape<2>(shape, cases, items, n_items, item_max, dt_fixed, n_sm, s);
    return cudaErrorInvalidValue;
}

size_t fluid_stage_blocks(const GridParams &g, int fp_bytes) {
    if (fp_bytes == 4) return g.dim == 3 ? zmarch_blocks(g) : ymarch_blocks(g);
    const dim3 d = g.dim == 3 ? stage_grid<3>(g)
                   : small_2d_fp64(g) ? stage_grid<2, true>(g) : stage_grid<2>(g);
    return (size_t)d.x * d.y * d.z;
}

size_t dt_init_blocks(const GridParams &g) {
    const int c = dt_cells_per_cta(g.N);
    return (size_t)((g.N + c - 1) / c);
}

size_t fluid_blockmax_count(const GridParams &g, int fp_bytes) {
    const size_t a = fluid_stage_blocks(g, fp_bytes), b = dt_init_blocks(g);
    return a > b ? a : b;
}

cudaError_t launch_stage1(const GridParams &g, int fp_bytes, const void *U, void *U1,
                          const FluidBuffers &fb, double dt_fixed, cudaStream_t s) {
    return dispatch<1>(g, fp_bytes, U, U, U1, fb, dt_fixed, s);
}

cudaError_t launch_stage2(const GridParams &g, int fp_bytes, const void *Un, const void *U1,
                          void *out, const FluidBuffers &fb, double dt_fixed, cudaStream_t s) {
    return dispatch<2>(g, fp_bytes, U1, Un, out, fb, dt_fixed, s);
}

cudaError_t launch_rhs(const GridParams &g, int fp_bytes, const void *U, void *L,
                       const FluidBuffers &fb, cudaStream_t s) {
    return dispatch<0>(g, fp_bytes, U, U, L, fb, 0.0, s);
}

template <int DIM, typename T>
static cudaError_t dt_init_t(const GridParams &g, const void *U, const FluidBuffers &fb, double *t,
                             long long *steps, cudaStream_t s) {
    dt_init_kernel<DIM, T><<<(unsigned)dt_init_blocks(g), NT, 0, s>>>(
        g, (const T *)U, fb.blockmax, fb.counter, fb.dt, fb.err, dt_cells_per_cta(g.N), t, steps);
    return cudaGetLastError();
}
cudaError_t launch_dt_init(const GridParams &g, int fp_bytes, const void *U,
                           const FluidBuffers &fb, cudaStream_t s, double *t, long long *steps) {
    if (g.dim == 3)
        return fp_bytes == 4 ? dt_init_t<3, float>(g, U, fb, t, steps, s)
                             : dt_init_t<3, double>(g, U, fb, t, steps, s);
    return fp_bytes == 4 ? dt_init_t<2, float>(g, U, fb, t, steps, s)
                         : dt_init_t<2, double>(g, U, fb, t, steps, s);
}

}  // namespace ibmk

#include "flux_ym.cuh"
