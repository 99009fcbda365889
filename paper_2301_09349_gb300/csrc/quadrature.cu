// Lagrangian quadrature of Sec. 2.2: the weights eps solve A eps = 1 with
// A_kl the overlap of the k-th and l-th interpolation kernels, so that
// interpolating a spread unit field returns 1 at every marker.  Taken in
// dimensionless form A~_kl = sum_j Phi_k(j) Phi_l(j), A~ eps~ = 1,
// eps = h^d eps~.
//
// Because Phi is a tensor product, A~_kl = prod_d sum_i phi(r_k,d(i))
// phi(r_l,d(i)) over the three support columns of k on each axis.  Rows are
// assembled in ELL form (column-major, one warp per marker, neighbours
// found through the marker bins in a fixed order).  The solution is FP64:
// residuals rhs - A~ x and the stopping test are formed in FP64, and only the
// corrections are FP32.  Up to 160 markers they come from a dense Cholesky
// factor on one CTA, in 2D with more than 64 markers and short rows from
// conjugate gradients first; above, from conjugate gradients on one CTA (up to
// 512 markers) or one thread-block cluster (up to 16384).  Systems that these
// cannot contract, and those of more than 16384 markers, go to Jacobi-
// preconditioned CG in FP64 on one CTA.  Fixed-order sums throughout: the
// result is bitwise reproducible; every loop is bounded.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>

#include "cluster_plan.h"
#include "internal.h"

namespace cg = cooperative_groups;

namespace ibmk {
namespace {

// The 1D weights of every marker at its owner cell and the two beside it,
// per axis: wphi[k][d][i] = phi((i - 1) + 1/2 - frac_d[k][d]) (Eq. 3-point
// delta), one thread per (marker, axis).  FP64 runs at a small fraction of
// the FP32 rate on this GPU, so the assembly multiplies these tabulated
// weights instead of evaluating phi for every pair of markers.
__global__ void support_weights_kernel(const MarkerBuffers m, int dim) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = t / 3, d = t - 3 * k;
    if (k >= m.ns || d >= dim) return;
    const double fk = m.frac_d[(long long)k * 3 + d];
#pragma unroll
    for (int i = 0; i < 3; ++i) m.wphi[(long long)k * 9 + d * 3 + i] = phi_d(((double)(i - 1) + 0.5) - fk);
}

// Row k of A~: one warp per marker, one lane per neighbour cell of its owner
// cell (the 5^d cells whose markers can overlap its support), visited in
// (z, y, x) order and bin order within a cell; a warp scan of the per-cell
// counts places every entry where a serial walk would, so the rows are the
// same whatever the warp size.  A~_kl = prod_d sum_i phi_k,d(i) phi_l,d(i)
// over the cells of both supports, from the tabulated weights: cell
// ck - 1 + i of marker k is cell j = ck - cl + i of marker l, and the terms
// with j outside [0, 2] are zero (|r| >= 3/2), so skipping them leaves every
// sum as it was with phi evaluated per pair.
template <int DIM>
__global__ void __launch_bounds__(128)
assemble_kernel(const GridParams g, const MarkerBuffers m, const QuadBuffers q,
                const unsigned *__restrict__ keys, const int *__restrict__ perm) {
    constexpr int NCELLS = DIM == 3 ? 125 : 25;
    const int lane = threadIdx.x & 31;
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (k >= m.ns) return;
    int ck[3] = {0, 0, 0};
    double wk[3][3];
    for (int d = 0; d < DIM; ++d) {
        ck[d] = m.cell[(long long)k * 3 + d];
        for (int i = 0; i < 3; ++i) wk[d][i] = m.wphi[(long long)k * 9 + d * 3 + i];
    }
    int base = 0;
    bool overflow = false;
    for (int r0 = 0; r0 < NCELLS; r0 += 32) {
        const int c = r0 + lane;
        int lo = 0, end = 0;
        if (c < NCELLS) {
            const int ox = c % 5 - 2, oy = (c / 5) % 5 - 2, oz = DIM == 3 ? c / 25 - 2 : 0;
            const int x = ck[0] + ox, y = ck[1] + oy, z = (DIM == 3 ? ck[2] : 0) + oz;
            const bool in = x >= 0 && y >= 0 && z >= 0 && x < g.n[0] && y < g.n[1] &&
                            (DIM == 2 || z < g.n[2]);
            if (in) {
                const unsigned key = cell_key(g, x, y, z);
                const int tc = (int)(key / (unsigned)g.cells_per_tile);
                int a = m.tile_off[tc], b = m.tile_off[tc + 1];
                const int tend = b;
                while (a < b) {
                    const int mid = (a + b) >> 1;
                    if (keys[mid] < key) a = mid + 1;
                    else b = mid;
                }
                lo = a;
                end = a;
                while (end < tend && keys[end] == key) ++end;
            }
        }
        const int cnt = end - lo;
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const int tot = __shfl_sync(0xffffffffu, incl, 31);
        int w = base + incl - cnt;
        for (int p = lo; p < end; ++p, ++w) {
            const int l = perm[p];
            double a = 1.0;
            for (int d = 0; d < DIM; ++d) {
                const int off = ck[d] - m.cell[(long long)l * 3 + d];
                const double *wl = m.wphi + (long long)l * 9 + d * 3;
                double sum = 0.0;
                for (int i = 0; i < 3; ++i) {
                    const int j = off + i;
                    if (j >= 0 && j <= 2) sum += wk[d][i] * wl[j];
                }
                a *= sum;
            }
            if (l == k) q.diag[k] = a;
            if (w < q.width) {
                q.col[(long long)w * q.cap + k] = l;
                q.val[(long long)w * q.cap + k] = a;
            } else {
                overflow = true;
            }
        }
        base += tot;
    }
    overflow = __any_sync(0xffffffffu, overflow);
    if (lane == 0) {
        q.cnt[k] = base < q.width ? base : q.width;
        if (overflow) record_error(m.err, ERR_CAPACITY);
    }
}

template <int NTH>
__device__ __forceinline__ double block_sum(double v, double *s_red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) s_red[w] = v;
    __syncthreads();
    double r = lane < NTH / 32 ? s_red[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
}

template <int NTH>
__device__ __forceinline__ double block_max(double v, double *s_red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = dmax_nonneg(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) s_red[w] = v;
    __syncthreads();
    double r = lane < NTH / 32 ? s_red[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r = dmax_nonneg(r, __shfl_xor_sync(0xffffffffu, r, o));
    return r;
}

template <int NTH>
__device__ __forceinline__ void spmv(int ns, const QuadBuffers &q, const double *x, double *y,
                                     int *err) {
    for (int k = threadIdx.x; k < ns; k += NTH) {
        const int c = q.cnt[k];
        double s = 0.0;
        for (int i = 0; i < c; ++i) {
            const int l = q.col[(long long)i * q.cap + k];
            if (in_bounds(l, ns, err)) s += q.val[(long long)i * q.cap + k] * x[l];
        }
        y[k] = s;
    }
}

// Jacobi-PCG on A~ x = rhs (all ones when rhs is null) by one CTA of NTH
// threads, from x (warm) or from zero; restarts from the true residual.
// Returns whether max|rhs - A~ x| <= tol; *iters and *resid report the run.
template <int NTH>
__device__ bool pcg_solve(int ns, const QuadBuffers &q, double *x, const double *__restrict__ rhs,
                          double tol, int maxit, int warm, double *s_red, int *iters,
                          double *resid, int *err) {
    double *r = q.r, *z = q.z, *p = q.p, *qv = q.q;
    if (!warm)
        for (int k = threadIdx.x; k < ns; k += NTH) x[k] = 0.0;
    __syncthreads();
    int it = 0;
    bool converged = false;
    double rmax = 0.0;
    for (int restart = 0; restart < 50 && it < maxit && !converged; ++restart) {
        spmv<NTH>(ns, q, x, qv, err);
        __syncthreads();
        double lm = 0.0;
        for (int k = threadIdx.x; k < ns; k += NTH) {
            r[k] = (rhs ? rhs[k] : 1.0) - qv[k];
            lm = dmax_nonneg(lm, fabs(r[k]));
        }
        rmax = block_max<NTH>(lm, s_red);
        if (rmax <= tol) { converged = true; break; }
        double lrz = 0.0;
        for (int k = threadIdx.x; k < ns; k += NTH) {
            z[k] = r[k] / q.diag[k];
            p[k] = z[k];
            lrz += r[k] * z[k];
        }
        double rz = block_sum<NTH>(lrz, s_red);
        while (it < maxit) {
            __syncthreads();
            spmv<NTH>(ns, q, p, qv, err);
            __syncthreads();
            double lpq = 0.0;
            for (int k = threadIdx.x; k < ns; k += NTH) lpq += p[k] * qv[k];
            const double alpha = rz / block_sum<NTH>(lpq, s_red);
            double lr = 0.0;
            for (int k = threadIdx.x; k < ns; k += NTH) {
                x[k] += alpha * p[k];
                r[k] -= alpha * qv[k];
                lr = dmax_nonneg(lr, fabs(r[k]));
            }
            const double rm = block_max<NTH>(lr, s_red);
            ++it;
            if (rm <= tol) break;
            double lrz2 = 0.0;
            for (int k = threadIdx.x; k < ns; k += NTH) {
                z[k] = r[k] / q.diag[k];
                lrz2 += r[k] * z[k];
            }
            const double rzn = block_sum<NTH>(lrz2, s_red);
            const double beta = rzn / rz;
            rz = rzn;
            for (int k = threadIdx.x; k < ns; k += NTH) p[k] = z[k] + beta * p[k];
        }
        __syncthreads();
    }
    if (!converged) {
        __syncthreads();
        spmv<NTH>(ns, q, x, qv, err);
        __syncthreads();
        double lm = 0.0;
        for (int k = threadIdx.x; k < ns; k += NTH) lm = dmax_nonneg(lm, fabs((rhs ? rhs[k] : 1.0) - qv[k]));
        rmax = block_max<NTH>(lm, s_red);
        converged = rmax <= tol;
    }
    *iters = it;
    *resid = rmax;
    return converged;
}

template <int NTH>
__global__ void __launch_bounds__(NTH)
pcg_kernel(int ns, const QuadBuffers q, double *x, const double *__restrict__ rhs, double tol,
           int maxit, int warm, int *err) {
    __shared__ double s_red[32];
    int it = 0;
    double rmax = 0.0;
    const bool converged =
        pcg_solve<NTH>(ns, q, x, rhs, tol, maxit, warm, s_red, &it, &rmax, err);
    if (threadIdx.x == 0) {
        *q.iters = it;
        *q.resid = rmax;
        if (!converged) record_error(err, ERR_NOCONV);
    }
}

// sums of a and b over the warp: lanes below 16 return a's, the others b's
__device__ __forceinline__ float warp_sum2(float a, float b, int lane) {
    float v = lane & 16 ? b : a;
    v += __shfl_xor_sync(0xffffffffu, lane & 16 ? a : b, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// the sums over the CTA's warps of the pairs part[w], part[32 + w] (zeros
// past the last warp), in every lane
__device__ __forceinline__ float2 part_sum2(const float *part, int lane) {
    const float *p = part + (lane & 16 ? 32 : 0) + (lane & 15);
    float v = p[0] + p[16];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const float w = __shfl_xor_sync(0xffffffffu, v, 16);
    return lane & 16 ? make_float2(w, v) : make_float2(v, w);
}
// The power of two at or below x: FP32 corrections are solved for r / cg_unit(max
// |r|), so that they give the same bits at every scale of the right-hand side
// (the adjoint's may have any) and nothing underflows.
__device__ __forceinline__ double cg_unit(double x) {
    return __longlong_as_double(__double_as_longlong(x) & 0x7ff0000000000000ll);
}
// 1 / cg_unit(x) (an FP64 division is a chain of some 40 operations of 64 cycles)
__device__ __forceinline__ double cg_per_unit(double x) {
    return __longlong_as_double(0x7fe0000000000000ll - (__double_as_longlong(x) & 0x7ff0000000000000ll));
}
// residuals whose unit and its reciprocal are normal numbers (not NaN, not inf)
__device__ __forceinline__ bool cg_in_range(double rmax) { return rmax > 1e-290 && rmax < 1e290; }
// r.u at which max|r| has fallen far enough: by `inner` from rmax's own r.u,
// or (the diagonal of A~ is at most one) to a tenth of tol in the mean square
// (r and tol in units of cg_unit)
__device__ __forceinline__ float cg_stop(float ru, float inner, int ns, double tol) {
    const float t = 0.1f * (float)tol;
    return fmaxf(ru * inner * inner, (float)ns * t * t);
}

// When FP32 corrections give up.  A first pass takes 17 to 72 iterations with one
// marker per cell (200 to 16000 markers), 90 to 600 with 1.4 markers per cell;
// the next one 1.1 to 4 times as many, on a residual that the first has left
// where A~ is weakest.  A nearly singular A~ (two markers 0.01 to 0.9 cells apart
// in one cell, condition 1e8 and more) shows itself there: eight iterations
// beyond the first pass's its r.u has grown by 200 and more, where it is below
// 0.05 of its start in the others (one that went on took up to 1000 iterations,
// all of them lost).  Besides, a first pass of more iterations than unknowns and
// a later one of over four times the first are ended, and a pass that does not
// contract the residual by four is the last.  A whole set_markers, before these
// limits -> now, and by the FP64 solver alone: 5000 markers, two of them 0.1
// cells apart, 7.5 -> 2.8 ms (2.9), 700 0.97 -> 0.77 (0.69), 300 markers on 150
// cells 14.4 -> 4.2 (3.9).
//
// The FP64 solver then starts where the call started (from zero if its guess is
// no better): what FP32 got wrong lies along the near-null vectors, where it
// costs the FP64 solver more than the corrections save (200 markers, two of them
// 0.9 cells apart: 108 iterations from zero, no convergence from the corrected
// values).  After two contracting passes A~ is well conditioned, and it goes on
// from the last good values.  maxit bounds the FP32 iterations, and those of the
// FP64 solver, which then has all of maxit: FP32 passes take 1.1 to 9 times its
// iterations, so that counting them as well would refuse what it solves within
// maxit.
struct CgPass {
    int left, look;   // iterations left, and how many will be when r.u is looked at
};
__device__ __forceinline__ CgPass cg_pass(int outer, int first, int ns, int left) {
    if (outer == 0) return CgPass{min(ns, left), 0};
    const int last = min(4 * first + 32, left);
    return CgPass{last, max(last - first - 8, 0)};
}

// The FP64 solver for what FP32 could not contract, from x: by the CTA's NTH
// threads, or 256 of them up to 2048 markers (5 us an iteration at 200 markers, 7
// with 512: its block sums and barriers).  A call, so that it takes no registers
// from the corrections (inlined, 2 % of their time).
template <int NTH>
__device__ __noinline__ bool pcg_takes_over(int ns, const QuadBuffers &q, double *x,
                                            const double *rhs, double tol, int maxit, double *s_red,
                                            int *iters, double *resid, int *err) {
    if (ns > 2048) return pcg_solve<NTH>(ns, q, x, rhs, tol, maxit, 1, s_red, iters, resid, err);
    return pcg_solve<256>(ns, q, x, rhs, tol, maxit, 1, s_red, iters, resid, err);
}
__device__ __forceinline__ bool pcg_idle(int ns, int tid) { return ns <= 2048 && tid >= 256; }

// BCG_MAX to CL_MAX markers: FP32 conjugate gradients inside FP64 iterative
// refinement, on one thread-block cluster.
//
// The FP64 PCG on one CTA (above) is bound by the FP64 pipe of a single SM
// (about two operations per cycle; 85 k nonzeros of a 2842-marker sphere take
// 25 us of it per iteration) and by the L2 latency of the ELL rows: 10.36 ms
// for that sphere, 3.56 ms for 713 markers.  Here the rows are dealt to the
// CTAs of a cluster (8, or 16 above CL_WIDE markers), 2^j threads per row,
// which hold their FP32 entries in registers (past CL_REG in shared memory,
// past that the ELL rows serve); the correction
// equation A~ d = r is solved in FP32 (Jacobi preconditioner, the
// single-reduction form of Chronopoulos and Gear) to CL_INNER of its
// residual, and r = rhs - A~ x is formed in FP64 from the ELL rows, so the
// solution and the stopping test max|r| <= tol are those of the FP64 solver.
// Per iteration: the product from a replicated copy of u, the warps' partial
// sums sent to every CTA through distributed shared memory, a cluster
// barrier, the vector updates, u sent to every CTA, a second barrier: what
// bounds it now are the two exchanges (on a GB300 a cluster barrier behind
// remote stores takes ~1000 cycles with 8 CTAs and, with all of u travelling,
// ~2400 with 16).  2842 markers 10.36 -> 0.69 ms, 713 markers 3.56 -> 0.34 ms
// (one CTA of 1024 threads, whose gathers meet in the banks: 0.55).  Every CTA reduces the same partials in the same order, so all take
// the same branches and the result is bitwise reproducible.  A system that
// FP32 cannot contract (near-singular A~: two markers in one cell placed
// without dedup) goes to the FP64 PCG in the same launch.
constexpr int CL_SM = 16;                // entries of a thread in shared memory
constexpr float CL_INNER = 1e-5f;
constexpr int CL_OUTER_MAX = 24;
template <int NTH> constexpr int CL_REG = NTH <= 512 ? 24 : 12;   // entries in registers

// u of every row (16-byte aligned), the CTAs' FP64 maxima and partial sums,
// the threads' entries past their registers
template <int NTH>
size_t cluster_smem(const ClusterShape &c) {
    return sizeof(float) * (size_t)c.ctas * c.rows + (sizeof(double) + sizeof(float2)) * c.ctas +
           (sizeof(float) + sizeof(unsigned short)) * (size_t)CL_SM * NTH;
}

template <int NTH>
__global__ void __launch_bounds__(NTH, 1)
cluster_cg_kernel(int ns, const ClusterShape sh, const QuadBuffers q, double *x,
                  const double *__restrict__ rhs, double tol, int maxit, int warm, int *err) {
    constexpr int REG = CL_REG<NTH>;
    extern __shared__ __align__(16) double smem_cl[];
    cg::cluster_group cl = cg::this_cluster();
    const int C = sh.ctas, R = sh.rows, LG = sh.lpr_log, LPR = 1 << LG;
    const int rank = (int)cl.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sub = tid & (LPR - 1), row = tid >> LG, k = rank * R + row;
    const bool own = row < R && k < ns, on = 32 * warp < (R << LG);
    float *su = reinterpret_cast<float *>(smem_cl);                    // [C * R]
    double *smax = reinterpret_cast<double *>(su + C * R);             // [C]
    float2 *spart = reinterpret_cast<float2 *>(smax + C);              // [C] (r.u, w.u)
    float *sval = reinterpret_cast<float *>(spart + C);                // [CL_SM][NTH]
    unsigned short *scol = reinterpret_cast<unsigned short *>(sval + CL_SM * NTH);
    __shared__ float s_warp[64];
    __shared__ double s_red[32];
    // what a pass needs at its ends only, out of the registers: r.u at its
    // start, max|r| before it, its iterations, those so far and of the first
    __shared__ struct {
        double rprev;
        float ru0;
        int last, it, first;
    } s_pass;
    if (tid < 64) s_warp[tid] = 0.0f;
    // entry j of this thread: number sub + j LPR of its row
    const int cnt = own ? q.cnt[k] : 0;
    const int mine = cnt > sub ? (cnt - sub + LPR - 1) >> LG : 0;
    auto entry = [&](int j, float &v, int &l) {
        v = 0.0f;
        l = 0;
        if (j < mine) {
            const long long at = (long long)(sub + (j << LG)) * q.cap + k;
            l = q.col[at];
            v = (float)q.val[at];
            if (!in_bounds(l, ns, err)) { l = 0; v = 0.0f; }
        }
    };
    float rv[REG];
    unsigned rc[REG / 2];
#pragma unroll
    for (int j = 0; j < REG; j += 2) {
        int l0, l1;
        entry(j, rv[j], l0);
        entry(j + 1, rv[j + 1], l1);
        rc[j / 2] = (unsigned)l0 | ((unsigned)l1 << 16);
    }
    for (int j = REG; j < min(mine, REG + CL_SM); ++j) {
        float v;
        int l;
        entry(j, v, l);
        sval[(j - REG) * NTH + tid] = v;
        scol[(j - REG) * NTH + tid] = (unsigned short)l;
    }
    const float inv = own ? (float)(1.0 / q.diag[k]) : 0.0f;
    // a row's first thread holds its value, in x; the first guess and the value
    // at the start of a pass wait in the FP64 solver's workspace
    const bool writes = own && sub == 0;
    bool guess = warm != 0;
    if (tid == 0) s_pass.it = s_pass.first = 0;
    if (writes) {
        if (!warm) x[k] = 0.0;
        q.z[k] = x[k];
    }
    __threadfence();
    cl.sync();

    // (r.u, w.u) over the cluster: the CTA's own first, one 8-byte store to
    // every CTA, a cluster barrier; the CTAs' values summed in one order by
    // every warp
    auto reduce_all = [&](float a, float b) {
        if (on) {
            const float t = warp_sum2(a, b, lane);
            if ((lane & 15) == 0) s_warp[2 * (lane & 16) + warp] = t;
        }
        __syncthreads();
        if (warp == 0) {
            const float2 v = part_sum2(s_warp, lane);
            if (lane < C) cl.map_shared_rank(spart, lane)[rank] = v;
        }
        cl.sync();
        const float2 v = (lane & 15) < C ? spart[lane & 15] : make_float2(0.0f, 0.0f);
        float s1 = lane & 16 ? v.y : v.x;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        const float s2 = __shfl_xor_sync(0xffffffffu, s1, 16);
        return lane & 16 ? make_float2(s2, s1) : make_float2(s1, s2);
    };
    // this CTA's rows of u to every CTA
    auto send_u = [&](float u) {
        if (row < R && sub == 0) su[rank * R + row] = u;
        __syncthreads();
        const int n4 = R / 4;
        float4 *part4 = reinterpret_cast<float4 *>(su + rank * R);
        for (int i = tid; i < n4 * C; i += NTH) {
            const int t = i / n4, j = i - t * n4;
            if (t != rank) cl.map_shared_rank(part4, t)[j] = part4[j];
        }
        cl.sync();
    };

    bool converged = false, over = false;   // over: the last pass was given up
    double rmax = 0.0;
    for (int outer = 0;; ++outer) {
        // r = rhs - A~ x in FP64 from the ELL rows; x was written by its rows'
        // owners before the last cluster barrier
        double a = 0.0;
#pragma unroll 4
        for (int i = sub; i < cnt; i += LPR) {
            const int l = __ldg(q.col + (long long)i * q.cap + k);
            if (in_bounds(l, ns, err)) a += __ldg(q.val + (long long)i * q.cap + k) * __ldcg(x + l);
        }
        for (int o = LPR / 2; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        const double r64 = own ? (rhs ? rhs[k] : 1.0) - a : 0.0;
        rmax = block_max<NTH>(fabs(r64), s_red);
        if (tid < C) cl.map_shared_rank(smax, tid)[rank] = rmax;
        cl.sync();
        rmax = lane < C ? smax[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            rmax = dmax_nonneg(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
        if (rmax <= tol) { converged = true; break; }
        // no contraction, or a value FP32 cannot hold: the FP64 solver
        if (outer == 0 && !(rmax < 1.0)) guess = false;   // worse than none
        const bool failed = outer > 0 && (over || !(rmax < 0.25 * s_pass.rprev));
        if (failed || !cg_in_range(rmax) || outer == CL_OUTER_MAX ||
            s_pass.it >= maxit) {
            if (writes && (s_pass.it >= maxit || outer - (failed ? 1 : 0) < 2)) x[k] = guess ? q.z[k] : 0.0;
            else if (writes && failed) x[k] = q.r[k];
            break;
        }
        if (writes) q.r[k] = x[k];
        CgPass pass = cg_pass(outer, s_pass.first, ns, maxit - s_pass.it);
        // the correction d, from zero (a row's threads all hold its values)
        float r = (float)(r64 * cg_per_unit(rmax)), u = r * inv, p = 0.0f, sv = 0.0f, d = 0.0f,
              gam = 1.0f, alpha = 1.0f, stop = 0.0f;
        send_u(u);
        if (tid == 0) {   // (every thread is past the tests above)
            s_pass.rprev = rmax;
            s_pass.last = pass.left;
        }
        for (bool first = true;; first = false) {
            float w = 0.0f;
            if (on) {
                float w1 = 0.0f;
#pragma unroll
                for (int j = 0; j < REG; j += 2) {
                    if (j >= mine) break;
                    w += rv[j] * su[rc[j / 2] & 0xffffu];
                    w1 += rv[j + 1] * su[rc[j / 2] >> 16];
                }
                for (int j = REG; j < mine; ++j) {
                    if (j < REG + CL_SM) {
                        w += sval[(j - REG) * NTH + tid] * su[scol[(j - REG) * NTH + tid]];
                    } else {
                        float v;
                        int l;
                        entry(j, v, l);
                        w += v * su[l];
                    }
                }
                w += w1;
                for (int o = LPR / 2; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
            }
            const float2 tot = reduce_all(sub == 0 ? r * u : 0.0f, sub == 0 ? w * u : 0.0f);
            const float g1 = tot.x, del = tot.y;
            if (first) {
                stop = cg_stop(g1, CL_INNER, ns, tol * cg_per_unit(s_pass.rprev));
                if (tid == 0) s_pass.ru0 = g1;
            }
            if (g1 <= stop) break;
            const float beta = first ? 0.0f : __fdividef(g1, gam);
            const float den = first ? del : del - beta * __fdividef(g1, alpha);
            if (!(den > 0.0f) || pass.left == pass.look) {   // (a NaN sum ends here too)
                over = pass.left == 0 || (pass.left == pass.look && g1 > s_pass.ru0);
                if (over || !(den > 0.0f)) break;
                pass.look = 0;
            }
            --pass.left;
            alpha = __fdividef(g1, den);
            gam = g1;
            p = u + beta * p;
            sv = w + beta * sv;
            d += alpha * p;
            r -= alpha * sv;
            u = r * inv;
            send_u(u);
        }
        if (tid == 0) {
            s_pass.it += s_pass.last - pass.left;
            if (outer == 0) s_pass.first = s_pass.it;
        }
        // the next residual reads every CTA's rows
        if (writes) x[k] += (double)d * cg_unit(s_pass.rprev);
        __threadfence();
        cl.sync();
    }
    __threadfence();
    cl.sync();   // no CTA leaves while another may still write to it
    if (rank != 0) return;
    int n = 0;
    if (!converged) {
        if (pcg_idle(ns, tid)) return;
        converged = pcg_takes_over<NTH>(ns, q, x, rhs, tol, maxit, s_red, &n, &rmax, err);
    }
    if (tid == 0) {
        *q.iters = s_pass.it + n;
        *q.resid = rmax;
        if (!converged) record_error(err, ERR_NOCONV);
    }
}

template <int NTH>
cudaLaunchConfig_t cluster_config(const ClusterShape &sh, cudaLaunchAttribute *at, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)sh.ctas);
    cfg.blockDim = dim3(NTH);
    cfg.dynamicSmemBytes = cluster_smem<NTH>(sh);
    cfg.stream = s;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = (unsigned)sh.ctas;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

// Whether the device can hold one cluster of `ctas` CTAs of the kernel at its
// largest (16 need as many SMs with room in one GPC, which a partition of the
// device may lack).
template <int NTH> bool cluster_fits(int ctas) {
    const void *fn = (const void *)cluster_cg_kernel<NTH>;
    const ClusterShape sh{ctas, NTH < CL_ROWS ? NTH : CL_ROWS, 0};
    if (func_smem_attr(fn, cluster_smem<NTH>(sh)) != cudaSuccess) return false;
    if (ctas > CL_CTAS &&
        cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    cudaLaunchAttribute at{};
    const cudaLaunchConfig_t cfg = cluster_config<NTH>(sh, &at, nullptr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) == cudaSuccess) return n > 0;
    cudaGetLastError();   // not a launch error of the caller's
    return false;
}

// CTAs of the widest cluster that both kernels can run as (16, 8 or 0), asked
// of a device once.
int widest_cluster() {
    static std::atomic<int> of_device[64];   // 0: not yet asked, else CTAs + 1
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    int w = dev < 64 ? of_device[dev].load() : 0;
    if (w == 0) {
        auto both = [](int ctas) { return cluster_fits<512>(ctas) && cluster_fits<1024>(ctas); };
        w = 1 + (both(CL_CTAS_WIDE) ? CL_CTAS_WIDE : both(CL_CTAS) ? CL_CTAS : 0);
        if (dev < 64) of_device[dev].store(w);
    }
    return w - 1;
}

template <int NTH>
cudaError_t launch_cluster_cg(int ns, const ClusterShape &sh, const QuadBuffers &qb, double *x,
                              const double *rhs, double tol, int maxit, int warm, int *err,
                              cudaStream_t s) {
    const cudaError_t e = func_smem_attr((const void *)cluster_cg_kernel<NTH>, cluster_smem<NTH>(sh));
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at{};
    const cudaLaunchConfig_t cfg = cluster_config<NTH>(sh, &at, s);
    return cudaLaunchKernelEx(&cfg, cluster_cg_kernel<NTH>, ns, sh, qb, x, rhs, tol, maxit, warm, err);
}

// 161 to BCG_MAX markers: the same method on one CTA, one thread per row in
// bin order (neighbouring lanes gather neighbouring u-values: few bank
// conflicts), the row's first FP32 entries in its registers.  An iteration is
// one product, one block reduction (two sums folded into one butterfly, ten
// shuffles) and two block barriers of ~200 cycles each: 1.2 us at 388
// markers, where a cluster of eight CTAs took 2.5 us, its two cluster
// barriers with their remote stores costing more than the wider product
// saves.  388-marker moving sphere: 1116 us (FP64 PCG) -> 167 us per step;
// the gathers' bank conflicts bound it (one copy of u: 221 us).
constexpr int BCG_MAX = 512;
constexpr int BCG_SM = 24;              // entries of a thread in shared memory
constexpr int BCG_REP = 8;              // copies of u: lane l gathers from copy l % 8, so only four
                                        // lanes of a warp can meet in a bank
constexpr int BCG_OUTER_MAX = 24;
constexpr float BCG_INNER = 1e-5f;
constexpr int BCG_REG = 32;             // entries of a thread in registers

constexpr size_t BCG_SMEM = sizeof(double) * BCG_MAX +
                            (sizeof(float) + sizeof(unsigned short)) * (size_t)BCG_SM * BCG_MAX +
                            sizeof(float) * BCG_REP * BCG_MAX + sizeof(unsigned short) * BCG_MAX;

__global__ void __launch_bounds__(BCG_MAX, 1)
block_cg_kernel(int ns, const QuadBuffers q, double *x, const double *__restrict__ rhs, double tol,
                int maxit, int warm, int *err) {
    constexpr int NTH = BCG_MAX, REG = BCG_REG;
    extern __shared__ __align__(16) double smem_b[];
    double *sx = smem_b;                                          // [NTH] solution, marker order
    float *sval = reinterpret_cast<float *>(sx + NTH);            // [BCG_SM][NTH]
    float *su = sval + BCG_SM * NTH;                              // [NTH][BCG_REP] u, row order
    unsigned short *scol = reinterpret_cast<unsigned short *>(su + BCG_REP * NTH);   // [BCG_SM][NTH]
    unsigned short *srow = scol + BCG_SM * NTH;                   // [NTH] row of a marker
    __shared__ float s_part[64];
    __shared__ double s_red[32];
    __shared__ float s_ru0;   // r.u at the start of a pass
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool own = tid < ns, on = 32 * warp < ns;               // a row; a warp with rows
    const int k = own ? (q.order ? q.order[tid] : tid) : 0;
    const int cnt = own ? q.cnt[k] : 0;
    if (tid < 64) s_part[tid] = 0.0f;
    bool guess = warm != 0;   // x holds the first guess until the end
    if (own) {
        srow[k] = (unsigned short)tid;
        sx[k] = warm ? x[k] : 0.0;
    }
    __syncthreads();
    // the row's entries: FP32 value and row of the column's marker
    auto entry = [&](int i, float &v, int &l) {
        v = 0.0f;
        l = own ? tid : 0;
        if (i < cnt) {
            const int c = q.col[(long long)i * q.cap + k];
            if (in_bounds(c, ns, err)) {
                v = (float)q.val[(long long)i * q.cap + k];
                l = srow[c];
            }
        }
    };
    float rv[REG];
    unsigned rc[REG / 2];
#pragma unroll
    for (int j = 0; j < REG; j += 2) {
        int l0, l1;
        entry(j, rv[j], l0);
        entry(j + 1, rv[j + 1], l1);
        rc[j / 2] = (unsigned)l0 | ((unsigned)l1 << 16);
    }
    for (int j = REG; j < min(cnt, REG + BCG_SM); ++j) {
        float v;
        int l;
        entry(j, v, l);
        sval[(j - REG) * NTH + tid] = v;
        scol[(j - REG) * NTH + tid] = (unsigned short)l;
    }
    const float inv = own ? (float)(1.0 / q.diag[k]) : 0.0f;
    const float *const suc = su + (lane & (BCG_REP - 1));   // this lane's copy
    auto put_u = [&](float u) {
        if (!own) return;
        float4 *d4 = reinterpret_cast<float4 *>(su + BCG_REP * tid);
        d4[0] = d4[1] = make_float4(u, u, u, u);
    };
    static_assert(BCG_REP == 8, "put_u writes eight copies");
    __syncthreads();

    int it = 0, first_its = 0;
    bool converged = false, over = false;   // over: the last pass was given up
    double rmax = 0.0, rprev = 0.0;
    for (int outer = 0;; ++outer) {
        // r = rhs - A~ x in FP64 from the ELL rows
        double a = 0.0;
#pragma unroll 4
        for (int i = 0; i < cnt; ++i) {
            const int l = __ldg(q.col + (long long)i * q.cap + k);
            if (in_bounds(l, ns, err)) a += __ldg(q.val + (long long)i * q.cap + k) * sx[l];
        }
        const double r64 = own ? (rhs ? rhs[k] : 1.0) - a : 0.0;
        rmax = block_max<NTH>(fabs(r64), s_red);
        if (rmax <= tol) { converged = true; break; }
        if (outer == 0 && !(rmax < 1.0)) guess = false;   // worse than none
        const bool failed = outer > 0 && (over || !(rmax < 0.25 * rprev));
        if (failed || !cg_in_range(rmax) || outer == BCG_OUTER_MAX || it >= maxit) {
            // (each row's value is its owner's alone from here on)
            if (own && (it >= maxit || outer - (failed ? 1 : 0) < 2)) sx[k] = guess ? x[k] : 0.0;
            else if (own && failed) sx[k] = q.r[k];
            break;
        }
        rprev = rmax;
        if (own) q.r[k] = sx[k];   // (the FP64 solver's workspace)
        CgPass pass = cg_pass(outer, first_its, ns, maxit - it);
        it += pass.left;
        float r = (float)(r64 * cg_per_unit(rmax)), u = r * inv, p = 0.0f, sv = 0.0f, d = 0.0f,
              gam = 1.0f, alpha = 1.0f, stop = 0.0f;
        put_u(u);
        __syncthreads();
        for (bool first = true;; first = false) {
            float w = 0.0f;
            if (on) {
                float w1 = 0.0f;
#pragma unroll
                for (int j = 0; j < REG; j += 2) {
                    w += rv[j] * suc[BCG_REP * (rc[j / 2] & 0xffffu)];
                    w1 += rv[j + 1] * suc[BCG_REP * (rc[j / 2] >> 16)];
                }
                for (int j = REG; j < cnt; ++j) {
                    if (j < REG + BCG_SM) {
                        w += sval[(j - REG) * NTH + tid] * suc[BCG_REP * scol[(j - REG) * NTH + tid]];
                    } else {
                        float v;
                        int l;
                        entry(j, v, l);
                        w += v * suc[BCG_REP * l];
                    }
                }
                w += w1;
                const float t = warp_sum2(r * u, w * u, lane);
                if ((lane & 15) == 0) s_part[2 * (lane & 16) + warp] = t;
            }
            __syncthreads();
            const float2 tot = part_sum2(s_part, lane);
            const float g1 = tot.x;
            if (first) {
                stop = cg_stop(g1, BCG_INNER, ns, tol * cg_per_unit(rprev));
                if (tid == 0) s_ru0 = g1;
            }
            if (g1 <= stop) break;
            const float beta = first ? 0.0f : __fdividef(g1, gam);
            const float den = first ? tot.y : tot.y - beta * __fdividef(g1, alpha);
            if (!(den > 0.0f) || pass.left == pass.look) {   // (a NaN sum ends here too)
                over = pass.left == 0 || (pass.left == pass.look && g1 > s_ru0);
                if (over || !(den > 0.0f)) break;
                pass.look = 0;
            }
            --pass.left;
            alpha = __fdividef(g1, den);
            gam = g1;
            p = u + beta * p;
            sv = w + beta * sv;
            d += alpha * p;
            r -= alpha * sv;
            u = r * inv;
            put_u(u);
            __syncthreads();
        }
        it -= pass.left;
        if (outer == 0) first_its = it;
        if (own) sx[k] += (double)d * cg_unit(rprev);
        __syncthreads();
    }
    if (own) x[k] = sx[k];
    __syncthreads();
    if (!converged) {
        if (pcg_idle(ns, tid)) return;
        int n = 0;
        converged = pcg_takes_over<NTH>(ns, q, x, rhs, tol, maxit, s_red, &n, &rmax, err);
        it += n;
    }
    if (tid == 0) {
        *q.iters = it;
        *q.resid = rmax;
        if (!converged) record_error(err, ERR_NOCONV);
    }
}

cudaError_t launch_block_cg(int ns, const QuadBuffers &qb, double *x, const double *rhs, double tol,
                            int maxit, int warm, int *err, cudaStream_t s) {
    cudaError_t e = func_smem_attr((const void *)block_cg_kernel, BCG_SMEM);
    if (e != cudaSuccess) return e;
    block_cg_kernel<<<1, BCG_MAX, BCG_SMEM, s>>>(ns, qb, x, rhs, tol, maxit, warm, err);
    return cudaGetLastError();
}

// Small systems (up to CHOL_MAX markers) on one CTA.  In 2D, above SCG_MIN
// markers and with rows of at most SCG_ROW entries, corrections come from FP32
// conjugate gradients first (small_cg); a system they do not contract by ten per
// pass, and every other one, is factored.  A~ is then copied dense, in FP32, into
// shared memory from the ELL rows.  FP64 runs at a small fraction of the FP32 rate on this GPU, so
// the O(ns^3) work is done in FP32: a blocked right-looking Cholesky
// A~ = L L^T over 32-column panels (one warp factors the panel's diagonal
// block without block barriers, one thread per row solves the rows below
// it, 4 x 4 register tiles update the trailing matrix: three barriers per
// panel), then the inverses of the 32 x 32 diagonal blocks of L, one warp
// each.  The FP64 solution comes from iterative refinement,
// x += L^-T L^-1 (rhs - A~ x), with the residual taken in FP64 from the
// ELL rows (only their nonzeros) and the two triangular solves blocked by
// the same panels (each diagonal block applied through its inverse); it
// contracts by about cond(A~) times the FP32 rounding per pass and stops
// at the FP64 residual's rounding floor: when the residual is within
// CHOL_FLOOR of the right-hand side's size, stops falling, or reaches zero
// (the first test saves the pass that would only confirm the floor).  Fixed
// order throughout, so the result is bitwise reproducible.
// If the refinement stops above tol or a pivot is not positive (a system
// too ill-conditioned for the FP32 factor), the same CTA runs the FP64
// Jacobi-PCG instead; ERR_NOCONV only if that fails too.
constexpr int CHOL_T = 512;
constexpr int CHOL_W = CHOL_T / 32;
#ifndef IBM_CHOL_MAX
#define IBM_CHOL_MAX 160
#endif
constexpr int CHOL_MAX = IBM_CHOL_MAX;
constexpr int CHOL_PB = 32;                                  // panel width
static_assert((CHOL_MAX + CHOL_PB - 1) / CHOL_PB <= CHOL_W, "one warp per diagonal block");
constexpr int CHOL_REFINE_MAX = 40;
constexpr double CHOL_FLOOR = 4.0 * 2.220446049250313e-16;   // 4 ulp of 1

// the first CHOL_EC entries of every row of A~ are kept in shared memory for
// the residuals of the refinement (rows hold ~10-60 entries; the rest are
// read from the ELL arrays in global memory)
constexpr int CHOL_EC = 32;

// x [ns] and the cached row values [CHOL_EC][ns] in FP64, then the FP32
// factors [ns][ns | 1], 1/L_jj, r and t, then the cached columns [CHOL_EC][ns]
// and the row lengths [ns]
size_t chol_smem(int ns) {
    return sizeof(double) * (size_t)ns * (1 + CHOL_EC) +
           sizeof(float) * ((size_t)ns * (ns | 1) + 3 * (size_t)ns) +
           sizeof(int) * (size_t)ns * (CHOL_EC + 1);
}

// Cholesky of the diagonal block [c0, c0 + w) in place, by one warp: lane r
// holds row c0 + r of the block in registers; 1 / L_kk into dinv, *bad set
// on a pivot that is not positive.  The row shifts left by one column per
// step (a[l] holds column k + l at step k), so the pivot column is always
// a[0] and every step runs the same compact loop body.  Step k hands the
// pivot column L_{k+l,k} to the lanes through col (32 floats, 16-byte
// aligned, this warp's alone): each lane stores its entry at l = lane - k
// and reads the column back as eight 16-byte broadcast loads, where 31
// shuffles (one per entry) set the step's latency.  Same operations in the
// same order as a shuffle form.
__device__ __forceinline__ void chol_diag_block(float *__restrict__ F, int ld, int c0, int w,
                                                float *__restrict__ dinv, int lane, int *bad,
                                                float *__restrict__ col) {
    float a[CHOL_PB];
#pragma unroll
    for (int l = 0; l < CHOL_PB; ++l)
        a[l] = (lane < w && l <= lane) ? F[(size_t)(c0 + lane) * ld + c0 + l] : 0.0f;
#pragma unroll 1
    for (int k = 0; k < w; ++k) {
        const float d = __shfl_sync(0xffffffffu, a[0], k);
        // pivots from the hardware reciprocal square root (a few ulp; the
        // factor only has to make the FP64 refinement contract): 18.7 k ->
        // 13.5 k cycles per 32-column block against IEEE sqrt and division
        const bool good = d > 0.0f;
        const float inv = good ? rsqrtf(d) : 1.0f;
        const float sd = good ? d * inv : 1.0f;
        float lk = a[0];   // zero on the lanes above the diagonal
        if (lane == k) {
            lk = sd;
            dinv[c0 + k] = inv;
            if (!good) *bad = 1;
        } else if (lane > k) {
            lk = a[0] * inv;
        }
        if (lane >= k && lane < w) F[(size_t)(c0 + lane) * ld + c0 + k] = lk;
        // col[l] = L_{k+l,k}; the entries past 31 - k are stale and unused
        if (lane >= k) col[lane - k] = lk;
        __syncwarp();
        float c[CHOL_PB];
#pragma unroll
        for (int v = 0; v < CHOL_PB / 4; ++v) {
            const float4 q = reinterpret_cast<const float4 *>(col)[v];
            c[4 * v] = q.x;
            c[4 * v + 1] = q.y;
            c[4 * v + 2] = q.z;
            c[4 * v + 3] = q.w;
        }
        __syncwarp();   // every lane has read col before the next step writes it
#pragma unroll
        for (int l = 1; l < CHOL_PB; ++l)
            if (lane >= k + l) a[l] -= lk * c[l];
#pragma unroll
        for (int l = 0; l < CHOL_PB - 1; ++l) a[l] = a[l + 1];
        a[CHOL_PB - 1] = 0.0f;
    }
}

// rows i >= c0 + w of panel [c0, c0 + w): L_i = A_i L_D^-T, one thread per row
__device__ __forceinline__ void chol_panel_rows(float *__restrict__ F, int ld, int c0, int w,
                                                int ns, const float *__restrict__ dinv, int tid) {
    for (int i = c0 + w + tid; i < ns; i += CHOL_T) {
        float *row = F + (size_t)i * ld + c0;
        float v[CHOL_PB];
#pragma unroll
        for (int k = 0; k < CHOL_PB; ++k) v[k] = k < w ? row[k] : 0.0f;
#pragma unroll
        for (int k = 0; k < CHOL_PB; ++k) {
            if (k < w) {
                const float *lk = F + (size_t)(c0 + k) * ld + c0;
                float acc = v[k];
#pragma unroll
                for (int l = 0; l < k; ++l) acc -= v[l] * lk[l];
                v[k] = acc * dinv[c0 + k];
            }
        }
#pragma unroll
        for (int k = 0; k < CHOL_PB; ++k)
            if (k < w) row[k] = v[k];
    }
}

// trailing update A_ij -= sum_k L_ik L_jk over the panel's columns, for
// c1 <= j <= i < ns, in 2 x 2 tiles (tile pairs tj <= ti, one per thread;
// 4 x 4 tiles kept fewer warps busy: 2.6 us more per moving-cylinder step)
__device__ __forceinline__ void chol_trailing(float *__restrict__ F, int ld, int c0, int w, int ns,
                                              int tid) {
    const int c1 = c0 + w, m = ns - c1, nt = (m + 1) / 2, npairs = nt * (nt + 1) / 2;
    for (int p = tid; p < npairs; p += CHOL_T) {
        int ti = (int)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
        while ((ti + 1) * (ti + 2) / 2 <= p) ++ti;
        while (ti * (ti + 1) / 2 > p) --ti;
        const int tj = p - ti * (ti + 1) / 2;
        const int i0 = c1 + 2 * ti, j0 = c1 + 2 * tj;
        float acc[2][2];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int q = 0; q < 2; ++q) acc[r][q] = 0.0f;
        for (int k = 0; k < w; ++k) {
            float a[2], b[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                a[r] = i0 + r < ns ? F[(size_t)(i0 + r) * ld + c0 + k] : 0.0f;
                b[r] = j0 + r < ns ? F[(size_t)(j0 + r) * ld + c0 + k] : 0.0f;
            }
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int q = 0; q < 2; ++q) acc[r][q] += a[r] * b[q];
        }
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int i = i0 + r, j = j0 + q;
                if (i < ns && j <= i) F[(size_t)i * ld + j] -= acc[r][q];
            }
    }
}

// inverse of the diagonal block [b0, b0 + wb) of L by one warp (lane =
// column c): X_rc for r > c goes to F[c][r], above the diagonal; X_cc is
// dinv[c] already
__device__ __forceinline__ void chol_diag_inverse(float *__restrict__ F, int ld, int b0, int wb,
                                                  const float *__restrict__ dinv, int lane) {
    float xc[CHOL_PB];
#pragma unroll
    for (int r = 0; r < CHOL_PB; ++r) {
        float acc = r == lane ? 1.0f : 0.0f;
        if (r < wb) {
            const float *lr = F + (size_t)(b0 + r) * ld + b0;
#pragma unroll
            for (int l = 0; l < r; ++l) acc -= lr[l] * xc[l];
            acc *= dinv[b0 + r];
        }
        xc[r] = acc;
    }
    if (lane < wb) {
        float *out = F + (size_t)(b0 + lane) * ld + b0;
#pragma unroll
        for (int r = 0; r < CHOL_PB; ++r)
            if (r > lane && r < wb) out[r] = xc[r];
    }
}

// FP32 conjugate gradients for the correction A~ d = r32 of a small system
// (the threads of the first ceil(ns / 32) warps, one row each; the other
// warps wait): Jacobi preconditioner, single-reduction form, until the
// residual has fallen by SCG_INNER.  The surface systems of one marker per cell are
// well conditioned (about four iterations per decimal digit), and an
// iteration costs ~600 cycles against ~118 k for the dense factor of 97
// markers: 61.5 -> 40.8 us per step of the moving cylinder.  The row's first SCG_REG
// FP32 entries sit in registers.  Curves have five to nine entries per row;
// surfaces have over twenty and a condition number four times theirs, where
// the dense factor is the faster (62 iterations per pass at 120 markers), so
// systems with a row of more than SCG_ROW entries are factored at once.
// false when it did not get there in SCG_ITS iterations (the caller then
// factors A~).
constexpr int SCG_ROW = 12;   // longest row for which it is tried: see above
constexpr int SCG_MIN = 64;   // one or two panels factor sooner (61 markers, cold: 171 us for a
                              // whole set_markers against 176)
constexpr int SCG_REG = 8, SCG_ITS = 48, SCG_W = (CHOL_MAX + 31) / 32;
constexpr float SCG_INNER = 1e-5f;
__device__ __forceinline__ bool small_cg(int ns, const QuadBuffers &q, int k, int cnt,
                                         const float (&rv)[SCG_REG], const int (&rc)[SCG_REG],
                                         float inv, const float *__restrict__ ev32,
                                         const int *__restrict__ ec, float r,
                                         float *__restrict__ su, float *__restrict__ part,
                                         float &d, int &it) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = (ns + 31) / 32, nth = 32 * nw;
    auto bar = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(nth) : "memory"); };
    float stop = 0.0f;
    float u = r * inv, p = 0.0f, sv = 0.0f, gam = 1.0f, alpha = 1.0f;
    d = 0.0f;
    if (k < ns) su[k] = u;
    bar();
    for (int n = 0;; ++n) {
        float w = 0.0f;
#pragma unroll
        for (int i = 0; i < SCG_REG; ++i) w += rv[i] * su[rc[i]];
        for (int i = SCG_REG; i < cnt; ++i) {
            if (i < CHOL_EC) {
                w += ev32[i * ns + k] * su[ec[i * ns + k]];
            } else {
                const int l = q.col[(long long)i * q.cap + k];
                w += (float)q.val[(long long)i * q.cap + k] * su[l];
            }
        }
        const float t = warp_sum2(r * u, w * u, lane);
        if ((lane & 15) == 0) part[2 * warp + (lane >> 4)] = t;
        bar();
        float g1 = 0.0f, del = 0.0f;
#pragma unroll
        for (int i = 0; i < SCG_W; ++i) {   // the slots past nw hold zeros
            const float2 v = reinterpret_cast<const float2 *>(part)[i];
            g1 += v.x;
            del += v.y;
        }
        if (n == 0) stop = g1 * SCG_INNER * SCG_INNER;
        if (g1 <= stop) return true;
        const float beta = n == 0 ? 0.0f : __fdividef(g1, gam);
        const float den = n == 0 ? del : del - beta * __fdividef(g1, alpha);
        if (!(den > 0.0f) || n == SCG_ITS) return false;   // (a NaN sum too)
        alpha = __fdividef(g1, den);
        gam = g1;
        p = u + beta * p;
        sv = w + beta * sv;
        d += alpha * p;
        r -= alpha * sv;
        u = r * inv;
        if (k < ns) su[k] = u;
        ++it;
        bar();
    }
}

// one CTA per launch: the register file is the CTA's alone, so the
// registers a thread may take are bounded for one resident block (the
// diagonal-block factor keeps a 32-float row per lane)
template <bool CG>
__global__ void __launch_bounds__(CHOL_T, 1)
chol_kernel(int ns, const QuadBuffers q, double *x, const double *__restrict__ rhs, double tol,
            int maxit, int warm, int *err) {
    // rows have an odd stride, so a warp walking a column (consecutive rows)
    // or threads walking their own rows hit distinct banks
    const int ld = ns | 1;
    extern __shared__ __align__(16) double sD[];
    double *sx = sD;                                 // [ns] solution
    double *ev = sx + ns;                            // [CHOL_EC][ns] cached row values
    float *F = reinterpret_cast<float *>(ev + (size_t)CHOL_EC * ns);
                                                     // [ns][ld]: L on and below the diagonal,
                                                     // the inverses X_II of its 32 x 32
                                                     // diagonal blocks transposed above it
    float *dinv = F + (size_t)ns * ld;               // [ns] 1 / L_jj, the diagonal of X_II
    float *r32 = dinv + ns;                          // [ns] residual in FP32
    float *st = r32 + ns;                            // [ns] the triangular solves' vector
    int *ec = reinterpret_cast<int *>(st + ns);      // [CHOL_EC][ns] cached row columns
    int *ecnt = ec + (size_t)CHOL_EC * ns;           // [ns] row lengths
    __shared__ double s_red[CHOL_T / 32];
    __shared__ int s_bad;
    __shared__ __align__(16) float s_col[CHOL_PB];
    __shared__ __align__(8) float s_part[2 * SCG_W];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_bad = 0;
    if (tid < 2 * SCG_W) s_part[tid] = 0.0f;
    // the rows' first CHOL_EC entries and their lengths, kept for the
    // residuals; without the conjugate gradients (whose FP32 values take F's
    // place) the lower triangle of A~ too (the upper stays zero)
    if (!CG) {
        for (int i = tid; i < ns * ld; i += CHOL_T) F[i] = 0.0f;
        __syncthreads();
    }
    for (int k = tid; k < ns; k += CHOL_T) {
        const int c = q.cnt[k];
        ecnt[k] = c;
        for (int i = 0; i < (CG ? min(c, CHOL_EC) : c); ++i) {
            int l = q.col[(long long)i * q.cap + k];
            double v = q.val[(long long)i * q.cap + k];
            if (!in_bounds(l, ns, err)) { l = k; v = 0.0; }
            if (CG || i < CHOL_EC) {
                ec[(size_t)i * ns + k] = l;
                ev[(size_t)i * ns + k] = v;
            }
            if (!CG && l <= k && v != 0.0) F[(size_t)k * ld + l] = (float)v;
        }
        sx[k] = warm ? x[k] : 0.0;
    }
    // the right-hand side's size, the scale of the residual's floor
    double rscale = 1.0;
    if (rhs) {
        double lr = 0.0;
        for (int k = tid; k < ns; k += CHOL_T) lr = dmax_nonneg(lr, fabs(rhs[k]));
        rscale = block_max<CHOL_T>(lr, s_red);   // synchronizes
    }
    __syncthreads();
    // r = rhs - A~ x in FP64 from the ELL rows (one thread per row) into r32 in
    // units of cg_unit(rscale), its largest entry returned (synchronizes)
    auto residual = [&]() {
        double lm = 0.0;
        for (int k = tid; k < ns; k += CHOL_T) {
            const int c = ecnt[k];
            const int cc = min(c, CHOL_EC);
            double sum = 0.0;
            // the cached entries in batches of four (loads first, then the
            // terms in row order), the rest from the ELL arrays
            for (int i0 = 0; i0 < cc; i0 += 4) {
                int l[4];
                double v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool in = i0 + u < cc;
                    l[u] = in ? ec[(size_t)(i0 + u) * ns + k] : 0;
                    v[u] = in ? ev[(size_t)(i0 + u) * ns + k] : 0.0;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (i0 + u < cc) sum += v[u] * sx[l[u]];
            }
            for (int i = CHOL_EC; i < c; ++i) {
                const int l = q.col[(long long)i * q.cap + k];
                if (in_bounds(l, ns, err)) sum += q.val[(long long)i * q.cap + k] * sx[l];
            }
            const double r = (rhs ? rhs[k] : 1.0) - sum;
            r32[k] = (float)(r * cg_per_unit(rscale));
            lm = dmax_nonneg(lm, fabs(r));
        }
        return block_max<CHOL_T>(lm, s_red);
    };
    double rmax = 0.0, rprev = 0.0;
    int it = 0;
    bool done = false;   // the residual is at its floor
    if (CG && !__syncthreads_or(tid < ns && ecnt[tid] > SCG_ROW)) {
        // corrections by FP32 conjugate gradients first
        float rv[SCG_REG], inv = 0.0f;
        int rc[SCG_REG];
        float *ev32 = F;
#pragma unroll
        for (int i = 0; i < SCG_REG; ++i) { rv[i] = 0.0f; rc[i] = 0; }
        int cnt = 0;
        if (tid < ns) {
            cnt = ecnt[tid];
            inv = (float)(1.0 / q.diag[tid]);
            for (int i = 0; i < min(cnt, CHOL_EC); ++i) ev32[(size_t)i * ns + tid] = (float)ev[(size_t)i * ns + tid];
#pragma unroll
            for (int i = 0; i < SCG_REG; ++i)
                if (i < cnt) {
                    rv[i] = ev32[(size_t)i * ns + tid];
                    rc[i] = ec[(size_t)i * ns + tid];
                }
        }
        for (int outer = 0;; ++outer) {
            rmax = residual();
            if (!(rmax > 0.0) || rmax <= CHOL_FLOOR * rscale ||
                (outer > 0 && rmax <= 64.0 * CHOL_FLOOR * rscale && !(rmax < 0.5 * rprev))) {
                done = true;
                break;
            }
            // no contraction by ten, or nothing FP32 can hold: factor A~
            if (!(rmax < 1e30 * rscale) || (outer > 0 && !(rmax < 0.1 * rprev)) ||
                outer == CHOL_REFINE_MAX)
                break;
            rprev = rmax;
            const double m = rmax * cg_per_unit(rscale);   // r32's largest entry
            float d = 0.0f;
            bool got = true;
            if (warp < (ns + 31) / 32) {
                got = small_cg(ns, q, tid, cnt, rv, rc, inv, ev32, ec,
                               tid < ns ? r32[tid] * (float)cg_per_unit(m) : 0.0f, st,
                               s_part, d, it);
                if (got && tid < ns) sx[tid] += (double)d * (cg_unit(m) * cg_unit(rscale));
            }
            if (__syncthreads_or(!got)) break;
        }
    }
    if (!done) {
    if (CG) {
        // the dense factor: the lower triangle of A~ (the upper stays zero),
        // and the refinement from where the call started (what FP32 did not
        // contract may be of any size along the near-null vectors)
        for (int k = tid; k < ns; k += CHOL_T) sx[k] = warm ? x[k] : 0.0;
        for (int i = tid; i < ns * ld; i += CHOL_T) F[i] = 0.0f;
        __syncthreads();
        for (int k = tid; k < ns; k += CHOL_T) {
            const int c = ecnt[k], cc = min(c, CHOL_EC);
            for (int i = 0; i < cc; ++i) {
                const int l = ec[(size_t)i * ns + k];
                if (l <= k) F[(size_t)k * ld + l] = (float)ev[(size_t)i * ns + k];
            }
            for (int i = CHOL_EC; i < c; ++i) {
                const int l = q.col[(long long)i * q.cap + k];
                if (in_bounds(l, ns, err) && l <= k)
                    F[(size_t)k * ld + l] = (float)q.val[(long long)i * q.cap + k];
            }
        }
        __syncthreads();
    }
    // blocked Cholesky over 32-column panels, then the diagonal blocks' inverses
    for (int c0 = 0; c0 < ns; c0 += CHOL_PB) {
        const int w = min(CHOL_PB, ns - c0);
        if (warp == 0) chol_diag_block(F, ld, c0, w, dinv, lane, &s_bad, s_col);
        __syncthreads();
        if (c0 + w < ns) {
            chol_panel_rows(F, ld, c0, w, ns, dinv, tid);
            __syncthreads();
            chol_trailing(F, ld, c0, w, ns, tid);
            __syncthreads();
        }
    }
    if (warp * CHOL_PB < ns)
        chol_diag_inverse(F, ld, warp * CHOL_PB, min(CHOL_PB, ns - warp * CHOL_PB), dinv, lane);
    __syncthreads();
    // refinement: r = rhs - A~ x in FP64, x += L^-T L^-1 r in FP32
    for (it = 0;; ++it) {
        rmax = residual();
        if (!(rmax > 0.0) || rmax <= CHOL_FLOOR * rscale || (it > 0 && !(rmax < 0.5 * rprev)) ||
            it == CHOL_REFINE_MAX)
            break;
        rprev = rmax;
        // t = L^-1 r: per panel, t_I = X_II t_I (warp 0), then the rows
        // below take -L_iI t_I
        for (int i = tid; i < ns; i += CHOL_T) st[i] = r32[i];
        __syncthreads();
        for (int b0 = 0; b0 < ns; b0 += CHOL_PB) {
            const int b1 = min(b0 + CHOL_PB, ns);
            // (loops of the panel width with predicated terms: the loads of
            // every term issue together; same terms in the same order as
            // loops that stop at the ragged end)
            if (warp == 0) {
                const int i = b0 + lane;
                float y = 0.0f;
                if (i < b1) {
                    y = dinv[i] * st[i];
#pragma unroll
                    for (int j = 0; j < CHOL_PB - 1; ++j) {
                        const int cq = b0 + j;
                        if (cq < i) y += F[(size_t)cq * ld + i] * st[cq];
                    }
                }
                __syncwarp();
                if (i < b1) st[i] = y;
            }
            __syncthreads();
            for (int i = b1 + tid; i < ns; i += CHOL_T) {
                const float *row = F + (size_t)i * ld;
                float a0 = st[i], a1 = 0.0f;
#pragma unroll
                for (int j = 0; j < CHOL_PB / 2; ++j) {
                    const int cq = b0 + 2 * j;
                    if (cq + 2 <= b1) {
                        a0 -= row[cq] * st[cq];
                        a1 -= row[cq + 1] * st[cq + 1];
                    } else if (cq < b1) {
                        a0 -= row[cq] * st[cq];
                    }
                }
                st[i] = a0 + a1;
            }
            __syncthreads();
        }
        // z = L^-T t: per panel from the last, z_I = X_II^T t_I (warp 0),
        // then the rows above take -L_Ic^T z_I
        for (int b0 = ((ns - 1) / CHOL_PB) * CHOL_PB; b0 >= 0; b0 -= CHOL_PB) {
            const int b1 = min(b0 + CHOL_PB, ns);
            if (warp == 0) {
                const int c = b0 + lane;
                float z = 0.0f;
                if (c < b1) {
                    const float *row = F + (size_t)c * ld;
                    z = dinv[c] * st[c];
#pragma unroll
                    for (int j = 1; j < CHOL_PB; ++j) {
                        const int i = b0 + j;
                        if (i > c && i < b1) z += row[i] * st[i];
                    }
                }
                __syncwarp();
                if (c < b1) st[c] = z;
            }
            __syncthreads();
            for (int c = tid; c < b0; c += CHOL_T) {
                float a0 = st[c], a1 = 0.0f;
#pragma unroll
                for (int j = 0; j < CHOL_PB / 2; ++j) {
                    const int i = b0 + 2 * j;
                    if (i + 2 <= b1) {
                        a0 -= F[(size_t)i * ld + c] * st[i];
                        a1 -= F[(size_t)(i + 1) * ld + c] * st[i + 1];
                    } else if (i < b1) {
                        a0 -= F[(size_t)i * ld + c] * st[i];
                    }
                }
                st[c] = a0 + a1;
            }
            __syncthreads();
        }
        for (int c = tid; c < ns; c += CHOL_T) sx[c] += (double)st[c] * cg_unit(rscale);
        __syncthreads();
    }
    }   // !done
    for (int k = tid; k < ns; k += CHOL_T) x[k] = sx[k];
    bool ok = !s_bad && rmax <= tol;
    if (!ok) {
        // too ill-conditioned for the FP32 factor (e.g. two markers in one
        // cell, placed without dedup): the FP64 Jacobi-PCG takes over, from
        // the refined x when it is finite
        __shared__ double s_red32[32];
        const bool warm_x = !s_bad && rmax < 1.0;
        ok = pcg_solve<CHOL_T>(ns, q, x, rhs, tol, maxit, warm_x, s_red32, &it, &rmax, err);
    }
    if (tid == 0) {
        *q.iters = it;
        *q.resid = rmax;
        if (!ok) record_error(err, ERR_NOCONV);
    }
}

}  // namespace

int quad_row_width(int dim) { return dim == 3 ? 125 * 4 : 25 * 4; }

// A~ x = rhs (rhs == nullptr: all ones), warm-started if asked.  One CTA up
// to BCG_MAX markers, one cluster to CL_MAX (both sides of each line measured
// at the kernels), the FP64 PCG above and where no cluster can be placed
static cudaError_t launch_quadrature_solve_w(int dim, int ns, const QuadBuffers &qb, const double *rhs,
                                            double *x, double tol, int maxit, int warm, int *err,
                                            cudaStream_t s) {
    if (ns <= 0) return cudaSuccess;
    if (ns <= CHOL_MAX) {
        // conjugate gradients are worth a try where rows may be short (curves
        // in 2D) and there is more to factor than two panels; a try that is
        // sure to fail costs 103 markers in 3D 78 -> 84 us
        const auto kernel = dim == 2 && ns > SCG_MIN ? chol_kernel<true> : chol_kernel<false>;
        cudaError_t e = func_smem_attr((const void *)kernel, chol_smem(CHOL_MAX));
        if (e != cudaSuccess) return e;
        kernel<<<1, CHOL_T, chol_smem(ns), s>>>(ns, qb, x, rhs, tol, maxit, warm, err);
    } else if (ns <= BCG_MAX) {
        return launch_block_cg(ns, qb, x, rhs, tol, maxit, warm, err, s);
    } else {
        const ClusterShape sh = ns <= CL_MAX ? cluster_shape(ns, widest_cluster()) : ClusterShape{0, 0, 0};
        if (sh.ctas > 0)
            return sh.rows <= 512
                       ? launch_cluster_cg<512>(ns, sh, qb, x, rhs, tol, maxit, warm, err, s)
                       : launch_cluster_cg<1024>(ns, sh, qb, x, rhs, tol, maxit, warm, err, s);
        if (ns <= 2048)
            pcg_kernel<256><<<1, 256, 0, s>>>(ns, qb, x, rhs, tol, maxit, warm, err);
        else
            pcg_kernel<1024><<<1, 1024, 0, s>>>(ns, qb, x, rhs, tol, maxit, warm, err);
    }
    return cudaGetLastError();
}

cudaError_t launch_quadrature(const GridParams &g, const MarkerBuffers &m, const QuadBuffers &qb,
                              double tol, int maxit, int warm, cudaStream_t s, int have_weights) {
    if (m.ns <= 0) return cudaSuccess;
    const unsigned *keys = m.keys[m.sorted];
    const int *perm = m.perm[m.sorted];
    if (!have_weights) support_weights_kernel<<<(m.ns * 3 + 127) / 128, 128, 0, s>>>(m, g.dim);
    const int nb = (m.ns * 32 + 127) / 128;   // one warp per marker
    if (g.dim == 3) assemble_kernel<3><<<nb, 128, 0, s>>>(g, m, qb, keys, perm);
    else assemble_kernel<2><<<nb, 128, 0, s>>>(g, m, qb, keys, perm);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    QuadBuffers q = qb;
    q.order = perm;   // the solvers may take the rows in bin order
    return launch_quadrature_solve_w(g.dim, m.ns, q, nullptr, m.eps, tol, maxit, warm, m.err, s);
}

// A~ x = rhs with the matrix assembled by the last launch_quadrature (the
// adjoint of the weights); x starts from zero.
cudaError_t launch_quadrature_solve(int dim, int ns, const QuadBuffers &qb, const double *rhs, double *x,
                                    double tol, int maxit, int *err, cudaStream_t s) {
    return launch_quadrature_solve_w(dim, ns, qb, rhs, x, tol, maxit, 0, err, s);
}

}  // namespace ibmk
