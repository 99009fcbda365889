// drcp and drsqrt (paper_2301_09349_gb300/csrc/common.cuh) against 1/x and
// 1/sqrt(x) in extended precision: both ends of every 16th binade over the
// range they are stated for, random mantissas, and a dense run through the
// binades [1, 2) and [2, 4).  Prints the seeds' and the results' largest
// errors; fails above the stated bounds (2^-18 relative, 2 ulp).
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>

#include "common.cuh"

__global__ void evaluate(int n, const double *x, double *rcp, double *rsq, double *rcp_seed,
                         double *rsq_seed) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    rcp[i] = ibmk::drcp(x[i]);
    rsq[i] = ibmk::drsqrt(x[i]);
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(rcp_seed[i]) : "d"(x[i]));
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(rsq_seed[i]) : "d"(x[i]));
}

static double ulps(double got, long double want) {
    int e;
    frexpl(want, &e);
    return (double)(fabsl((long double)got - want) / ldexpl(1.0L, e - 53));
}

int main() {
    std::vector<double> x;
    uint64_t s = 88172645463325252ull;   // xorshift64
    auto rnd = [&]() {
        s ^= s << 13;
        s ^= s >> 7;
        s ^= s << 17;
        return s;
    };
    auto make = [&](int e, uint64_t mant) {   // 2^e (1 + mant 2^-52)
        const uint64_t b = ((uint64_t)(e + 1023) << 52) | (mant & ((1ull << 52) - 1));
        double d;
        memcpy(&d, &b, 8);
        x.push_back(d);
    };
    for (int e = -1021; e <= 1020; ++e) {
        if (e % 16 == 0)
            for (uint64_t k = 0; k < 64; ++k) {
                make(e, k);
                make(e, ~k);
            }
        for (int k = 0; k < 256; ++k) make(e, rnd());
    }
    const int dense = 1 << 20;
    for (int i = 0; i < dense; ++i) {
        make(0, ((uint64_t)i << 32) | (rnd() >> 32));
        make(1, ((uint64_t)i << 32) | (rnd() >> 32));
    }
    const int regular = (int)x.size();
    const double special[] = {0.0, -0.0, INFINITY, NAN, -1.0};
    for (double v : special) x.push_back(v);
    const int n = (int)x.size();
    double *d;
    if (cudaMalloc(&d, sizeof(double) * 5 * (size_t)n) != cudaSuccess) return 2;
    cudaMemcpy(d, x.data(), sizeof(double) * n, cudaMemcpyHostToDevice);
    evaluate<<<(n + 255) / 256, 256>>>(n, d, d + n, d + 2 * n, d + 3 * n, d + 4 * n);
    std::vector<double> out(4 * (size_t)n);
    if (cudaMemcpy(out.data(), d + n, sizeof(double) * 4 * n, cudaMemcpyDeviceToHost) != cudaSuccess)
        return 2;
    cudaFree(d);
    double u[2] = {0.0, 0.0}, seed[2] = {0.0, 0.0};
    for (int i = 0; i < regular; ++i) {
        const long double v = x[i], want[2] = {1.0L / v, 1.0L / sqrtl(v)};
        for (int f = 0; f < 2; ++f) {
            u[f] = fmax(u[f], ulps(out[(size_t)f * n + i], want[f]));
            seed[f] = fmax(seed[f], (double)fabsl(out[(size_t)(2 + f) * n + i] / want[f] - 1.0L));
        }
    }
    // 1 / -1, and no root of it; no value at 0, infinity and NaN
    bool special_ok = out[regular + 4] == -1.0 && std::isnan(out[n + regular + 4]);
    for (int f = 0; f < 2; ++f)
        for (int i = 0; i < 4; ++i) special_ok = special_ok && std::isnan(out[(size_t)f * n + regular + i]);
    std::printf("drcp %.3f ulp (seed 2^%.2f), drsqrt %.3f ulp (seed 2^%.2f), NaN at 0, inf and NaN: %d\n",
                u[0], std::log2(seed[0]), u[1], std::log2(seed[1]), (int)special_ok);
    const bool ok = u[0] <= 2.0 && u[1] <= 2.0 && seed[0] <= std::ldexp(1.0, -18) &&
                    seed[1] <= std::ldexp(1.0, -18) && special_ok;
    return ok ? 0 : 1;
}
