// How the rows of a quadrature system are dealt to a thread-block cluster
// (host-only C++, no CUDA dependency, so it is unit-tested on the CPU).
#pragma once

namespace ibmk {

constexpr int CL_CTAS = 8, CL_CTAS_WIDE = 16;   // portable, and an opt-in of the kernel
constexpr int CL_WIDE = 1536;            // above, the product of 8 CTAs outweighs 16's exchange
constexpr int CL_ROWS = 1024;            // rows of a CTA, one thread each
constexpr int CL_MAX = CL_CTAS_WIDE * CL_ROWS;   // (16-bit columns)

struct ClusterShape {
    int ctas;       // CTAs of the cluster; 0: no cluster takes the system
    int rows;       // rows per CTA, a multiple of 4
    int lpr_log;    // log2 of the threads per row
};

// widest: CTAs of the widest cluster that may be launched (16, 8, or 0 for
// none)
inline ClusterShape cluster_shape(int ns, int widest) {
    ClusterShape c;
    c.ctas = ns > CL_WIDE && widest >= CL_CTAS_WIDE ? CL_CTAS_WIDE : CL_CTAS;
    c.rows = ((ns + c.ctas - 1) / c.ctas + 3) / 4 * 4;   // chunks of u move as 16-byte words
    c.lpr_log = 0;
    if (widest < CL_CTAS || c.rows > CL_ROWS) return ClusterShape{0, 0, 0};
    while (c.lpr_log < 4 && (2 << c.lpr_log) * c.rows <= 512) ++c.lpr_log;
    return c;
}

}  // namespace ibmk
