// Host-only check of the rows' distribution over a cluster
// (paper_2301_09349_gb300/csrc/cluster_plan.h) for every marker count: each row
// has a CTA and its threads, the portable width takes what fits it, and a
// device without clusters gets none.
#include <cstdio>

#include "cluster_plan.h"

#define CHECK(c)                                                       \
    do {                                                               \
        if (!(c)) {                                                    \
            std::printf("FAILED %s at %d markers, %d CTAs\n", #c, ns, widest); \
            return 1;                                                  \
        }                                                              \
    } while (0)

int main() {
    using namespace ibmk;
    const int widths[] = {0, 8, 16};
    for (int widest : widths)
        for (int ns = 161; ns <= CL_MAX; ++ns) {
            const ClusterShape c = cluster_shape(ns, widest);
            const bool takes = widest == 16 || (widest == 8 && ns <= 8 * CL_ROWS);
            CHECK((c.ctas > 0) == takes);
            if (!takes) continue;
            CHECK(c.ctas <= widest);
            CHECK(c.ctas == (ns > CL_WIDE ? widest : 8));
            CHECK((long long)c.ctas * c.rows >= ns && c.rows % 4 == 0 && c.rows <= CL_ROWS);
            const int threads = c.rows <= 512 ? 512 : 1024;
            CHECK(c.lpr_log >= 0 && c.lpr_log <= 4 && (c.rows << c.lpr_log) <= threads);
        }
    std::printf("cluster plan ok\n");
    return 0;
}
