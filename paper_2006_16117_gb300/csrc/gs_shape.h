// The launch shape of the cluster form of Gram–Schmidt (gs_cluster.cu).
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <limits>

namespace sim {

constexpr int GC_MAXV = 64;   // basis vectors per call (cnt)
constexpr int GC_MAXE = 20;   // rows per thread: two CTAs' pieces of w fit an SM

struct GsShape {
    int Cg = 0, E = 0, NT = 256;  // CTAs per cluster, rows and threads
    size_t smem = 0;
    double cost = std::numeric_limits<double>::infinity();  // estimated clocks
};

// Cluster size and rows per thread: as many CTAs a job as the GPU holds at two per
// SM, at most 16 (the hardware's limit), no more than there are rows for and no more
// than fits(cluster size, threads, bytes of dynamic shared memory) says the device
// places; an infinite cost if there is no such shape.  The estimate charges each SM's
// FP64 instructions 64 clocks a warp on its four schedulers and 2,500 clocks a pass for
// the sums across the cluster.
template <class Fits>
GsShape gs_cluster_shape(int64_t n, int cnt, int passes, int nactive, int sms, Fits fits) {
    auto up = [](int64_t a, int64_t b) { return (a + b - 1) / b; };
    GsShape s;
    s.NT = n <= 128 * 16 ? 128 : 256;
    const int64_t need = up(n, (int64_t)s.NT * GC_MAXE);
    if (need > 16 || cnt > GC_MAXV) return s;
    const int64_t room = std::max(1, 2 * sms / std::max(1, nactive));
    for (int64_t C = std::max(need, std::min(std::min<int64_t>(16, room), up(n, s.NT))); C >= need; --C) {
        const int E = (int)up(n, (int64_t)s.NT * C);
        const int Cg = (int)up(n, (int64_t)s.NT * E);
        const size_t smem = (size_t)E * s.NT * 16;
        if (!fits(Cg, s.NT, smem)) continue;
        s.Cg = Cg;
        s.E = E;
        s.smem = smem;
        const double per_warp = E * (4.0 * cnt * passes + 6.0) + 1.2 * cnt * passes + 20.0;
        const double per_sm = std::ceil((double)nactive * Cg / sms);
        s.cost = per_warp * 64.0 * (s.NT / 128) * per_sm + (passes + 1.0) * 2500.0;
        break;
    }
    return s;
}

}  // namespace sim
