"""Cluster shapes of Gram-Schmidt and of the fused separable apply on a device that
places smaller clusters than the largest: a smaller shape, or none (the other form
then runs), and the unrestricted shape where everything fits."""
import native_program


def test_shapes_within_what_the_device_places(tmp_path):
    out = native_program.run(tmp_path, r'''
#include <cstdio>
#include <cmath>
#include "gs_shape.h"
#include "separable_fused_shape.h"
int main() {
    for (int most : {16, 8, 5, 1, 0})
        for (int64_t n : {1, 127, 2048, 2049, 40000, 81920, 81921})
            for (int jobs : {1, 40, 400}) {
                const sim::GsShape s = sim::gs_cluster_shape(n, 8, 2, jobs, 152, [&](int C, int, size_t) { return C <= most; });
                printf("gs %d %ld %d %d %d %d %d\n", most, (long)n, jobs, s.Cg, s.E, s.NT, (int)std::isinf(s.cost));
            }
    for (int most : {16, 8, 5, 1, 0})
        for (int N0 : {1, 9, 60, 250, 2048})
            for (int N1 : {2, 131, 250})
                for (int jobs : {1, 64}) {
                    const sim::FusedShape f = sim::fused_shape_that_fits(N0, N1, jobs, 152, [&](const sim::FusedShape& g) { return g.C <= most; });
                    printf("sep %d %d %d %d %d %d %d\n", most, N0, N1, f.C, f.Rc, f.Cc, (int)f.smem);
                }
}
''')
    best = {}
    for row in out.splitlines():
        kind, *v = row.split()
        v = list(map(int, v))
        if kind == "gs":
            most, n, jobs, C, E, threads, none = v
            assert none == (C == 0) and C <= most
            if C:
                assert 1 <= E <= 20 and (C - 1) * E * threads < n <= C * E * threads
                assert none == 0
            else:  # only where no cluster that is placed holds the rows
                assert -(-n // (20 * (128 if n <= 2048 else 256))) > most
            if most == 16:
                best[n, jobs] = C
            assert C == best[n, jobs] or C < best[n, jobs]
        else:
            most, N0, N1, C, Rc, Cc, smem = v
            assert C <= most
            if C:
                assert C * Rc >= N1 and C * Cc >= N0 and smem <= 220 * 1024
            if most == 0:
                assert C == 0
    assert best[40000, 1] == 16  # beyond the portable size where there is room
