"""A single pass overrides the selective second one, in the cluster form and in the
grid form of the Gram-Schmidt step alike (gs.h)."""
import native_program
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SOURCE = r'''
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "gs.h"
using namespace sim;
template <class T> T* dev(size_t n) {
    T* p;
    SIM_CUDA(cudaMalloc(&p, n * sizeof(T)));
    SIM_CUDA(cudaMemset(p, 0, n * sizeof(T)));
    return p;
}
int main(int, char** v) {
    const int64_t n = atoll(v[1]);
    const int cnt = 3, J = 2, pw = cnt + 2;
    // basis e_0, e_1, e_2; w = e_0 + 2 e_1 + 2^-10 e_5: the first pass cuts its norm far
    // enough for the selective test to want a second one
    std::vector<double2> basis(J * cnt * n, make_double2(0, 0)), w(J * n, make_double2(0, 0));
    for (int j = 0; j < J; ++j) {
        for (int i = 0; i < cnt; ++i) basis[(j * cnt + i) * n + i].x = 1;
        w[j * n].x = 1, w[j * n + 1].x = 2, w[j * n + 5].x = 0x1p-10;
    }
    GSArgs a;
    double2* b = dev<double2>(basis.size());
    SIM_CUDA(cudaMemcpy(b, basis.data(), basis.size() * sizeof(double2), cudaMemcpyHostToDevice));
    a.basis = b, a.bstride = cnt * n;
    a.w = dev<double2>(w.size()), a.wstride = n;
    SIM_CUDA(cudaMemcpy(a.w, w.data(), w.size() * sizeof(double2), cudaMemcpyHostToDevice));
    a.hcol = dev<double2>(J * (cnt + 1)), a.hstride = cnt + 1;
    a.cnt = cnt, a.n = n;
    const int act[J] = {0, 1};
    int* d_act = dev<int>(J);
    SIM_CUDA(cudaMemcpy(d_act, act, sizeof act, cudaMemcpyHostToDevice));
    a.active = d_act;
    a.single = 1, a.dgks = 1;
    a.part = dev<double2>(gs_grid_partials(n, J, pw)), a.pw = pw;
    a.hsum = dev<double2>(2 * J * pw), a.fin = dev<double>(J), a.need = dev<int>(J), a.ticket = dev<int>(J), a.J = J;
    const bool grid = !(gs_cluster_cost(n, cnt, 2, J) <= gs_grid_cost(n, cnt, 2, J));
    gram_schmidt(a, J, nullptr);
    SIM_CUDA(cudaDeviceSynchronize());
    std::vector<double2> h(J * (cnt + 1));
    SIM_CUDA(cudaMemcpy(w.data(), a.w, w.size() * sizeof(double2), cudaMemcpyDeviceToHost));
    SIM_CUDA(cudaMemcpy(h.data(), a.hcol, h.size() * sizeof(double2), cudaMemcpyDeviceToHost));
    printf("%d\n", (int)grid);
    for (int j = 0; j < J; ++j) {
        int others = 0;
        for (int64_t i = 0; i < n; ++i) others += i != 5 && (w[j * n + i].x != 0 || w[j * n + i].y != 0);
        printf("%g %d %g %g %g %g\n", w[j * n + 5].x, others, h[j * 4].x, h[j * 4 + 1].x, h[j * 4 + 2].x, h[j * 4 + 3].x * 1024);
    }
}
'''


@pytest.mark.parametrize("n,grid", [(100, 0), (200000, 1)])
def test_single_pass_overrides_the_selective_one(tmp_path, n, grid):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    form, *jobs = native_program.run(tmp_path, SOURCE, n).splitlines()
    assert int(form) == grid  # the size meant for that form takes it
    assert jobs == ["1 0 1 2 0 1"] * 2
