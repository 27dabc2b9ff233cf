// Batched Gram–Schmidt arguments (krylov.cu, gs_cluster.cu, gs_grid.cu).
#pragma once

#include "internal.h"

namespace sim {

// What the orthogonalisation's last step does for the inner FGMRES, once the
// coefficients and the norm are known (gs_finish.cuh): START begins a cycle (the
// norm is γ), STEP applies the Givens rotations to column i, updates the residual
// estimate and, when the cycle ends with this column, solves R y = g.
struct GmArgs {
    enum { NONE = 0, START = 1, STEP = 2 };
    int mode = NONE;
    int k = 0, i = 0;       // restart length; column of a STEP
    int first = 0;          // START: first cycle of the solve
    double tol = 0.0;
    int max_iter = 0;
    double2 *Hg = nullptr, *cs = nullptr, *sn = nullptr, *g = nullptr, *y = nullptr;
    double* scal = nullptr;
    int* istat = nullptr;
};

// Vectors of job `job`: basis vector i at basis + job*bstride + i*n; w at
// w + job*wstride, read from src + job*sstride instead if src is set (w is then
// only written).  Coefficients go to hcol + job*hstride, the norm to hcol[cnt].
struct GSArgs {
    const double2* basis = nullptr;
    int64_t bstride = 0;
    double2* w = nullptr;
    int64_t wstride = 0;
    const double2* src = nullptr;
    int64_t sstride = 0;
    double2* hcol = nullptr;
    int64_t hstride = 0;
    int cnt = 0;
    int64_t n = 0;
    const int* active = nullptr;
    // Arnoldi breakdown test (optional): H base / stride / ld and column j
    const double2* Hfull = nullptr;
    int64_t Hstride = 0;
    int Hld = 0;
    int j = 0;
    double btol = 0.0;
    int* meff = nullptr;      // per job (optional)
    int* istat = nullptr;     // per job IS_N ints (optional): IS_BROKEN flag
    int* h_istat = nullptr;   // host copy of istat's flags that the host waits for
    // selective reorthogonalisation (Daniel-Gragg-Kaufman-Stewart): the second
    // pass runs only if the first one cut the norm of w below 1/sqrt(2) of it
    int dgks = 0;
    // one pass only (the classical Gram-Schmidt printed in Sec. 2); overrides dgks
    int single = 0;
    GmArgs gm;
    // scratch of the grid kernels (gs_grid.cu)
    double2* part = nullptr;  // partial sums: gs_grid_partials()
    int pw = 0;               // values per chunk
    double2* hsum = nullptr;  // [2][J][pw] totals of the two passes
    double* fin = nullptr;    // [J] scale of the result
    int* need = nullptr;      // [J] second pass wanted
    int* ticket = nullptr;    // [J] zero between launches
    int J = 0;
};

// The orthogonalisation of nactive jobs: w against cnt basis vectors, norm,
// breakdown test, normalisation, FGMRES step.  Picks one of the two forms below.
void gram_schmidt(const GSArgs& a, int nactive, cudaStream_t st);

// Estimated clocks of the two forms, and the second one's launches.
double gs_cluster_cost(int64_t n, int cnt, int passes, int nactive);  // infinite: out of its range
double gs_grid_cost(int64_t n, int cnt, int passes, int nactive);
void gs_grid(const GSArgs& a, int nactive, cudaStream_t st);
// Rows per CTA of the grid form and the partial sums it needs for any number of
// active jobs up to J.
int64_t gs_grid_partials(int64_t n, int J, int pw);

}  // namespace sim
