"""The fused separable preconditioner of 2-D grids at the edges of its tiles, stages
and clusters: the same solution in the same number of steps (give or take one, FP32
either way) as the separate mode products on the CUDA cores."""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spla

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims", [(2, 2), (2, 9), (5, 3), (16, 16), (31, 17), (33, 64), (65, 48), (97, 131), (250, 250)])
def test_fused_apply_equals_the_separate_products(dims):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2006_16117_gb300 as sim
    from workloads import cdr_axes, cdr_csr, cdr_separable_eigenvalues

    beta = (1.0, 0.5)
    rng = np.random.default_rng(dims[0])
    n = int(np.prod(dims))
    react = 0.3 * np.sqrt(rng.uniform(size=n)) * np.exp(2j * np.pi * rng.uniform(size=n))
    A = cdr_csr(dims, beta, react)
    lam = np.sort(cdr_separable_eigenvalues(dims, beta).real)
    sigma = lam[len(lam) // 3] + 0.37 + 0.2j
    r = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    ref = spla.splu((A.to_scipy() - sigma * sp.identity(n)).tocsc()).solve(r)
    its = []
    for tc in (0, 1):
        s = sim.Sim(A, None, sim.sim_default_options(precision="mixed", separable_tensor_cores=tc))
        s.set_separable(dims, cdr_axes(dims, beta))
        x, iters, rel = s.shifted_solve(sigma, torch.from_numpy(r).cuda())
        s.close()
        assert rel <= 1e-12
        assert np.linalg.norm(x.cpu().numpy() - ref) <= 1e-9 * np.linalg.norm(ref)
        its.append(iters)
    assert abs(its[0] - its[1]) <= 1, its
