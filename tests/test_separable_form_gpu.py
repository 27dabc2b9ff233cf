"""Which form the separable preconditioner takes: the fused kernel for few jobs of a
2-D grid that a cluster holds in mixed precision, the separate products otherwise."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims,precision,cores,fused", [((60, 60), "mixed", 1, True), ((250, 250), "mixed", 1, True),
                                                        ((60, 60), "mixed", 0, False), ((60, 60), "fp64", 1, False),
                                                        ((2100, 2), "mixed", 1, False), ((12, 12, 12), "mixed", 1, False)])
def test_fused_where_it_applies(dims, precision, cores, fused):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2006_16117_gb300 as sim
    from workloads import cdr_axes, cdr_csr

    beta = (1.0, 0.5, 0.25)[: len(dims)]
    n = int(np.prod(dims))
    s = sim.Sim(cdr_csr(dims, beta, np.zeros(n)), None,
                sim.sim_default_options(precision=precision, separable_tensor_cores=cores))
    try:
        s.set_separable(dims, cdr_axes(dims, beta))
        sim.kernel_timing(True)
        s.shifted_solve(10.0 + 0.5j, torch.ones(n, dtype=torch.complex128, device="cuda"))
        torch.cuda.synchronize()
        one, every = sim.kernel_stats("sep_fused"), sim.kernel_stats("separable")
    finally:
        sim.kernel_timing(False)
        s.close()
    assert every["launches"] > 0
    assert (one["launches"] if one else 0) == (every["launches"] if fused else 0)
