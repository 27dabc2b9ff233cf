"""set_separable keeps the fused kernel's padded table only where that kernel can
run: FP64, one and three axes and axes no cluster holds do without it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision,dims", [("fp64", (2000, 2)), ("mixed", (2500, 2)), ("mixed", (2500,)), ("mixed", (2000, 2, 1))])
def test_no_padded_table_where_nothing_reads_it(precision, dims):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2006_16117_gb300 as sim
    from workloads import cdr_axes, cdr_csr

    def used(dims):
        beta = (1.0, 0.5, 0.25)[: len(dims)]
        n = int(np.prod(dims))
        s = sim.Sim(cdr_csr(dims, beta, np.zeros(n)), None, sim.sim_default_options(precision=precision))
        try:
            before = torch.cuda.mem_get_info()[0]
            s.set_separable(dims, cdr_axes(dims, beta))
            return before - torch.cuda.mem_get_info()[0]
        finally:
            s.close()

    used((4,) * len(dims))  # the kernels are loaded
    # Q in FP64 and FP32 and its two FP32 parts, 20 bytes an entry; the padded copy
    # would be 4 more.  2 MiB a buffer for the allocator's granularity
    n2 = max(dims) ** 2
    got = used(dims)
    assert got <= 20 * n2 + 7 * 2**21, (got, n2)
    assert 20 * n2 + 7 * 2**21 < 24 * n2
