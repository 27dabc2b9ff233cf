"""sim_apply_shifted straight on the caller's vectors: separate, in place, overlapping
and misaligned ones give the same product, for every kind of B."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1, 255, 256, 257, 1000])
@pytest.mark.parametrize("kind", ["identity", "diag", "general"])
def test_apply_in_place_overlapping_and_misaligned(n, kind):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2006_16117_gb300 as simlib

    rng = np.random.default_rng(n)
    A = sp.random(n, n, density=min(1.0, 6.0 / n), random_state=1, format="csr", dtype=np.float64) + 2j * sp.identity(n)
    A = sp.csr_matrix(A)
    A.sort_indices()
    B = None
    if kind == "diag":
        B = sp.csr_matrix(sp.diags(rng.uniform(1, 2, n)).astype(np.complex128))
    elif kind == "general":
        B = sp.csr_matrix(sp.identity(n) + 0.25 * sp.random(n, n, density=min(1.0, 2.0 / n), random_state=2)).astype(np.complex128)
        B.sort_indices()
    csr = lambda M: None if M is None else (M.indptr, M.indices, M.data)  # noqa: E731
    s = simlib.Sim(csr(A), csr(B))
    L = simlib.lib()
    x = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    sigma = 0.7 - 0.3j
    ref = A @ x - sigma * (x if B is None else B @ x)
    tol = 1e-13 * max(1.0, np.max(np.abs(ref)))

    def apply(px, py):
        assert L.sim_apply_shifted(s.h, sigma.real, sigma.imag, px, py) == 0
        torch.cuda.synchronize()

    buf = torch.zeros(2 * (2 * n + 8), dtype=torch.float64, device="cuda")
    xr = torch.from_numpy(x.view(np.float64)).cuda()
    read = lambda off: buf[off: off + 2 * n].cpu().numpy().view(np.complex128)  # noqa: E731
    for xo, yo in ((0, 2 * n + 2), (0, 0), (2, 0), (0, 2), (1, 2 * n + 4), (0, 2 * n + 3), (3, 1)):
        buf.zero_()
        buf[xo: xo + 2 * n] = xr
        apply(buf.data_ptr() + 8 * xo, buf.data_ptr() + 8 * yo)
        assert np.max(np.abs(read(yo) - ref)) <= tol, (xo, yo)
    s.close()
