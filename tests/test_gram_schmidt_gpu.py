"""The Gram-Schmidt step over its forms (a cluster per job, the whole GPU) and
their shapes: location and multiplicities of a separable operator with known
eigenvalues, from vectors shorter than a CTA to vectors no cluster holds."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nx,ny", [(9, 7), (16, 8), (43, 3), (64, 32), (89, 23), (64, 65), (201, 203)])
def test_location_of_known_eigenvalues(precision, nx, ny):
    _check(precision, nx, ny, 3)


def test_long_vectors():
    _check("mixed", 291, 289, 2)


def _check(precision, nx, ny, count):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2006_16117_gb300 as sim

    beta = (1.0, 0.5)
    axes, lams = [], []
    for N, b in zip((nx, ny), beta):
        h = 1.0 / (N + 1)
        sub, dg, sup = -1 / h**2 - b / (2 * h), 2 / h**2, -1 / h**2 + b / (2 * h)
        axes.append((sub, dg, sup))
        lams.append(dg + 2 * np.sqrt(sub * sup) * np.cos(np.arange(1, N + 1) * np.pi / (N + 1)))
    lam = np.sort((lams[0][:, None] + lams[1][None, :]).ravel())
    import scipy.sparse as sp

    d1 = [sp.diags([s * np.ones(N - 1), d * np.ones(N), u * np.ones(N - 1)], [-1, 0, 1])
          for N, (s, d, u) in zip((nx, ny), axes)]
    A = sp.csr_matrix(sp.kron(sp.identity(ny), d1[0]) + sp.kron(d1[1], sp.identity(nx)), dtype=np.complex128)
    A.sort_indices()
    gaps = np.diff(lam)
    c = count
    while gaps[c - 1] < 1.0:
        c += 1
    region = (lam[0] - 2.0, 0.5 * (lam[c - 1] + lam[c]), -0.3, 0.7)
    s = sim.Sim((A.indptr, A.indices, A.data), None, sim.sim_default_options(precision=precision, mult_k=4))
    try:
        s.set_separable((nx, ny), axes)
        rng = np.random.default_rng(nx)
        s.set_region(region, rng.standard_normal(nx * ny) + 1j * rng.standard_normal(nx * ny))
        s.solve_all_levels()
        eig, mult = s.eigenvalues(), s.multiplicity()
        assert eig.size == c and np.max(np.abs(eig - lam[:c])) <= 1e-6  # the final squares' side
        assert np.array_equal(mult, np.ones(c, dtype=int))
        assert s.stats()["max_inner_residual"] <= 1e-10  # mult_inner_tol, the looser of the two
    finally:
        s.close()
