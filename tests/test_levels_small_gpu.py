"""The Schur form of a shift and the rank of a Gram matrix at their smallest and
largest orders."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def simlib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2006_16117_gb300 as sim

    return sim


def _locate(simlib, A, region, f, **options):
    s = simlib.Sim(A, None, simlib.sim_default_options(**options))
    try:
        s.set_region(region, f)
        marked = s.solve_all_levels()
        return marked, s.eigenvalues(), s.multiplicity(), s.stats()
    finally:
        s.close()


@pytest.mark.parametrize("n", [1, 2, 3, 5, 8])
def test_krylov_spaces_of_order_n(simlib, n):
    """A diagonal matrix of order n breaks the Arnoldi process down at n steps, so
    the Schur form has order n; the eigenvalues are known, all simple."""
    rng = np.random.default_rng(n)
    lam = np.sort_complex(0.37 + np.arange(n) * 0.9 + 1j * rng.uniform(-0.2, 0.6, n))
    A = (np.arange(n + 1, dtype=np.int32), np.arange(n, dtype=np.int32), lam)
    region = (0.0, float(n), -0.3, 0.7)
    f = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    runs = [_locate(simlib, A, region, f, level_solver=k) for k in (0, 1)]
    for marked, eig, mult, st in runs:
        assert marked == runs[0][0]
        assert eig.size == n and np.max(np.abs(eig - lam)) <= 1e-6  # the final squares' side
        assert np.array_equal(mult, np.ones(n, dtype=int))
    assert runs[1][3]["direct_level_evaluations"] == 0


@pytest.mark.parametrize("m", [33, 51])
def test_schur_orders(simlib, m):
    """Orders that are no multiple of a warp, up to the largest: the Schur levels
    mark the same squares as the direct solves."""
    from workloads import cd2d_csr, cd2d_eigenvalues, complex_gaussian
    from workloads.configs import window_region

    A = cd2d_csr(12, (1.0, 0.5))
    region = window_region(np.sort(cd2d_eigenvalues(12, (1.0, 0.5)).real), 60, 8)
    runs = [_locate(simlib, A, region, complex_gaussian(A.n, 0), m=m, level_solver=k) for k in (0, 1)]
    assert runs[0][0] == runs[1][0]
    assert runs[0][1].size == 8 and np.array_equal(runs[0][1], runs[1][1])
    assert np.array_equal(runs[1][2], np.ones(8, dtype=int))


@pytest.mark.parametrize("k", [1, 2, 7, 32, 64])
def test_rank_of_k_vectors(simlib, k):
    """The multiplicity of a triple eigenvalue with k random vectors, doubled to at
    least four of them: 3 (and 1 for its simple neighbour)."""
    lam = np.array([1.0, 1.0, 1.0, 2.2, 3.1, 4.4, 5.2, 6.3]) + 0.15j
    A = (np.arange(9, dtype=np.int32), np.arange(8, dtype=np.int32), lam)
    f = np.random.default_rng(3).standard_normal(8) + 0.5j
    _, eig, mult, _ = _locate(simlib, A, (0.5, 2.5, -0.3, 0.7), f, mult_k=k)
    assert np.max(np.abs(eig - [1.0 + 0.15j, 2.2 + 0.15j])) <= 1e-6
    assert mult.tolist() == [3, 1]
