"""The block solve's forms at their edges: one to sixteen right-hand sides a shift,
clusters of one CTA whose rows take several chunks, blocks too long for their
inputs to be fetched ahead."""
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


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("T", [2, 18, 34, 66, 258])
@pytest.mark.parametrize("nodes", [4, 5, 16, 64])
def test_many_shifts(simlib, precision, T, nodes):
    """Φ = ||Σ_j w_j (A - z_j)^{-1} f||² of up to 64 nodes solved together, against
    dense inverses.  Each solve leaves a relative residual of 1e-12 (2e-12 with its
    own rounding), so its error is at most ||(A - z_j)^{-1}|| times that."""
    from oracle.grad import circle_nodes
    from test_factor_gpu import _block_matrix

    blocks = 8 if T < 66 else 3  # eight or more: both sides of the elimination
    if T == 258 and nodes > 5:
        pytest.skip("dense inverses of that order")
    A = _block_matrix(T, blocks, 60 + T)
    A.sort_indices()
    n = A.shape[0]
    f = np.random.default_rng(5).standard_normal(n) + 0.5j
    c, r = 3.0 * np.sqrt(2.0 * T), 1.5 * np.sqrt(2.0 * T)
    z, w = circle_nodes(c, r, nodes)
    x, dx = 0.0, 0.0
    for zj, wj in zip(z, w):
        inv = np.linalg.inv(A.toarray() - zj * np.identity(n))
        x = x + wj * (inv @ f)
        dx += abs(wj) * np.linalg.norm(inv, 2) * 2e-12 * np.linalg.norm(f)
    s = simlib.Sim((A.indptr, A.indices, A.data), None, simlib.sim_default_options(precision=precision))
    phi = s.projection_norm(c, r, f, nodes, True)
    s.close()
    ref = np.linalg.norm(x)
    assert abs(phi - ref**2) <= 2.0 * ref * dx + dx * dx


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("grid,k", [(12, 2), (12, 3), (12, 8), (30, 2), (30, 4), (30, 5), (30, 16), (101, 3), (101, 8)])
def test_right_hand_sides_of_a_shift(simlib, precision, grid, k):
    """k random vectors a shift (2, 4 or 8 at a time share the factor): simple
    eigenvalues, every solve to its tolerance in a few iterations."""
    from test_levels_small_gpu import _locate
    from workloads import cd2d_csr, cd2d_eigenvalues, complex_gaussian
    from workloads.configs import window_region

    A = cd2d_csr(grid, (1.0, 0.5))
    lam = np.sort(cd2d_eigenvalues(grid, (1.0, 0.5)).real)
    region = window_region(lam, 10, 3)
    _, eig, mult, st = _locate(simlib, A, region, complex_gaussian(A.n, 0), precision=precision, mult_k=k)
    assert np.max(np.min(np.abs(lam[None, :] - eig[:, None]), axis=1)) <= 1e-6
    assert np.array_equal(mult, np.ones(eig.size, dtype=int)) and eig.size >= 1
    assert st["max_gmres_iterations"] <= 8


def test_more_groups_than_a_launch_carries(simlib):
    """Many shifts with 64 vectors each: the table of groups goes through device
    memory instead of the launch's parameters."""
    from test_levels_small_gpu import _locate
    from workloads import cd2d_csr, cd2d_eigenvalues, complex_gaussian
    from workloads.configs import window_region

    A = cd2d_csr(12, (1.0, 0.5))
    lam = np.sort(cd2d_eigenvalues(12, (1.0, 0.5)).real)
    region = window_region(lam, 20, 90)
    _, eig, mult, st = _locate(simlib, A, region, complex_gaussian(A.n, 0), precision="mixed", mult_k=64)
    assert st["num_shifts"] * 64 > 512
    assert np.max(np.min(np.abs(lam[None, :] - eig[:, None]), axis=1)) <= 1e-6
    assert np.array_equal(mult, np.ones(eig.size, dtype=int)) and eig.size >= 80
