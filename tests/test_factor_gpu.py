"""The block factorisation at the edges of its panels, warps and cluster shapes:
blocks whose pivots are scattered over their rows, ragged last blocks, several
couplings per row, against sparse LU."""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spla

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _block_matrix(T, blocks, seed):
    """Half-width T exactly: dense diagonal blocks, dominant on a permutation of
    their diagonal so that no pivot sits on it, couplings of one to three entries
    per row to both neighbours, and a ragged last block."""
    rng = np.random.default_rng(seed)
    n = blocks * T + max(1, T // 3)
    i, j = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    ib, jb, il, jl = i // T, j // T, i % T, j % T
    G = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    diag = ib == jb
    off = ((ib == jb + 1) & (il <= jl) & (jl <= il + 2)) | ((jb == ib + 1) & (jl <= il) & (il <= jl + 2))
    A = np.where(diag, G, 0) + np.where(off, 0.5 * G, 0)
    for a in range(0, n, T):
        m = min(T, n - a)
        A[a + rng.permutation(m), a + np.arange(m)] += 3.0 * np.sqrt(2.0 * T)
    return sp.csr_matrix(A)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("T", [2, 4, 8, 10, 16, 18, 30, 32, 34, 64, 66, 96, 128, 130, 160, 256, 258, 280])
def test_factor_of_permuted_blocks(precision, T):
    _check(_block_matrix(T, 4, 40 + T), T, 5, precision)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("T", [2, 18, 34])
@pytest.mark.parametrize("blocks", [1, 2, 3, 5])
def test_chains_of_few_blocks(precision, T, blocks):
    """Two to six block rows: sides of the two-ended elimination of uneven
    length, down to one block and none."""
    _check(_block_matrix(T, blocks, 90 + T), T, blocks + 1, precision)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [1, 2])
def test_a_single_block(precision, n):
    A = sp.csr_matrix(np.array([[2.0 + 1j, 0.5], [-0.25j, 3.0]])[:n, :n])
    _check(A, 2, 1, precision)


def _check(A, T, nb, precision):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2006_16117_gb300 as simlib

    A.sort_indices()
    n = A.shape[0]
    s = simlib.Sim((A.indptr, A.indices, A.data), None, simlib.sim_default_options(precision=precision))
    assert s.stats()["block_size"] == T and s.stats()["num_blocks"] == nb
    rng = np.random.default_rng(7)
    r = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    sigma = 0.3 - 0.2j
    x, iters, rel = s.shifted_solve(sigma, torch.from_numpy(r).cuda())
    ref = spla.splu((A - sigma * sp.identity(n)).tocsc()).solve(r)
    assert rel <= 1e-12
    # condition below 1e3: an FP64 factorisation leaves one refinement step, an FP32
    # one gains at least three digits a step
    assert iters <= (3 if precision == "fp64" else 5)
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 1e-9 * np.linalg.norm(ref)
    s.close()
