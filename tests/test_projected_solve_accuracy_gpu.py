"""The direct projected solves, (I + (sigma - z) H) y = beta e_1 at every node of a
square, are as accurate as plain elimination in FP64: the residual's factor
|y_m| / ||y|| against extended precision."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _hessenberg(m, rng):
    """H of a Krylov space whose m Ritz values lie around sigma: (m+1, m)."""
    import scipy.linalg as sl

    g = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    gap = np.cumsum(rng.uniform(0.5, 6.0, m)) * np.where(np.arange(m) % 2 == 0, 1.0, -1.0)
    d = 1.0 / (gap - 0.2j)
    q, _ = np.linalg.qr(g(m, m))
    M = q @ (np.diag(d) + np.triu(0.02 * g(m, m), 1) * np.abs(d)) @ q.conj().T
    H = np.zeros((m + 1, m), dtype=np.complex128)
    H[:m] = sl.hessenberg(M)
    H[np.tril_indices(m + 1, -2, m)] = 0.0
    H[m, m - 1] = 1e-4
    return H, gap - 0.2j


def _factor(H, alpha, dtype):
    """|y_m| / ||y|| of every alpha by elimination with adjacent row exchanges in `dtype`."""
    m = H.shape[1]
    A = alpha.astype(dtype)[:, None, None] * H[:m].astype(dtype)
    A[:, np.arange(m), np.arange(m)] += 1
    r = np.zeros((alpha.size, m), dtype)
    r[:, 0] = 1
    for k in range(m - 1):
        swap = np.abs(A[:, k + 1, k]) > np.abs(A[:, k, k])
        for X in (A, r):
            X[swap, k], X[swap, k + 1] = X[swap, k + 1].copy(), X[swap, k].copy()
        f = A[:, k + 1, k] / A[:, k, k]
        A[:, k + 1, k:] -= f[:, None] * A[:, k, k:]
        r[:, k + 1] -= f * r[:, k]
    for j in range(m - 1, -1, -1):
        r[:, j] /= A[:, j, j]
        r[:, :j] -= A[:, :j, j] * r[:, j: j + 1]
    return np.abs(r[:, -1]) / np.sqrt((np.abs(r) ** 2).sum(1))


@pytest.mark.parametrize("m", [12, 31, 32, 33, 50])
def test_as_accurate_as_plain_elimination(m):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2006_16117_gb300 as sim

    rng = np.random.default_rng(m)
    H, gap = _hessenberg(m, rng)
    count, sigma = 128, 1000.0 + 0.2j
    sides = 0.25 * 2.0 ** -rng.integers(0, 10, count).astype(np.float64)
    centers = sigma + gap[rng.integers(0, m, count)] + 2 * sides * (rng.uniform(-1, 1, count) + 1j * rng.uniform(-1, 1, count))
    rho = sim.eval_squares(H, m, 1.0, sigma, centers, sides)[1]
    rho = rho.cpu().numpy() if torch.is_tensor(rho) else np.asarray(rho)
    off = sides[:, None] / np.sqrt(2.0) * np.exp(2j * np.pi * np.arange(8) / 8)
    alpha = sigma - (centers[:, None] + off)
    size = (np.abs(alpha) * 1e-4).astype(np.longdouble)
    of = lambda dtype: (size * _factor(H, alpha.ravel(), dtype).reshape(alpha.shape)).max(1)  # noqa: E731
    ref, plain = of(np.clongdouble), of(np.complex128)
    err = lambda v: float(np.median(np.abs(v - ref) / ref))  # noqa: E731
    # the same number of roundings but for a reciprocal and a product in a division's
    # place; half again leaves room for the median's own scatter over 128 squares
    assert err(rho) <= 1.5 * err(plain), (err(rho), err(plain))
