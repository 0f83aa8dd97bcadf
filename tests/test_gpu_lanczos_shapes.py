"""GPU: the orthogonalisation and step kernels of the Lanczos solver at the set
counts where their lane mapping changes (one set, rows packed into a warp,
exactly one warp of sets, more than one, the compile-time 64, the most allowed)
and at few and many iterations, against dense eigenvalues of the same matrices.

The solver stops at residual bounds of 1e-9 |theta|, so its eigenvalues are
within that of the dense ones, and the vectors' residuals within twice it.
"""
import numpy as np
import pytest

from paper_1412_5989_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cih():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_5989_gb300 import cih as mod
    return mod


def dense(rowptr, col, val, dim):
    H = torch.zeros((dim, dim), dtype=torch.float64, device="cuda")
    i = torch.repeat_interleave(torch.arange(dim, device="cuda"), rowptr[1:] - rowptr[:-1])
    H[i, col.long()] = val.double()
    return torch.triu(H) + torch.triu(H, 1).t()


@pytest.mark.parametrize("space,K", [((2, 2, 2, 0), K) for K in (1, 2, 3, 5, 16, 31, 32, 33, 64, 65, 100, 256)] +
                         [((3, 3, 2, 0), 1), ((3, 3, 2, 0), 7), ((3, 3, 2, 0), 64), ((1, 1, 2, 4), 3), ((2, 3, 0, 1), 2),
                          ((2, 2, 0, 0), 4), ((2, 3, 4, 5), 1)])
def test_against_dense(cih, space, K):
    B = cih.Basis(*space)
    T = torch.from_numpy(synth.tbme_tables(B.tbme_len, range(K))).cuda()
    rowptr, nnz = B.count()
    col, val = B.fill(rowptr, nnz, T)
    nev = min(5, B.dim)
    ev, vec, conv = B.lanczos(rowptr, col, val, nev=nev, max_iter=400, tol=1e-9)
    assert conv
    for k in sorted({0, K // 2, K - 1}):
        H = dense(rowptr, col, val[k], B.dim)
        w = torch.linalg.eigvalsh(H)[:nev].cpu().numpy()
        assert np.all(np.abs(ev[k] - w) <= 1e-9 * np.maximum(1.0, np.abs(w)))
        v = vec[k]
        assert abs(float(v.norm()) - 1.0) < 1e-12
        assert float((H @ v - ev[k, 0] * v).norm()) <= 2e-9 * max(1.0, abs(w[0]))


@pytest.mark.parametrize("iters", [1, 2, 3, 7])
def test_iteration_limit(cih, iters):
    """The limit ends the run there, with the Ritz values of that many steps
    (the same as of a NumPy Lanczos from the documented start vector)."""
    B = cih.Basis(3, 3, 2, 0)
    T = torch.from_numpy(synth.tbme_table(B.tbme_len, 3)).cuda()
    rowptr, nnz = B.count()
    col, val = B.fill(rowptr, nnz, T)
    ev, vec, conv = B.lanczos(rowptr, col, val, nev=2, max_iter=iters, tol=1e-12)
    assert not conv
    H = dense(rowptr, col, val[0], B.dim).cpu().numpy()
    z = np.arange(B.dim, dtype=np.uint64) + np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    z ^= z >> np.uint64(31)
    V = [1.0 + 0.5 * (z >> np.uint64(11)).astype(np.float64) / 9007199254740992.0]
    V[0] /= np.linalg.norm(V[0])
    Q = np.stack(V)
    for _ in range(iters - 1):
        w = H @ Q[-1]
        for _ in range(2):
            w -= Q.T @ (Q @ w)
        Q = np.vstack([Q, w / np.linalg.norm(w)])
    th = np.linalg.eigvalsh(Q @ H @ Q.T)[:2]
    got = ev[0][: len(th)]
    assert np.all(np.abs(got - th) <= 1e-10 * np.abs(th))
    assert np.all(np.isnan(ev[0][len(th):]))
