"""GPU: fills of few rows.  Where the rows leave the GPU idle, a row's elements are
filled by two or three CTAs, and the sums of several sets are made side by side.
Both leave the bits as they are: against one CTA a row, against one-set fills,
and against the oracle.
"""
import numpy as np
import pytest

import oracle
from paper_1412_5989_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cih():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_5989_gb300 import cih as mod
    return mod


# 12 to 10,817 rows: three, two and one CTA a row on 152 SMs of 32 warps; one species,
# one particle, more pairs than the pair queue
SPACES = [(1, 0, 5, 1), (2, 2, 2, 0), (3, 0, 4, 1), (0, 4, 4, 0), (9, 5, 1, 0), (2, 3, 4, 5), (8, 1, 3, 1), (3, 4, 3, 1)]


@pytest.mark.parametrize("space", SPACES)
@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 6, 7, 8, 9, 12, 15, 16, 20, 22, 64])
def test_parts_same_bits(cih, space, K):
    B = cih.Basis(*space)
    T = torch.from_numpy(synth.tbme_tables(B.tbme_len, range(K))).cuda()
    til = cih.tbme_interleave(T)
    e = torch.from_numpy(synth.single_particle_energies(sum(B.n_orb), 3)).cuda()
    rowptr, nnz = B.count()

    def fills():
        return [B.fill(rowptr, nnz, T, e_sp=e), B.fill_interleaved(rowptr, nnz, til, K, e_sp=e),
                B.fill_batched(rowptr, nnz, til, K, e_sp=e)]

    got = fills()
    step = max(1, B.dim // 3)
    parts = [B.fill_rows(rowptr, r, min(B.dim, r + step), T, e_sp=e) for r in range(0, B.dim, step)]
    assert torch.equal(torch.cat([c for c, _ in parts]), got[0][0])
    assert torch.equal(torch.cat([v for _, v in parts], dim=1), got[0][1])
    B.set_launch(16, 1)                          # half the CTAs at once: fewer parts
    for (c, v), (c1, v1) in zip(got, fills()):
        assert torch.equal(c, c1) and torch.equal(v, v1)
    if K < 16 and B.dim < 8192:                  # (a larger basis may take another order for some set counts)
        for k in range(K):
            c1, v1 = B.fill(rowptr, nnz, T[k], e_sp=e)
            assert torch.equal(c1, got[0][0]) and torch.equal(v1[0], got[0][1][k])
            assert torch.equal(v1[0], got[1][1][k]) and torch.equal(v1[0], got[2][1][:, k])
    S = oracle.Space(*space)
    for k in {0, K - 1}:
        _, _, col_o, val_o = S.rows(np.arange(B.dim), T[k].cpu().numpy(), esp=e.cpu().numpy())
        np.testing.assert_array_equal(got[0][0].cpu().numpy(), col_o)
        for v in (got[0][1][k], got[1][1][k], got[2][1][:, k]):
            assert np.all(np.abs(v.cpu().numpy().astype(np.float64) - val_o) <= 1e-5 * (np.abs(val_o) + 1.0))
    B.check()
