"""GPU: the forms of the one-set fill.  A fill over many rows prepares a working
copy of the table (own-species sums, pn groups as full squares); a fill of few
rows, or one without memory for the copy, reads the table itself.  Both give the
same bits, and the whole matrix agrees with the oracle, on spaces with one
species, one particle of a species, many levels, odd A and unequal species.
"""
import numpy as np
import pytest

import oracle
from paper_1412_5989_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SPACES = [(3, 0, 4, 1), (0, 4, 3, 0), (1, 1, 5, 0), (1, 4, 3, 1), (4, 1, 3, 1), (2, 6, 2, 0), (6, 2, 2, 0), (3, 3, 2, 4),
          (2, 2, 5, 0), (5, 6, 1, 1), (9, 3, 1, 0), (1, 0, 5, 1), (2, 3, 0, 1),
          (4, 4, 2, 0), (1, 2, 7, 1), (2, 6, 3, 4), (6, 2, 3, 4), (2, 2, 6, 4), (0, 4, 6, 0), (4, 0, 6, 0),
          # large enough for the copy to be prepared
          (3, 3, 4, 0), (2, 5, 4, 1), (5, 2, 4, 1)]


@pytest.fixture(scope="module")
def cih():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_5989_gb300 import cih as mod
    return mod


@pytest.mark.parametrize("space", SPACES)
@pytest.mark.parametrize("energies", ["ho", "table", "onebody"])
def test_prepared_fill(cih, space, energies):
    B = cih.Basis(*space)
    S = oracle.Space(*space)
    t = synth.tbme_table(B.tbme_len, 11)
    T = torch.from_numpy(t).cuda()
    rowptr, nnz = B.count()
    B.set_count_mode(True)
    assert torch.equal(B.count()[0], rowptr)
    B.set_count_mode(False)
    n_orb = sum(B.n_orb)
    if energies == "onebody":
        t1 = synth.onebody_table(B.onebody_len, 5) * 10.0
        col, val = B.fill_onebody(rowptr, nnz, T, torch.from_numpy(t1).cuda())
        S.set_onebody(t1)
        _, _, col_o, val_o = S.rows(np.arange(B.dim), t)
    else:
        e = synth.single_particle_energies(n_orb, 3) if energies == "table" else None
        e_d = None if e is None else torch.from_numpy(e).cuda()
        col, val = B.fill(rowptr, nnz, T, e_sp=e_d)
        _, _, col_o, val_o = S.rows(np.arange(B.dim), t, esp=e)
        # shards of a few rows read the table itself
        step = max(1, B.dim // 40)
        parts = [B.fill_rows(rowptr, r, min(B.dim, r + step), T, e_sp=e_d) for r in range(0, B.dim, step)]
        assert torch.equal(torch.cat([c for c, _ in parts]), col)
        assert torch.equal(torch.cat([v for _, v in parts], dim=1), val)
    B.check()
    np.testing.assert_array_equal(col.cpu().numpy(), col_o)
    got = val[0].cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - val_o) <= 1e-5 * (np.abs(val_o) + 1.0))


@pytest.mark.parametrize("space", [(3, 3, 2, 0), (4, 4, 2, 0), (2, 6, 3, 4), (4, 0, 6, 0), (4, 5, 2, 1), (3, 3, 4, 0),
                                   (3, 4, 4, 1)])
@pytest.mark.parametrize("K", [2, 3, 4, 5, 7])
def test_few_sets(cih, space, K):
    """Fewer than eight sets: passes of up to four sets through the working copy.
    The bits are the same in every layout and from shards of a few rows; where the
    copy is prepared for these sets and not for one, or the other way round, a
    set's sums have another order than its own one-set fill's."""
    B = cih.Basis(*space)
    T = torch.from_numpy(synth.tbme_tables(B.tbme_len, range(K))).cuda()
    e = torch.from_numpy(synth.single_particle_energies(sum(B.n_orb), 3)).cuda()
    rowptr, nnz = B.count()
    col, val = B.fill(rowptr, nnz, T, e_sp=e)
    for k in range(K):
        c1, v1 = B.fill(rowptr, nnz, T[k], e_sp=e)
        assert torch.equal(c1, col)
        if B.dim < 8192:
            assert torch.equal(v1[0], val[k])
        assert bool(((v1[0] - val[k]).abs() <= 1e-6 * (val[k].abs() + 1.0)).all())
    til = cih.tbme_interleave(T)
    c2, v2 = B.fill_interleaved(rowptr, nnz, til, K, e_sp=e)
    c3, v3 = B.fill_batched(rowptr, nnz, til, K, e_sp=e)
    assert torch.equal(c2, col) and torch.equal(v2, val)
    assert torch.equal(c3, col) and torch.equal(v3.t(), val)
    step = max(1, B.dim // 30)
    parts = [B.fill_rows(rowptr, r, min(B.dim, r + step), T, e_sp=e) for r in range(0, B.dim, step)]
    assert torch.equal(torch.cat([c for c, _ in parts]), col)
    assert torch.equal(torch.cat([v for _, v in parts], dim=1), val)
    B.check()


def test_prepared_fill_in_a_graph(cih):
    """The working copy of a captured fill belongs to the graph: replays read the
    table anew."""
    B = cih.Basis(3, 3, 4, 0)
    rowptr, nnz = B.count()
    T = torch.from_numpy(synth.tbme_table(B.tbme_len, 1)).cuda()
    col, val = B.fill(rowptr, nnz, T)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        B.fill(rowptr, nnz, T, stream=s, col=col, val=val)
    T.copy_(torch.from_numpy(synth.tbme_table(B.tbme_len, 2)).cuda())
    for _ in range(3):
        val.zero_()
        g.replay()
    torch.cuda.synchronize()
    got = val.clone()
    assert torch.equal(got, B.fill(rowptr, nnz, T)[1])
    B.check()
