"""GPU: a fill's bits do not depend on its rows.  A fill of few sets over many rows
sums through a working copy of the tables; a shard of few rows sums in the row
kernel, which makes the sums that the order could change again in the other form's
order.  Both are compared bit for bit, on tables for which the order matters.
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


def tables(kind, K, n, n1):
    """K two-body tables and a one-body table."""
    g = torch.Generator(device="cuda").manual_seed(7)
    t = torch.randn((K, n), generator=g, device="cuda")
    t1 = torch.randn(n1, generator=g, device="cuda", dtype=torch.float64) * 10.0
    if kind == "spread":                        # more binary orders than a double-float pair holds
        t = t * 10.0 ** (torch.rand((K, n), generator=g, device="cuda") * 16.0 - 8.0)
    elif kind == "halves":                      # sums of ones and half last bits, decided by terms of 2^-46
        t = 1.0 + torch.randint(-(1 << 20), 1 << 20, (K, n), generator=g, device="cuda") * 2.0 ** -23
        t1 = t1 * 2.0 ** -46
    elif kind == "small":                       # low parts down to the smallest subnormals
        t = t * 2.0 ** -118
        t1 = t1 * 2.0 ** -118
    elif kind == "nonfinite":
        t[torch.rand((K, n), generator=g, device="cuda") < 0.01] = float("inf")
        t[torch.rand((K, n), generator=g, device="cuda") < 0.01] = float("nan")
        t[torch.rand((K, n), generator=g, device="cuda") < 0.05] = -0.0
    return t.to(torch.float32).contiguous(), t1


def same(a, b):
    """Equal bits; NaN equals NaN."""
    nan = torch.isnan(a)
    return torch.equal(nan, torch.isnan(b)) and torch.equal(a.view(torch.int32)[~nan], b.view(torch.int32)[~nan])


# space, set counts whose fills of all rows go through the copy
SPACES = [((4, 5, 2, 1), (2, 3, 4)), ((3, 3, 4, 0), (1, 2, 3, 4)), ((5, 2, 4, 1), (1, 2, 3, 4)), ((3, 4, 4, 1), (1, 2, 3, 4, 5, 7)),
          ((10, 3, 2, 1), (1, 2, 3, 4)), ((16, 3, 1, 1), (2, 3, 4)), ((1, 6, 4, 1), (2, 3, 4)), ((6, 1, 4, 1), (2, 3, 4)),
          ((2, 2, 7, 0), (2, 3, 4))]


@pytest.mark.parametrize("space,copied", SPACES)
@pytest.mark.parametrize("kind", ["normal", "spread", "halves", "small", "nonfinite"])
def test_shards_same_bits(cih, space, copied, kind):
    B = cih.Basis(*space)
    rowptr, nnz = B.count()
    T, _ = tables(kind, 8, B.tbme_len, B.onebody_len)
    e = torch.rand(sum(B.n_orb), dtype=torch.float64, device="cuda") * (2.0 ** -46 if kind == "halves" else 50.0)
    step = max(1, B.dim // 40)
    for K in (1, 2, 3, 4, 5, 7, 8):
        t = T[:K].contiguous()
        n0 = cih.kernel_launches()
        col, val = B.fill(rowptr, nnz, t, e_sp=e)
        assert (cih.kernel_launches() - n0 > 1) == (K in copied)
        if K == 1:
            one = [B.fill(rowptr, nnz, T[k], e_sp=e)[1][0] for k in range(7)]
        if K < 8 and (1 in copied) == (K in copied):                # the same way for one set: the same bits
            assert all(same(val[k], one[k]) for k in range(K))
        n0 = cih.kernel_launches()
        parts = [B.fill_rows(rowptr, r, min(B.dim, r + step), t, e_sp=e) for r in range(0, B.dim, step)]
        assert cih.kernel_launches() - n0 == len(parts)          # shards of a fortieth: the row kernel
        assert torch.equal(torch.cat([c for c, _ in parts]), col)
        assert same(torch.cat([v for _, v in parts], dim=1), val)
    B.check()


@pytest.mark.parametrize("space", [(1, 6, 4, 1), (6, 1, 4, 1), (10, 3, 2, 1), (16, 3, 1, 1), (2, 2, 7, 0), (2, 3, 6, 1)])
@pytest.mark.parametrize("onebody", [False, True])
def test_copy_against_the_oracle(cih, space, onebody):
    """Few particles of a species, many of one, many levels: every element of two sets."""
    B = cih.Basis(*space)
    S = oracle.Space(*space)
    t = synth.tbme_tables(B.tbme_len, range(2))
    T = torch.from_numpy(t).cuda()
    rowptr, nnz = B.count()
    n0 = cih.kernel_launches()
    if onebody:
        t1 = synth.onebody_table(B.onebody_len, 5) * 10.0
        col, val = B.fill_onebody(rowptr, nnz, T, torch.from_numpy(t1).cuda())
        S.set_onebody(t1)
        e = None
    else:
        e = synth.single_particle_energies(sum(B.n_orb), 3)
        col, val = B.fill(rowptr, nnz, T, e_sp=torch.from_numpy(e).cuda())
    assert cih.kernel_launches() - n0 == 2
    for k in range(2):
        _, _, col_o, val_o = S.rows(np.arange(B.dim), t[k], esp=e)
        np.testing.assert_array_equal(col.cpu().numpy(), col_o)
        assert np.all(np.abs(val[k].cpu().numpy().astype(np.float64) - val_o) <= 1e-5 * (np.abs(val_o) + 1.0))
    B.check()


def test_walk_order_same_bits(cih):
    """At least 2^19 rows: the copy's form takes the rows of 16 proton sub-dets side by side."""
    B = cih.Basis(2, 6, 6, 4)
    assert B.dim >= 1 << 19
    rowptr, nnz = B.count()
    T, _ = tables("halves", 1, B.tbme_len, B.onebody_len)
    e = torch.rand(sum(B.n_orb), dtype=torch.float64, device="cuda") * 2.0 ** -46
    whole = B.fill(rowptr, nnz, T[0], e_sp=e)
    bounds = cih.shard_bounds(rowptr.cpu(), 100)
    for k in (0, 1, 37, 98, 99):
        r0, r1 = int(bounds[k]), int(bounds[k + 1])
        a, b = int(rowptr[r0]), int(rowptr[r1])
        c, v = B.fill_rows(rowptr, r0, r1, T[0], e_sp=e)
        assert torch.equal(c, whole[0][a:b]) and same(v[0], whole[1][0, a:b])
    B.check()
