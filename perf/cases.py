"""What a user of this library has it do, as measurable cases.

A case names an operation (``op``), a space (protons Z, neutrons N, Nmax, 2M)
and a number of interaction sets K.  The operations are the public entry
points in the order a study uses them:

  build     a new basis, the count pass and the fill: the whole construction
            of one matrix from its two-body table
  fill      the fill alone, on a basis and row pointers in hand (another
            interaction on the same nucleus), with per-orbital energies
  onebody   the same with a one-body table in place of the energies
  batched   K interactions sharing one structure, element-major values
  host      tables from and matrix to page-locked host memory
  spmv      y = H x for K matrices (element-major values when K > 1)
  lanczos   the five lowest eigenvalues and the lowest vector of each matrix
  grad      the adjoint: d E0 / d (table entry) for given vectors
  eigen     E0 and its gradient through autograd (build, Lanczos, adjoint)
  batch     uneven instances: count, admission, build, Lanczos, adjoint

``exact`` states the results in 64 bits with plain torch: determinants are
enumerated, pairs are found by counting common orbitals, and matrix elements
come from the positions of the moved orbitals.
"""
from __future__ import annotations

import functools
import random

import numpy as np
import torch

from paper_1412_5989_gb300 import cih

HW = 20.0
NEV = 5

# (Z, N, Nmax, 2M): the spaces of this repository's configurations and tests,
# and neighbours of them: one species alone, few particles at high Nmax, many
# at low, odd A and odd 2M.  The last number is the stored nonzeros of one
# matrix in thousands.
SPACES = (
    (2, 2, 2, 0, 1), (2, 2, 3, 4, 4), (2, 3, 2, 1, 6), (3, 0, 4, 1, 18), (3, 3, 2, 0, 35), (1, 1, 6, 0, 71),
    (0, 4, 4, 0, 97), (1, 2, 5, 1, 100), (3, 4, 2, 1, 113), (2, 3, 4, 5, 156), (1, 2, 6, 1, 370), (4, 5, 2, 1, 714),
    (3, 4, 3, 1, 1100), (5, 5, 2, 0, 1377), (2, 2, 6, 0, 1399), (3, 3, 4, 4, 1453), (2, 5, 4, 1, 3187), (4, 5, 3, 5, 4632),
    (3, 4, 4, 1, 8011), (2, 3, 6, 1, 9144), (3, 3, 5, 0, 12683), (2, 5, 5, 1, 20068), (4, 4, 4, 4, 20724), (4, 4, 4, 0, 28937),
    (2, 6, 5, 0, 35965), (3, 4, 5, 1, 47127), (3, 3, 6, 0, 60237), (4, 5, 4, 1, 64323), (5, 5, 4, 4, 109001), (5, 6, 4, 5, 139524),
    (2, 6, 6, 4, 158634), (5, 6, 4, 1, 207050),
)


def listed():
    return [
        # the smallest build: a light nucleus, one table; launches and host set-up decide
        {"name": "build_3p3n_nmax2", "op": "build", "space": "3,3,2,0", "K": 1},
        # the headline workload, from nothing to 925 M stored nonzeros
        {"name": "build_4p4n_nmax6", "op": "build", "space": "4,4,6,0", "K": 1},
        # a new interaction on a basis in hand, with per-orbital energies: an ordinary fill
        {"name": "fill_4p4n_nmax4", "op": "fill", "space": "4,4,4,0", "K": 1},
        # odd A, odd 2M, kinetic-energy table, three interactions side by side (set-major)
        {"name": "onebody_5p6n_nmax4_k3", "op": "onebody", "space": "5,6,4,1", "K": 3},
        # an ensemble of 64 interactions on one structure: the batched configuration
        {"name": "batched_4p4n_nmax4_k64", "op": "batched", "space": "4,4,4,0", "K": 64},
        # a matrix for a host program: tables from and arrays to page-locked memory
        {"name": "host_4p4n_nmax4", "op": "host", "space": "4,4,4,0", "K": 1},
        # the adjoint at the headline size
        {"name": "grad_4p4n_nmax6", "op": "grad", "space": "4,4,6,0", "K": 1},
        # one product with the headline matrix: a caller's own eigensolver
        {"name": "spmv_4p4n_nmax6", "op": "spmv", "space": "4,4,6,0", "K": 1},
        # the smallest solve: every step of it is latency
        {"name": "lanczos_3p3n_nmax2", "op": "lanczos", "space": "3,3,2,0", "K": 1},
        # an ensemble of 64 matrices solved together (a mid-size nucleus: a solve takes some 140 products)
        {"name": "lanczos_3p4n_nmax4_k64", "op": "lanczos", "space": "3,4,4,1", "K": 64},
        # one optimisation step on an interaction: E0 forward, d E0 / d table backward
        {"name": "eigen_4p4n_nmax4", "op": "eigen", "space": "4,4,4,0", "K": 1},
        # the uneven batch: three nuclei, count to gradient in one call
        {"name": "batch_uneven", "op": "batch", "space": "3,3,6,0;4,4,4,0;5,6,4,1", "K": 1},
    ]


def draw(rng: random.Random):
    op = rng.choice(("build", "fill", "onebody", "batched", "host", "spmv", "lanczos", "grad", "eigen", "batch"))
    # values of one pass, in thousands; the solvers read the matrix a hundred times or more
    room = {"batched": 1850000, "spmv": 1850000, "lanczos": 210000, "host": 210000, "eigen": 65000}.get(op, 210000)
    want = 10 ** rng.uniform(0.5, 5.4)                       # stored nonzeros in thousands, spread over their logarithm
    near = sorted((s for s in SPACES if s[4] <= room), key=lambda s: abs(np.log(s[4] / want)))
    sp = rng.choice(near[:4])
    most = max(1, min({"batched": 64, "spmv": 64, "lanczos": 32, "fill": 8, "onebody": 8, "grad": 4}.get(op, 1), room // sp[4]))
    K = int(round(2 ** rng.uniform(0, np.log2(most)))) if most > 1 else 1
    text = "%d,%d,%d,%d" % sp[:4]
    if op == "batch":
        others = [s for s in SPACES if s[4] <= 70000]
        text = ";".join("%d,%d,%d,%d" % rng.choice(others)[:4] for _ in range(rng.randint(2, 4)))
    return {"op": op, "space": text, "K": K}


def _spaces(case):
    return [tuple(int(x) for x in s.split(",")) for s in case["space"].split(";")]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) + 77)


def _tables(B, K, g):
    """K two-body tables, N(0, 1) float32 per entry."""
    return torch.randn((K, max(B.tbme_len, 1)), generator=g, device="cuda")[:, : B.tbme_len].contiguous()


def prepare(case, seed):
    g, op, K = _gen(seed), case["op"], case["K"]
    if op == "batch":
        items = []
        for sp in _spaces(case):
            B = cih.Basis(*sp)
            items.append((B, _tables(B, K, g)))
        return {"op": op, "items": items}
    sp = _spaces(case)[0]
    B = cih.Basis(*sp)
    s = {"op": op, "K": K, "space": sp, "B": B, "T": _tables(B, K, g)}
    if op == "build":
        s["B"] = None                                        # run makes its own
        return s
    if op == "eigen":
        s["T"].requires_grad_(True)
        return s
    s["rowptr"], s["nnz"] = B.count()
    if op == "fill":
        s["e_sp"] = torch.rand(B.n_orb[0] + B.n_orb[1], generator=g, device="cuda", dtype=torch.float64) * 100.0
    elif op == "onebody":
        s["t1"] = torch.randn(B.onebody_len, generator=g, device="cuda", dtype=torch.float64) * 10.0
    elif op == "grad":
        psi = torch.randn((K, B.dim), generator=g, device="cuda", dtype=torch.float64)
        s["psi"] = psi / psi.norm(dim=1, keepdim=True)
    if op in ("fill", "onebody"):                            # output arrays reused from one interaction to the next
        s["col"] = torch.empty(s["nnz"], dtype=torch.int32, device="cuda")
        s["val"] = torch.empty((K, s["nnz"]), dtype=torch.float32, device="cuda")
    elif op in ("batched", "spmv", "lanczos") and K > 1:
        s["Til"] = cih.tbme_interleave(s["T"])
        s["col"] = torch.empty(s["nnz"], dtype=torch.int32, device="cuda")
        s["val"] = torch.empty((s["nnz"], K), dtype=torch.float32, device="cuda")
        if op != "batched":
            B.fill_batched(s["rowptr"], s["nnz"], s["Til"], K, HW, col=s["col"], val=s["val"])
    elif op == "batched":
        s["Til"] = cih.tbme_interleave(s["T"])
        s["col"] = torch.empty(s["nnz"], dtype=torch.int32, device="cuda")
        s["val"] = torch.empty((s["nnz"], 1), dtype=torch.float32, device="cuda")
    elif op in ("spmv", "lanczos"):
        s["col"], s["val"] = B.fill(s["rowptr"], s["nnz"], s["T"], HW)
    if op == "spmv":
        x = torch.randn((B.dim, K) if K > 1 else (B.dim,), generator=g, device="cuda", dtype=torch.float64)
        s["x"] = x / x.norm(dim=0)
    elif op == "host":
        s["T"] = s["T"].cpu().pin_memory()
        s["rowptr_h"] = torch.empty(B.dim + 1, dtype=torch.int64).pin_memory()
        s["col_h"] = torch.empty(s["nnz"], dtype=torch.int32).pin_memory()
        s["val_h"] = torch.empty((K, s["nnz"]), dtype=torch.float32).pin_memory()
    return s


def run(s):
    op = s["op"]
    if op == "build":
        B = cih.Basis(*s["space"])
        rowptr, nnz = B.count()
        col, val = B.fill(rowptr, nnz, s["T"], HW)
        return rowptr, col, val
    if op == "fill":
        return s["B"].fill(s["rowptr"], s["nnz"], s["T"], HW, s["e_sp"], col=s["col"], val=s["val"])
    if op == "onebody":
        return s["B"].fill_onebody(s["rowptr"], s["nnz"], s["T"], s["t1"], col=s["col"], val=s["val"])
    if op == "batched":
        return s["B"].fill_batched(s["rowptr"], s["nnz"], s["Til"], s["K"], HW, col=s["col"], val=s["val"])
    if op == "host":
        s["B"].build_to_host(s["T"], s["rowptr_h"], s["col_h"], s["val_h"], HW)
        return s["rowptr_h"], s["col_h"], s["val_h"]
    if op == "spmv":
        return s["B"].spmv(s["rowptr"], s["col"], s["val"], s["x"], element_major=s["K"] > 1)
    if op == "lanczos":
        ev, vec, _ = s["B"].lanczos(s["rowptr"], s["col"], s["val"], NEV, 300, 1e-8, element_major=s["K"] > 1)
        return ev, vec
    if op == "grad":
        return s["B"].tbme_grad(s["rowptr"], s["psi"])
    if op == "eigen":
        e0 = cih.lowest_eigenvalue(s["B"], s["T"], HW)
        return e0.detach(), torch.autograd.grad(e0.sum(), s["T"])[0]
    _, got = cih.solve_batch(s["items"], HW, NEV, 300, 1e-8)
    return [(r["evals"], r["grad"]) for r in got]


@functools.lru_cache(maxsize=None)
def _sizes(sp):
    B = cih.Basis(*sp)
    return B.dim, B.count()[1], B.tbme_len


def work(case):
    """Bytes: outputs written once, inputs (tables, vectors, a matrix where it
    is an input) read once.  Operations: a multiply and an add per stored
    nonzero and use.  A solve to five converged pairs cannot do without some
    forty products; each reads the matrix, which exceeds the cache but for the
    small spaces."""
    op, K = case["op"], case["K"]
    total = {"bytes": 0, "flops": 0}
    for sp in _spaces(case):
        dim, nnz, tl = _sizes(sp)
        matrix, tables, m = nnz * (4 + 4 * K) + 8 * (dim + 1), 4 * tl * K, min(40, dim)
        b, f = {
            "build": (matrix + tables, 0), "fill": (matrix + tables, 0), "onebody": (matrix + tables, 0),
            "batched": (matrix + tables, 0), "host": (matrix + tables, 0),
            "grad": (8 * K * (dim + tl), 2 * K * nnz),
            "spmv": (matrix + 16 * K * dim, 4 * K * nnz),
            "lanczos": (m * matrix + 8 * K * dim, 4 * K * nnz * m),
            "eigen": ((m + 1) * matrix + 2 * tables, 4 * K * nnz * m + 2 * K * nnz),
            "batch": ((m + 1) * matrix + 3 * tables, 4 * K * nnz * m + 2 * K * nnz),
        }[op]
        total["bytes"] += b
        total["flops"] += f
    return total


# ---- the same results in 64 bits, in plain torch -----------------------------

def _min_quanta(Z):
    q, n = 0, 0
    while Z > 0:
        k = min(Z, (n + 1) * (n + 2))
        q, Z, n = q + k * n, Z - k, n + 1
    return q, n - 1                                          # quanta, highest shell (-1: none)


def _orbitals(Z, Nmax):
    if Z == 0:
        return []
    top = _min_quanta(Z)[1] + Nmax
    return [(N, l, j, m) for N in range(top + 1) for l in range(N % 2, N + 1, 2) for j in (2 * l - 1, 2 * l + 1) if j > 0
            for m in range(-j, j + 1, 2)]


def _subdets(orb, Z, cap):
    """Every subset of Z orbitals with at most `cap` quanta: (2M, parity, N, bits, members), ascending."""
    out = []

    def go(k, left, q, m, bits, members):
        if left == 0:
            out.append((m, q % 2, q, bits, members))
            return
        for a in range(k, len(orb) - left + 1):
            if q + orb[a][0] * left > cap:                   # orbitals are ordered by shell
                break
            go(a + 1, left - 1, q + orb[a][0], m + orb[a][3], bits | 1 << a, members + (a,))

    go(0, Z, 0, 0, 0, ())
    return sorted(out)


@functools.lru_cache(maxsize=2)
def _plain(sp):
    """Occupied orbitals of every basis state, the pair table (group offset and
    size, place in the group, sign of the order given) and the one-body layout."""
    Z, N, Nmax, twoM = sp
    op, on = _orbitals(Z, Nmax), _orbitals(N, Nmax)
    q0p, q0n = _min_quanta(Z)[0], _min_quanta(N)[0]
    lim = q0p + q0n + Nmax
    P, Q = _subdets(op, Z, lim - q0n), _subdets(on, N, lim - q0p)
    by = {}
    for n in Q:
        by.setdefault((n[0], n[1]), []).append(n)
    rows = [p[4] + tuple(len(op) + b for b in n[4]) for p in P
            for n in by.get((twoM - p[0], (lim - p[2]) % 2), ()) if p[2] + n[2] <= lim]
    orb = op + on
    T = len(orb)
    off, size = np.full((T, T), -1, np.int64), np.zeros((T, T), np.int64)
    place, sign = np.zeros((T, T), np.int64), np.ones((T, T), np.int64)
    at = 0
    spans = {"pp": (range(len(op)),) * 2, "nn": (range(len(op), T),) * 2, "pn": (range(len(op)), range(len(op), T))}
    for ch, (first, second) in spans.items():
        zz, nn = {"pp": (Z - 2, N), "nn": (Z, N - 2), "pn": (Z - 1, N - 1)}[ch]
        if zz < 0 or nn < 0:
            continue
        most = lim - _min_quanta(zz)[0] - _min_quanta(nn)[0]
        groups = {}
        for a in first:
            for b in second:
                if a < b and orb[a][0] + orb[b][0] <= most:
                    groups.setdefault((orb[a][3] + orb[b][3], (orb[a][0] + orb[b][0]) % 2), []).append((a, b))
        for key in sorted(groups):
            members = groups[key]
            for u, (a, b) in enumerate(members):
                off[a, b] = off[b, a] = at
                size[a, b] = size[b, a] = len(members)
                place[a, b] = place[b, a] = u
                sign[b, a] = -1
            at += len(members) * (len(members) + 1) // 2
    one = np.full((T, T), -1, np.int64)
    at = 0
    for species in (range(len(op)), range(len(op), T)):
        groups = {}
        for a in species:
            groups.setdefault((orb[a][3], orb[a][0] % 2), []).append(a)
        for key in sorted(groups):
            for u, a in enumerate(groups[key]):
                for c in groups[key][u:]:
                    one[a, c] = one[c, a] = at
                    at += 1
    dev = {k: torch.from_numpy(v).cuda() for k, v in (("off", off), ("size", size), ("place", place), ("sign", sign), ("one", one))}
    dev["occ"] = torch.tensor(rows, dtype=torch.int64, device="cuda")
    dev["shell"] = torch.tensor([o[0] for o in orb], dtype=torch.float64, device="cuda")
    return dev


def _entry(D, a, b, c, d):
    """Table index and sign of V_{ab,cd}."""
    u, v = D["place"][a, b], D["place"][c, d]
    lo, hi, n = torch.minimum(u, v), torch.maximum(u, v), D["size"][a, b]
    return D["off"][a, b] + lo * n - lo * (lo - 1) // 2 + (hi - lo), D["sign"][a, b] * D["sign"][c, d]


def _chunks(D):
    """The stored elements (i, j), j >= i, of a run of rows, and their terms:
    yields i, j, [(elements, table index, sign)], [(elements, a, c, sign)]."""
    occ = D["occ"]
    dim, A = occ.shape
    full = torch.zeros((dim, D["shell"].numel()), device="cuda").scatter_(1, occ, 1.0)
    step = max(64, min(2048, (1 << 28) // max(dim, 1)))
    pairs = torch.triu_indices(A, A, 1, device="cuda")
    for r0 in range(0, dim, step):
        r1 = min(dim, r0 + step)
        common = full[r0:r1] @ full.t()
        i, j = torch.nonzero(common >= A - 2 - 0.5, as_tuple=True)
        i = i + r0
        keep = j >= i
        i, j = i[keep], j[keep]
        oi, oj = occ[i], occ[j]
        eq = oi[:, :, None] == oj[:, None, :]
        bi, bj = ~eq.any(2), ~eq.any(1)                      # moved orbitals of the bra and of the ket
        n = bi.sum(1)
        places = torch.arange(A, device="cuda")
        two, terms, ones = [], [], []
        e = torch.nonzero(n == 2)[:, 0]
        if e.numel():
            pi, pj = torch.nonzero(bi[e])[:, 1].view(-1, 2), torch.nonzero(bj[e])[:, 1].view(-1, 2)
            a, c = oi[e].gather(1, pi), oj[e].gather(1, pj)
            idx, sg = _entry(D, a[:, 0], a[:, 1], c[:, 0], c[:, 1])
            terms.append((e, idx, sg * (1 - 2 * ((pi.sum(1) + pj.sum(1)) % 2))))
        e = torch.nonzero(n == 1)[:, 0]
        if e.numel():
            pi, pj = torch.nonzero(bi[e])[:, 1], torch.nonzero(bj[e])[:, 1]
            a, c = oi[e, pi], oj[e, pj]
            ph = 1 - 2 * ((pi + pj) % 2)
            ones.append((e, a, c, ph))
            for k in range(A):
                use = pi != k
                spect = oi[e, k][use]
                idx, sg = _entry(D, a[use], spect, c[use], spect)
                terms.append((e[use], idx, sg * ph[use]))
        e = torch.nonzero(n == 0)[:, 0]
        for k in range(A):
            ones.append((e, oi[e, k], oi[e, k], torch.ones_like(e)))
        for x, y in pairs.t().tolist():
            idx, sg = _entry(D, oi[e, x], oi[e, y], oi[e, x], oi[e, y])
            terms.append((e, idx, sg))
        yield i, j, terms, ones


def _exact_matrix(sp, T, e_sp=None, t1=None):
    """(rowptr, col, values (K, nnz) float64) of the stored half."""
    D = _plain(sp)
    t = T.double()
    energies = HW * (D["shell"] + 1.5) if e_sp is None else e_sp
    cols, vals, counts = [], [], torch.zeros(D["occ"].shape[0], dtype=torch.int64, device="cuda")
    for i, j, terms, ones in _chunks(D):
        v = torch.zeros((i.numel(), t.shape[0]), dtype=torch.float64, device="cuda")
        for e, idx, sg in terms:
            v.index_add_(0, e, t[:, idx].t() * sg[:, None])
        for e, a, c, sg in ones:
            if t1 is not None:
                v.index_add_(0, e, (t1[D["one"][a, c]] * sg)[:, None].expand(-1, t.shape[0]))
            elif e.numel():
                v.index_add_(0, e, torch.where(a == c, energies[a], 0.0)[:, None].expand(-1, t.shape[0]))
        cols.append(j.to(torch.int32))
        vals.append(v)
        counts.index_add_(0, i, torch.ones_like(i))
    rowptr = torch.zeros(counts.numel() + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = counts.cumsum(0)
    return rowptr, torch.cat(cols), torch.cat(vals).t()


def _exact_grad(sp, psi):
    D = _plain(sp)
    g = torch.zeros((psi.shape[0], _sizes(sp)[2]), dtype=torch.float64, device="cuda")
    for i, j, terms, _ in _chunks(D):
        w = psi[:, i] * psi[:, j] * torch.where(i == j, 1.0, 2.0).double()
        for e, idx, sg in terms:
            g.index_add_(1, idx, w[:, e] * sg)
    return g


def _product(rowptr, col, val, x):
    """H x in float64 from the stored half; val (nnz,), x (dim,)."""
    y = torch.zeros_like(x)
    nnz, dim, step = col.numel(), x.numel(), 1 << 26
    for k in range(0, nnz, step):
        at = torch.arange(k, min(nnz, k + step), device="cuda")
        i = torch.searchsorted(rowptr, at, right=True) - 1
        c, v = col[k:k + step].long(), val[k:k + step].double()
        y.index_add_(0, i, v * x[c])
        y.index_add_(0, c, torch.where(c != i, v * x[i], 0.0))
    return y


def _eigen(rowptr, col, val, nev):
    """The nev lowest eigenvalues and the lowest vector, by Lanczos with full
    reorthogonalisation on the whole matrix, to 1e-12."""
    dim = rowptr.numel() - 1
    i = torch.repeat_interleave(torch.arange(dim, device="cuda"), rowptr[1:] - rowptr[:-1])
    c, v = col.long(), val.double()
    off = i != c
    H = torch.sparse_coo_tensor(torch.stack((torch.cat((i, c[off])), torch.cat((c, i[off])))),
                                torch.cat((v, v[off])), (dim, dim)).coalesce().to_sparse_csr()
    if dim <= 3000:
        w, U = torch.linalg.eigh(H.to_dense())
        return w[:nev].cpu(), U[:, 0]
    most = min(dim, 400)
    V = torch.zeros((most + 1, dim), dtype=torch.float64, device="cuda")
    x = torch.arange(dim, dtype=torch.float64, device="cuda")
    V[0] = 1.0 + 0.25 * torch.sin(1.7 * x)
    V[0] /= V[0].norm()
    al, be = [], []
    for m in range(most):
        w = H @ V[m]
        a = 0.0
        for _ in range(2):
            h = V[: m + 1] @ w
            w -= h @ V[: m + 1]
            a += float(h[m])
        al.append(a)
        be.append(float(w.norm()))
        done = m + 1 == most or be[-1] < 1e-11
        if m % 10 == 9 or done:
            b = torch.diag(torch.tensor(be[:-1], dtype=torch.float64), 1)
            th, Z = torch.linalg.eigh(torch.diag(torch.tensor(al, dtype=torch.float64)) + b + b.t())
            if done or (m >= nev and float((be[-1] * Z[-1, :nev].abs()).max()) < 1e-11 * max(1.0, float(th[0].abs()))):
                break
        V[m + 1] = w / be[-1]
    u = Z[:, 0].cuda() @ V[: len(al)]
    return th[:nev], u / u.norm()


def _exact_solve(sp, T):
    """Eigenvalues and gradient for one set, from the values as stored (rounded to FP32)."""
    rowptr, col, val = _exact_matrix(sp, T)
    w, u = _eigen(rowptr, col, val[0].float(), NEV)
    return w, _exact_grad(sp, u[None])


def exact(case, seed):
    op, K = case["op"], case["K"]
    sizes = [_sizes(sp) for sp in _spaces(case)]
    nnz = sum(s[1] for s in sizes)
    s = prepare(case, seed)
    if op == "batch":
        out = []
        for (B, T), sp, (dim, n, _) in zip(s["items"], _spaces(case), sizes):
            if n > 30_000_000 or dim < NEV:
                out.append((None, None))
                continue
            w, g = _exact_solve(sp, T.detach())
            out.append((w[None], g))
        return out if any(w is not None for w, _ in out) else None
    sp = _spaces(case)[0]
    if op == "spmv":
        val = s["val"] if K > 1 else s["val"].t()
        x = s["x"] if K > 1 else s["x"][:, None]
        if nnz * K > 2_000_000_000:
            return None
        y = torch.stack([_product(s["rowptr"], s["col"], val[:, k].contiguous(), x[:, k].contiguous()) for k in range(K)], 1)
        return y if K > 1 else y[:, 0]
    if op == "lanczos":
        # the lowest vector is defined up to its sign; no value is given for it
        if nnz > 30_000_000 or K > 8 or sizes[0][0] < NEV:
            return None
        val = s["val"] if K > 1 else s["val"].t()
        return torch.stack([_eigen(s["rowptr"], s["col"], val[:, k].contiguous(), NEV)[0] for k in range(K)]), None
    if nnz > 30_000_000:
        return None
    if op == "grad":
        return _exact_grad(sp, s["psi"])
    if op == "eigen":
        w, g = _exact_solve(sp, s["T"].detach())
        return w[:1], g
    T = s["T"].cuda()
    rowptr, col, val = _exact_matrix(sp, T, s.get("e_sp"), s.get("t1"))
    if op in ("build", "host"):
        return rowptr, col, val
    return (col, val) if op != "batched" else (col, val.t())
