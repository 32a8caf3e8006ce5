"""Edges of the interpolation and condensation kernels: tile remainders, the
smallest and largest of their ranges, residues at both ends of [0, p).
Integer work: every comparison is bit-exact."""
import numpy as np
import pytest

from helpers import ensure_lib, evals_tensor
from oracle import modular

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _u32(t):
    from paper_2010_12117_gb300.binding import as_u32
    return as_u32(t)


def _values(coeffs, nodes, p):
    """Values of the polynomial with coefficient tensor ``coeffs`` (python
    ints) at the product grid of ``nodes`` (per variable), mod p."""
    t = coeffs.astype(object)
    for v, xs in enumerate(nodes):
        V = np.array([[pow(x, e, p) for e in range(t.shape[v])] for x in xs], dtype=object)
        t = np.moveaxis(np.tensordot(V, t, axes=(1, v)) % p, 0, v)
    return t


@pytest.mark.parametrize("n,degs,D", [
    (3, (7,), (0,)), (3, (7,), (6,)),              # no whole coset: 1 and 7 nodes of one
    (3, (7,), (7,)), (3, (7,), (14,)),             # one coset; one and 7 of the next
    (8, (7,), (55,)), (9, (7,), (62,)),            # 7 cosets; 7 and 7 nodes
    (5, (3,), (15,)), (5, (3,), (14,)), (6, (3,), (18,)),  # cosets of 4: remainders 0, 3, 3
    (9, (1,), (9,)), (9, (1,), (8,)),              # cosets of 2
    (1, (0, 3), (0, 3)),                           # a variable without degree
    (24, (3, 1), (72, 24)),                        # rows of 25 words, 73 strided columns
    (32, (1, 6), (32, 192)),                       # rows of 193 words
    (6, (2, 3, 1), (11, 17, 5)),                   # three passes, every remainder
    (2, (5, 200), (10, 399)),                      # 50 cosets of 8
])
def test_interp_recovers_coefficients(n, degs, D):
    from paper_2010_12117_gb300.binding import Plan
    P = 2
    pl = Plan(n, degs, P, det_degs=D)
    rng = np.random.default_rng(sum(D) + n)
    box = tuple(x + 1 for x in D)
    vals, want = [], []
    for q, p in enumerate(pl.primes):
        c = rng.integers(0, p, box)
        c.flat[0], c.flat[-1] = p - 1, p - 1
        nodes = [[pow(pl.roots[q][v], e, p) for e in pl.node_exps[v]] for v in range(len(D))]
        vals.append(_values(c, nodes, p).reshape(-1).astype(np.uint32))
        want.append(c.reshape(-1).astype(np.uint32))
    det = torch.from_numpy(np.concatenate(vals).view(np.int32)).cuda()
    res = torch.empty(P * pl.C, dtype=torch.int32, device="cuda")
    pl.interp(det, 0, P, res, pl.workspace(P))
    assert np.array_equal(_u32(res), np.concatenate(want))


def test_interp_wide_passes_match_small_ones():
    """Many columns (whole 64-column tiles and a ragged one) against the same
    columns interpolated one prime at a time through another tile size."""
    from paper_2010_12117_gb300.binding import Plan
    n, degs, P = 16, (3, 2, 1), 9
    pl = Plan(n, degs, P)
    gen = torch.Generator(device="cuda").manual_seed(5)
    det = torch.cat([torch.randint(0, p, (pl.G,), generator=gen, dtype=torch.int32, device="cuda")
                     for p in pl.primes])
    res = torch.empty(P * pl.C, dtype=torch.int32, device="cuda")
    one = torch.empty_like(res)
    pl.interp(det, 0, P, res, pl.workspace(P))
    for q in range(P):
        pl.interp(det[q * pl.G:(q + 1) * pl.G], q, q + 1, one[q * pl.C:(q + 1) * pl.C], pl.workspace(1))
    assert torch.equal(res, one)


@pytest.mark.parametrize("n", list(range(2, 33)))
def test_condense_residues_at_the_ends(n):
    """Entries from {0, 1, p - 2, p - 1}: the largest sums of products the
    fast pass reduces, zero pivots and zero block determinants at every step,
    on the smallest and the largest primes a plan of 68 primes holds (one of
    them above the limit of the five-product reduction)."""
    from paper_2010_12117_gb300.binding import Plan
    pl = Plan(n, (1,), 68)
    picks = [0, 40, 67]  # 1863319553, a smaller prime, the first above 1865126253
    assert pl.primes[67] > 1865126253 >= max(pl.primes[:67])
    rng = np.random.default_rng(n)
    for q in picks:
        p = pl.primes[q]
        pool = np.array([0, 1, p - 2, p - 1], dtype=np.uint64)
        mats = pool[rng.integers(0, 4, (1, pl.G, n, n))]
        mats[0, 0] = p - 1                                            # rank 1
        mats[0, 1] = np.where(np.eye(n, dtype=bool), p - 1, pool[1])  # p - 1 on the diagonal, 1 elsewhere
        det = torch.empty(pl.G, dtype=torch.int32, device="cuda")
        pl.condense(evals_tensor(mats, pl.G), q, q + 1, det)
        want = [modular.det_mod_p(mats[0, g].astype(object).tolist(), p) for g in range(pl.G)]
        assert _u32(det).tolist() == want, (n, p)


def _check_nodes(pl, terms, got, nodes, q):
    """``got(g)`` against the sum of ``terms`` (coefficient, exponents) at
    node g of prime q."""
    p, ws = pl.primes[q], pl.roots[q]
    for g in nodes:
        s = [pl.node_exps[v][i] for v, i in enumerate(modular.grid_index(g, pl.M))]
        want = sum(c * pow(ws[0], s[0] * e[0], p) * pow(ws[1], s[1] * e[1], p) *
                   (pow(ws[2], s[2] * e[2], p) if len(e) > 2 else 1) for c, e in terms) % p
        assert got(g) == want, (q, g)


@pytest.mark.parametrize("lin", range(1, 9))
@pytest.mark.parametrize("rows,full", [(361, False), (545, False), (544, False), (97, False), (4, True)])
def test_eval_x1_pass(lin, rows, full):
    """The first variable's pass with 1 to 8 coefficients: one, two and four
    columns per thread, rows on and off the 32-byte grid, ragged ends of rows
    and of cosets, and the power-of-two grid."""
    from paper_2010_12117_gb300.binding import Plan
    n, P = 24, 3
    d2 = max(1, -(-(rows - 1) // n))
    D1 = n * (lin - 1) - (3 if lin > 2 else 0)
    pl = Plan(n, (lin - 1, d2), P, full_grid=full, det_degs=(D1, rows - 1))
    rng = np.random.default_rng(100 * lin + rows)
    c = rng.integers(-2 ** 31, 2 ** 31, (n * n, lin, d2 + 1)).astype(np.int32)
    coeffs = torch.from_numpy(c.reshape(-1)).cuda()
    evals = torch.empty(P * n * n * pl.G, dtype=torch.int32, device="cuda")
    pl.eval(coeffs, 0, P, evals, pl.workspace(P))
    ev = evals.reshape(P, n * n, pl.G)
    nodes = sorted({0, pl.M[1] - 1, pl.G - pl.M[1], pl.G - 1, *(int(x) for x in rng.integers(0, pl.G, 12))})
    for q in (0, P - 1):
        for e in (0, int(rng.integers(1, n * n - 1)), n * n - 1):
            row = _u32(ev[q, e])
            terms = [(int(c[e, i, j]), (i, j)) for i in range(lin) for j in range(d2 + 1)]
            _check_nodes(pl, terms, lambda g: int(row[g]), nodes, q)


def test_eval_rows_beyond_32_bit_offsets():
    """One entry of 15 x 8191 x 8191 nodes: its rows span more than 4 GB."""
    from paper_2010_12117_gb300.binding import Plan
    n, degs = 2, (7, 4095, 4095)
    pl = Plan(n, degs, 1)
    pl.set_entry_map(np.array([0, -1, -1, 0], dtype=np.int32), 1)
    rng = np.random.default_rng(8)
    terms = [(int(rng.integers(-2 ** 31, 2 ** 31)), tuple(int(rng.integers(0, d + 1)) for d in degs)) for _ in range(6)]
    coeffs = torch.zeros([d + 1 for d in degs], dtype=torch.int32, device="cuda")
    for c, e in terms:
        coeffs[e] = c
    evals = torch.empty(pl.entries * pl.G, dtype=torch.int32, device="cuda")
    pl.eval(coeffs.reshape(-1), 0, 1, evals, pl.workspace(1))
    assert int(evals[pl.G:].count_nonzero()) == 0  # the zero entry
    nodes = [0, pl.G - 1, *(int(x) for x in rng.integers(0, pl.G, 60))]
    got = evals[torch.tensor(nodes, device="cuda")].cpu().numpy().view(np.uint32)
    at = dict(zip(nodes, got.tolist()))
    _check_nodes(pl, terms, at.__getitem__, nodes, 0)
