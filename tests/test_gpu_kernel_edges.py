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
