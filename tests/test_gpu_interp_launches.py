"""Interpolation passes by the kernels that large and small passes take: four coefficients per thread, one with its
tables in shared memory, one with them in global memory, every coset size and remainder.  Integer work: every
coefficient equals the one the values were made from."""
import numpy as np
import pytest

from helpers import ensure_lib

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _values(c, nodes, p):
    """Values on the product grid of ``nodes`` of the polynomial with coefficients ``c``, by Horner's rule."""
    t = c.astype(np.uint64)
    for v, xs in enumerate(nodes):
        t = np.moveaxis(t, v, 0)
        x = np.array(xs, dtype=np.uint64).reshape((-1,) + (1,) * (t.ndim - 1))
        acc = np.zeros((len(xs),) + t.shape[1:], dtype=np.uint64)
        for e in range(t.shape[0] - 1, -1, -1):
            acc = (acc * x + t[e]) % np.uint64(p)
        t = np.moveaxis(acc, 0, v)
    return t


def _check(n, degs, D, P):
    from paper_2010_12117_gb300.binding import Plan, as_u32
    pl = Plan(n, degs, P, det_degs=D)
    rng = np.random.default_rng(sum(D) + 7 * n)
    det = np.empty((P, pl.G), dtype=np.uint32)
    want = {}
    for q, p in enumerate(pl.primes):
        if q not in (0, P // 2, P - 1):  # any values do: their coefficients are not compared
            det[q] = rng.integers(0, p, pl.G)
            continue
        c = rng.integers(0, p, tuple(x + 1 for x in D))
        c.flat[0], c.flat[-1] = p - 1, p - 1
        nodes = [[pow(pl.roots[q][v], e, p) for e in pl.node_exps[v]] for v in range(len(D))]
        det[q] = _values(c, nodes, p).reshape(-1)
        want[q] = c.reshape(-1).astype(np.uint32)
    dev = torch.from_numpy(det.reshape(-1).view(np.int32)).cuda()
    res = torch.empty(P * pl.C, dtype=torch.int32, device="cuda")
    pl.interp(dev, 0, P, res, pl.workspace(P))
    got = as_u32(res).reshape(P, pl.C)
    for q, w in want.items():
        assert np.array_equal(got[q], w), (n, degs, D, q, np.flatnonzero(got[q] != w)[:8])


@pytest.mark.parametrize("n,d,nodes", [
    (32, 1, 16), (32, 1, 19), (32, 1, 20), (32, 1, 23),  # cosets of 2: 8 to 11 whole ones, remainders 0, 1, 0, 1
    (32, 3, 32), (32, 3, 39), (32, 3, 41), (32, 3, 46),  # cosets of 4: remainders 0, 3, 1, 2
    (32, 7, 64), (32, 7, 77), (32, 7, 81), (32, 7, 95),  # cosets of 8: remainders 0, 5, 1, 7
])
def test_large_passes(n, d, nodes):
    """24 primes of ``nodes`` x 1000 nodes: more than 256 threads' work per SM in each pass, 1000 strided columns
    (a ragged tile) and then rows of 1000 words."""
    _check(n, (d, 32), (nodes - 1, 999), 24)


@pytest.mark.parametrize("n,degs,D,P", [
    (10, (7,), (63,), 2), (11, (7,), (71,), 2), (11, (7,), (74,), 1),  # 8 and 9 whole cosets: the staging limit
    (24, (7,), (168,), 4), (32, (3,), (96,), 1), (32, (1,), (32,), 1), (32, (2,), (63,), 3),
    (10, (50,), (479,), 1), (10, (50,), (497,), 1), (11, (50,), (519,), 2),  # tables on both sides of 16 KB
    (8, (5, 200), (40, 1600), 1), (24, (40, 3), (960, 72), 3),  # few columns of long rows, few long strided ones
    (19, (200,), (3800,), 2), (2, (7, 7), (14, 14), 3), (2, (4, 4), (8, 8), 1), (3, (1, 7, 0), (3, 20, 0), 2),
])
def test_small_passes(n, degs, D, P):
    _check(n, degs, D, P)
