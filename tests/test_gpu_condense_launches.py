"""The condensation kernels of small launches, large launches and large primes, each on whole launches: a pool of
distinct matrices spread over the nodes, most warps without a zero pivot, some of them full of zero pivots, a ragged
last CTA.  Integer work: every determinant equals the oracle's."""
import numpy as np
import pytest

from helpers import ensure_lib, random_residue_mats
from oracle import modular

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _pool(n, p, rng):
    """(matrices [48][n][n], determinants): 24 random, 8 with entries next to p, then 16 that meet zero pivots."""
    mats = random_residue_mats(rng, 1, 48, n, [p])[0]
    mats[24:32] = np.uint64(p - 1) - rng.integers(0, 1000, (8, n, n)).astype(np.uint64)
    mats[32:40] = np.array([0, 1, p - 2, p - 1], dtype=np.uint64)[rng.integers(0, 4, (8, n, n))]
    for k in range(40, 46):  # zeros that move the first pivot, a zero leading block, a zero second block
        mats[k, :1 + k % 3, :1 + k % 3] = 0
    if n > 4:
        mats[45, 2:4, 2:4] = mats[45, :2, :2] = 0
    mats[46, n - 1] = mats[46, 0]
    mats[47] = np.triu(mats[47])
    return mats, [modular.det_mod_p(m.astype(object).tolist(), p) for m in mats]


def _grid(matrices):
    """Degrees of a two-variable grid of at least ``matrices`` nodes, hardly more."""
    a = int(matrices ** 0.5)
    return a - 1, -(-matrices // a) - 1


def _check(n, matrices, primes, nprimes, lo):
    """Launch condensation of ``matrices`` nodes for primes [lo, lo + len(primes)) of a plan of ``nprimes``."""
    from paper_2010_12117_gb300.binding import Plan, as_u32
    D = _grid(matrices)
    pl = Plan(n, tuple(max(1, -(-x // n)) for x in D), nprimes, det_degs=D)
    assert matrices <= pl.G < matrices + 2000
    hi = lo + primes
    evals = torch.empty(primes, n * n, pl.G, dtype=torch.int32, device="cuda")
    want = []
    g = np.arange(pl.G)
    odd = (g // 32) % 9 == 5  # warps (of one lane per matrix) with zero pivots
    pick = torch.from_numpy(np.where(odd, 32 + g % 16, (g * 7 + g // 32) % 32)).cuda()
    for q in range(lo, hi):
        mats, dets = _pool(n, pl.primes[q], np.random.default_rng(1000 * n + q))
        pool = torch.from_numpy(mats.reshape(48, n * n).T.astype(np.uint32).view(np.int32).copy()).cuda()
        torch.index_select(pool, 1, pick, out=evals[q - lo])
        want.append(np.array(dets, dtype=np.uint32)[pick.cpu().numpy()])
    det = torch.empty(primes * pl.G, dtype=torch.int32, device="cuda")
    pl.condense(evals.reshape(-1), lo, hi, det)
    got = as_u32(det).reshape(primes, pl.G)
    for q in range(primes):
        bad = np.flatnonzero(got[q] != want[q])
        assert bad.size == 0, (n, matrices, lo + q, bad[:8])


@pytest.mark.parametrize("n", [2, 10, 14, 15, 17, 18, 19, 21, 23, 25, 26, 27, 28, 32])
@pytest.mark.parametrize("matrices", [97, 25000])
def test_primes_on_both_sides_of_the_fold_limit(n, matrices):
    """Primes 66 .. 68 of the table: one below the limit of the three- and five-product sums, two above it."""
    _check(n, matrices, 3, 70, 66)


@pytest.mark.parametrize("n", [10, 15])
def test_long_ranges_split_at_the_fold_limit(n):
    """More than 2^18 matrices below the limit: the part above it is a launch of its own."""
    _check(n, 270_000, 2, 69, 66)


def _launches(n, prime):
    """(smallest, largest) launch up to 140000 matrices of every kernel of order n."""
    from paper_2010_12117_gb300 import binding
    sizes = [97, 7000, 7297, 9700, 9729, 14500, 14593, 19400, 19457, 21800, 21889, 32700, 32769, 65000, 65537,
             131000, 131073, 140000]
    kernels = {}
    for m in sizes:
        kernels.setdefault(binding.condense_launch(n, m, prime), []).append(m)
    return sorted({m for ms in kernels.values() for m in (ms[0], next((x for x in ms[1:] if x > 21900), ms[-1]))})


@pytest.mark.parametrize("n", range(1, 33))
def test_every_kernel_of_an_order(n):
    """Each kernel the launch rule names for order n, in its smallest launch and one of several waves."""
    for matrices in _launches(n, 0):
        _check(n, matrices, 1, 1 + n % 3, n % 3)
