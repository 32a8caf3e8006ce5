"""First-variable evaluation passes large enough to be split by the length of their rows: every split, with whole
outputs compared with 64-bit arithmetic.  Integer work: every comparison is bit-exact."""
import numpy as np
import pytest

from helpers import ensure_lib

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


N = 32
FILL = 152 * 4096   # columns that fill the chip
BYTES = 128_000_000  # outputs from which rows off the sector grid have splits of their own


def _powers(pl, q, v, count):
    p = pl.primes[q]
    rows = [[pow(pow(pl.roots[q][v], e, p), i, p) for e in pl.node_exps[v]] for i in range(count)]
    return torch.tensor(rows, dtype=torch.int64, device="cuda")


def _check(lin, rows, full=False, large=False):
    """Coefficients at both ends of int32; ``rows`` nodes of x_2, a ragged number of cosets of x_1; as many primes as
    fill the chip, or as make a ``large`` output."""
    from paper_2010_12117_gb300.binding import Plan
    d2 = max(1, -(-(rows - 1) // N))
    lp = 1 << max(0, lin - 1).bit_length()
    D0 = min(N * (lin - 1), 2 * lp + (2 if lp > 2 else 0))
    if large and lin > 1:  # all the nodes of x_1 but a ragged few
        D0 = N * (lin - 1) - (1 if lin == 2 else 3)
    P = -(-FILL // (N * N * rows))
    if large:
        P = -(-BYTES // (4 * N * N * rows * (D0 + 1)))
    pl = Plan(N, (lin - 1, d2), P, full_grid=full, det_degs=(D0, rows - 1))
    assert not large or 4 * pl.P * N * N * pl.G >= BYTES
    rng = np.random.default_rng(100 * lin + rows)
    c = rng.integers(-2 ** 31, 2 ** 31, (N * N, lin, d2 + 1)).astype(np.int32)
    c[0], c[-1] = -2 ** 31, 2 ** 31 - 1
    coeffs = torch.from_numpy(c).cuda()
    evals = torch.full((pl.P, N * N, pl.M[0], pl.M[1]), -1, dtype=torch.int32, device="cuda")
    pl.eval(coeffs.reshape(-1), 0, pl.P, evals.reshape(-1), pl.workspace(pl.P))
    for q in sorted({0, pl.P - 1}):
        p = pl.primes[q]
        x, y = _powers(pl, q, 0, lin), _powers(pl, q, 1, d2 + 1)
        want = torch.zeros(evals.shape[1:], dtype=torch.int64, device="cuda")
        for i in range(lin):
            part = torch.zeros(N * N, pl.M[1], dtype=torch.int64, device="cuda")
            for j in range(d2 + 1):
                part = (part + (coeffs[:, i, j].long() % p)[:, None] * y[j]) % p
            want = (want + x[i][None, :, None] * part[:, None, :]) % p
        assert torch.equal(evals[q].long() & 0xffffffff, want), (lin, rows, q)


@pytest.mark.parametrize("lin", [1, 2, 3, 4, 5, 6, 8])
@pytest.mark.parametrize("rows", [33, 65, 127, 129, 511, 513,  # off the sector grid: one, two, four columns
                                  40, 64, 120, 128, 136, 1024])  # on it: flattened, two columns
def test_node_grid(lin, rows):
    _check(lin, rows)


@pytest.mark.parametrize("lin", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("rows", [13, 31, 47, 65, 79,  # flattened, a limit on the CTAs per SM
                                  49, 63, 81, 95,     # a row's warps one CTA's
                                  97, 127, 129, 383,  # two columns per thread, 64 and 256 threads
                                  385, 1023, 1025])   # four
def test_outputs_larger_than_l2(lin, rows):
    _check(lin, rows, large=True)


@pytest.mark.parametrize("lin", [1, 4])
def test_long_rows_on_the_grid(lin):
    """At most four coefficients of x_1: four columns per thread."""
    _check(lin, 8192)


@pytest.mark.parametrize("lin", [2, 3, 5, 8])
@pytest.mark.parametrize("rows", [64, 128, 512])
def test_power_of_two_grid(lin, rows):
    _check(lin, rows, full=True)


@pytest.mark.parametrize("tail", [(608,), (1024,), (96, 84)])
def test_windows_of_rows(tail):
    """Slabs of nodes of x_1 (rows of 609 nodes; of 1025 and 8245, padded to the grid) against one evaluation of all
    of them."""
    from paper_2010_12117_gb300.binding import Plan
    pl = Plan(N, (3,) + tuple(-(-x // N) for x in tail), 1, det_degs=(26,) + tail)
    rng = np.random.default_rng(sum(tail))
    c = torch.from_numpy(rng.integers(-2 ** 31, 2 ** 31, N * N * pl.E).astype(np.int32)).cuda()
    evals = torch.empty(N * N * pl.G, dtype=torch.int32, device="cuda")
    want, got = (torch.empty(pl.G, dtype=torch.int32, device="cuda") for _ in range(2))
    pl.eval(c, 0, 1, evals, pl.workspace(1))
    pl.condense(evals, 0, 1, want)
    for slab in (4, 12):
        got.fill_(-1)
        ws = torch.empty(pl.stream_ws_words(slab), dtype=torch.int32, device="cuda")
        pl.eval_condense(c, 0, 1, got, ws)
        assert torch.equal(got, want), slab
