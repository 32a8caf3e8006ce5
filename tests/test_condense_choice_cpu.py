"""Which condensation kernel a launch takes (a host rule on order, matrices and primes)."""
import pytest

from helpers import ensure_lib

FOLD3_MAX = 1865126253  # the largest prime whose three- and five-product sums reduce in one step


@pytest.fixture(scope="module")
def binding():
    ensure_lib()
    from paper_2010_12117_gb300 import binding
    return binding


SIZES = [1, 100, 5000, 19456, 19457, 300_000, 100_000_000]


@pytest.mark.parametrize("n", [10, 15, 17, 18, 19, 21, 23])
@pytest.mark.parametrize("matrices", SIZES)
def test_large_primes_keep_triples(binding, n, matrices):
    """Pairs and quads redo every matrix of a prime above FOLD3_MAX; these orders have triples, which take any prime."""
    assert binding.prime_table()[67] > FOLD3_MAX >= max(binding.prime_table()[:67])
    assert binding.condense_launch(n, matrices, binding.prime_table()[67])[1] == 3
    assert binding.condense_launch(n, matrices, FOLD3_MAX + 1)[1] == 3
    large = binding.condense_launch(n, 10 ** 9, FOLD3_MAX)
    assert large[1] == binding.condense_columns(n) == 4


@pytest.mark.parametrize("n", range(25, 29))
@pytest.mark.parametrize("matrices", SIZES)
def test_large_primes_redo_with_eight_lanes(binding, n, matrices):
    assert binding.condense_launch(n, matrices, FOLD3_MAX + 1)[0] == 8


def test_every_choice_is_a_launchable_kernel(binding):
    columns = set()
    for n in range(1, 33):
        columns.add(binding.condense_columns(n))
        for matrices in SIZES:
            for prime in (0, FOLD3_MAX, FOLD3_MAX + 1, 2 ** 31 - 1):
                lanes, cols, ctas, threads = binding.condense_launch(n, matrices, prime)
                assert lanes in (1, 2, 4, 8) and 2 <= cols <= 4 and ctas >= 1
                assert threads % 32 == 0 and threads % lanes == 0
                assert -(-n // lanes) * n <= 256  # words of a lane's registers
    assert columns == {2, 3, 4}
    for bad in ((0, 1), (33, 1), (5, 0), (5, -1)):
        with pytest.raises(binding.PolydetError):
            binding.condense_launch(*bad)
    for bad in (0, 33):
        with pytest.raises(binding.PolydetError):
            binding.condense_columns(bad)


SMALL = {8: (0, 65536), 9: (0, 32768), 10: (0, 131072), 13: (0, 19456), 16: (0, 65536), 19: (14593, 19456),
         23: (0, 14592), 25: (0, 7296), 26: (0, 7296), 27: (0, 7296), 28: (0, 7296), 31: (0, 21888), 32: (0, 65536)}


@pytest.mark.parametrize("n", range(1, 33))
def test_small_launches_have_their_own_range(binding, n):
    """Orders whose small launches take another kernel do so inside their range and nowhere else."""
    large = binding.condense_launch(n, 10 ** 9)
    lo, hi = SMALL.get(n, (0, -1))
    end = 9728 if n in (25, 28) else hi  # a second choice follows the first
    for m in (1, 100, 4800, 7296, 7297, 9728, 9729, 14592, 14593, 19300, 19456, 19457, 21888, 21889, 32768, 32769,
              65536, 65537, 131072, 131073, 200_000):
        own = binding.condense_launch(n, m)
        if lo <= m <= end:
            assert n == 31 or own != large, (n, m)  # order 31 differs in where the pivots are folded
        else:
            assert own == large, (n, m)


@pytest.mark.parametrize("n", [16, 23, 26, 32])
@pytest.mark.parametrize("matrices", [30, 100, 1200, 2400, 4800, 7200])
def test_launches_below_a_wave_take_small_ctas(binding, n, matrices):
    """Three CTAs of 128 threads per SM: short of a wave, larger CTAs leave some SMs with twice the warps of others,
    and four CTAs have fewer registers per thread."""
    assert binding.condense_launch(n, matrices)[2:] == (3, 128)


def test_large_primes_do_not_redo_what_triples_pass(binding):
    for n in range(1, 33):
        if binding.condense_columns(n) == 3:
            for matrices in SIZES:
                assert binding.condense_launch(n, matrices, FOLD3_MAX + 1)[1] == 3, (n, matrices)
