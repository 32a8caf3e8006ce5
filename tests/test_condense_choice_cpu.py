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
