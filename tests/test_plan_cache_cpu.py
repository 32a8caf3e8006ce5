"""What is kept per shape can be given back."""
from helpers import ensure_lib


def test_plan_cache_clear_gives_back_the_shape_constants():
    ensure_lib()
    from paper_2010_12117_gb300 import binding
    binding._shape_consts[(3, (1,), (3,), 2, False)] = ((5, 7), [(1,), (2,)], [(0, 1, 2, 3)])
    binding.plan_cache_clear()
    assert not binding._shape_consts
    binding.plan_cache_clear()
