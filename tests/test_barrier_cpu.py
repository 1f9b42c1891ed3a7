"""The counter of the barrier that a launch's CTAs meet at, on the host: a CTA
passes exactly when all have arrived, also where the 32-bit count wraps (long
circuits: a chain of 600 CTAs after 7 million steps)."""
import pytest

from paper_2502_10685_gb300 import _lib


@pytest.mark.parametrize("ctas", [1, 2, 64, 128, 224, 600, 608, 1216])
def test_ctas_wait_for_all_also_where_the_count_wraps(ctas):
    L = _lib.load()
    steps = {0, 1, 1000, 2 ** 31 - 1}
    for wrap in (2 ** 31, 2 ** 32, 2 ** 33):
        steps |= {wrap // ctas + d for d in range(-3, 4)}
    for step in sorted(s for s in steps if 0 <= s < 2 ** 31):
        assert L.stab_selftest_barrier(ctas, step) == 0, step


def test_arguments_out_of_range():
    L = _lib.load()
    for ctas, step in ((0, 0), (2 ** 20 + 1, 0), (4, -1), (4, 2 ** 31)):
        assert L.stab_selftest_barrier(ctas, step) == -2
