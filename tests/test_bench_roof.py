"""bench.py's bound of the tridiagonal reduction, on the CPU: bytes where the matrices
do not fit the SMs' shared memory, integer multiply-adds where they do."""
import os
import sys
from types import SimpleNamespace

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def roof(decomps, searches, steps=2):
    wl = SimpleNamespace(searches=[SimpleNamespace(n=n) for n in searches])
    return bench.reduction_roof(wl, decomps, steps, 6800.0, 152, 2000.0)


def test_batch_is_bound_by_bytes():
    bound, amount, rate, unit = roof({50: 10, 1000: 20, 2000: 40}, [50] * 10 + [1000] * 20 + [2000] * 40)
    assert bound == "hbm" and unit == "GB/s" and rate == 6.8e12
    assert abs(amount - 16 * (10 * 1000 ** 3 + 20 * 2000 ** 3) / 3) < 1e-6 * amount


def test_one_search_in_shared_memory_is_bound_by_multiply_adds():
    bound, amount, rate, _ = roof({1000: 4}, [1000])
    assert bound == "alu" and abs(rate - 28 * 152 * 2e9) < 1
    assert abs(amount - 9 * 2 * 1000 ** 3 / 3) < 1e-6 * amount


def test_the_reduction_has_no_flop_count():
    assert "reduction" not in bench.stage_flops({1000: 4})
