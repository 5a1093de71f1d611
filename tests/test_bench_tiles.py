"""The benchmark's count of the per-energy formation's tiles: halves of 128 x 256 tiles that hold no entry (i <= j < n)
are left out by the kernel and not counted."""
import importlib.util
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("bench_for_tiles", os.path.join(ROOT, "bench.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


@pytest.mark.parametrize("n", [1, 127, 128, 129, 256, 257, 331, 384, 385, 640, 1000, 1492])
def test_halves_that_hold_an_entry(bench, n):
    halves = sum(any(128 * ib <= j for j in range(128 * h, min(n, 128 * h + 128)))
                 for ib in range(-(-n // 128)) for h in range(-(-n // 128)))
    assert bench._pe_tiles(n) == halves / 2


def test_stated_counts(bench):
    assert bench._pe_tiles(1000) == 18 and bench._pe_tiles(331) == 3 and bench._pe_tiles(231) == 1.5
