"""Host logic of bench.py: when the density pass's candidate tests are counted for mobile
homes only (the library's frozen split)."""
import importlib.util
import os

import pytest

from paper_1903_10134_gb300 import inputs as I

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _bench():
    spec = importlib.util.spec_from_file_location("bench", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


@pytest.mark.parametrize("precision, n, thread, frozen, want", [
    (1, 38912, True, (1,), False), (1, 38913, True, (1,), True), (1, 500000, False, (1,), False),
    (1, 500000, True, (), False), (0, 1000, True, (1,), True), (0, 1000, False, (1,), False)])
def test_split_is_counted_where_it_runs(precision, n, thread, frozen, want):
    p = I.MDPDParams(box=(10.0, 10.0, 10.0), ntypes=2, frozen_types=frozen).copy(precision=precision)
    assert _bench().density_splits(p, n, thread) is want
