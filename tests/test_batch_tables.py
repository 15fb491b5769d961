"""Pair tables handed over for all replicas of a batch: one 8 x 8 table per replica, or
ValueError (never a broadcast over replicas or over a table's rows)."""
import numpy as np
import pytest

from paper_1903_10134_gb300 import inputs as I
from paper_1903_10134_gb300 import mdpd as M


def _params(n):
    return [I.MDPDParams(box=(4.0 + r, 4.0, 4.0)) for r in range(n)]


def _tables(*shape):
    k = int(np.prod(shape))
    return [np.arange(k, dtype=np.float64).reshape(shape) + q * k for q in range(3)]


@pytest.mark.parametrize("n, shape", [(1, (8, 8)), (4, (8, 8)), (8, (8, 8)), (10, (8, 8)),
                                      (4, (1, 8, 8)), (4, (3, 8, 8)), (2, (2, 8, 1)),
                                      (2, (2, 1, 8)), (2, (2, 7, 8)), (2, (8,)),
                                      (2, (2, 1, 8, 8))])
def test_other_shapes_are_refused(n, shape):
    with pytest.raises(ValueError):
        M._c_params_list(_params(n), _tables(*shape))


@pytest.mark.parametrize("n, shape", [(1, (1, 8, 8)), (4, (4, 8, 8)), (3, (5, 8, 8)), (2, (2, 9, 8))])
def test_each_replica_gets_its_own_table(n, shape):
    tabs = _tables(*shape)
    c = M._c_params_list(_params(n), tabs)
    for r in range(n):
        assert c[r].box[0] == 4.0 + r
        for name, t in zip(("A", "B", "gamma"), tabs):
            assert np.array_equal(np.array(getattr(c[r], name)), t[r, :8, :8])


def test_without_tables_the_objects_own_are_taken():
    ps = _params(3)
    for r, p in enumerate(ps):
        p.set_pair(0, 1, A=-30.0 - r, B=20.0 + r, gamma=4.0 + r)
    c = M._c_params_list(ps)
    for r, p in enumerate(ps):
        for name in ("A", "B", "gamma"):
            assert np.array_equal(np.array(getattr(c[r], name)), np.asarray(getattr(p, name)))
