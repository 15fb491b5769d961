"""Replicas with frozen types under the default kernel variant: each equals its system
run alone to the bit, densities of the frozen particles included (no frozen split there,
whose fixed-point sums a batch does not form)."""
import numpy as np
import pytest

from paper_1903_10134_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# (particles, box, frozen types): FP64 below and above the size of shared homes; FP32 the
# same, above it with few and with many mobile particles
CASES = {
    0: [(1500, (6.1, 6.4, 6.7), (1,)), (11000, (12.3, 12.1, 13.0), (0, 2))],
    1: [(2300, (7.3, 7.1, 7.7), (2,)), (39100, (19.0, 18.2, 18.9), (0, 1))],
}


@pytest.mark.parametrize("precision", [0, 1])
def test_replicas_with_frozen_types_equal_their_systems_bitwise(precision):
    from paper_1903_10134_gb300 import mdpd as M
    ws = []
    for k, (n, box, frozen) in enumerate(CASES[precision]):
        w = I.tiny(n, box, 60 + k, periodic=(1, k, 1), ntypes=3, precision=precision, dt=1e-4,
                   frozen_types=frozen)
        w.vel[np.isin(w.type, frozen)] = 0.0
        ws.append(w)
    b = M.Batch.from_workloads(ws)
    b.step(2)
    for r, w in enumerate(ws):
        x, v, _, rho = b.replica_state(r)
        with M.System(w.params, w.pos, w.vel, w.type, w.seed) as s:
            s.step(2)
            xs, vs, _, rhos = s.state()
        assert np.array_equal(rho, rhos), r
        assert np.array_equal(x, xs) and np.array_equal(v, vs), r
    b.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_autotune_times_the_split_where_it_differs(precision):
    """With frozen particles (and, in FP32, more than fit the chip at once) the two list
    variants are timed apart; elsewhere one timing stands for both."""
    from paper_1903_10134_gb300 import mdpd as M
    n, box, frozen = CASES[precision][1]
    for fz in ((), frozen):
        w = I.tiny(n, box, 64, ntypes=3, precision=precision, dt=1e-4, frozen_types=fz)
        with M.System(w.params, w.pos, w.vel, w.type, w.seed) as s:
            s.set_option(M.OPT_KERNELS, M.KERNELS_SCAN)
            res = s.autotune(3)
            chosen, ms = res
            if fz:
                assert chosen == (M.KERNELS_NLIST if ms[0] < ms[1] else M.KERNELS_NLIST_THREAD)
            else:
                assert ms[0] == ms[1] and chosen == M.KERNELS_NLIST
