"""Homes that four lanes share (FP32, few mobile particles) next to homes of one lane."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1903_10134_gb300 import inputs as I

pytestmark = pytest.mark.gpu

RHO_TOL = {0: 1e-13, 1: 2e-6}


@pytest.mark.parametrize("rho_self", [0, 1])
def test_replicas_of_a_large_batch_equal_their_systems_bitwise(rho_self):
    """Alone, a replica's homes have four lanes; in a batch of 36,000 one, which sums
    the same groups of rows.  One replica is dense enough for more hits than the four
    lanes keep."""
    from paper_1903_10134_gb300 import mdpd as M
    boxes = [(6.3, 5.2, 7.4)] * 16 + [(3.0, 3.4, 3.2), (9.9, 4.0, 5.5)]
    ws = [I.tiny(2003 - r, b, 90 + r, periodic=(1, r % 2, 1), precision=1, dt=1e-4, rho_self=rho_self)
          for r, b in enumerate(boxes)]
    b = M.Batch.from_workloads(ws)
    b.step(2)
    for r in (0, 1, 16, 17):
        w = ws[r]
        x, v, _, rho = b.replica_state(r)
        with M.System(w.params, w.pos, w.vel, w.type, w.seed) as s:
            s.step(2)
            xs, vs, _, rhos = s.state()
        assert np.array_equal(rho, rhos), r
        assert np.array_equal(x, xs) and np.array_equal(v, vs), r
    b.close()


@pytest.mark.parametrize("box", [(8.1, 6.4, 7.7), (4.2, 3.1, 3.9)])
def test_frozen_split_with_shared_homes(box):
    """Mobile homes of four lanes in the frozen split, at a usual density and at one
    with more hits than the lanes keep: densities, wall density, partner count."""
    from paper_1903_10134_gb300 import mdpd as M
    w = I.tiny(2400, box, 81, periodic=(1, 1, 0), ntypes=3, precision=1, frozen_types=(2,))
    w.vel[w.type == 2] = 0.0
    o = O.Oracle(w.params.copy(precision=0), w.pos, w.vel, w.type, w.seed)
    with M.System(w.params, w.pos, w.vel, w.type, w.seed) as s, \
            M.System(w.params, w.pos, w.vel, w.type, w.seed) as d:
        s.set_option(M.OPT_WALL_DENSITY, 1)
        d.set_option(M.OPT_KERNELS, M.KERNELS_SCAN)
        _, rho = s.forces()
        d.forces()
        assert s.pair_count() == d.pair_count()
        assert np.abs(rho - o.rho).max() <= RHO_TOL[1] * o.rho.max()
        phi, ref = s.wall_density(), o.wall_density()
        assert np.abs(phi - ref).max() <= 2e-5 * (1.0 + ref.max())


@pytest.mark.parametrize("n, box, frozen", [(39100, (19.0, 18.2, 18.9), (1,)),
                                            (39100, (12.1, 11.0, 13.2), (1, 2))])
def test_frozen_split_above_the_size_of_shared_homes(n, box, frozen):
    """More slots than fit the chip at once, but few enough mobile ones: the split with
    four lanes a home, at a usual density and at one with more hits than they keep."""
    from paper_1903_10134_gb300 import mdpd as M
    w = I.tiny(n, box, 82, periodic=(1, 0, 1), ntypes=3, precision=1, frozen_types=frozen)
    w.vel[np.isin(w.type, frozen)] = 0.0
    o = O.Oracle(w.params.copy(precision=0), w.pos, w.vel, w.type, w.seed, use_cells=1)
    with M.System(w.params, w.pos, w.vel, w.type, w.seed) as s, \
            M.System(w.params, w.pos, w.vel, w.type, w.seed) as d:
        s.set_option(M.OPT_WALL_DENSITY, 1)
        d.set_option(M.OPT_KERNELS, M.KERNELS_SCAN)
        _, rho = s.forces()
        d.forces()
        assert s.pair_count() == d.pair_count()
        assert np.abs(rho - o.rho).max() <= RHO_TOL[1] * o.rho.max()
        phi, ref = s.wall_density(), o.wall_density()
        assert np.abs(phi - ref).max() <= 2e-5 * (1.0 + ref.max())


def test_replicas_of_a_large_fp64_batch_equal_their_systems_bitwise():
    """The same in FP64, where a home has four lanes in systems below 9,728 particles:
    alone four, in a batch of 11,000 one."""
    from paper_1903_10134_gb300 import mdpd as M
    ws = [I.tiny(1391 - r, (6.3, 5.2, 7.4) if r else (3.0, 3.4, 3.2), 70 + r, periodic=(1, r % 2, 1),
                 precision=0, dt=1e-4, rho_self=r % 2) for r in range(8)]
    b = M.Batch.from_workloads(ws)
    b.step(2)
    for r in (0, 1, 2, 7):
        w = ws[r]
        x, v, _, rho = b.replica_state(r)
        with M.System(w.params, w.pos, w.vel, w.type, w.seed) as s:
            s.step(2)
            xs, vs, _, rhos = s.state()
        assert np.array_equal(rho, rhos), r
        assert np.array_equal(x, xs) and np.array_equal(v, vs), r
    b.close()


@pytest.mark.parametrize("box", [(8.1, 6.4, 7.7), (4.2, 3.1, 3.9)])
def test_frozen_split_with_shared_homes_fp64(box):
    """The frozen split's mobile homes in FP64 with four lanes, also at a density with
    more hits than the lanes keep."""
    from paper_1903_10134_gb300 import mdpd as M
    w = I.tiny(2400, box, 83, periodic=(1, 1, 0), ntypes=3, precision=0, frozen_types=(2,))
    w.vel[w.type == 2] = 0.0
    o = O.Oracle(w.params, w.pos, w.vel, w.type, w.seed)
    with M.System(w.params, w.pos, w.vel, w.type, w.seed) as s:
        s.set_option(M.OPT_WALL_DENSITY, 1)
        _, rho = s.forces()
        assert np.abs(rho - o.rho).max() <= RHO_TOL[0] * o.rho.max()
        assert np.abs(s.wall_density() - o.wall_density()).max() <= 1e-12 * (1.0 + o.wall_density().max())
