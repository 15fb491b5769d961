"""The filtered density pass against the direct scan (which shares none of its
code) and the oracle, at lattices where its windows, runs and masks have edges."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1903_10134_gb300 import inputs as I

pytestmark = pytest.mark.gpu

RHO_TOL = {0: 1e-13, 1: 2e-6}

# box, periodic, particles, extra parameters
CASES = {
    "three_cells": ((3.0, 3.9, 3.99), (1, 1, 1), 250, {}),
    "windows_4_5_6": ((4.0, 5.3, 6.9), (1, 1, 1), 900, {}),
    "windows_7_8_9": ((7.2, 8.0, 9.7), (1, 1, 1), 3400, {}),
    "open_x": ((5.5, 4.2, 4.4), (0, 1, 1), 600, {}),
    "one_and_two_cells": ((1.9, 2.7, 6.0), (0, 0, 0), 180, {}),
    "wide_r_d": ((6.1, 5.0, 4.7), (1, 1, 0), 860, {"rd": 1.0}),
    "scaled": ((14.6, 11.0, 9.1), (1, 0, 1), 640, {"rc": 2.3, "rd": 1.7, "box_lo": (-3.0, 5.0, 11.0)}),
    "long_runs": ((4.0, 3.5, 3.2), (1, 1, 1), 1500, {}),      # over 32 candidates a run
    "longer_runs": ((3.2, 3.1, 3.0), (1, 0, 1), 4000, {}),    # more masks than places
    "single": ((3.0, 3.0, 3.0), (1, 1, 1), 1, {}),
}


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("case", sorted(CASES))
def test_filtered_density_matches_scan_and_oracle(case, precision):
    from paper_1903_10134_gb300 import mdpd as M
    box, per, n, kw = CASES[case]
    w = I.tiny(n, box, 77, periodic=per, ntypes=2, precision=precision, **kw)
    o = O.Oracle(w.params.copy(precision=0), w.pos, w.vel, w.type, w.seed)
    a = M.System(w.params, w.pos, w.vel, w.type, w.seed)
    b = M.System(w.params, w.pos, w.vel, w.type, w.seed)
    b.set_option(M.OPT_KERNELS, M.KERNELS_SCAN)
    (_, ra), (_, rb) = a.forces(), b.forces()
    assert a.pair_count() == b.pair_count()
    assert np.abs(ra - o.rho).max() <= RHO_TOL[precision] * max(o.rho.max(), 1.0)
    assert np.abs(rb - o.rho).max() <= RHO_TOL[precision] * max(o.rho.max(), 1.0)
    a.close()
    b.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_frozen_split_densities_and_wall_density(precision):
    """Mobile homes only, scattering to frozen ones, with the wall density: a box
    with a third of its particles frozen, odd cell counts, faces in y."""
    from paper_1903_10134_gb300 import mdpd as M
    w = I.tiny(1800, (7.3, 5.2, 8.4), 78, periodic=(1, 0, 1), ntypes=3, precision=precision,
               frozen_types=(1,))
    w.vel[w.type == 1] = 0.0
    o = O.Oracle(w.params.copy(precision=0), w.pos, w.vel, w.type, w.seed)
    s = M.System(w.params, w.pos, w.vel, w.type, w.seed)
    s.set_option(M.OPT_WALL_DENSITY, 1)
    _, rho = s.forces()
    assert np.abs(rho - o.rho).max() <= RHO_TOL[precision] * o.rho.max()
    phi, ref = s.wall_density(), o.wall_density()
    assert np.abs(phi - ref).max() <= (1e-12 if precision == 0 else 2e-5 * (1.0 + ref.max()))
    s.close()
