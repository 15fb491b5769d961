"""How many lanes share a home follows from the number of homes of the pass.  Without the
frozen split every particle is one, whether its type is frozen or not: the densities of a
system equal, to the bit, those of the same particles with no frozen type, in the step's
pass and in the adjoint's (four lanes sum in groups, one lane does not).  The frozen type's
particles have the highest ids, so that a cell, which puts its frozen particles last, keeps
one order."""
import numpy as np
import pytest

from paper_1903_10134_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision, n, box", [
    (0, 9728, (12.3, 11.1, 12.0)), (0, 9729, (12.3, 11.1, 12.0)), (0, 17000, (14.3, 13.1, 15.0)),
    (1, 38912, (19.0, 18.2, 18.9)), (1, 38913, (19.0, 18.2, 18.9)), (1, 70001, (23.0, 22.2, 22.9))])
def test_frozen_types_do_not_change_the_sums(precision, n, box):
    import torch
    from paper_1903_10134_gb300 import adjoint as AD, mdpd as M
    w = I.tiny(n, box, 71, periodic=(1, 1, 0), ntypes=2, precision=precision)
    w.type[:] = np.arange(n) >= n // 2
    rho = []
    for frozen in ((), (1,)):
        p = w.params.copy(frozen_types=frozen)
        vel = w.vel.copy()
        vel[np.isin(w.type, frozen)] = 0.0
        with M.System(p, w.pos, vel, w.type, w.seed) as s:
            step = s.state()[3]
            ones = torch.ones(n, dtype=torch.float64, device="cuda")
            AD.eval_vjp(s, rhobar=ones)
            rho.append((step, s.state()[3]))
    for a, b in zip(*rho):
        assert np.array_equal(a, b)
