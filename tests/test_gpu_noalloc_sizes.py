"""mdpd_density_noalloc where its kernels change route or could go wrong: one particle, a
partial warp, both sides of the size at which four lanes share a particle (FP32), axes of
one and two cells, cells longer than r_c, a box away from the origin, and particles some
box lengths outside a periodic axis, against the FP64 oracle.

Tolerance: that of the other tests of this entry point (FP64 1e-13, FP32 2e-6 of the
largest density).  A box at distance D from the origin, or a particle wrapped from D away,
adds the rounding of its double coordinates, D 2^-52 each, times the density's largest
slope, 3 w(0) / r_d summed over the partners (at most four times the largest density per
unit length here): 16 D 2^-52 for two particles in three coordinates.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1903_10134_gb300 import inputs as I

pytestmark = pytest.mark.gpu

RHO_TOL = {0: 1e-13, 1: 2e-6}

CASES = {
    "one": (1, (3.0, 3.0, 3.0), (0, 0, 0), (1, 1, 1)),
    "partial_warp": (31, (1.0, 3.0, 0.7), (0, 0, 0), (0, 1, 0)),
    "thin": (1500, (1.9, 12.4, 2.7), (0, 0, 0), (0, 1, 0)),
    "far_origin": (2000, (7.9, 3.99, 5.0), (-40.25, 17.5, 300.0), (1, 1, 0)),
    "four_lanes": (16000, (14.0, 13.0, 12.5), (-1.0, 0, 2.0), (1, 0, 1)),
    "one_lane": (16001, (14.0, 13.0, 12.5), (-1.0, 0, 2.0), (1, 0, 1)),
    "dense": (4000, (4.0, 5.0, 4.5), (0, 0, 0), (1, 1, 1)),
}


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("case", sorted(CASES))
def test_noalloc_sizes(case, precision):
    import torch
    from paper_1903_10134_gb300 import mdpd as M
    n, box, lo, periodic = CASES[case]
    rng = np.random.default_rng(41)
    p = I.MDPDParams(box=box, box_lo=lo, periodic=periodic).copy(precision=precision)
    pos = I.uniform_positions(n, lo, np.add(lo, box), rng)
    given = pos.copy()
    for k in range(3):
        if periodic[k]:
            given[:, k] += box[k] * rng.integers(-2, 3, n)
    ref = O.Oracle(p, pos, np.zeros_like(pos), np.zeros(n, np.int32), 1, use_cells=n > 4000).density()
    far = max(abs(v) + 3 * b for v, b in zip(lo, box))
    rho = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
    pos_t = torch.from_numpy(given).to("cuda")
    stream = torch.cuda.current_stream()
    M.mdpd_density_noalloc(p, pos_t, rho, stream)
    err = np.abs(rho.cpu().numpy() - ref).max()
    assert err <= (RHO_TOL[precision] + 16 * far * 2.0 ** -52) * ref.max(), err
