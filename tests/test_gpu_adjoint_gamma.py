"""The gamma gradient of an evaluation is linear in d = d(sigma)/d(gamma) = sqrt(kT / 2 gamma)
at fixed positions, velocities, cotangents and random draws: S1 + d S2.  From two
temperatures at which d is a binary fraction it follows for any other; a d rounded to FP32
would show as a factor of the whole of S2.

Isolated pairs at rest, and cotangents along each pair's random force, so that S2 is a sum
of terms of one sign, in which the terms' own roundings average out and a common factor's
does not.  Tolerance: a term in FP32 is off by less than four half units of 2^-23, that is
4 x 2^-24 of it, with signs at random; 8,192 of them leave less than
4 x 2^-24 / sqrt(8192) = 2.6e-9 of S2, and three gradients are compared: 2^-27 = 7.5e-9.
The temperatures are those whose d, rounded to FP32, is off by more than 5e-8."""
import numpy as np
import pytest

from paper_1903_10134_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _pairs(rng):
    """16^3 pairs 0.2 to 0.9 apart, more than r_c from one another."""
    g = np.stack(np.meshgrid(*[np.arange(16)] * 3, indexing="ij"), -1).reshape(-1, 3) * 2.5 + 1.25
    e = rng.normal(size=g.shape)
    e /= np.linalg.norm(e, axis=1, keepdims=True)
    half = 0.5 * rng.uniform(0.2, 0.9, (len(g), 1)) * e
    return np.concatenate([g + half, g - half]), e


@pytest.mark.parametrize("precision", [0, 1])
def test_gamma_gradient_is_linear_in_the_random_scale(precision):
    import torch
    from paper_1903_10134_gb300 import adjoint as AD, mdpd as M
    rng = np.random.default_rng(17)
    x, e = _pairs(rng)
    n = len(x)
    p = I.MDPDParams(box=(40.0,) * 3, dt=1.0 / 64).copy(precision=precision)
    p.gamma[:] = 2.0                            # d = sqrt(kT) / 2
    kTs = [kT for kT in rng.uniform(1.0, 1.2, 200)
           if abs(np.float64(np.float32(0.5 * np.sqrt(kT))) / (0.5 * np.sqrt(kT)) - 1.0) > 5e-8][:8]
    with M.System(p, x, np.zeros_like(x), np.zeros(n, np.int32), 9) as s:
        def at(kT):
            M.mdpd_set_params(s.h, p.copy(kT=kT))

        at(1.0)
        f1 = s.forces()[0]
        at(4.0)
        random = (s.forces()[0] - f1)[:n // 2]
        side = 0.5 * np.sign((random * e).sum(1, keepdims=True)) * e
        abar = torch.from_numpy(np.concatenate([side, -side])).to("cuda")

        def gradient(kT):
            at(kT)
            return float(AD.eval_vjp(s, abar)[2][2, 0, 0])

        g1, g4 = gradient(1.0), gradient(4.0)   # d = 1/2, 1
        s2 = (g4 - g1) / 0.5
        assert len(kTs) == 8 and s2 > 0.0
        for kT in kTs:
            want = g1 + (0.5 * np.sqrt(kT) - 0.5) * s2
            assert abs(gradient(kT) - want) <= 2.0 ** -27 * s2, kT
