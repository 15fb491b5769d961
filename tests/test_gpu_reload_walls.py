"""Walled systems whose state is loaded without an evaluation (mdpd_set_state_accel) and
whose frozen-frozen density part must then be recomputed, because the parameters or the
kernel variant change before the next step: the step equals, to the bit, that of a handle
on which the change came before the load.

FP64, and FP32 with more slots than FP32 gives shared homes to, where the frozen split
runs."""
import numpy as np
import pytest

from paper_1903_10134_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_10134_gb300 import mdpd
    mdpd.lib()
    return mdpd


def _rock(precision):
    return I.rock(nvox=32 if precision == 0 else 64, porosity=0.3, g=0.5, seed=5,
                  precision=precision)


def _load(M, s, saved):
    x, v, acc, steps = saved
    M.mdpd_set_step(s.h, steps)
    M.mdpd_set_state_accel(s.h, x, v, acc)


def _saved(M, s):
    x, v, _, _ = s.state()
    return x, v, M.mdpd_get_accel(s.h), M.mdpd_step_count(s.h)


def _same(a, b):
    for p, q in zip(a.state(), b.state()):
        assert np.array_equal(p, q)


@pytest.mark.parametrize("kernels", [0, 2])
@pytest.mark.parametrize("precision", [0, 1])
def test_parameters_changed_after_a_load(M, precision, kernels):
    w = _rock(precision)
    other = w.params.copy(g=(0.1, 0.2, 0.0))
    with M.System.from_workload(w) as a, M.System.from_workload(w) as b:
        assert precision == 0 or a.n > 38912
        for s in (a, b):
            s.set_option(M.OPT_KERNELS, kernels)
            s.step(3)
        saved = _saved(M, a)
        _load(M, a, saved)
        M.mdpd_set_params(a.h, other)
        M.mdpd_set_params(b.h, other)
        _load(M, b, saved)
        for k in (1, 2):
            a.step(k)
            b.step(k)
            _same(a, b)


@pytest.mark.parametrize("kernels", [0, 2])
@pytest.mark.parametrize("precision", [0, 1])
def test_list_variant_chosen_after_a_load_under_scan(M, precision, kernels):
    w = _rock(precision)
    with M.System.from_workload(w) as a, M.System.from_workload(w) as b:
        for s in (a, b):
            s.set_option(M.OPT_KERNELS, M.KERNELS_SCAN)
            s.step(3)
        saved = _saved(M, a)
        _load(M, a, saved)
        a.set_option(M.OPT_KERNELS, kernels)
        b.set_option(M.OPT_KERNELS, kernels)
        _load(M, b, saved)
        for k in (1, 2):
            a.step(k)
            b.step(k)
            _same(a, b)
