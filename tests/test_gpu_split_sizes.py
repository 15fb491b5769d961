"""The frozen split in FP32 at the sizes where it runs (above 38,912 slots), with a rock of
28,000 mobile particles (a home has four lanes) and with one of 57,000 (one lane, one round
of homes a block, list columns counted within it); and the allocation-free densities on
both sides of the size at which four lanes share a particle.

Tolerances are those of the parity tests (densities 2e-6 of the largest, forces 1e-5 of
max(|f|, rms f) in FP32; densities 1e-13 in FP64)."""
import os
import subprocess
import sys

import numpy as np
import pytest

from oracle import oracle as O
from paper_1903_10134_gb300 import inputs as I

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SIZES = [64, 80]
RHO_TOL = {0: 1e-13, 1: 2e-6}
FORCE_TOL = 1e-5


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_10134_gb300 import mdpd
    mdpd.lib()
    return mdpd


def _rock(M, nvox, direct=False):
    """A rock under the frozen split (one more launch a step than without)."""
    w = I.rock(nvox=nvox, g=0.5, seed=5)
    s = M.System.from_workload(w)
    without = M.mdpd_describe(s.h)[1]
    s.set_option(M.OPT_KERNELS, M.KERNELS_NLIST_THREAD)
    assert M.mdpd_describe(s.h)[1] == without + 1
    assert s.n > 38912 and (w.n > 38912) == (nvox == 80)
    if direct:
        s.set_option(M.OPT_GRAPH, 0)
    return w, s


def _same(a, b):
    for p, q in zip(a.state(), b.state()):
        assert np.array_equal(p, q)


@pytest.mark.parametrize("nvox", SIZES)
def test_densities_and_forces_track_the_oracle(M, nvox):
    """Also with the walls loaded unmoved, with one wall particle moved (the frozen-frozen
    part is formed anew), and moved back."""
    w, s = _rock(M, nvox)
    s.step(6)
    x, v, t, rho = s.state()
    acc = M.mdpd_get_accel(s.h)
    walls = np.flatnonzero(t == w.wall_type)
    mob = t != w.wall_type
    x2 = x.copy()
    x2[walls[len(walls) // 2]] += np.array([0.05, -0.03, 0.02])
    ref = {}
    for k, xs in enumerate((x, x2)):
        ref[k] = O.Oracle(w.params.copy(precision=0), xs, v, t, w.seed, use_cells=True,
                          step=M.mdpd_step_count(s.h))
    assert np.abs(rho - ref[0].rho).max() <= RHO_TOL[1] * ref[0].rho.max()
    for k in (0, 1, 1, 0):
        M.mdpd_set_state_accel(s.h, x2 if k else x, v, acc)
        f, rho = s.forces()
        o = ref[k]
        assert np.abs(rho - o.rho).max() <= RHO_TOL[1] * o.rho.max()
        size = np.linalg.norm(o.a[mob], axis=1)
        rms = np.sqrt(np.mean(size ** 2))
        err = np.linalg.norm(f[mob] - o.a[mob], axis=1) / np.maximum(size, rms)
        assert err.max() <= FORCE_TOL
    s.close()


@pytest.mark.parametrize("nvox", SIZES)
def test_graph_direct_and_resume_bitwise(M, nvox):
    _, a = _rock(M, nvox)
    _, b = _rock(M, nvox, direct=True)
    for s in (a, b):
        s.step(19)
    _same(a, b)
    x, v, _, _ = a.state()
    acc, steps = M.mdpd_get_accel(a.h), M.mdpd_step_count(a.h)
    _, c = _rock(M, nvox)
    M.mdpd_set_step(c.h, steps)
    M.mdpd_set_state_accel(c.h, x, v, acc)
    a.step(11)
    c.step(11)
    _same(a, c)
    for s in (a, b, c):
        s.close()


def run_rocks(path):
    """Steps under the split, results saved to path (npz)."""
    from paper_1903_10134_gb300 import mdpd
    res = {}
    for nvox in SIZES:
        _, s = _rock(mdpd, nvox)
        s.step(10)
        for name, a in zip("xvtr", s.state()):
            res[f"{name}{nvox}"] = a
        s.close()
    np.savez(path, **res)


def test_debug_build_matches_release_bitwise(M, tmp_path):
    """The index checks of the debug build report nothing and change nothing."""
    from paper_1903_10134_gb300 import _build
    _build.build(debug=True)
    code = ("import sys; sys.path[:0] = [%r, %r]; import test_gpu_split_sizes as T; "
            "from paper_1903_10134_gb300 import mdpd; assert mdpd.debug_build(); "
            "T.run_rocks(%r)" % (ROOT, HERE, str(tmp_path / "debug.npz")))
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, MDPD_DEBUG="1", PYTHONPATH=ROOT + os.pathsep + HERE))
    assert r.returncode == 0, r.stdout + r.stderr
    run_rocks(tmp_path / "release.npz")
    a, b = np.load(tmp_path / "debug.npz"), np.load(tmp_path / "release.npz")
    assert sorted(a.files) == sorted(b.files)
    for k in a.files:
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("precision, n", [(0, 9728), (0, 9729), (1, 38912), (1, 38913)])
def test_noalloc_on_both_sides_of_shared_homes(M, precision, n):
    import torch
    box, lo, periodic = (18.4, 19.1, 19.7), (-1.0, 0.5, 2.0), (1, 0, 1)
    if precision == 0:
        box = tuple(0.62 * b for b in box)
    p = I.MDPDParams(box=box, box_lo=lo, periodic=periodic).copy(precision=precision)
    pos = I.uniform_positions(n, lo, np.add(lo, box), np.random.default_rng(43))
    ref = O.Oracle(p, pos, np.zeros_like(pos), np.zeros(n, np.int32), 1, use_cells=True).density()
    rho = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
    M.mdpd_density_noalloc(p, torch.from_numpy(pos).to("cuda"), rho, torch.cuda.current_stream())
    assert np.abs(rho.cpu().numpy() - ref).max() <= RHO_TOL[precision] * ref.max()
