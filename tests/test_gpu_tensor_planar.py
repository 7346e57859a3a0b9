"""The tensor mode's separate real and imaginary operands, at the sizes where their split can slip:
K ranges of an odd number of half slices (the last slice of a CTA half used, a split of the forward
product starting inside a slice), odd rows (pairs of pixels, pairs of traps), a single pixel column
or row, and the coefficients of vanishing fields.

Tolerances: a field is a mean of N unit products, each within 4e-6 (two FP16 parts, FP32 sums: the
bound of the product alone) plus 5e-7 (the phasors' sine and cosine) plus 5e-7 (the tables) of its
64-bit value; the phases are held to the same bound as the mode's other tests.
"""
import numpy as np
import pytest

import oracle
from paper_0907_4027_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

ABS_V = 5e-6
TOL_S = 4e-6


@pytest.fixture(scope="module")
def hot():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0907_4027_gb300 import _build
    _build.build()
    from paper_0907_4027_gb300 import hot as h
    return h


def check_step(gpu_phi, w, coef):
    ophi, S = oracle.backproject(w.geom, w.xyz, coef, want_S=True)
    d = np.abs(np.angle(np.exp(1j * (gpu_phi.astype(np.float64) - ophi))))
    bad = np.abs(S) * d > TOL_S * np.sum(np.abs(coef))
    assert not bad.any(), f"{bad.sum()} pixels"


@pytest.mark.parametrize("W,H,M", [(96, 5, 16), (97, 130, 17), (160, 64, 33), (31, 129, 31), (1, 200, 32), (300, 1, 97),
                                   (1000, 700, 300), (1281, 515, 95)])
def test_ragged_slices_and_pairs(hot, W, H, M):
    w = wl.random_case(W, H, M, seed=3 * W + H + M, precision="tensor")
    with hot.Hologram.from_workload(w) as h:
        h.gsw(0)
        V0, _ = h.fields()
        h.gsw(1)
        V1, _ = h.fields()
        phi1 = h.phase("f32")
    assert np.abs(V0 - oracle.forward(w.geom, w.xyz, w.phi0)).max() < ABS_V
    assert np.abs(V1 - oracle.forward(w.geom, w.xyz, phi1.astype(np.float64))).max() < ABS_V
    _, coef = oracle.update_weights(V0, np.ones(M))
    check_step(phi1, w, coef)


@pytest.mark.parametrize("only", [False, True])
def test_vanishing_fields(hot, only):
    """Phases 0 everywhere and a trap half a turn a pixel away: its field is an exact zero, its weight
    stays and its coefficient is the weight (Sec. 3); alone, or among others."""
    w = wl.random_case(128, 64, 1 if only else 40, seed=9, precision="tensor")
    w.phi0[:] = 0.0
    w.xyz[0] = (0.5 * w.wavelength * w.focal / w.pitch, 0.0, 0.0)
    with hot.Hologram.from_workload(w) as h:
        h.gsw(0)
        V0, _ = h.fields()
        h.gsw(1)
        _, w1 = h.fields()
        phi1 = h.phase("f32")
    assert V0[0] == 0
    w2, coef = oracle.update_weights(V0, np.ones(w.M))
    assert w1[0] == 1.0 and np.allclose(w1, w2, rtol=1e-5)
    check_step(phi1, w, coef)
