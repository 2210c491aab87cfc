"""Folding of the gradient onto the physical grid at the sizes where its kernels
change course: one or two points on an axis, no layer, and rows and planes on
either side of the 32 x 32 elements of a CTA."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nbl", [0, 3])
@pytest.mark.parametrize("shape", [(5, 1, 1), (1, 33, 2), (3, 31, 32), (2, 34, 33)])
def test_folded_gradient(shape, nbl):
    import paper_2004_10519_gb300 as wp
    nx, ny, nz = shape
    rng = np.random.default_rng(nz)
    vp = rng.uniform(1.5, 3.0, shape).astype(np.float32)
    dt = synth.cfl_dt(10.0, 3.0)
    src = np.zeros((1, 3), np.float32)
    rec = np.array([[(nx - 1) * 10.0, (ny - 1) * 10.0, (nz - 1) * 10.0], [0, 0, 0]], np.float32)
    p = synth.Problem(synth.ACOUSTIC, nx, ny, nz, nbl, 10.0, 4, 24, dt, {"vp": vp}, src,
                      synth.ricker(60.0, dt, 24)[None], rec)
    d = rng.standard_normal((2, 24)).astype(np.float32)
    g, J = wp.Propagator.from_problem(p).gradient(p.wavelet, p.src, p.rec, d)
    g_ref, J_ref = oracle.Problem(p).gradient(d)
    assert abs(J - J_ref) <= 1e-5 * J_ref
    assert np.linalg.norm(g - g_ref) <= 1e-4 * np.linalg.norm(g_ref)
