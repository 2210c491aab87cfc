"""Diverging fields (check_nan = 0) hold what plain division gives: large finite
numbers and infinities, not NaN, above the range of the shared-reciprocal quotient."""
import numpy as np
import pytest

from test_gpu_rows import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("adjoint", [False, True])
@pytest.mark.parametrize("nz", [41, 40])
def test_tti_step_of_a_diverging_field(nz, adjoint, monkeypatch):
    import paper_2004_10519_gb300 as wp
    p = problem("tti", nz, nt=8)
    out = []
    for no_tma in (False, True):
        if no_tma:
            monkeypatch.setenv("WAVEPROP_NO_TMA", "1")
        prop = wp.Propagator.from_problem(p, check_nan=0)
        rng = np.random.default_rng(2)
        state = [(rng.standard_normal(prop.grid) * 1e30 * 10.0 ** rng.uniform(0, 7.3, prop.grid)).astype(np.float32)
                 for _ in range(prop.nfields)]
        prop.set_state(state)
        prop.step(1, adjoint=adjoint)
        out.append(prop.get_state())
        prop.close()
    assert max(np.nanmax(np.abs(f[np.isfinite(f)])) for f in out[1]) > 1e36
    for a, b in zip(*out):
        if nz == 41:                 # padded rows follow the pipelined passes bit for bit
            np.testing.assert_array_equal(a, b)
        else:
            ok = np.isfinite(b) & (np.abs(b) < 3e38)
            assert np.isfinite(a[ok]).all()
