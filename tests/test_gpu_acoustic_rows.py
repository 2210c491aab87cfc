"""Acoustic handles whose rows are padded compute what the direct pass computes on
packed rows (WAVEPROP_NO_TMA=1), bit for bit over a whole record: the quotient in
the absorbing layer depends on the position alone, so a rounding of its own adds up
there from step to step."""
import numpy as np
import pytest

from test_gpu_rows import problem

pytestmark = pytest.mark.gpu


def calls(p, wp, snap):
    prop = wp.Propagator.from_problem(p, snap_mode=snap)
    # receivers one cell below the top layer
    x = p.h * np.arange(0, p.nx, 3)
    rec = np.array([(a, b, p.h) for a in x for b in p.h * np.arange(0, p.ny, 4)], np.float32)
    tr = prop.forward(p.wavelet, p.src, rec)
    launches = prop.last_launches()
    out = [tr] + prop.get_state()
    g, J = prop.gradient(p.wavelet, p.src, rec, 0.5 * tr)
    out += [g, np.float64(J), prop.adjoint(tr, p.src, rec)]
    prop.close()
    return out, launches


@pytest.mark.parametrize("so", [4, 8, 12, 16])
@pytest.mark.parametrize("nz", [41, 42, 43])
def test_padded_rows_keep_the_bits_of_the_direct_pass(nz, so, monkeypatch):
    import paper_2004_10519_gb300 as wp
    p = problem("acoustic", nz, so=so, nt=150, nbl=6, shape=(45, 37))
    p.src = np.array([[p.nx * p.h / 2 + 0.3, p.ny * p.h / 2 - 0.8, 2 * p.h]], np.float32)
    snap = wp.SNAP_CKPT_FP32 if nz == 42 else wp.SNAP_FULL_FP32
    padded, n = calls(p, wp, snap)
    assert n < 2 * p.nt                            # one pass a step: sources and receivers are in it
    monkeypatch.setenv("WAVEPROP_NO_TMA", "1")
    direct, n = calls(p, wp, snap)
    assert n >= 3 * p.nt - 2
    assert np.abs(direct[0]).max() > 0 and np.abs(direct[3]).max() > 0
    for a, b in zip(padded, direct):
        np.testing.assert_array_equal(a, b)


def test_a_diverging_field_overflows_to_infinity(monkeypatch):
    """Quotients above the range of the shared-reciprocal form."""
    import paper_2004_10519_gb300 as wp
    p = problem("acoustic", 41, nt=8)
    out = []
    for no_tma in (False, True):
        if no_tma:
            monkeypatch.setenv("WAVEPROP_NO_TMA", "1")
        prop = wp.Propagator.from_problem(p, check_nan=0)
        rng = np.random.default_rng(2)
        state = [(rng.standard_normal(prop.grid) * 1e30 * 10.0 ** rng.uniform(0, 7.5, prop.grid)).astype(np.float32)
                 for _ in range(prop.nfields)]
        prop.set_state(state)
        prop.step(1)
        out.append(prop.get_state())
        prop.close()
    assert np.isinf(out[1][0]).any() and np.isfinite(out[1][0]).any()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
