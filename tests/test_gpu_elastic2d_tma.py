"""The TMA-fed 2D elastic passes against the plain-load ones (WAVEPROP_NO_TMA=1)
and the FP64 oracle: every point of a few steps from a state without zeros, on
both tile heights, with grid edges on and beside the tiles' (64 z, 16 or 32 x)
and rows that need padding; sources and receivers inside the passes."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


# physical sizes; the computational grid has 8 more: 152 tiles of 64 x 32 from 1216 x 256 on
SHAPES = [(24, 56), (25, 57), (23, 119), (41, 122), (7, 20), (1208, 248), (1215, 251)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("so", [4, 8, 12, 16])
def test_every_point(so, shape, monkeypatch):
    import paper_2004_10519_gb300 as wp
    p = synth.elastic2d_small(shape=shape, nbl=4, so=so, nt=20)
    p.rec = np.vstack([p.rec, [[(p.nx + 3) * p.h, 0, (p.nz + 3) * p.h], [-4 * p.h, 0, -4 * p.h]]]).astype(np.float32)
    out = {}
    for tag in ("tma", "plain"):
        if tag == "plain":
            monkeypatch.setenv("WAVEPROP_NO_TMA", "1")
        prop = wp.Propagator.from_problem(p)
        state = synth.random_state(5, prop.grid, 3)
        prop.set_state(state)
        prop.step(4)
        out[tag] = prop.get_state()
        tr = prop.forward(p.wavelet, p.src, p.rec)
        many = np.vstack([p.src] + [p.src[:1] + np.float32([[0.3 + i, 0, 0.4 + i]]) for i in range(4)])
        wav = np.vstack([p.wavelet, np.zeros((4, p.nt), np.float32)])
        np.testing.assert_array_equal(prop.forward(wav, many, p.rec), tr)      # injection kernel: the same bits
        out[tag] += [tr, prop.adjoint(tr, p.src, p.rec)]
        prop.close()
    # FP32 rounding of a few steps in another order
    for a, b in zip(out["tma"], out["plain"]):
        assert np.linalg.norm(a.astype(np.float64) - b) <= 2e-6 * np.linalg.norm(b.astype(np.float64))   # (0 where no wave has come)
        assert np.max(np.abs(a - b)) <= 1e-5 * np.max(np.abs(b))
    if shape[0] < 100:
        assert rel(out["tma"][5], oracle.Problem(p).forward()) <= 1e-5
