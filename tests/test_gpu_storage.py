"""Forward steps write stored levels into the storage itself (full storage, the
full-storage tail and recomputed segments), which then serves as the state.
The final state after a saved run is that of a plain one, and every storage
form gives the gradient of full storage bit for bit (FP32 recomputation is
exact), for the shortest runs, where every level is the first or the last, too."""
import numpy as np
import pytest

from test_gpu_rows import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nt", [2, 3, 4, 9])
@pytest.mark.parametrize("kind", ["tti", "tti_sp", "elastic", "acoustic"])
def test_storage_forms_agree(kind, nt, monkeypatch):
    import paper_2004_10519_gb300 as wp
    p = problem(kind, 40, nt=nt)
    p.rec = np.vstack([p.rec, p.src + np.float32(11.0) * np.array([[1, 0, -1]], np.float32)]).astype(np.float32)
    d = np.random.default_rng(2).standard_normal((p.rec.shape[0], nt)).astype(np.float32)
    ref = wp.Propagator.from_problem(p)
    tr = ref.forward(p.wavelet, p.src, p.rec)
    state = ref.get_state()
    out = {}
    for tag, mode, K, tail in (("full", wp.SNAP_FULL_FP32, 0, None), ("tail", wp.SNAP_CKPT_FP32, 0, None),
                               ("part", wp.SNAP_CKPT_FP32, 2, "2"), ("segments", wp.SNAP_CKPT_FP32, 2, "0")):
        if tail is None:
            monkeypatch.delenv("WAVEPROP_CKPT_TAIL", raising=False)
        else:
            monkeypatch.setenv("WAVEPROP_CKPT_TAIL", tail)
        prop = wp.Propagator.from_problem(p, snap_mode=mode, ckpt_interval=K)
        np.testing.assert_array_equal(prop.forward(p.wavelet, p.src, p.rec, save=True), tr)
        for a, b in zip(prop.get_state(), state):
            np.testing.assert_array_equal(a, b)
        g, _ = prop.backward(d, nsrc=1)
        out[tag] = [g, prop.gradient(p.wavelet, p.src, p.rec, tr - d)[0]]
        np.testing.assert_array_equal(prop.forward(p.wavelet, p.src, p.rec), tr)      # the handle's arrays are whole
        prop.close()
    for tag in ("tail", "part", "segments"):
        for a, b in zip(out[tag], out["full"]):
            np.testing.assert_array_equal(a, b)
