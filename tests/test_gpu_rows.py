"""Grids whose rows are not whole 16-byte units (computational NZ % 4 = 1, 2, 3)
run on the TMA-fed passes with padded rows.  Every point of a few steps from a
state without zeros agrees with the pipelined passes (WAVEPROP_NO_TMA=1), the
state comes back in packed rows, gradients meet the oracle's tolerance, shots
batch bitwise, and the calls that stay on the pipelined passes keep their bits."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

KINDS = ["tti", "tti_sp", "elastic", "acoustic"]


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def problem(kind, nz, so=8, nt=24, nbl=4, shape=(29, 35), h=10.0):
    nx, ny = shape
    seed = 3 + nz
    if kind == "elastic":
        m, vmax = synth.random_elastic(nx, ny, nz, seed, 3.0), None
    elif kind == "acoustic":
        m, vmax = {"vp": np.ascontiguousarray(synth.layered_vp(nx, ny, nz, seed, noise_sigma=3.0), np.float32)}, None
    else:
        m = synth.layered_tti(nx, ny, nz, seed, noise_sigma=3.0, smooth_sigma=1.5)
        vmax = float(np.max(m["vp"] * np.sqrt(1 + 2 * m["eps"])))
    dt = synth.cfl_dt(h, vmax or float(m["vp"].max()))
    src = np.array([[nx * h / 2 + 0.3, ny * h / 2 - 0.8, (nz + nbl - 1) * h - 6.0]], np.float32)
    rec = synth.carpet_receivers(5.0, 6.0, 3.3 * h, 7, 8, (nz + nbl - 1) * h)      # the last node of each row
    code = {"elastic": synth.ELASTIC, "acoustic": synth.ACOUSTIC}.get(kind, synth.TTI)
    return synth.Problem(code, nx, ny, nz, nbl, h, so, nt, dt, m, src,
                         synth.ricker(40.0, dt, nt)[None], rec, tti_op=int(kind == "tti_sp"))


@pytest.mark.parametrize("nz", [41, 42, 43, 5])
@pytest.mark.parametrize("kind", KINDS)
def test_every_point_agrees_with_the_pipelined_passes(kind, nz, monkeypatch):
    import paper_2004_10519_gb300 as wp
    p = problem(kind, nz)
    out = {}
    for tag in ("padded", "pipelined"):
        if tag == "pipelined":
            monkeypatch.setenv("WAVEPROP_NO_TMA", "1")
        prop = wp.Propagator.from_problem(p)
        state = synth.random_state(prop.nfields, prop.grid, 7)
        prop.set_state(state)
        for a, b in zip(prop.get_state(), state):
            np.testing.assert_array_equal(a, b)
        prop.step(3)
        out[tag] = prop.get_state()
        prop.set_state(state)
        prop.step(4, adjoint=True)
        out[tag] += prop.get_state()
        prop.close()
    for a, b in zip(out["padded"], out["pipelined"]):
        if kind.startswith("tti"):           # the centred TTI passes follow each other's rounding
            np.testing.assert_array_equal(a, b)
        else:                                # FP32 rounding of a few steps, as their traces are held to
            assert rel(a, b) <= 2e-6
            assert np.max(np.abs(a - b)) <= 1e-5 * np.max(np.abs(b))


@pytest.mark.parametrize("nz", [41, 42, 43])
@pytest.mark.parametrize("kind", ["tti", "elastic", "acoustic"])
def test_gradient_parity(kind, nz):
    import paper_2004_10519_gb300 as wp
    p = problem(kind, nz)
    o = oracle.Problem(p)
    ref = o.forward()
    d = (0.5 * ref).astype(np.float32)
    prop = wp.Propagator.from_problem(p, snap_mode=wp.SNAP_CKPT_FP32)
    assert rel(prop.forward(p.wavelet, p.src, p.rec), ref) <= 1e-5
    g, J = prop.gradient(p.wavelet, p.src, p.rec, d)
    g_ref, J_ref = o.gradient(d)
    assert abs(J - J_ref) <= 1e-5 * J_ref
    for a, b in zip(np.reshape(g, (-1,) + prop.shape), np.reshape(g_ref, (-1,) + prop.shape)):
        assert rel(a, b) <= 1e-4
    prop.close()


@pytest.mark.parametrize("kind", ["tti", "elastic"])
def test_batched_shots_are_bitwise_single_calls(kind):
    import paper_2004_10519_gb300 as wp
    ps = [problem(kind, 41, shape=s) for s in ((29, 35), (22, 31))]
    props = [wp.Propagator.from_problem(p, snap_mode=wp.SNAP_CKPT_FP32) for p in ps]
    W, S, R = [p.wavelet for p in ps], [p.src for p in ps], [p.rec for p in ps]
    ones = [q.forward(*a) for q, a in zip(props, zip(W, S, R))]
    for a, b in zip(wp.forward_batch(props, W, S, R), ones):
        np.testing.assert_array_equal(a, b)
    D = [0.5 * t for t in ones]
    grads = [q.gradient(*a)[0] for q, a in zip(props, zip(W, S, R, D))]
    for a, b in zip(wp.gradient_batch(props, W, S, R, D)[0], grads):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("kind", ["tti", "tti_sp", "elastic", "acoustic"])
def test_calls_that_keep_the_pipelined_bits(kind, monkeypatch):
    """16-bit checkpoints, every TTI sweep, and the gradient of every TTI parameter."""
    import paper_2004_10519_gb300 as wp
    p = problem(kind, 43)
    out = {}
    for tag in ("default", "pipelined"):
        if tag == "pipelined":
            monkeypatch.setenv("WAVEPROP_NO_TMA", "1")
        prop = wp.Propagator.from_problem(p, snap_mode=wp.SNAP_CKPT_BF16)
        tr = prop.forward(p.wavelet, p.src, p.rec)
        out[tag] = [tr, prop.gradient(p.wavelet, p.src, p.rec, 0.5 * tr)[0]]
        full = wp.Propagator.from_problem(p)
        if kind.startswith("tti"):
            out[tag] += [full.adjoint(tr, p.src, p.rec), full.gradient(p.wavelet, p.src, p.rec, 0.5 * tr)[0]]
        if kind == "tti":
            out[tag].append(full.gradient_aniso(p.wavelet, p.src, p.rec, 0.5 * tr)[0])
    for a, b in zip(out["default"], out["pipelined"]):
        np.testing.assert_array_equal(a, b)


def test_staggered_pair_gradient_is_still_refused():
    import paper_2004_10519_gb300 as wp
    p = problem("tti_sp", 41)
    prop = wp.Propagator.from_problem(p)
    with pytest.raises(wp.PropError) as e:
        prop.gradient_aniso(p.wavelet, p.src, p.rec, np.zeros((p.rec.shape[0], p.nt), np.float32))
    assert e.value.code == wp.PROP_EINVAL


@pytest.mark.parametrize("kind", ["tti", "elastic"])
def test_noalloc_modelling_is_bitwise_the_handle(kind):
    import ctypes as C
    import paper_2004_10519_gb300 as wp
    p = problem(kind, 41)
    ref = wp.Propagator.from_problem(p).forward(p.wavelet, p.src, p.rec)
    q = wp.PropDesc(p.kind, p.nx, p.ny, p.nz, p.nbl, p.h, p.so, p.nt, p.dt, 0.0, 0, 0, 0, 0)
    model = p.model_list()
    ptr = lambda a: C.c_void_p(a.ctypes.data)
    out = np.zeros_like(ref)
    L = wp.lib()
    L.prop_forward_noalloc.argtypes = [C.POINTER(wp.PropDesc), C.POINTER(C.c_void_p), C.c_void_p, C.c_void_p, C.c_int,
                                       C.c_void_p, C.c_int, C.c_void_p, C.c_void_p]
    rc = L.prop_forward_noalloc(C.byref(q), (C.c_void_p * len(model))(*[ptr(a) for a in model]), ptr(p.wavelet),
                                ptr(p.src), 1, ptr(p.rec), p.rec.shape[0], ptr(out), None)
    assert rc == 0, L.prop_last_error(None)
    np.testing.assert_array_equal(out, ref)
