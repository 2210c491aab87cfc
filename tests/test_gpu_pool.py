"""The library's pool of device memory: blocks are freed after the work of the
stream that used them, whatever other threads do meanwhile."""
import glob
import os
import threading

import numpy as np
import pytest

from test_gpu_rows import problem

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2004_10519_gb300", "csrc")


def test_no_device_wide_synchronisation():
    """It is refused while any stream of the device is captured, by another thread too: what it was to wait for
    would not have been waited for."""
    for f in glob.glob(os.path.join(CSRC, "*")):
        with open(f) as src:
            assert "cudaDeviceSynchronize" not in src.read(), f


@pytest.mark.gpu
def test_frees_beside_captures_of_another_thread(monkeypatch):
    import paper_2004_10519_gb300 as wp
    monkeypatch.setenv("WAVEPROP_GRAPHS", "1")           # prop_step must capture
    p, q = problem("tti", 41), problem("elastic", 40, shape=(40, 33))
    state = [np.random.default_rng(5).standard_normal((37, 43, 49), np.float32) for _ in range(4)]

    def steps(prop):
        out = []
        for n in (4, 5, 7):
            prop.set_state(state)
            prop.step(n)
            out += prop.get_state()
            prop.trim()                                   # other buffers next time, so another capture
        return out

    def gradients(prop):
        out = []
        for scale in (0.5, 0.25, 0.0):
            out.append(prop.gradient(q.wavelet, q.src, q.rec, scale * d)[0])
            prop.trim()
        return out

    a, b = wp.Propagator.from_problem(p), wp.Propagator.from_problem(q, snap_mode=wp.SNAP_CKPT_FP32)
    assert a.grid == state[0].shape
    d = b.forward(q.wavelet, q.src, q.rec)
    serial = steps(a), gradients(b)
    got, errors = {}, []

    def run(name, f, prop):
        try:
            got[name] = [f(prop) for _ in range(8)]
        except Exception as e:                            # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=run, args=x) for x in (("steps", steps, a), ("gradients", gradients, b))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for name, ref in zip(("steps", "gradients"), serial):
        for round_ in got[name]:
            for x, y in zip(round_, ref):
                np.testing.assert_array_equal(x, y)


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _acoustic(wp, nt, n=192):
    vp = np.full((n, n, n), 2.0, np.float32)
    return wp.Propagator(wp.PROP_ACOUSTIC, (n, n, n), 4, 10.0, 4, nt, [vp], snap_mode=wp.SNAP_FULL_FP32)


def _gradient(prop, nt):
    wav = np.ones((1, nt), np.float32)
    at = np.full((1, 3), 500.0, np.float32)
    return prop.gradient(wav, at, at, np.zeros((1, nt), np.float32))[0]


@pytest.mark.gpu
def test_a_destroyed_handle_returns_its_memory_beside_others():
    import paper_2004_10519_gb300 as wp
    other, warm = _acoustic(wp, 4), _acoustic(wp, 4)
    _gradient(warm, 4)
    warm.close()
    other.trim()                                          # what the call's buffers left goes too
    before = _free()
    prop = _acoustic(wp, 40)                              # model and state: four fields of 31 MB
    assert before - _free() > 60 << 20
    prop.close()
    assert before - _free() < 8 << 20
    prop = _acoustic(wp, 40)
    _gradient(prop, 40)                                   # leaves the buffers of a call
    held = _free()
    prop.close()
    assert _free() - held > 100 << 20                     # its own memory and the adjoint state's, at least
    other.trim()
    assert before - _free() < 8 << 20                     # and all that is unused
    other.close()


@pytest.mark.gpu
def test_allocation_takes_what_the_pool_holds_unused():
    """A block larger than what the device has free and than any that the pool holds, but not than both."""
    import torch
    import paper_2004_10519_gb300 as wp
    a, b = _acoustic(wp, 60), _acoustic(wp, 80)
    _gradient(b, 80)                                      # modules, and what the answer is
    ref = _gradient(b, 80)
    b.trim()
    full = _free()
    _gradient(a, 60)
    assert full - _free() > 1500 << 20                    # 59 levels of 32 MB, now unused
    rest = torch.empty(_free() - (1 << 30), dtype=torch.uint8, device="cuda")
    assert _free() < 1100 << 20
    np.testing.assert_array_equal(_gradient(b, 80), ref)  # 79 levels
    del rest
    torch.cuda.empty_cache()
    a.trim()
    b.trim()
    assert _free() > full - (300 << 20)                   # the work arrays went too; models stay
