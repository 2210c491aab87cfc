"""Receivers sampled and sources added inside the forward passes: the same bits
as the kernels that do it for many source cells (reached here by further
sources with a zero wavelet), with sources and receivers on both sides of tile
and chunk edges and on the grid's first and last points."""
import numpy as np
import pytest

from test_gpu_rows import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz", [64, 41, 43])
@pytest.mark.parametrize("kind", ["tti", "elastic", "acoustic"])
def test_in_pass_sources_and_receivers(kind, nz):
    import paper_2004_10519_gb300 as wp
    p = problem(kind, nz, nt=12, shape=(41, 57))
    h, b = p.h, p.nbl
    at = lambda *q: [(c - b) * h for c in q]         # metres of a computational grid point
    NX, NY, NZ = p.nx + 2 * b, p.ny + 2 * b, nz + 2 * b
    for points in ([at(20, 15.5, 31), at(0, 0, 0), at(NX - 1, NY - 1, NZ - 1)],      # 2 + 1 + 1 cells
                   [at(7.5, 31.5, 31.25)],                                            # 8, across every edge
                   [at(NX - 1, 16, NZ - 1.5), at(8, 32, 32), at(9, 31, 32), at(9, 32.5, 33)]):
        src = np.array(points, np.float32)
        n = len(points)
        wav = np.vstack([(0.5 + 0.25 * i) * p.wavelet for i in range(n)]).astype(np.float32)
        rec = np.array(points + [at(x, y, z) for x in (0, 7.5, NX - 1) for y in (15.5, NY - 1) for z in (31.5, NZ - 1)] +
                       [at(3 + 0.01 * i, 20, 5) for i in range(400)], np.float32)
        far = np.array([at(30.5, 10.5, 10.5), at(31.5, 12.5, 12.5)], np.float32)
        prop = wp.Propagator.from_problem(p)
        a = prop.forward(wav, src, rec)
        sa = prop.get_state()
        c = prop.forward(np.vstack([wav, np.zeros((2, p.nt), np.float32)]), np.vstack([src, far]), rec)
        np.testing.assert_array_equal(a, c)
        assert np.abs(a).max() > 0
        for x, y in zip(sa, prop.get_state()):
            np.testing.assert_array_equal(x, y)
        prop.close()
