"""Which calls run on which passes, counted by their launches: comparisons of the
TMA-fed and the pipelined family compare two families, and the handles that stay on
packed rows do stay there."""
import numpy as np
import pytest

from test_gpu_rows import problem

pytestmark = pytest.mark.gpu

PASSES = {"acoustic": 1, "tti": 2, "elastic": 2}


def forward(wp, p, **kw):
    prop = wp.Propagator.from_problem(p, **kw)
    tr = prop.forward(p.wavelet, p.src, p.rec)
    n = prop.last_launches()
    prop.close()
    return tr, n


@pytest.mark.parametrize("nz", [40, 41, 42, 43])
@pytest.mark.parametrize("kind", sorted(PASSES))
def test_a_forward_step_is_its_passes(kind, nz, monkeypatch):
    """Whole and padded rows: sources and receivers are in the passes; many source cells, and the pipelined passes,
    take kernels of their own for them."""
    import paper_2004_10519_gb300 as wp
    p, steps = problem(kind, nz), PASSES[kind]
    assert steps * p.nt <= forward(wp, p)[1] < (steps + 1) * p.nt
    q = problem(kind, nz)
    for n, own in ((6, 0), (9, 1)):                # nodes 14 .. 17 and 14 .. 18: 16 cells, the most that a pass takes, 20
        q.src = np.vstack([p.src + np.float32([[3.3 * i, 0, -20]]) for i in range(n)]).astype(np.float32)
        q.wavelet = np.vstack([p.wavelet] * n)
        assert (steps + own) * p.nt <= forward(wp, q)[1] < (steps + own + 1) * p.nt
    monkeypatch.setenv("WAVEPROP_NO_TMA", "1")
    assert (steps + 2) * p.nt <= forward(wp, p)[1] < (steps + 3) * p.nt


@pytest.mark.parametrize("kind", sorted(PASSES))
def test_short_rows_are_not_padded(kind):
    """Computational nz 13: three floats of padding would be more than an eighth."""
    import paper_2004_10519_gb300 as wp
    p = problem(kind, 5)
    n = forward(wp, p)[1]
    assert (PASSES[kind] + 2) * p.nt <= n < (PASSES[kind] + 3) * p.nt


@pytest.mark.parametrize("kind", ["elastic", "acoustic"])
def test_16_bit_checkpoints_on_ragged_rows_stay_pipelined(kind):
    import paper_2004_10519_gb300 as wp
    p = problem(kind, 41)
    n = forward(wp, p, snap_mode=wp.SNAP_CKPT_BF16)[1]
    assert (PASSES[kind] + 2) * p.nt <= n < (PASSES[kind] + 3) * p.nt


@pytest.mark.parametrize("nz,same", [(40, False), (41, True), (42, True), (43, True)])
def test_staggered_pair_on_ragged_rows_stays_pipelined(nz, same, monkeypatch):
    """Both families take as many launches; they differ in last bits."""
    import paper_2004_10519_gb300 as wp
    p = problem("tti_sp", nz)
    a = forward(wp, p)[0]
    monkeypatch.setenv("WAVEPROP_NO_TMA", "1")
    assert np.array_equal(a, forward(wp, p)[0]) == same
