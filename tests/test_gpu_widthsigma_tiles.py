"""Per-width MADs where the selection's tiles end (15360 starts, 16384 for trials whose
sums need 64 bits), with widths that are and are not multiples of 16, trials of both
kinds in one call, enough tiles that a block takes several, and medians in the coarse
bins or beyond the first pass; exact against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

WIDTHS = np.array([1, 3, 8, 16, 17, 160, 1024], np.int32)


def rows(nout):
    rng = np.random.default_rng(nout)
    D = rng.normal(0, 30, (6, nout)).round().astype(np.int64)
    D[1] = D[1] * 900 + np.cumsum(rng.integers(-9, 10, nout))       # second and third digits
    D[2] = np.where(np.arange(nout) % 5 < 2, 700, 0)                # MAD 0: the coarse bins
    D[3] = np.where(np.arange(nout) % 5 < 2, 100_000, 0)            # beyond the first pass
    for d in (4, 5):                                                # sums of 64 bits
        D[d, rng.integers(0, nout, 40)] += (1 << 24) * (1 if d == 4 else -1)
    return D.astype(np.int32)


@pytest.mark.parametrize("nout", [1025, 15_359, 15_360, 15_361, 30_737, 140_001])
def test_tiles(nout):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_00398_gb300 as hp
    D = rows(nout)
    p = hp.Plan(64, 1500.0, -1.0, 1e-3, np.zeros(6, np.float32), WIDTHS, 6.0, width_sigma=1)
    hp.detect(p, torch.from_numpy(D).cuda(), nout)
    assert hp.hp_plan_sync_status(p) == hp.HP_OK
    sg, md = (t.cpu().numpy() for t in hp.hp_width_sigmas(p))
    win = oracle.baseline_window(2.0, 1e-3)
    for d in range(6):
        m_o, s_o = oracle.width_sigma(oracle.subtract_baseline(D[d], 0, win), WIDTHS)
        assert np.array_equal(md[d], m_o), (d, md[d], m_o)
        assert np.array_equal(sg[d], s_o), d
