"""Statistics and detection of few or short series: every span of the |y| histogram's
threads (32, 64 or 256 samples, by padding and block count), at its blocks' edges and
below one block; exact against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

WIDTHS = np.array([1, 2, 4, 12, 16], np.int32)
DISTINCT = 5      # rows; the trials repeat them
# spans of 32: a block of 8192 samples; of 64: 16384; of 256: 65536
CASES = [(5, 40), (5, 8191), (5, 8192), (5, 8193), (45, 24_576),
         (600, 700), (310, 16_384), (310, 16_387), (300, 65_536), (150, 131_071)]


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("ndm,nout", CASES)
def test_short_series(ndm, nout, mode):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_00398_gb300 as hp
    rng = np.random.default_rng(nout + mode)
    rows = rng.normal(0, 40, (DISTINCT, nout)).round().astype(np.int32)
    rows += (np.arange(nout) // 50 % 40).astype(np.int32)           # a baseline to follow
    rows[3] *= 200                                                  # a MAD above 4096: refined
    for d in range(DISTINCT):
        at = int(rng.integers(0, max(1, nout - 30)))
        rows[d, at:at + 25] += 400
    raw_o, sig_o, mad_o = oracle.search_trials(rows, 0, 1e-3, WIDTHS, 5.0, baseline_mode=mode,
                                               baseline_s=0.3)
    which = np.arange(ndm) % DISTINCT
    p = hp.Plan(16, 1500.0, -1.0, 1e-3, np.zeros(ndm, np.float32), WIDTHS, 5.0,
                baseline_mode=mode, baseline_s=0.3)
    raw_g, sig_g, mad_g = hp.detect(p, torch.from_numpy(rows[which]).cuda(), nout)
    assert np.array_equal(mad_g, mad_o[which]) and np.array_equal(sig_g, sig_o[which])
    assert mad_o[3] > 4096 or nout == 40
    want = [[] for _ in range(DISTINCT)]
    for r in raw_o:
        want[int(r["dm_idx"])].append((int(r["sample"]), int(r["width_idx"]), int(r["S"])))
    got = [[] for _ in range(ndm)]
    for r in raw_g:
        got[int(r["dm_idx"])].append((int(r["sample"]), int(r["width_idx"]), int(r["S"])))
    assert len(raw_o) > 0 or nout == 40
    for d in range(ndm):
        assert sorted(got[d]) == sorted(want[d % DISTINCT]), d
