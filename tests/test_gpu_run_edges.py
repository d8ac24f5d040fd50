"""Runs above threshold where the 32-bit detection hands them on: from lane to lane
(16 starts), warp to warp (512), chunk to chunk (2048) and out of a segment (a multiple
of 2048), up to the end of the series, and more candidates in one chunk than it
collects before appending.  Raw candidates exact against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

NOUT = 9 * 2048 + 700           # two segments at this size (at least four chunks each)
WIDTHS = np.array([1, 2, 3, 8, 12, 16, 40, 64, 160], np.int32)


def _series(kind, rng, ndm):
    D = rng.integers(-2, 3, size=(ndm, NOUT)).astype(np.int64)      # (few values: many ties)
    if kind == "comb":              # a run of one start per raised sample
        D[:, 3000:7000:3] += 30
    elif kind == "end":
        for d in range(ndm):
            D[d, NOUT - 1 - 37 * d:] += 12
    else:                           # plateaus of `kind` samples around the hand-over points
        for d in range(ndm):
            for at in (16, 512, 2048, 3 * 2048 + 16, 4 * 2048, 5 * 2048, 6 * 2048 + 512):
                a = max(at + int(rng.integers(-2, 3)) - (kind if d % 2 else kind // 2), 0)
                D[d, a:a + kind] += 6 + d % 3
    return D.astype(np.int32)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("kind", [1, 15, 17, 511, 513, 1500, "comb", "end"])
def test_runs_over_edges(kind, mode):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_00398_gb300 as hp
    ndm = 6
    D = _series(kind, np.random.default_rng(3 + mode), ndm)
    # a window of many plateaus' length: they stay above the baseline
    raw_o, sig_o, mad_o = oracle.search_trials(D, 0, 1e-3, WIDTHS, 3.0, baseline_mode=mode,
                                               baseline_s=6.0)
    assert len(raw_o) > 0
    p = hp.Plan(16, 1500.0, -1.0, 1e-3, np.zeros(ndm, np.float32), WIDTHS, 3.0,
                baseline_mode=mode, baseline_s=6.0)
    raw_g, sig_g, mad_g = hp.detect(p, torch.from_numpy(D).cuda(), NOUT)
    assert np.array_equal(mad_g, mad_o) and np.array_equal(sig_g, sig_o)
    key = lambda rs: sorted((int(r["dm_idx"]), int(r["sample"]), int(r["width_idx"]), int(r["S"]))
                            for r in rs)
    assert key(raw_g) == key(raw_o)
