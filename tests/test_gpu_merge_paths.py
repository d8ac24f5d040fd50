"""hp_merge and hp_merge_static over the paths of the merge: the one-block path (up
to 2048 candidates) and the general one, components by running maxima (any width a
friend's, t_gap >= 0) and friend scans otherwise, at list sizes around the sort's and
the scans' block edges, against the oracle's merge (exact clusters)."""
import numpy as np
import pytest

import oracle
from tests.raw_lists import raw_list

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 33, 64, 65, 1023, 1025, 2047, 2048, 2049, 3073, 8192, 8193, 40_001]
NDM, NOUT = 60, 30_000


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_00398_gb300 as hp
    from paper_2512_00398_gb300 import synth
    recs, sigma = raw_list(21, 42_000, ndm=NDM, nout=NOUT, nw=8, members=(5, 60), dm_spread=3,
                           t_spread=60)
    return torch, hp, synth.widths_pow2(128), recs, sigma


def _same(got, want):
    key = lambda c: (int(c["dm_idx"]), int(c["sample"]), int(c["width_idx"]))
    assert [key(c) for c in got] == [key(c) for c in want]
    for f in ("members", "dm_lo", "dm_hi", "t_lo", "t_hi"):
        assert np.array_equal(got[f].astype(np.int64), want[f].astype(np.int64)), f
    # one FP64 value, rounded to FP32 once
    assert np.abs(got["snr"].astype(np.float64) - want["snr"]).max() <= 1e-4


# default; gaps; a gap past every sample; negative gaps (overlaps); few widths friends
TOLERANCES = [(1, 0, 8), (0, 0, 8), (3, 25, 7), (1, 10 ** 15, 8), (70, 0, 8), (1, -3, 8), (2, 5, 1),
              (1, 0, 0)]
# (the oracle's scans of the longest list take too long for the last four)
CASES = [(n, *t) for t in TOLERANCES for n in SIZES if n <= 8193 or t in TOLERANCES[:4]]


@pytest.mark.parametrize("n,dm_tol,t_gap,w_tol", CASES)
def test_paths(env, n, dm_tol, t_gap, w_tol):
    torch, hp, widths, recs, sigma = env
    r = recs[:n]
    want = oracle.merge(oracle.raw_with_snr(r, sigma, widths), widths, dm_tol=dm_tol, t_gap=t_gap,
                        w_tol=w_tol)
    p = hp.Plan(16, 1500.0, -1.0, 1e-3, np.arange(NDM, dtype=np.float32), widths, 6.0,
                raw_capacity=65536, dm_tol=dm_tol, t_gap=t_gap, w_tol=w_tol)
    host = np.zeros(n, hp.RAW_DTYPE)
    for f in ("dm_idx", "width_idx", "sample", "S"):
        host[f] = r[f]
    raw = torch.from_numpy(host.view(np.uint8).copy()).cuda()
    cnt = torch.tensor([n], dtype=torch.int64, device="cuda")
    sig = torch.from_numpy(sigma.astype(np.float64)).cuda()
    data, count = hp.hp_merge(p, raw, cnt, sig, capacity=want.size + 3)
    assert hp.hp_plan_sync_status(p) == hp.HP_OK and int(count.item()) == want.size
    _same(hp.cands_to_numpy(data, count), want)
    if dm_tol < 70:
        data, count = hp.hp_merge_static(raw, cnt, sig, widths, dm_tol=dm_tol, t_gap=t_gap, w_tol=w_tol,
                                         capacity=want.size + 3)
        assert int(count.item()) == want.size
        _same(hp.cands_to_numpy(data, count), want)
    p.close()


def test_empty_and_truncated(env):
    torch, hp, widths, recs, sigma = env
    p = hp.Plan(16, 1500.0, -1.0, 1e-3, np.arange(NDM, dtype=np.float32), widths, 6.0,
                raw_capacity=65536)
    host = np.zeros(3000, hp.RAW_DTYPE)
    for f in ("dm_idx", "width_idx", "sample", "S"):
        host[f] = recs[:3000][f]
    raw = torch.from_numpy(host.view(np.uint8).copy()).cuda()
    sig = torch.from_numpy(sigma.astype(np.float64)).cuda()
    none = torch.zeros(1, dtype=torch.int64, device="cuda")
    _, count = hp.hp_merge(p, raw, none, sig)
    assert int(count.item()) == 0
    # a count past the buffer: its entries merged, the overflow reported
    many = torch.tensor([5000], dtype=torch.int64, device="cuda")
    data, count = hp.hp_merge(p, raw, many, sig)
    assert hp.hp_plan_sync_status(p) == hp.HP_ERR_CAND_OVERFLOW
    want = oracle.merge(oracle.raw_with_snr(recs[:3000], sigma, widths), widths)
    _same(hp.cands_to_numpy(data, count), want)
    p.close()
