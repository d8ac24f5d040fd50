"""The list lengths at which the merge leaves its one block for the whole GPU (1280
candidates, 1088 with friend scans, fewer with many trials in reach) and takes two
candidates a thread (1025), against the oracle; and a dense list whose friend scans one
block would make alone."""
import numpy as np
import pytest

import oracle
from tests.raw_lists import raw_list
from tests.test_gpu_merge_paths import _same

pytestmark = pytest.mark.gpu
NDM, NOUT = 400, 200_000


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_00398_gb300 as hp
    from paper_2512_00398_gb300 import synth
    return torch, hp, synth.widths_pow2(4096)


def _upload(torch, hp, recs, sigma):
    host = np.zeros(recs.size, hp.RAW_DTYPE)
    for f in ("dm_idx", "width_idx", "sample", "S"):
        host[f] = recs[f]
    return (torch.from_numpy(host.view(np.uint8).copy()).cuda(),
            torch.tensor([recs.size], dtype=torch.int64, device="cuda"),
            torch.from_numpy(sigma.astype(np.float64)).cuda())


def _plan(hp, widths, **kw):
    return hp.Plan(16, 1500.0, -1.0, 1e-3, np.arange(NDM, dtype=np.float32), widths, 6.0,
                   raw_capacity=65536, **kw)


# (any width a friend's, or friend scans)
@pytest.mark.parametrize("dm_tol,w_tol,limit", [
    (0, 13, 1280), (1, 13, 1280), (1, 13, 1024), (16, 13, 1024), (70, 13, 234), (399, 13, 41),
    (0, 1, 1088), (1, 1, 1088), (1, 1, 1024), (9, 1, 910), (70, 1, 117), (399, 1, 32)])
def test_around_the_limit(env, dm_tol, w_tol, limit):
    torch, hp, widths = env
    recs, sigma = raw_list(31, 1500, ndm=NDM, nout=NOUT, nw=13, members=(5, 60), dm_spread=3, t_spread=60)
    with _plan(hp, widths, dm_tol=dm_tol, w_tol=w_tol) as p:
        for n in (limit - 1, limit, limit + 1):
            raw, cnt, sig = _upload(torch, hp, recs[:n], sigma)
            want = oracle.merge(oracle.raw_with_snr(recs[:n], sigma, widths), widths, dm_tol=dm_tol, w_tol=w_tol)
            data, count = hp.hp_merge(p, raw, cnt, sig)
            assert hp.hp_plan_sync_status(p) == hp.HP_OK
            _same(hp.cands_to_numpy(data, count), want)


def test_dense_friend_scans_use_the_whole_gpu(env):
    """2000 clustered candidates, 64 trials in reach: as fast as with 100 isolated ones
    more, which one block's shared memory never held."""
    torch, hp, widths = env
    recs, sigma = raw_list(3, 2000, ndm=NDM, nout=NOUT, nw=13)
    far = np.zeros(100, recs.dtype)
    far["dm_idx"], far["sample"], far["S"] = 0, 10 * NOUT + 10_000 * np.arange(100), 50
    us = []
    with _plan(hp, widths, dm_tol=64, w_tol=1) as p:
        for r in (recs, np.concatenate([recs, far])):
            raw, cnt, sig = _upload(torch, hp, r, sigma)
            out = hp.new_cand_buf(1 << 16)
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            best = np.inf
            for _ in range(5):
                e[0].record()
                for _ in range(5):
                    hp.hp_merge(p, raw, cnt, sig, out=out)
                e[1].record()
                torch.cuda.synchronize()
                best = min(best, e[0].elapsed_time(e[1]) * 200.0)
            us.append(best)
    assert us[0] < 1.5 * us[1], us
