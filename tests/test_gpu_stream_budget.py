"""Device memory of a stream whose plan takes the pattern rows: device_bytes counts their
tables, so a budget of that many bytes holds the same stream again; a budget without room
for them holds the same slots, on byte rows."""
import numpy as np
import pytest

from paper_2512_00398_gb300 import synth
from tests.test_gpu_patterns import hp                                # noqa: F401

pytestmark = pytest.mark.gpu
NCH, G, NB = 1024, 8192, 3


@pytest.fixture(scope="module")
def plan(hp):                                                         # noqa: F811
    dms = np.linspace(0.0, 30.0, 48).astype(np.float32)
    p = hp.Plan(NCH, 1500.0, -500.0 / 4096, 49.152e-6, dms, synth.widths_pow2(16), 6.0)
    yield p
    p.close()


def _open(hp, plan, **kw):                                            # noqa: F811
    """(step slots, beam slots, device bytes) of a stream, and the stream."""
    st = hp.Stream(plan, nbeams=NB, gulp=G, cand_capacity=256, **kw)
    s = st.stats()
    return (s["max_batch"], s["beam_slots"], s["device_bytes"]), st


def test_device_bytes_reopen_the_stream(hp, plan):                    # noqa: F811
    want, st = _open(hp, plan)
    st.close()
    assert want[:2] == (NB, NB)
    got, st = _open(hp, plan, hbm_budget=want[2])
    st.close()
    assert got == want


def test_slots_come_before_the_pattern_tables(hp, plan):              # noqa: F811
    import torch
    want, st = _open(hp, plan)
    st.close()
    got, st = _open(hp, plan, hbm_budget=want[2] - 1)
    assert got[:2] == want[:2] and got[2] < want[2]
    # two gulps of every beam: the whole file's window of each is as the search's own
    n = 2 * G
    rng = np.random.Generator(np.random.PCG64(3))
    x = [rng.integers(0, 40, size=(n, NCH), dtype=np.uint8) for _ in range(NB)]
    for b in range(NB):
        x[b][3000 + 100 * b:3004 + 100 * b] += 90
        for g in range(2):
            st.push(b, x[b][g * G:(g + 1) * G])
    found = {}
    while len(found) < 2 * NB:
        info, c = st.poll(timeout_ms=60000)
        assert info["status"] == hp.HP_OK
        found[info["beam"], info["gulp_index"]] = c
    st.close()
    for b in range(NB):
        # the first gulp's window starts at 0 and its series is the file's
        got = found[b, 0]
        want = hp.search(plan, torch.from_numpy(x[b][:G]).cuda())
        near = lambda c: c[np.abs(c["sample"] - 3000 - 100 * b) < 8]   # noqa: E731
        assert len(near(want)) > 0 and np.array_equal(near(got), near(want))
