"""Device memory of a stream whose plan takes the pattern rows: device_bytes counts their
tables, so a budget of that many bytes holds the same stream again."""
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
