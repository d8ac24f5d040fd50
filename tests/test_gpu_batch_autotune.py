"""A batch's autotuning times the launches that its searches make: a short file whose
pattern-row tiles are shared by several blocks keeps the tile shape that shares them (the
same tiles whole take about twice as long, and other shapes win against those)."""
import numpy as np
import pytest

from tests.test_gpu_patterns import hp                                # noqa: F401
from tests.test_gpu_table_upload import _plan

pytestmark = pytest.mark.gpu


def test_short_file_keeps_shared_tiles(hp):                           # noqa: F811
    import torch
    nchans = 2048
    dms = np.linspace(0.0, 60.0, 200).astype(np.float32)
    with _plan(hp, dms, nchans) as p, _plan(hp, dms, nchans) as q:
        fb = torch.randint(0, 256, (8192 + p.max_delay, nchans), dtype=torch.uint8, device="cuda")
        want = hp.search(q, fb)
        assert q.dedisp_kernel() > 1
        b = hp.Batch([p])
        config, ms = b.autotune([fb])
        got = b.search([fb])[0]
        b.close()
        assert config == 17 and ms > 0 and p.dedisp_kernel() > 1
        assert np.array_equal(got, want)
