"""A call whose input is the first that the pattern rows pay for builds their tables, also
while another stream is being captured: that capture goes on."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_patterns import hp                                # noqa: F401
from tests.test_gpu_table_upload import BW, TSAMP, _plan

pytestmark = pytest.mark.gpu


def test_tables_built_beside_a_capture(hp):                           # noqa: F811
    import torch
    nchans, nout = 96, 60 * 2048 + 9        # (3000 samples: byte rows)
    dms = np.linspace(0.0, 600.0, 48).astype(np.float32)
    delays = oracle.delays(nchans, 1500.0, BW, TSAMP, dms)
    rng = np.random.Generator(np.random.PCG64(23))
    x = rng.integers(0, 256, size=(nout + int(delays.max()), nchans), dtype=np.uint8)
    fb = torch.from_numpy(x).cuda()
    with _plan(hp, dms, nchans) as p:
        p.bind_workspace(x.shape[0])
        hp.dedisperse(p, fb[:3000 + p.max_delay])
        allocs = hp.hp_plan_stats(p)["device_allocs"]
        out = torch.empty((48, nout + 3 & ~3), dtype=torch.int32, device="cuda")
        y = torch.zeros(4, device="cuda")
        side = torch.cuda.Stream()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):                                     # (global capture mode)
            y += 1
            hp.hp_dedisperse(p, fb, stream=side, out=out)
            y += 1
        g.replay()
        torch.cuda.synchronize()
        assert y.tolist() == [2.0] * 4
        assert hp.hp_plan_stats(p)["device_allocs"] == allocs + 1     # the tables
        assert np.array_equal(out[:, :nout].cpu().numpy(), oracle.dedisperse(x, delays))
