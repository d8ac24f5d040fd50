"""The choice of the dedispersion kernel on trial grids that widen with the DM: their last
tiles share few partial sums and end a short launch, so byte rows run although the average
tile would be cheaper as pattern rows (1.4 to 2.3 times as slow there); where the last
tiles share enough, pattern rows."""
import numpy as np
import pytest

import oracle
from paper_2512_00398_gb300 import synth
from tests.test_gpu_patterns import hp                                # noqa: F401

pytestmark = pytest.mark.gpu
TSAMP = 49.152e-6


def _grid(nchans, ndm, dm_hi, nout):
    o = synth.Observation(nchans=nchans, f_top=1500.0, chan_bw=-500.0 / nchans, tsamp=TSAMP,
                          nsamps=nout + 3000, mean=128.0, sigma=12.0)
    return synth.dm_list_smearing(o, 0.0, dm_hi, ndm)


# (whole tiles, parts of tiles; the widest grid in two waves)
@pytest.mark.parametrize("nchans,ndm,dm_hi,nout,patterns", [
    (512, 240, 312.0, 8000, False), (256, 120, 75.0, 20000, False), (512, 240, 312.0, 22900, False),
    (512, 375, 234.0, 8000, False), (1024, 24, 31.0, 20000, True), (4096, 375, 488.0, 40000, True)])
def test_kernel_on_a_widening_grid(hp, nchans, ndm, dm_hi, nout, patterns):   # noqa: F811
    import torch
    dms = _grid(nchans, ndm, dm_hi, nout)
    with hp.Plan(nchans, 1500.0, -500.0 / nchans, TSAMP, dms, synth.widths_pow2(16), 6.0) as p:
        rng = np.random.Generator(np.random.PCG64(ndm))
        x = rng.integers(0, 256, size=(nout + p.max_delay, nchans), dtype=np.uint8)
        fb = torch.from_numpy(x).cuda()
        got = hp.hp_dedisperse(p, fb)
        torch.cuda.synchronize()
        assert (p.dedisp_kernel() > 0) == patterns
        # the first and the last trial, which differ most
        delays = oracle.delays(nchans, 1500.0, -500.0 / nchans, TSAMP, dms)
        for d in (0, ndm - 1):
            want = np.zeros(nout, np.int64)
            for c in range(nchans):
                want += x[delays[d, c]:delays[d, c] + nout, c]
            assert np.array_equal(got[d, :nout].cpu().numpy(), want)
