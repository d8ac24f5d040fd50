"""The kernel that each plan's dedispersion took (hp_plan_dedisp_kernel), at the shapes of
the pattern-row tests -- so that those compare the kernel they name -- and its sums where
the byte rows are kept."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_patterns import hp                                # noqa: F401
from tests.test_gpu_table_upload import BW, TSAMP, _plan

pytestmark = pytest.mark.gpu
WHOLE = [(64, 48, 60 * 2048, 0, 60), (64, 47, 60 * 2048 + 1, 0, 60), (65, 49, 45 * 2048 - 1, 0, 60),
         (66, 48, 60 * 2048 - 1023, 0, 60), (67, 48, 60 * 2048 - 1025, 0, 60),
         (259, 48, 59 * 2048 + 3, 0, 60), (5, 48, 60 * 2048 + 5, 0, 60), (256, 48, 60 * 2048 + 7, 0, 30),
         (515, 48, 60 * 2048 + 7, 0, 30), (203, 48, 60 * 2048 + 11, 0, 0),
         (203, 48, 60 * 2048 + 11, 500, 530), (203, 48, 60 * 2048 + 11, 3000, 3060)]
PARTS = [(1024, 24, 3 * 2048 + 5), (1027, 47, 2048), (1101, 49, 2049), (2048, 25, 1000),
         (1024, 48, 8 * 2048 - 1023), (4096, 30, 700), (640, 72, 52 * 2048 + 3), (1024, 48, 3000)]


def _kernel(hp, nchans, ndm, nout, lo, hi, config=None):              # noqa: F811
    import torch
    with _plan(hp, np.linspace(lo, hi, ndm).astype(np.float32), nchans) as p:
        with pytest.raises(hp.HPError):
            p.dedisp_kernel()                      # nothing was dedispersed yet
        if config is not None:
            p.set_param("dedisp_config", config)
        hp.hp_dedisperse(p, torch.zeros((nout + p.max_delay, nchans), dtype=torch.uint8, device="cuda"))
        torch.cuda.synchronize()
        return p.dedisp_kernel()


@pytest.mark.parametrize("shape", WHOLE)
def test_pattern_rows(hp, shape):                                     # noqa: F811
    assert _kernel(hp, *shape) >= 1
    assert _kernel(hp, *shape, config=12) == 0


@pytest.mark.parametrize("shape", PARTS)
def test_shared_tiles(hp, shape):                                     # noqa: F811
    assert _kernel(hp, *shape, 0, 30) > 1


# (unlike trials; a single wave of byte rows)
@pytest.mark.parametrize("nchans,bw,ndm,hi,nout", [(128, -1.953125, 100, 400, 70001),
                                                   (96, BW, 48, 600, 3001)])
def test_byte_rows_kept(hp, nchans, bw, ndm, hi, nout):               # noqa: F811
    import torch
    from paper_2512_00398_gb300 import synth
    dms = np.linspace(0, hi, ndm).astype(np.float32)
    delays = oracle.delays(nchans, 1500.0, bw, TSAMP, dms)
    rng = np.random.Generator(np.random.PCG64(nchans))
    x = rng.integers(0, 256, size=(nout + int(delays.max()), nchans), dtype=np.uint8)
    with hp.Plan(nchans, 1500.0, bw, TSAMP, dms, synth.widths_pow2(16), 6.0) as p:
        assert np.array_equal(hp.dedisperse(p, torch.from_numpy(x).cuda()), oracle.dedisperse(x, delays))
        assert p.dedisp_kernel() == 0


def test_batch_and_subband_plans(hp):                                 # noqa: F811
    import torch
    x = torch.zeros((6000, 1024), dtype=torch.uint8, device="cuda")
    dms = np.linspace(0.0, 30.0, 48).astype(np.float32)
    with _plan(hp, dms, 1024) as p, _plan(hp, dms, 1024) as q:
        q.set_param("subband_chans", 64)
        b = hp.Batch([p, q])
        for _ in range(3):                         # eager, captured, replayed
            b.search([x, x])
            assert p.dedisp_kernel() > 1 and q.dedisp_kernel() == 0
        b.close()
