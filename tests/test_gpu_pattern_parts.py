"""Pattern-row tiles shared by several blocks: the last time columns of a launch whose
last wave would be nearly empty, or all of a short input's.  Exact sums against the
oracle at tile edges (24 trials x 2048 samples), odd channel counts, the largest
samples, next to whole tiles in one launch, and under capture."""
import numpy as np
import pytest

import oracle
from paper_2512_00398_gb300 import synth
from tests.test_gpu_patterns import _kernels, hp                      # noqa: F401

pytestmark = pytest.mark.gpu
BW, TSAMP = -500.0 / 4096, 49.152e-6


def _plan(hp, nchans, ndm, dm_hi):
    dms = np.linspace(0.0, dm_hi, ndm).astype(np.float32)
    return dms, hp.Plan(nchans, 1500.0, BW, TSAMP, dms, synth.widths_pow2(16), 6.0)


# (the last: 53 time columns of three tiles, 159 blocks where 152 fit)
@pytest.mark.parametrize("nchans,ndm,nout,fill", [
    (1024, 24, 3 * 2048 + 5, None), (1027, 47, 2048, None), (1101, 49, 2049, None),
    (2048, 25, 1000, None), (1024, 48, 8 * 2048 - 1023, 255), (4096, 30, 700, 255),
    (640, 72, 52 * 2048 + 3, None)])
def test_parts_exact(hp, nchans, ndm, nout, fill):                    # noqa: F811
    import torch
    dms, p = _plan(hp, nchans, ndm, 30.0)
    rng = np.random.Generator(np.random.PCG64(nchans))
    n = nout + p.max_delay
    x = (rng.integers(0, 256, size=(n, nchans), dtype=np.uint8) if fill is None
         else np.full((n, nchans), fill, np.uint8))
    fb = torch.from_numpy(x).cuda()
    want = oracle.dedisperse(x, oracle.delays(nchans, 1500.0, BW, TSAMP, dms))
    out = []
    names = _kernels(lambda: out.append(hp.dedisperse(p, fb)))
    assert not names or any("dedisp_patterns_kernel<true>" in k for k in names)
    assert np.array_equal(out[0], want)
    # a second call adds to zeros again
    assert np.array_equal(hp.dedisperse(p, fb), want)
    p.close()


def test_parts_captured(hp):                                          # noqa: F811
    import torch
    nchans, ndm, nout = 1024, 48, 3000
    rng = np.random.Generator(np.random.PCG64(5))
    _, p1 = _plan(hp, nchans, ndm, 30.0)
    _, p2 = _plan(hp, nchans, ndm, 30.0)
    p2.set_param("dedisp_config", 12)                                 # byte rows
    x = rng.integers(0, 40, size=(nout + p1.max_delay, nchans), dtype=np.uint8)
    x[1000:1004] += 90
    fb = torch.from_numpy(x).cuda()
    want = hp.search(p2, fb)
    b = hp.Batch([p1])
    for _ in range(3):                                                # eager, captured, replayed
        got = b.search([fb])[0]
        assert len(want) > 0 and np.array_equal(got, want)
    b.close()
