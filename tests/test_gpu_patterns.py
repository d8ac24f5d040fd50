"""The pattern-row dedispersion kernel: exact sums at the edges of its tiles (24
trials x 2048 samples in two halves, groups of 1 to 4 channels, 16-bit sums added
to the 32-bit ones every 256 channels) against the oracle, and the shapes that the
rule gives to it.  The inputs are long enough for the byte rows to need a second
wave of blocks, which is when the rule prefers the pattern rows."""
import numpy as np
import pytest

import oracle
from paper_2512_00398_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hp():
    import torch
    import paper_2512_00398_gb300 as m
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    m.lib()
    return m


def _kernels(fn):
    import torch
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        fn()
        torch.cuda.synchronize()
    return [e.name for e in prof.events()]


def _run(hp, nchans, ndm, nout, dm_lo, dm_hi, fill=None, seed=0):
    import torch
    bw = -500.0 / 4096
    dms = np.linspace(dm_lo, dm_hi, ndm).astype(np.float32)
    p = hp.Plan(nchans, 1500.0, bw, 49.152e-6, dms, synth.widths_pow2(16), 6.0)
    n = nout + p.max_delay
    rng = np.random.Generator(np.random.PCG64(seed))
    x = (rng.integers(0, 256, size=(n, nchans), dtype=np.uint8) if fill is None
         else np.full((n, nchans), fill, np.uint8))
    fb = torch.from_numpy(x).cuda()
    out = []
    names = _kernels(lambda: out.append(hp.dedisperse(p, fb)))
    assert not names or any("dedisp_patterns" in k for k in names)
    want = oracle.dedisperse(x, oracle.delays(nchans, 1500.0, bw, 49.152e-6, dms))
    assert np.array_equal(out[0], want)
    # the byte rows of another tile shape
    p.set_param("dedisp_config", 12)
    assert np.array_equal(hp.dedisperse(p, fb), want)
    p.close()


# (24 or 48 trials: whole DM tiles; 47 and 49: a partial last one and a third)
@pytest.mark.parametrize("nchans,ndm,nout", [
    (64, 48, 60 * 2048), (64, 47, 60 * 2048 + 1), (65, 49, 45 * 2048 - 1), (66, 48, 60 * 2048 - 1023),
    (67, 48, 60 * 2048 - 1025), (259, 48, 59 * 2048 + 3), (5, 48, 60 * 2048 + 5)])
def test_tile_edges(hp, nchans, ndm, nout):
    _run(hp, nchans, ndm, nout, 0.0, 60.0, seed=nchans)


@pytest.mark.parametrize("nchans", [256, 257, 515])
def test_largest_sums(hp, nchans):
    """All samples 255: every 16-bit field reaches its largest value before it is
    added to the 32-bit sums (256 channels x 255 = 65 280)."""
    _run(hp, nchans, 48, 60 * 2048 + 7, 0.0, 30.0, fill=255)


@pytest.mark.parametrize("dm_lo,dm_hi", [(0.0, 0.0), (500.0, 530.0), (3000.0, 3060.0)])
def test_delay_ranges(hp, dm_lo, dm_hi):
    """One pattern for every trial; large first delays; steep ones, whose rows and
    sets are split."""
    _run(hp, 203, 48, 60 * 2048 + 11, dm_lo, dm_hi, seed=7)


def test_unlike_trials_keep_byte_rows(hp):
    """128 channels over 250 MHz, 4 pc cm^-3 between trials: nearly every trial has
    patterns of its own."""
    import torch
    dms = np.linspace(0, 400, 100).astype(np.float32)
    p = hp.Plan(128, 1500.0, -1.953125, 64e-6, dms, synth.widths_pow2(16), 6.0)
    fb = torch.randint(0, 256, (p.max_delay + 70000, 128), dtype=torch.uint8, device="cuda")
    names = _kernels(lambda: hp.dedisperse(p, fb))
    assert not any("dedisp_patterns" in k for k in names)
    p.close()
