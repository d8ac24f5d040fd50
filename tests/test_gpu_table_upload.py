"""The constant tables of a plan's first call on a non-blocking stream: complete before
the kernel that reads them starts, and written after whatever the stream still does to
memory that a stream-ordered allocator hands out again."""
import numpy as np
import pytest

import oracle
from paper_2512_00398_gb300 import synth
from tests.test_gpu_patterns import hp                                # noqa: F401

pytestmark = pytest.mark.gpu
BW, TSAMP = -500.0 / 4096, 49.152e-6


@pytest.fixture(scope="module")
def case():
    nchans, nout = 640, 53 * 2048 + 3
    dms = np.linspace(0.0, 30.0, 72).astype(np.float32)
    delays = oracle.delays(nchans, 1500.0, BW, TSAMP, dms)
    rng = np.random.Generator(np.random.PCG64(17))
    x = rng.integers(0, 256, size=(nout + int(delays.max()), nchans), dtype=np.uint8)
    return dms, x, oracle.dedisperse(x, delays)


def _plan(hp, dms, nchans):                                           # noqa: F811
    return hp.Plan(nchans, 1500.0, BW, TSAMP, dms, synth.widths_pow2(16), 6.0)


# (tile shape 17 takes the pattern rows here, 12 the byte rows)
@pytest.mark.parametrize("config", [17, 12])
def test_first_call_on_a_side_stream(hp, case, config):               # noqa: F811
    import torch
    dms, x, want = case
    fb = torch.from_numpy(x).cuda()
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    for _ in range(8):                                                # a new plan each time
        with _plan(hp, dms, x.shape[1]) as p:
            p.set_param("dedisp_config", config)
            with torch.cuda.stream(s):
                assert np.array_equal(hp.dedisperse(p, fb), want)


@pytest.mark.parametrize("config", [17, 12])
def test_tables_in_memory_the_stream_still_writes(hp, case, config):  # noqa: F811
    import torch
    dms, x, want = case
    fb = torch.from_numpy(x).cuda()
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with _plan(hp, dms, x.shape[1]) as p:
        p.set_param("dedisp_config", config)
        p.use_torch_allocator()
        with torch.cuda.stream(s):
            # freed while the stream still fills it: the tables are cut from it
            big = torch.empty(1 << 30, dtype=torch.uint8, device="cuda")
            for _ in range(200):
                big.fill_(255)
            del big
            assert np.array_equal(hp.dedisperse(p, fb), want)
