"""hp_plan_prepare: the call with an input of the prepared length allocates nothing and is
captured with the kernel that it would take outside, also after a shorter first call."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_patterns import hp                                # noqa: F401
from tests.test_gpu_table_upload import BW, TSAMP, _plan

pytestmark = pytest.mark.gpu
NCHANS, NOUT = 96, 60 * 2048 + 9            # (3000 samples: byte rows)


@pytest.fixture(scope="module")
def case():
    dms = np.linspace(0.0, 600.0, 48).astype(np.float32)
    delays = oracle.delays(NCHANS, 1500.0, BW, TSAMP, dms)
    rng = np.random.Generator(np.random.PCG64(41))
    x = rng.integers(0, 256, size=(NOUT + int(delays.max()), NCHANS), dtype=np.uint8)
    return dms, x, oracle.dedisperse(x, delays)


@pytest.mark.parametrize("prepared", [True, False])
def test_captured_after_a_shorter_call(hp, case, prepared):           # noqa: F811
    import torch
    dms, x, want = case
    fb = torch.from_numpy(x).cuda()
    with _plan(hp, dms, NCHANS) as p:
        p.bind_workspace(x.shape[0])
        hp.dedisperse(p, fb[:3000 + p.max_delay])
        assert p.dedisp_kernel() == 0
        if prepared:
            p.prepare(x.shape[0])
        allocs = hp.hp_plan_stats(p)["device_allocs"]
        out = torch.empty((48, NOUT + 3 & ~3), dtype=torch.int32, device="cuda")
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            hp.hp_dedisperse(p, fb, out=out)
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert hp.hp_plan_stats(p)["device_allocs"] == allocs
        assert (p.dedisp_kernel() >= 1) == prepared
        assert np.array_equal(out[:, :NOUT].cpu().numpy(), want)


def test_prepared_plan_allocates_nothing(hp, case):                   # noqa: F811
    import torch
    dms, x, want = case
    fb = torch.from_numpy(x).cuda()
    with _plan(hp, dms, NCHANS) as p:
        p.prepare(x.shape[0])
        allocs = hp.hp_plan_stats(p)["device_allocs"]
        assert np.array_equal(hp.dedisperse(p, fb), want)
        assert hp.hp_plan_stats(p)["device_allocs"] == allocs
        for n in (0, p.max_delay + int(p.widths[-1])):
            with pytest.raises(hp.HPError):
                p.prepare(n)
