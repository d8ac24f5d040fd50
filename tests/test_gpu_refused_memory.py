"""Device memory that is refused: the call that needed it reports it once, the calls after
it run, and a plan whose pattern-row tables find no room keeps the byte rows."""
import ctypes as C

import numpy as np
import pytest

from paper_2512_00398_gb300 import synth
from tests.test_gpu_patterns import hp                                # noqa: F401
from tests.test_gpu_table_upload import case, _plan                   # noqa: F401

pytestmark = pytest.mark.gpu


def _ask_for_terabytes(hp, plan):                                     # noqa: F811
    """Detection of 2^32 samples x 1000 trials: the scratch is refused (by cudaMalloc of
    the library's own runtime) before anything is launched."""
    import torch
    buf = torch.zeros(64, dtype=torch.int64, device="cuda")
    out = hp._lib_mod.CandBuf(C.c_void_p(buf.data_ptr()), 1, C.c_void_p(buf.data_ptr()))
    return hp.lib().hp_detect(plan.handle, C.c_void_p(buf.data_ptr()), 1 << 32, 1 << 32, None,
                              C.byref(out), None, None)


@pytest.fixture()
def huge(hp):                                                         # noqa: F811
    with hp.Plan(4, 1500.0, -1.0, 64e-6, np.arange(1000, dtype=np.float32), synth.widths_pow2(16),
                 6.0) as p:
        yield p


def test_a_refused_call_leaves_no_error_behind(hp, case, huge):       # noqa: F811
    import torch
    dms, x, want = case
    with _plan(hp, dms, x.shape[1]) as p:
        fb = torch.from_numpy(x).cuda()
        for _ in range(2):
            assert _ask_for_terabytes(hp, huge) == hp.HP_ERR_OOM
            assert np.array_equal(hp.dedisperse(p, fb), want)


class Refusing:
    """Memory from torch; the tables of the pattern rows (the third request: constant
    tables, scratch, pattern tables) are refused, after a refused cudaMalloc of the
    library's own."""

    def __init__(self, hp, huge):                                     # noqa: F811
        self.hp, self.huge, self.asked = hp, huge, 0

    def alloc(self, n):
        import torch
        self.asked += 1
        if self.asked >= 3:
            assert _ask_for_terabytes(self.hp, self.huge) == self.hp.HP_ERR_OOM
            return 0
        return torch.cuda.caching_allocator_alloc(n)

    def free(self, ptr, n):
        import torch
        torch.cuda.caching_allocator_delete(ptr)


def test_no_room_for_the_pattern_tables(hp, case, huge):              # noqa: F811
    import torch
    dms, x, want = case
    with _plan(hp, dms, x.shape[1]) as p:
        hook = Refusing(hp, huge)
        p.use_allocator(hook.alloc, hook.free)
        fb = torch.from_numpy(x).cuda()
        for _ in range(3):
            assert np.array_equal(hp.dedisperse(p, fb), want)
        assert hook.asked == 3                     # refused once, not asked for again
        p.use_torch_allocator()                    # with room
        assert np.array_equal(hp.dedisperse(p, fb), want)
        assert hp.hp_plan_stats(p)["device_allocs"] == 2 + 3
