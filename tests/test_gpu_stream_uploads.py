"""Uploads beside the step before: gulps much shorter than the delay tail, so that each
upload goes into the ring slot which that step's transpose reads as its oldest, pushed
all at once from pinned memory; every gulp's clusters equal the streamed oracle's."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_stream import _plan, _same, env                  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gulp,nbeams,max_batch", [(1024, 3, 3), (1024, 3, 1), (2048, 1, 1)])
def test_short_gulps_all_at_once(env, gulp, nbeams, max_batch):       # noqa: F811
    torch, hp = env
    from paper_2512_00398_gb300 import workloads
    ngulps = 16384 // gulp
    ws = workloads.stream_tiny(nbeams=nbeams, ngulps=4, gulp=4096)
    pinned = [torch.from_numpy(w.generate().data).pin_memory() for w in ws]
    data = [t.numpy() for t in pinned]
    st = hp.Stream(_plan(hp, ws[0]), nbeams=nbeams, gulp=gulp, max_batch=max_batch)
    for g in range(ngulps):
        for b in range(nbeams):
            st.push(b, data[b][g * gulp:(g + 1) * gulp])
    for b in range(nbeams):
        st.end_beam(b)
    got = {}
    while len(got) < ngulps * nbeams:
        r = st.poll(timeout_ms=120000)
        assert r is not None, "stream stalled"
        info, c = r
        assert info["status"] == hp.HP_OK
        got[(info["beam"], info["gulp_index"])] = c
    st.close()
    found = 0
    for b, w in enumerate(ws):
        o = w.obs
        for r in oracle.stream_search(data[b], gulp, o.f_top, o.chan_bw, o.tsamp, w.dm_list, w.widths,
                                      w.threshold):
            _same(got[(b, r["g"])], r["clusters"])
            found += len(r["clusters"])
    assert found > 0
