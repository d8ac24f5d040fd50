"""Steps of a stream that hold gulps of unlike lengths (a beam's first window beside a
later one of another): one dedispersion launch each, and the beams' own results."""
import numpy as np
import pytest

from paper_2512_00398_gb300 import synth
from tests.test_gpu_patterns import _kernels, hp                      # noqa: F401

pytestmark = pytest.mark.gpu
# 96 channels, delays of 57 000 samples: first windows of 2593 samples (byte rows alone),
# later ones of 60 015 (pattern rows when two are together)
NCH, G, NG = 96, 60000, 6


def _run(hp, plan, data, order):                                      # noqa: F811
    st = hp.Stream(plan, nbeams=2, gulp=G, cand_capacity=1 << 14)
    got = {}
    for i, (b, g) in enumerate(order):
        st.push(b, data[b][g * G:(g + 1) * G])
        if i == 0:                                 # a step of its own
            info, c = st.poll(timeout_ms=60000)
            got[b, g] = (info["batch_size"], c)
    while len(got) < len(order):
        info, c = st.poll(timeout_ms=60000)
        assert info["status"] == hp.HP_OK
        got[info["beam"], info["gulp_index"]] = (info["batch_size"], c)
    steps = st.stats()["steps"]
    st.close()
    return got, steps


def test_first_windows_beside_later_ones(hp):                         # noqa: F811
    import torch
    dms = np.linspace(23500.0, 23600.0, 48).astype(np.float32)
    rng = np.random.Generator(np.random.PCG64(29))
    with hp.Plan(NCH, 1500.0, -500.0 / 1024, 49.152e-6, dms, synth.widths_pow2(16), 6.0) as plan:
        data = []
        for b in range(2):
            noise = rng.integers(0, 40, size=(NG * G, NCH), dtype=np.uint8)
            for t in range(700 + 100 * b, NG * G - 60000, 9001):      # pulses of the middle trial
                noise[t + plan.delays()[24], np.arange(NCH)] += 90
            x = torch.empty(noise.shape, dtype=torch.uint8, pin_memory=True)
            x.copy_(torch.from_numpy(noise))
            data.append(x)
        alone, _ = _run(hp, plan, data, [(0, g) for g in range(NG)])
        other, _ = _run(hp, plan, data, [(1, g) for g in range(NG)])
        alone.update(other)
        mixed = []
        order = [(0, g) for g in range(NG)] + [(1, g) for g in range(NG)]
        names = _kernels(lambda: mixed.append(_run(hp, plan, data, order)))
        got, steps = mixed[0]
        assert got[1, 0][0] == 2                   # beam 1's first gulp shared its step
        dedisp = [k for k in names if "dedisp_rows_kernel" in k or "dedisp_patterns_kernel" in k]
        assert len(dedisp) == steps < len(order)
        assert sum(len(c) for _, c in got.values()) > 0
        for k, (_, c) in got.items():
            assert np.array_equal(c, alone[k][1]), k
