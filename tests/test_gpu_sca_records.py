"""Launches of the automaton that end before the first record their buffer has
no room for: 6700 rings of two tiles take 0.5 MB a record, so 64 MB hold 125,
and with a record every sweep a launch is one of 125 sweeps.  Sums, counters at
the records and lattices of the first and last samples against the oracle, on
both sides of each launch's end, in one call, in steps and with a gap."""
import numpy as np
import pytest

import oracle
from paper_1012_0385_gb300 import asep as A

pytestmark = pytest.mark.gpu

th = oracle.threshold
UNITS, SAMPLES = 31, 6700


@pytest.mark.parametrize("chunks,times", [([255], list(range(0, 256))), ([100, 101, 54], list(range(1, 256))),
                                          ([255], list(range(0, 110)) + list(range(120, 256)))])
def test_more_records_than_the_buffer_holds(chunks, times):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kw = dict(L=256 * UNITS, p_thr=th(0.75), q_thr=th(0.25), seed=23)
    n = sum(chunks)
    with A.asep_create(A.make_params(schedule=A.ASEP_SCHED_SCA, samples_per_real=SAMPLES, **kw),
                       sample_times=times) as ctx:
        before = A.asep_get_info(ctx)["kernel_launches"]
        for k in chunks:
            A.asep_sweep(ctx, k)
        if chunks == [255] and times[-1] - times[0] == len(times) - 1:  # 125 + 125 + 5 sweeps and their records
            assert A.asep_get_info(ctx)["kernel_launches"] - before == 1 + 2 * 3
        words, _ = A.asep_state(ctx)
        sh, sh2, _ = A.asep_width(ctx)
        cur = A.asep_currents(ctx)
    for first in (0, SAMPLES - 1):
        P = oracle.Params(schedule=oracle.SCHED_SCA, samples_per_real=1, first_sample=first, **kw)
        ref = oracle.run(P, n, times)
        assert np.array_equal(words[first], ref.state[0])
        for t in range(len(times)):
            assert int(sh[t, first, 0]) == ref.sum_h[t, 0, 0]
            assert int(sh2[t, first, 0, 0]) + (int(sh2[t, first, 0, 1]) << 64) == ref.sum_h2[t, 0, 0]
            assert np.array_equal(cur[t, first], ref.extra["counters_at"][t, 0])
