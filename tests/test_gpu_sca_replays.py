"""asep_sweep of the automaton captured into a caller's CUDA graph: replays
run on from the device clock's sweep, so which sample times fall into one is
the device's to find -- none, some, and past the last, with records of every
observable, and the same for calls made after the replays."""
import numpy as np
import pytest

import oracle
from paper_1012_0385_gb300 import asep as A

pytestmark = pytest.mark.gpu

th = oracle.threshold
KINDS = {"ring": dict(p_thr=th(0.75), q_thr=th(0.25)), "any": dict(p_thr=th(0.8), q_thr=th(0.1)),
         "turning": dict(model=A.ASEP_MODEL_TWO_LANE, p_thr=th(0.8), q_thr=th(0.8), dis_kind=A.ASEP_DIS_TURNING,
                         dis_a_thr=th(0.4), dis_b_thr=th(0.3), dis_seed=3, init_kind=1, init_seed=5)}
TIMES = {"late": [200], "all": [0, 1, 3, 64, 65, 66, 127, 131, 200], "dense": list(range(0, 201, 2)) + [201], "none": []}


@pytest.fixture(scope="module", autouse=True)
def _device():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1012_0385_gb300 import build

    build.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("units", [1, 31, 70])
@pytest.mark.parametrize("times", sorted(TIMES))
@pytest.mark.parametrize("kind", sorted(KINDS))
def test_replays(kind, times, units):
    import torch

    kw = dict(schedule=A.ASEP_SCHED_SCA, L=256 * units, samples_per_real=2, seed=units, flags=A.ASEP_FLAG_PROFILE,
              **KINDS[kind])
    if TIMES[times]:
        kw.update(flags=A.ASEP_FLAG_PROFILE | A.ASEP_FLAG_AUTOCORR, autocorr_t0=TIMES[times][len(TIMES[times]) // 3])
    stream = torch.cuda.Stream()

    def outputs(ctx):
        out = [A.asep_profile(ctx), A.asep_counters(ctx), A.asep_currents(ctx)]
        return out + ([A.asep_autocorr(ctx)] if TIMES[times] else []) + list(A.asep_width(ctx))

    with A.asep_create(A.make_params(**kw), sample_times=TIMES[times], stream=stream.cuda_stream) as ctx:
        A.asep_sweep(ctx, 2)
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            A.asep_sweep(ctx, 65)
        with torch.cuda.stream(stream):
            for _ in range(3):  # sweeps 2..196
                graph.replay()
        A.asep_sweep(ctx, 13)   # and up to 210, past the last sample time
        with torch.cuda.stream(stream):
            graph.replay()      # up to 275
        words, _ = A.asep_state(ctx)
        profile = A.asep_profile(ctx)
        A.asep_load_state(ctx, words, 275)  # the host's clock as well
        got = outputs(ctx)
        assert np.array_equal(profile, got[0])
    with A.asep_create(A.make_params(**kw), sample_times=TIMES[times]) as ctx:
        A.asep_sweep(ctx, 275)
        assert np.array_equal(words, A.asep_state(ctx)[0])
        for x, y in zip(got, outputs(ctx)):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("times", ["late", "all", "dense"])
def test_captured_launches_are_as_long_as_others(times):
    """Two tiles a ring, 260 sweeps captured: three launches of the tiles, each
    with one for the records, however few sample times there are; a record
    buffer short of 128 records (6700 rings) cuts them to what it holds."""
    import torch

    for samples, most in [(2, 128), (6700, 125)]:
        kw = dict(schedule=A.ASEP_SCHED_SCA, L=256 * 31, samples_per_real=samples, seed=1, **KINDS["ring"])
        stream = torch.cuda.Stream()
        every = list(range(1, 400)) if samples > 2 else TIMES[times]
        with A.asep_create(A.make_params(**kw), sample_times=every, stream=stream.cuda_stream) as ctx:
            A.asep_sweep(ctx, 1)
            before = A.asep_get_info(ctx)["kernel_launches"]
            graph = torch.cuda.CUDAGraph()
            torch.cuda.synchronize()
            with torch.cuda.graph(graph, stream=stream):
                A.asep_sweep(ctx, 260)
            launches = A.asep_get_info(ctx)["kernel_launches"] - before
            assert launches <= 1 + 2 * -(-260 // most)
