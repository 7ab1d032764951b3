"""Calls of the automaton with more launches than a stream's queue takes return
while they run, and do what short calls do: with and without records, in launches
of 1, 3 and 128 sweeps, beyond 256 and beyond 8192 of them, on either half of
the edge buffer, and after a captured call."""
import time

import numpy as np
import pytest

import oracle
from paper_1012_0385_gb300 import asep as A

pytestmark = pytest.mark.gpu

th = oracle.threshold
KINDS = {"ring": dict(p_thr=th(0.75), q_thr=th(0.25)),
         "turning": dict(model=A.ASEP_MODEL_TWO_LANE, p_thr=th(0.8), q_thr=th(0.8), dis_kind=A.ASEP_DIS_TURNING,
                         dis_a_thr=th(0.4), dis_b_thr=th(0.3), dis_seed=3, init_kind=1, init_seed=5)}


@pytest.fixture(scope="module", autouse=True)
def _device():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1012_0385_gb300 import build

    build.build()
    torch.cuda.set_device(0)


def params(kind, units, samples=2):
    return A.make_params(schedule=A.ASEP_SCHED_SCA, L=256 * units, samples_per_real=samples, seed=units,
                         flags=A.ASEP_FLAG_PROFILE, **KINDS[kind])


def outputs(ctx):
    return [A.asep_state(ctx)[0], A.asep_counters(ctx), A.asep_currents(ctx), A.asep_profile(ctx), *A.asep_width(ctx)]


@pytest.mark.parametrize("units,samples", [(16, 8), (64, 8)])
def test_the_host_is_back_before_the_work_is_done(units, samples):
    with A.asep_create(params("ring", units, samples), sample_times=[1 << 18]) as ctx:
        A.asep_sweep(ctx, 40000)  # the first graph of a process takes its time
        A.asep_sync(ctx)
        start = time.perf_counter()
        A.asep_sweep(ctx, 1 << 20)
        back = time.perf_counter() - start
        A.asep_sync(ctx)
        done = time.perf_counter() - start
        assert back < 0.25 * done, (back, done)


@pytest.mark.parametrize("cap,n", [(1, 257), (1, 513), (1, 9001), (3, 1600), (0, 66000)])
@pytest.mark.parametrize("units", [16, 31, 70])
@pytest.mark.parametrize("kind", sorted(KINDS))
def test_long_calls_are_short_calls(kind, units, cap, n):
    for times in ([], [5, n - 1, n, n + 3], sorted(set(int(1.5 ** k) for k in range(30)) | {257, 258, n})):
        with A.asep_create(params(kind, units), sample_times=times) as ctx, \
                A.asep_create(params(kind, units), sample_times=times) as ref:
            A.asep_sweep(ctx, 1)
            A.asep_set_launch_sweeps(ctx, cap)
            A.asep_sweep(ctx, n)
            A.asep_sweep(ctx, 2)
            for k in range(0, n + 3, 16384):
                A.asep_sweep(ref, min(16384, n + 3 - k))
            assert A.asep_get_info(ctx)["sweep"] == A.asep_get_info(ref)["sweep"]
            for x, y in zip(outputs(ctx), outputs(ref)):
                assert np.array_equal(x, y)


@pytest.mark.parametrize("units", [16, 31])
def test_after_a_captured_call(units):
    import torch

    stream = torch.cuda.Stream()
    times = [3, 100, 700, 1500]
    with A.asep_create(params("ring", units), sample_times=times, stream=stream.cuda_stream) as ctx, \
            A.asep_create(params("ring", units), sample_times=times) as ref:
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            A.asep_sweep(ctx, 300)
        with torch.cuda.stream(stream):
            graph.replay()
            graph.replay()
        A.asep_set_launch_sweeps(ctx, 1)
        A.asep_sweep(ctx, 1000)  # 600 .. 1600, the host's clock at 300
        words, _ = A.asep_state(ctx)
        A.asep_load_state(ctx, words, 1600)
        A.asep_sweep(ref, 1600)
        for x, y in zip(outputs(ctx), outputs(ref)):
            assert np.array_equal(x, y)
