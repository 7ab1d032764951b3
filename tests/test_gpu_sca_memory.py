"""Automaton contexts of rings that one tile holds keep nothing beside what the
other schedules keep: no edge units, no parts of records; and what asep_plan
says is what a context holds, for one tile and for several."""
import pytest

import oracle
from paper_1012_0385_gb300 import asep as A

pytestmark = pytest.mark.gpu

th = oracle.threshold


@pytest.fixture(scope="module", autouse=True)
def _device():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1012_0385_gb300 import build

    build.build()
    torch.cuda.set_device(0)


def held(**kw):
    times = list(range(0, 9))
    prm = A.make_params(p_thr=th(0.75), q_thr=th(0.25), **kw)
    with A.asep_create(prm, sample_times=times) as ctx:
        n = A.asep_get_info(ctx)["device_bytes"]
    assert A.asep_plan(A.make_params(p_thr=th(0.75), q_thr=th(0.25), **kw), times)["device_bytes"] == n
    return n


@pytest.mark.parametrize("units,S", [(1, 20000), (16, 700), (30, 600), (62, 17000)])  # 62: two units a thread
def test_rings_of_one_tile(units, S):
    automaton = held(L=256 * units, samples_per_real=S, schedule=A.ASEP_SCHED_SCA)
    domain = held(L=256 * units, samples_per_real=S, domain_sites=32)
    assert automaton <= domain + 1024


def test_rings_of_several_tiles():
    one = held(L=256 * 31, samples_per_real=600, schedule=A.ASEP_SCHED_SCA)
    assert one > held(L=256 * 31, samples_per_real=600, domain_sites=32)


@pytest.mark.parametrize("model", [A.ASEP_MODEL_RING, A.ASEP_MODEL_TWO_LANE])
def test_records_of_rings_of_one_tile(model):
    """Every sweep recorded, over two launches, in steps that end inside them."""
    from test_gpu_parity import assert_same, oracle_params, run_gpu

    times = list(range(0, 141))
    kw = dict(L=256 * 30, schedule=A.ASEP_SCHED_SCA, samples_per_real=2, model=model, p_thr=th(0.75), q_thr=th(0.25),
              seed=4, flags=A.ASEP_FLAG_PROFILE | A.ASEP_FLAG_AUTOCORR, autocorr_t0=2)
    P = oracle_params(kw)
    assert_same(run_gpu(kw, [1, 130, 9], times), oracle.run(P, 140, times, autocorr_t0=2), P, times)
