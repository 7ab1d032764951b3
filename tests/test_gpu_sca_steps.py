"""Automaton contexts stepped a sweep at a time: a call is one launch of the
tiles and one that moves the clock (with the record, where there is one), the
tiles' edge units carry over from call to call, and a lattice that was replaced
in between (another seed, a loaded state) brings its own."""
import numpy as np
import pytest

import oracle
from paper_1012_0385_gb300 import asep as A

pytestmark = pytest.mark.gpu

th = oracle.threshold
KINDS = {"ring": dict(p_thr=th(0.75), q_thr=th(0.25)), "any": dict(p_thr=th(0.8), q_thr=th(0.1)),
         "turning": dict(model=A.ASEP_MODEL_TWO_LANE, p_thr=th(0.8), q_thr=th(0.8), dis_kind=A.ASEP_DIS_TURNING,
                         dis_a_thr=th(0.4), dis_b_thr=th(0.3), dis_seed=3, init_kind=1, init_seed=5)}


@pytest.fixture(scope="module", autouse=True)
def _device():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1012_0385_gb300 import build

    build.build()
    oracle.build()
    torch.cuda.set_device(0)


def params(kind, units, samples=2):
    return dict(schedule=A.ASEP_SCHED_SCA, L=256 * units, samples_per_real=samples, seed=units, **KINDS[kind])


@pytest.mark.parametrize("units,samples", [(16, 8), (61, 2), (61, 500)])
@pytest.mark.parametrize("kind", sorted(KINDS))
def test_launches_of_single_sweeps(kind, units, samples):
    for times, extra in [([], 0), (list(range(1, 40)), 0), ([5, 6, 20], 0)]:
        with A.asep_create(A.make_params(**params(kind, units, samples)), sample_times=times) as ctx:
            A.asep_sweep(ctx, 1)
            before = A.asep_get_info(ctx)["kernel_launches"]
            for _ in range(20):
                A.asep_sweep(ctx, 1)
            assert A.asep_get_info(ctx)["kernel_launches"] - before == 2 * 20


@pytest.mark.parametrize("chunks", [[1] * 9, [3, 1, 129, 1, 2], [128, 128]])
@pytest.mark.parametrize("units", [31, 70])
@pytest.mark.parametrize("kind", sorted(KINDS))
def test_steps_against_the_oracle(kind, units, chunks):
    from test_gpu_parity import assert_same, oracle_params, run_gpu

    n = sum(chunks)
    kw = params(kind, units)
    times = sorted({0, 1, 2, 4, n - 1, n})
    P = oracle_params(kw)
    assert_same(run_gpu(kw, chunks, times), oracle.run(P, n, times), P, times)


@pytest.mark.parametrize("kind", sorted(KINDS))
def test_replaced_lattices(kind):
    kw = params(kind, 70)
    with A.asep_create(A.make_params(**kw), sample_times=[7]) as ctx, \
            A.asep_create(A.make_params(**kw), sample_times=[7]) as ref:
        A.asep_sweep(ref, 7)
        words7, _ = A.asep_state(ref)
        A.asep_sweep(ref, 6)
        words13, _ = A.asep_state(ref)
        A.asep_sweep(ctx, 3)  # one launch: the edge units are in the other half
        A.asep_load_state(ctx, words7, 7)
        A.asep_sweep(ctx, 1)
        A.asep_sweep(ctx, 5)
        assert np.array_equal(A.asep_state(ctx)[0], words13)
        A.asep_reset(ctx, seed=kw["seed"], init_seed=kw.get("init_seed", 0))
        for k in (2, 1, 3, 1):
            A.asep_sweep(ctx, k)
        assert np.array_equal(A.asep_state(ctx)[0], words7)
        A.asep_set_plan(ctx, 32, 0)
        A.asep_sweep(ctx, 6)
        assert np.array_equal(A.asep_state(ctx)[0], words13)
