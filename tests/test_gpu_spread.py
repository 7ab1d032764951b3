"""Few samples: resident plans whose launches are spread over clusters, and
cluster plans of more CTAs than a sample needs -- bit-exact against the oracle
with every observable, on both sides of the 256-column line and for column
counts that leave the last CTA ragged; forced plans, balanced launches and
static batches keep the resident kernel and give the same lattices."""
import numpy as np
import pytest

import oracle
from paper_1012_0385_gb300 import asep as A

pytestmark = pytest.mark.gpu

th = oracle.threshold
D = 32  # 64 sites a column
MODELS = {
    "ring": dict(p_thr=th(0.75), q_thr=th(0.25), flags=A.ASEP_FLAG_PROFILE | A.ASEP_FLAG_AUTOCORR, autocorr_t0=3),
    "bimodal": dict(p_thr=A.ASEP_ALWAYS, dis_kind=A.ASEP_DIS_BIMODAL, dis_a_thr=th(0.4), dis_b_thr=th(0.3), dis_seed=3),
    "turning": dict(model=A.ASEP_MODEL_TWO_LANE, p_thr=A.ASEP_ALWAYS, q_thr=A.ASEP_ALWAYS, dis_kind=A.ASEP_DIS_TURNING,
                    dis_a_thr=th(0.3), dis_b_thr=th(0.4), dis_seed=4, init_kind=1, init_seed=2,
                    flags=A.ASEP_FLAG_PROFILE | A.ASEP_FLAG_AUTOCORR, autocorr_t0=3),
}


@pytest.fixture(scope="module", autouse=True)
def _device():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1012_0385_gb300 import build

    build.build()
    oracle.build()
    torch.cuda.set_device(0)


def params(model, G, S):
    return dict(L=2 * D * G, domain_sites=D, samples_per_real=S, seed=G + S, **MODELS[model])


@pytest.mark.parametrize("G,S", [(255, 1), (256, 2), (257, 1), (513, 2), (1000, 3), (1023, 1), (1024, 40), (1024, 67),
                                 (1025, 2), (2049, 1), (4100, 5)])
@pytest.mark.parametrize("model", sorted(MODELS))
def test_few_samples(model, G, S):
    from test_gpu_parity import assert_same, oracle_params, run_gpu

    kw = params(model, G, S)
    P = oracle_params(kw)
    ref = oracle.run(P, 7, [0, 3, 7], autocorr_t0=kw.get("autocorr_t0"))
    assert_same(run_gpu(kw, [2, 5], [0, 3, 7]), ref, P, [0, 3, 7])


@pytest.mark.parametrize("model", sorted(MODELS))
def test_the_plan_seen_and_forced(model):
    prm = A.make_params(**params(model, 1000, 2))
    states = []
    for k in range(4):
        with A.asep_create(prm, sample_times=[3, 6]) as ctx:
            assert A.asep_get_info(ctx)["cluster"] == 1  # the plan stays the resident one
            if k == 1:
                A.asep_set_plan(ctx, 1, 0)
            if k == 2:
                A.asep_set_balance(ctx, 2)
            if k == 3:
                A.asep_batch_sweep_static([ctx], [6])
            else:
                A.asep_sweep(ctx, 6)
            states.append(A.asep_state(ctx)[0])
    assert all(np.array_equal(states[0], s) for s in states[1:])


def test_batches_of_spread_contexts():
    kws = [params(m, G, S) for m, G, S in [("ring", 1024, 1), ("turning", 600, 3), ("bimodal", 100, 7), ("ring", 2048, 1)]]
    ctxs, alone = ([A.asep_create(A.make_params(**kw), sample_times=[3, 5]) for kw in kws] for _ in range(2))
    with A.asep_batch_create(max_jobs=8, max_items=16) as b:
        A.asep_batch_sweep(b, ctxs, [5, 3, 4, 2])
        A.asep_batch_graph(b, ctxs, [2, 2, 2, 2], 2)
    for ctx, ref, n in zip(ctxs, alone, [9, 7, 8, 6]):
        A.asep_set_plan(ref, 0, 0)
        A.asep_sweep(ref, n)
        assert np.array_equal(A.asep_state(ctx)[0], A.asep_state(ref)[0])
        assert all(np.array_equal(x, y) for x, y in zip(A.asep_width(ctx), A.asep_width(ref)))
        A.asep_destroy(ctx)
        A.asep_destroy(ref)
