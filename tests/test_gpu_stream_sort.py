"""The streamed tier's lane sort, bit-exact against the oracle where its
scratch just fits the tile's staged words and where it does not: ragged last
tiles around the limit (41 of 128 columns at D = 256, 81 at D = 128), tiles of
one column, and D = 64, whose rows never hold it."""
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
    oracle.build()
    torch.cuda.set_device(0)


MODELS = {
    "ring": dict(p_thr=th(0.75), q_thr=th(0.25)),
    "one_way_pq": dict(p_thr=th(0.9), dis_kind=A.ASEP_DIS_BIMODAL_PQ, dis_a_thr=th(0.4), dis_b_thr=th(0.3), dis_seed=3),
    "turning": dict(model=A.ASEP_MODEL_TWO_LANE, p_thr=A.ASEP_ALWAYS, q_thr=A.ASEP_ALWAYS, dis_kind=A.ASEP_DIS_TURNING,
                    dis_a_thr=th(0.3), dis_b_thr=th(0.4), dis_seed=4, init_kind=1, init_seed=2),
}


@pytest.mark.parametrize("D,C,last", [(256, 128, 1), (256, 128, 40), (256, 128, 41), (256, 128, 127), (128, 128, 80),
                                      (128, 128, 81), (128, 32, 31), (64, 96, 96), (2048, 32, 13)])
@pytest.mark.parametrize("model", sorted(MODELS))
def test_streamed_sort(model, D, C, last):
    from test_gpu_parity import assert_same, oracle_params, run_gpu

    kw = dict(L=2 * D * (2 * C + last), domain_sites=D, samples_per_real=2, seed=D + last, plan=(32, C), **MODELS[model])
    P = oracle_params({k: v for k, v in kw.items() if k != "plan"})
    assert_same(run_gpu(kw, [5], [0, 5]), oracle.run(P, 5, [0, 5]), P, [0, 5])
