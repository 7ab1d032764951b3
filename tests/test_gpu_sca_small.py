"""The automaton on rings cut into small tiles: on both sides of the number of
tiles up to which rings are cut further, down to the smallest tiles, with
every kind of threshold comparison -- bit-exact against the oracle."""
import pytest

import oracle
from paper_1012_0385_gb300 import asep as A

pytestmark = pytest.mark.gpu

th = oracle.threshold
KINDS = {
    "any": dict(p_thr=th(0.8), q_thr=th(0.2)),
    "shared": dict(p_thr=th(0.8), q_thr=th(0.8), dis_kind=A.ASEP_DIS_BIMODAL, dis_a_thr=th(0.5), dis_b_thr=th(0.16),
                   dis_c_thr=th(0.16)),
    "four": dict(p_thr=th(0.9), q_thr=th(0.3), dis_kind=A.ASEP_DIS_BIMODAL_PQ, dis_a_thr=th(0.5), dis_b_thr=th(0.16),
                 dis_c_thr=th(0.7)),
    "special": dict(p_thr=A.ASEP_ALWAYS, q_thr=0, dis_kind=A.ASEP_DIS_BIMODAL, dis_a_thr=th(0.5), dis_b_thr=th(0.3)),
    "turning": dict(model=A.ASEP_MODEL_TWO_LANE, p_thr=th(0.5), q_thr=th(0.3), dis_kind=A.ASEP_DIS_TURNING,
                    dis_a_thr=th(0.4), dis_b_thr=th(0.5), init_kind=1, init_seed=3),
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


# units of a ring, rings: tiles of four and of all units; 9 units in 3 tiles x 202 = 606 tiles, in 2 x 203; 61 units in
# 16 tiles x 38 = 608, 13 x 39 and 6 x 100; more rings than schedulers
@pytest.mark.parametrize("units,S", [(1, 3), (4, 5), (5, 5), (9, 202), (9, 203), (61, 38), (61, 39), (61, 100), (31, 609)])
@pytest.mark.parametrize("kind", sorted(KINDS))
def test_small_tiles(kind, units, S):
    from test_gpu_parity import assert_same, oracle_params, run_gpu

    kw = dict(L=256 * units, schedule=A.ASEP_SCHED_SCA, samples_per_real=S, dis_seed=2, seed=units + S, **KINDS[kind])
    P = oracle_params(kw)
    assert_same(run_gpu(kw, [3, 130], [0, 3, 60, 133]), oracle.run(P, 133, [0, 3, 60, 133]), P, [0, 3, 60, 133])
