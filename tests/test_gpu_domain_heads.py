"""The domain schedule's tables of random heads and its one-sided attempts,
bit-exact against the oracle on both sides of every choice: groups whose idle
buffer just holds the tables and just does not (with and without the lane
sort, several samples per CTA), rings with and without left hops, and lane
changes pooled over warps that hold columns of several samples."""
import pytest

import oracle
from paper_1012_0385_gb300 import asep as A

pytestmark = pytest.mark.gpu

th = oracle.threshold
RATES = {"right": (A.ASEP_ALWAYS, 0), "both": (th(0.75), th(0.25)), "left": (0, th(0.6))}


@pytest.fixture(scope="module", autouse=True)
def _device():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1012_0385_gb300 import build

    build.build()
    oracle.build()
    torch.cuda.set_device(0)


def check(kw, n, times):
    from test_gpu_parity import assert_same, oracle_params, run_gpu

    P = oracle_params(kw)
    assert_same(run_gpu(kw, [n], times), oracle.run(P, n, times), P, times)


# three samples a CTA: from 22 columns a sample (D = 256 and 32) and from 11 (D = 2048) the idle buffer holds their
# tables; 32 columns and more in steps of 32 are sorted (D = 32 has no room for the sort)
@pytest.mark.parametrize("D,G", [(256, 21), (256, 22), (256, 32), (256, 33), (32, 21), (32, 22), (32, 64), (2048, 10),
                                 (2048, 11)])
@pytest.mark.parametrize("rates", sorted(RATES))
def test_tables_of_heads(rates, D, G):
    p, q = RATES[rates]
    check(dict(L=2 * D * G, domain_sites=D, samples_per_real=3, p_thr=p, q_thr=q, seed=G + D), 4, [0, 1, 4])


@pytest.mark.parametrize("dis", [A.ASEP_DIS_BIMODAL, A.ASEP_DIS_BIMODAL_PQ])
@pytest.mark.parametrize("slow", [(th(0.3), 0), (th(0.3), th(0.1)), (A.ASEP_ALWAYS, 0)])
def test_quenched_rings_with_and_without_left_hops(dis, slow):
    for q in (0, th(0.2)):
        check(dict(L=64 * 2 * 20, domain_sites=64, n_realizations=2, samples_per_real=2, p_thr=th(0.9), q_thr=q,
                   dis_kind=dis, dis_a_thr=th(0.4), dis_b_thr=slow[0], dis_c_thr=slow[1], dis_seed=5, seed=8), 6, [0, 6])


@pytest.mark.parametrize("plan", [(0, 0), (2, 0), (32, 32)])
@pytest.mark.parametrize("dis", [A.ASEP_DIS_TURNING, A.ASEP_DIS_CROSSING])
@pytest.mark.parametrize("G", [5, 16, 96])
def test_lane_changes(dis, G, plan):
    if plan[0] and G < 96:
        pytest.skip("spread and streamed plans need more columns")
    check(dict(model=A.ASEP_MODEL_TWO_LANE, L=64 * 2 * G, domain_sites=64, samples_per_real=3, init_kind=1, init_seed=4,
               p_thr=th(0.7), q_thr=A.ASEP_ALWAYS, dis_kind=dis, dis_a_thr=th(0.6), dis_b_thr=th(0.5),
               dis_c_thr=th(0.2), dis_seed=G, seed=G + 1, plan=plan), 5, [0, 2, 5])
