"""The serial schedule's windows, bit-exact against the oracle under both
plans: rings so small that most of a window waits for one site, attempts
beyond one segment between two table clears, launches whose round numbers
pass their limit, and more samples than a CTA of warps holds."""
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
    "pq": dict(p_thr=th(0.9), q_thr=th(0.1), dis_kind=A.ASEP_DIS_BIMODAL_PQ, dis_a_thr=th(0.4), dis_b_thr=th(0.3),
               dis_c_thr=th(0.2), dis_seed=3),
    "crossing": dict(model=A.ASEP_MODEL_TWO_LANE, p_thr=A.ASEP_ALWAYS, dis_kind=A.ASEP_DIS_CROSSING, dis_a_thr=th(0.5),
                     dis_b_thr=th(0.4), dis_c_thr=th(0.1), dis_seed=4),
}


# 64 sites: every round short of free attempts, 2.6 M attempts in one launch (39 segments; over 100 000 rounds,
# beyond the 16-bit round numbers); 512 and 1024: the CTA's window as large as the sweep and half of it; 16384
# (two lanes 8192): the largest the CTA plan holds; 32768: warps only
@pytest.mark.parametrize("plan", [(1, 0), (2, 0)])
@pytest.mark.parametrize("L,S,n", [(64, 2, 60000), (128, 9, 1100), (512, 3, 300), (1024, 17, 70), (8192, 2, 9),
                                   (16384, 1, 9), (32768, 2, 5)])
@pytest.mark.parametrize("model", sorted(MODELS))
def test_serial_windows(model, L, S, n, plan):
    from test_gpu_parity import assert_same, oracle_params, run_gpu

    if plan[0] == 1 and L > (8192 if model == "crossing" else 16384):
        pytest.skip("beyond the one-CTA plan")
    kw = dict(schedule=A.ASEP_SCHED_SERIAL, L=L, samples_per_real=S, seed=L + S, plan=plan, **MODELS[model])
    P = oracle_params({k: v for k, v in kw.items() if k != "plan"})
    times = [0, n // 3, n]
    assert_same(run_gpu(kw, [n], times), oracle.run(P, n, times), P, times)
