"""The SCA's tiles (a warp per tile of a ring, up to 128 sweeps a launch with
one halo unit on either side), bit-exact against the oracle where they can go
wrong: rings of one unit and of one unit more or less than a tile, runs that
end on, before and after a launch, records inside them, and enough rings for
two units a thread."""
import numpy as np
import pytest

import oracle
from paper_1012_0385_gb300 import asep as A

pytestmark = pytest.mark.gpu

th = oracle.threshold
SCA = A.ASEP_SCHED_SCA
RATES = {"quarters": (th(0.75), th(0.25)), "halves": (th(0.5), th(0.5)), "two_planes": (th(0.25), th(0.5)),
         "twenty_bits": (th(0.6), th(0.3)), "one_sided": (th(0.8), 0), "deterministic": (A.ASEP_ALWAYS, 0)}
KINDS = {"bimodal": dict(dis_kind=A.ASEP_DIS_BIMODAL, dis_a_thr=th(0.3), dis_b_thr=th(0.15), dis_c_thr=th(0.05)),
         "pq": dict(dis_kind=A.ASEP_DIS_BIMODAL_PQ, dis_a_thr=th(0.5), dis_b_thr=th(0.16), dis_c_thr=th(0.16)),
         "turning": dict(model=A.ASEP_MODEL_TWO_LANE, dis_kind=A.ASEP_DIS_TURNING, dis_a_thr=th(0.4), dis_b_thr=th(0.3),
                         init_kind=1, init_seed=5),
         "crossing": dict(model=A.ASEP_MODEL_TWO_LANE, dis_kind=A.ASEP_DIS_CROSSING, dis_a_thr=th(0.5),
                          dis_b_thr=th(0.8), dis_c_thr=th(0.2), init_kind=1, init_seed=6)}


@pytest.fixture(scope="module", autouse=True)
def _device():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1012_0385_gb300 import build

    build.build()
    oracle.build()
    torch.cuda.set_device(0)


def check(kw, chunks, times):
    from test_gpu_parity import assert_same, oracle_params, run_gpu

    g = run_gpu(kw, chunks, times)
    P = oracle_params(kw)
    assert_same(g, oracle.run(P, sum(chunks), times), P, times)


@pytest.mark.parametrize("units,chunks", [(1, [129]), (29, [1, 127]), (30, [128]), (31, [130]), (60, [127, 2]),
                                          (61, [257])])
@pytest.mark.parametrize("rates", sorted(RATES))
def test_ring_tiles(rates, units, chunks):
    p, q = RATES[rates]
    n = sum(chunks)
    check(dict(schedule=SCA, L=256 * units, samples_per_real=2, p_thr=p, q_thr=q, seed=units + 7), chunks,
          [0, 3, min(n, 127), n])


@pytest.mark.parametrize("units,n", [(1, 40), (30, 130), (31, 129)])
@pytest.mark.parametrize("kind", sorted(KINDS))
def test_quenched_and_two_lane_tiles(kind, units, n):
    kw = dict(schedule=SCA, L=256 * units, n_realizations=2, samples_per_real=1, p_thr=th(0.8), q_thr=th(0.8),
              dis_seed=3, seed=units + 11)
    kw.update(KINDS[kind])
    check(kw, [n], [0, 5, n])


@pytest.mark.parametrize("units,samples", [(1, 16417), (62, 5473), (63, 5473)])
@pytest.mark.parametrize("rates", ["quarters", "halves", "two_planes"])
def test_two_units_a_thread(rates, units, samples):
    """Above 16416 one-unit tiles a thread holds two units; the first and last
    samples against the oracle."""
    p, q = RATES[rates]
    kw = dict(schedule=SCA, L=256 * units, samples_per_real=samples, p_thr=p, q_thr=q, seed=19)
    with A.asep_create(A.make_params(**kw), sample_times=[2, 131]) as ctx:
        A.asep_sweep(ctx, 131)
        words, _ = A.asep_state(ctx)
        sh, _, _ = A.asep_width(ctx)
        cnt = A.asep_counters(ctx)
    for first in (0, samples - 2):
        P = oracle.Params(schedule=oracle.SCHED_SCA, L=256 * units, samples_per_real=1, first_sample=first, p_thr=p,
                          q_thr=q, seed=19)
        ref = oracle.run(P, 131, [2, 131])
        assert np.array_equal(words[first], ref.state[0])
        assert [int(x) for x in sh[:, first, 0]] == [ref.sum_h[t, 0, 0] for t in range(2)]
        assert np.array_equal(cnt[first], ref.counters[0])
