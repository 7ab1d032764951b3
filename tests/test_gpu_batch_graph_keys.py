"""A batch's captured step is replayed only for the contexts, seeds, plans and
sweeps that it was captured with, and on their own descriptors: another step
of the same batch, a reset with another seed, another plan or new contexts in
the place of destroyed ones between two calls leave every lattice as the
context's own sweeps do."""
import numpy as np
import pytest

from paper_1012_0385_gb300 import asep as A

pytestmark = pytest.mark.gpu

th = A.asep_threshold
SHAPES = [dict(L=4096, domain_sites=64, samples_per_real=5, p_thr=th(0.7), q_thr=th(0.2)),
          dict(L=1 << 15, domain_sites=64, samples_per_real=2, p_thr=th(0.6)),  # 256 columns: launches are spread
          dict(model=A.ASEP_MODEL_TWO_LANE, L=2048, domain_sites=64, samples_per_real=3, dis_kind=A.ASEP_DIS_TURNING,
               dis_a_thr=th(0.3), dis_b_thr=th(0.2), p_thr=th(0.9), q_thr=th(0.9))]


@pytest.fixture(scope="module", autouse=True)
def _device():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1012_0385_gb300 import build

    build.build()
    torch.cuda.set_device(0)


def make(seed=1):
    return [A.asep_create(A.make_params(seed=seed + k, **kw), sample_times=[2, 5]) for k, kw in enumerate(SHAPES)]


def check(ctxs, sweeps, seeds):
    for ctx, n, seed, kw in zip(ctxs, sweeps, seeds, SHAPES):
        with A.asep_create(A.make_params(seed=seed, **kw), sample_times=[2, 5]) as ref:
            A.asep_sweep(ref, n)
            (words, sweep), (expect, at) = A.asep_state(ctx), A.asep_state(ref)
            assert sweep == at == n and np.array_equal(words, expect)
            assert np.array_equal(A.asep_counters(ctx), A.asep_counters(ref))
            assert all(np.array_equal(x, y) for x, y in zip(A.asep_width(ctx), A.asep_width(ref)))


def test_a_step_of_the_same_contexts_between():
    ctxs = make()
    with A.asep_batch_create(max_jobs=8, max_items=64) as b:
        A.asep_batch_graph(b, ctxs, [2, 2, 2], 1)
        A.asep_batch_sweep(b, ctxs, [1, 3, 4])
        A.asep_batch_graph(b, ctxs, [2, 2, 2], 2)
        check(ctxs, [7, 9, 10], [1, 2, 3])
    for c in ctxs:
        c.close()


def test_a_step_of_other_contexts_between():
    ctxs, others = make(), make(11)
    with A.asep_batch_create(max_jobs=8, max_items=64) as b:
        A.asep_batch_graph(b, ctxs, [2, 2, 2], 1)
        A.asep_batch_sweep(b, others[::-1], [3, 3, 3])
        A.asep_batch_graph(b, ctxs, [2, 2, 2], 1)
        A.asep_batch_graph(b, others, [1, 1, 1], 1)
        A.asep_batch_graph(b, ctxs, [2, 2, 2], 1)
        check(ctxs, [6, 6, 6], [1, 2, 3])
        check(others, [4, 4, 4], [11, 12, 13])
    for c in ctxs + others:
        c.close()


def test_another_seed_between():
    ctxs = make()
    with A.asep_batch_create(max_jobs=8, max_items=64) as b:
        A.asep_batch_graph(b, ctxs, [2, 2, 2], 2)
        for k, ctx in enumerate(ctxs):
            A.asep_reset(ctx, seed=70 + k)
        A.asep_batch_graph(b, ctxs, [2, 2, 2], 3)
        check(ctxs, [6, 6, 6], [70, 71, 72])
    for c in ctxs:
        c.close()


def test_another_plan_between():
    ctxs = make()
    with A.asep_batch_create(max_jobs=8, max_items=64) as b:
        A.asep_batch_graph(b, ctxs, [2, 2, 2], 1)
        A.asep_set_plan(ctxs[0], 1, 2)  # two samples a CTA
        A.asep_set_plan(ctxs[1], 4, 0)
        A.asep_batch_graph(b, ctxs, [2, 2, 2], 1)
        A.asep_set_plan(ctxs[1], 1, 0)
        A.asep_batch_graph(b, ctxs, [2, 2, 2], 1)
        check(ctxs, [6, 6, 6], [1, 2, 3])
    for c in ctxs:
        c.close()


def test_new_contexts_in_the_place_of_destroyed_ones():
    with A.asep_batch_create(max_jobs=8, max_items=64) as b:
        for seed in (1, 21, 41):  # the allocator hands out the same addresses again
            ctxs = make(seed)
            A.asep_batch_graph(b, ctxs, [2, 2, 2], 2)
            check(ctxs, [4, 4, 4], [seed, seed + 1, seed + 2])
            for c in ctxs:
                c.close()
