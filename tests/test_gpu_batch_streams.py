"""Batches whose cluster-tier contexts run beside one another: one, eight and
more than eight of them, with and without resident contexts, stepped and as a
graph; every lattice as the context's own sweeps leave it."""
import numpy as np
import pytest

from paper_1012_0385_gb300 import asep as A

pytestmark = pytest.mark.gpu

th = A.asep_threshold


def contexts(n_clusters, n_resident):
    out = []
    for k in range(n_clusters + n_resident):
        kw = dict(L=2 * 64 * (64 + 32 * (k % 5)), domain_sites=64, samples_per_real=1 + k % 3, p_thr=th(0.7),
                  q_thr=th(0.1 * (k % 2)), seed=100 + k)
        if k % 4 == 3:
            kw.update(model=A.ASEP_MODEL_TWO_LANE, dis_kind=A.ASEP_DIS_TURNING, dis_a_thr=th(0.3), dis_b_thr=th(0.2))
        ctx = A.asep_create(A.make_params(**kw), sample_times=[])
        if k < n_clusters:
            A.asep_set_plan(ctx, (2, 4, 8)[k % 3], 0)
        out.append(ctx)
    return out


@pytest.mark.parametrize("n_clusters,n_resident", [(1, 0), (8, 1), (19, 2)])
def test_cluster_contexts_side_by_side(n_clusters, n_resident):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctxs, alone = contexts(n_clusters, n_resident), contexts(n_clusters, n_resident)
    steps = [3 + k % 4 for k in range(len(ctxs))]
    steps[0] = 0 if n_clusters > 1 else 3  # nothing to do for one of them
    with A.asep_batch_create(max_jobs=len(ctxs), max_items=256) as b:
        A.asep_batch_sweep(b, ctxs, steps)
        A.asep_batch_sweep(b, ctxs, steps)
        A.asep_batch_graph(b, ctxs, steps, 2)
        for ctx, ref, n in zip(ctxs, alone, steps):
            if n:
                A.asep_sweep(ref, 4 * n)
            (words, sweep), (expect, at) = A.asep_state(ctx), A.asep_state(ref)
            assert sweep == at == 4 * n and np.array_equal(words, expect)
            assert np.array_equal(A.asep_counters(ctx), A.asep_counters(ref))
    for c in ctxs + alone:
        A.asep_destroy(c)
