"""Balanced launches whose slots are fewer than the groups, as many, and more:
narrow and wide groups, launches of a few chunks and of a ragged last one --
the lattices of one launch per group."""
import numpy as np
import pytest

from paper_1012_0385_gb300 import asep as A

pytestmark = pytest.mark.gpu

th = A.asep_threshold


@pytest.mark.parametrize("G,S", [(8, 700), (64, 500), (200, 310), (352, 330), (480, 170), (700, 160)])
def test_slots(G, S):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    prm = A.make_params(L=64 * G, domain_sites=32, samples_per_real=S, p_thr=th(0.75), q_thr=th(0.25), seed=G)
    out = []
    for chunk in (0, 2, 5):
        with A.asep_create(prm, sample_times=[4, 13]) as ctx:
            A.asep_set_plan(ctx, 1, 1)
            if chunk:
                A.asep_set_balance(ctx, chunk)
            A.asep_sweep(ctx, 13)
            out.append([A.asep_state(ctx)[0], A.asep_counters(ctx), *A.asep_width(ctx)])
    assert all(np.array_equal(x, y) for o in out[1:] for x, y in zip(out[0], o))
