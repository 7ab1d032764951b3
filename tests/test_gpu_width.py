"""W^2 = (L sum h^2 - (sum h)^2) / L^2 with one rounding, where 64 bits hold
the numerator and where they do not (a long ring filled on one side only)."""
import pytest

from paper_1012_0385_gb300 import asep as A

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,wide", [(64, False), (1 << 14, False), (3 << 14, False), (1 << 20, True)])
def test_width_of_a_step(L, wide):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    with A.asep_create(A.make_params(L=L, domain_sites=32, samples_per_real=2, p_thr=0, q_thr=0),
                       sample_times=[1]) as ctx:
        words, _ = A.asep_state(ctx)
        flat = words.reshape(2, -1).copy()
        flat[0, : L // 64], flat[0, L // 64:] = 0xFFFFFFFF, 0
        A.asep_load_state(ctx, flat.reshape(words.shape), 0)
        A.asep_sweep(ctx, 1)
        sh, sh2, w2 = A.asep_width(ctx)
    big = 0
    for s1, (lo, hi), w in zip(sh.ravel().tolist(), sh2.reshape(-1, 2).tolist(), w2.ravel().tolist()):
        num = L * (lo + (hi << 64)) - s1 * s1
        big = max(big, num)
        assert w == float(num // (L * L)) + float(num % (L * L)) / float(L * L)
    assert (big >= 1 << 64) == wide
