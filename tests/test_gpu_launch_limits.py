"""Small and large contexts of one kernel driven by several host threads: a
launch is never refused because another thread's smaller one set a lower
limit on the kernel's shared memory."""
import threading

import numpy as np
import pytest

from paper_1012_0385_gb300 import asep as A

pytestmark = pytest.mark.gpu

th = A.asep_threshold
DOMAIN = dict(domain_sites=256, p_thr=th(0.7), q_thr=th(0.2))
SERIAL = dict(schedule=A.ASEP_SCHED_SERIAL, p_thr=th(0.7), q_thr=th(0.2))
# name: (small, large, plan, balance chunk)
PAIRS = {
    "resident": (dict(L=1 << 14, **DOMAIN), dict(L=1 << 18, **DOMAIN), (1, 0), 0),
    "balanced": (dict(L=1 << 14, **DOMAIN), dict(L=1 << 18, **DOMAIN), (1, 0), 1),
    "streamed": (dict(L=1 << 16, **DOMAIN), dict(L=1 << 20, **DOMAIN), None, 0),  # tiles of 64 and of 1024 columns
    "serial_cta": (dict(L=1 << 8, **SERIAL), dict(L=1 << 14, **SERIAL), (1, 0), 0),
    "serial_warp": (dict(L=1 << 8, **SERIAL), dict(L=1 << 20, **SERIAL), (2, 0), 0),
    "batch": (dict(L=1 << 14, **DOMAIN), dict(L=1 << 17, **DOMAIN), (1, 0), 0),
}


@pytest.fixture(scope="module", autouse=True)
def _device():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1012_0385_gb300 import build

    build.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("name", sorted(PAIRS))
def test_threads_of_small_and_large_contexts(name):
    import torch

    small, large, plan, chunk = PAIRS[name]
    kws = [small, large] * 3
    errors, words = [], [None] * len(kws)
    start = threading.Barrier(len(kws))

    def work(k):
        torch.cuda.set_device(0)
        try:
            stream = torch.cuda.Stream()
            with A.asep_create(A.make_params(**kws[k]), sample_times=[], stream=stream.cuda_stream) as ctx:
                A.asep_set_plan(ctx, *(plan or (32, 64 if k % 2 == 0 else 1024)))
                A.asep_set_balance(ctx, chunk)
                b = A.asep_batch_create(max_jobs=1, max_items=8, stream=stream.cuda_stream) if name == "batch" else None
                start.wait(60)
                for i in range(1000):
                    if b is not None:
                        A.asep_batch_sweep(b, [ctx], [1])
                    else:
                        A.asep_sweep(ctx, 2 if chunk else 1)
                words[k] = A.asep_state(ctx)[0]
                if b is not None:
                    A.asep_batch_destroy(b)
        except Exception as e:  # reported by the test's own thread
            errors.append(f"context {k}: {e}")
            start.abort()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(kws))]
    for t in threads:
        t.start()
    for t in threads:
        t.join(120)
    assert not errors, errors
    assert all(np.array_equal(words[k], words[k % 2]) for k in range(len(kws)))
