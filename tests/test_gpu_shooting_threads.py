"""Shooting from two host threads at once, on two handles and streams whose launches take different
amounts of shared memory (58 KB and 0.2 KB of a block): every call gives what it gives alone."""
import threading
import time

import numpy as np
import pytest
import torch

from paper_2509_18497_gb300 import api, rgs, scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_18497_gb300 import build
    build.build()


def test_two_threads():
    jobs = []
    for n, lights in ((20, 300), (40, 1)):
        sc = scenes.random_cluster(n=n, seed=n, L=3, nb=1, n_lights=lights)
        d = api.upload(sc)
        pipe = api.Pipeline(pairs=True)
        pipe.build(d)
        pipe.trace(d)
        want = [x.cpu().numpy() for x in rgs.rgs_prog_refine(pipe.transport, 2)]
        jobs.append((pipe, want, torch.cuda.Stream()))
    torch.cuda.synchronize()
    errors = []
    end = time.monotonic() + 4.0

    def work(pipe, want, stream):
        try:
            with torch.cuda.stream(stream):
                while time.monotonic() < end and not errors:
                    for _ in range(20):
                        got = rgs.rgs_prog_refine(pipe.transport, 2, stream=stream)
                    for a, b in zip(got, want):
                        np.testing.assert_allclose(a.cpu().numpy(), b, rtol=1e-5, atol=1e-6)
        except Exception as e:  # noqa: BLE001 (handed to the test's thread)
            errors.append(e)

    threads = [threading.Thread(target=work, args=job) for job in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
