"""Infinite radiance of one source in the column layouts of the bounce: receivers that see it get an
infinity, as with three columns, and no other value changes.  A half tile takes two hits at a time and
repeats the last row of an odd count, which must not enter as 0 times infinity."""
import numpy as np
import pytest
import torch

from paper_2509_18497_gb300 import rgs, scenes

from gpu_helpers import run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_18497_gb300 import build
    build.build()


# 3 columns; a half tile alone; a whole tile and a half one; whole tiles
@pytest.mark.parametrize("precision", [rgs.RGS_FP32, rgs.RGS_BF16_FP32ACC])
@pytest.mark.parametrize("lights", [1, 4, 5, 12, 13, 20])
@pytest.mark.parametrize("L", [1, 2, 3])
def test_one_infinite_source(L, lights, precision):
    n, src = 120, 17
    sc = scenes.random_cluster(n=n, seed=4, L=L, nd=32, nb=1, n_lights=lights)
    sc["E"] = np.zeros((n, (L + 1) ** 2, 3))
    sc["E"][:, 0] = 0.5
    plain = run_gpu(sc, precision=precision, tensor_cores=0)["B"][:, 0]
    sc["E"][src, 0, 0] = 1.0
    sees = np.abs(run_gpu(sc, precision=precision, tensor_cores=0)["B"][:, 0, 0] - plain[:, 0]) > 0
    sees[src] = True
    assert 5 < sees.sum() < n
    sc["E"][src, 0, 0] = np.inf
    B = run_gpu(sc, precision=precision, tensor_cores=0)["B"][:, 0]
    first = np.arange(3 * lights) % 3 == 0  # the infinite channel
    assert np.isposinf(B[sees][:, first]).all()
    assert np.isfinite(B[~sees]).all() and np.isfinite(B[:, ~first]).all()
