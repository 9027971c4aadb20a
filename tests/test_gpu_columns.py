"""The column layouts of the bounce, opacity and adjoint gathers at their edges against the
FP64 oracle: 3-column and 12-column adjoint tiles (column counts that fill the last tile or
leave 3, 6 or 9 of its 12), full and half warps of columns, every SH degree, and rays
whose hits do not fill a group of rows.  Tolerances are those of the precision modes: FP32 1e-4,
BF16 rows 5e-3 (the rounding of a coefficient is 2^-9)."""
import numpy as np
import pytest
import torch

from paper_2509_18497_gb300 import rgs, scenes

from gpu_helpers import rel_l2, run_gpu, run_oracle

pytestmark = pytest.mark.gpu

TOL = {rgs.RGS_FP32: (1e-4, 1e-4), rgs.RGS_BF16_FP32ACC: (5e-3, 5e-3), rgs.RGS_BF16_FP32ACC_RESCORR: (1e-3, 5e-3)}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_18497_gb300 import build
    build.build()


@pytest.mark.parametrize("lights, L, nd, n", [
    (1, 3, 32, 90), (2, 2, 32, 70), (3, 0, 32, 120), (4, 1, 64, 60), (5, 3, 32, 97), (5, 2, 96, 61), (6, 1, 32, 150),
    (8, 2, 32, 80), (11, 0, 32, 75), (11, 3, 32, 50), (16, 2, 32, 66), (16, 3, 32, 1), (22, 1, 32, 41)])
def test_columns_against_the_oracle(lights, L, nd, n):
    sc = scenes.random_cluster(n=n, seed=n + lights, L=L, nd=nd, nb=3, n_lights=lights)
    sc = scenes.with_emission(sc, seed=5)
    W = np.random.default_rng(lights).normal(size=(n, (L + 1) ** 2, 3 * lights))
    o = run_oracle(sc, W=W)
    for prec, (tol, gtol) in TOL.items():
        g = run_gpu(sc, W=W, precision=prec, tensor_cores=0)
        assert rel_l2(g["B"], o["B"]) <= tol, (prec, rel_l2(g["B"], o["B"]))
        for key in ("dE", "dad", "dop"):
            assert rel_l2(g[key], o[key]) <= gtol, (prec, key, rel_l2(g[key], o[key]))
