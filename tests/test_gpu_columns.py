"""The column layouts of the bounce, opacity and adjoint gathers at their edges against the
FP64 oracle: 3-column and 12-column adjoint tiles (column counts that fill the last tile or
leave 3, 6 or 9 of its 12), full and half warps of columns, every SH degree, and rays
whose hits do not fill a group of rows.  Tolerances are those of the precision modes: FP32 1e-4,
BF16 rows 5e-3 (the rounding of a coefficient is 2^-9)."""
import numpy as np
import pytest
import torch

from paper_2509_18497_gb300 import api, rgs, scenes

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


@pytest.mark.parametrize("lights, L", [(1, 3), (1, 2), (1, 0), (2, 3), (4, 2), (5, 1), (5, 3)])
@pytest.mark.parametrize("form", ["with the bounces", "index in parts", "no opacity"])
def test_opacity_sums_against_the_oracle(lights, L, form):
    """The per-hit opacity sums formed with the transposed bounces, ray by ray where the index
    comes in parts (no memory for it in one), and the bounces alone."""
    sc = scenes.random_cluster(n=83, seed=lights + L, L=L, nd=64, nb=4, n_lights=lights)
    sc = scenes.with_emission(sc, seed=8)
    W = np.random.default_rng(3).normal(size=(83, (L + 1) ** 2, 3 * lights))
    o = run_oracle(sc, W=W)
    g = torch.as_tensor(np.ascontiguousarray(W, np.float32), device="cuda")
    for prec, (_, tol) in TOL.items():
        d = api.upload(sc)
        pipe = api.Pipeline(precision=prec, tensor_cores=0)
        pipe.build(d)
        pipe.trace(d)
        pipe.solve(d["E"], d["nb"])
        if form == "index in parts":
            rgs.rgs_set_memory_budget(pipe.transport, rgs.rgs_transport_info_get(pipe.transport)["device_bytes"])
        rgs.rgs_profile_reset()
        rgs.rgs_profile_enable(True)
        want = ("E", "albedo") if form == "no opacity" else ("E", "albedo", "opacity")
        out = rgs.rgs_adjoint(pipe.transport, g, want=want)
        torch.cuda.synchronize()
        rgs.rgs_profile_enable(False)
        rep = rgs.rgs_profile_report()
        raywise = sum(rep.get(k, (0, 0))[0] for k in ("k_opacity_g", "k_opacity_g_mc"))
        assert (raywise > 0) == (form == "index in parts")
        for key, v in zip(("dE", "dad", "dop"), out):
            if v is not None:
                assert rel_l2(v.double().cpu().numpy(), o[key]) <= tol, (prec, key)
