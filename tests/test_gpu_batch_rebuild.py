"""Batched solves of handles that are rebuilt in place, in buffers large enough to be used again:
with another opacity model, and with a lower and then the first SH degree again.  A launch plan
of the scenes as they were must not run on the scenes as they are.

Tolerance: per-scene solves of the same handles, 1e-5 relative L2 (FP32 sums in another order)."""
import pytest
import torch

from paper_2509_18497_gb300 import api, rgs, scenes

from gpu_helpers import rel_l2

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_18497_gb300 import build
    build.build()


def _batched_is_solved(pipes, L, model):
    ds = []
    for q, p in enumerate(pipes):
        sc = scenes.with_emission(scenes.random_cluster(n=300 + 50 * q, seed=q, L=L, nd=64, nb=3, n_lights=2), seed=q)
        d = api.upload(sc)
        p.alpha_model = model
        p.build(d)
        p.trace(d)
        ds.append(d)
    B, _ = rgs.rgs_solve_batched([p.transport for p in pipes], [d["E"] for d in ds], [d["nb"] for d in ds])
    held = [rgs.rgs_transport_info_get(p.transport)["device_bytes"] for p in pipes]
    for p, d, b in zip(pipes, ds, B):
        b = b.double().cpu().numpy()
        want = p.solve(d["E"], d["nb"])[0].double().cpu().numpy()
        assert rel_l2(b, want) <= TOL, (L, model, rel_l2(b, want))
    return held


def test_another_alpha_model():
    pipes = [api.Pipeline(), api.Pipeline()]
    held = _batched_is_solved(pipes, 3, rgs.RGS_ALPHA_GFSGS)
    assert _batched_is_solved(pipes, 3, rgs.RGS_ALPHA_GAUSS) == held
    assert _batched_is_solved(pipes, 3, rgs.RGS_ALPHA_GFSGS) == held


def test_another_degree():
    pipes = [api.Pipeline(), api.Pipeline()]
    held = _batched_is_solved(pipes, 3, rgs.RGS_ALPHA_GAUSS)
    for L in (2, 0, 3):
        assert _batched_is_solved(pipes, L, rgs.RGS_ALPHA_GAUSS) == held
