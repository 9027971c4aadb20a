"""What a memory budget decides.  A budget that holds the solve's iterates, 16 bytes a ray and the
transposed index keeps every iterate (so that geometry gradients are to be had); where the
adjoint's larger per-ray records would split the index for few columns, it takes the smaller ones,
and the larger ones where the index comes in parts anyway or there are many columns."""
import numpy as np
import pytest
import torch

from paper_2509_18497_gb300 import api, rgs, scenes

from gpu_helpers import rel_l2, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_18497_gb300 import build
    build.build()


@pytest.mark.parametrize("lights", [1, 2, 8, 16])
def test_budget_of_every_iterate(lights):
    n, nd, nb, C = 2000, 64, 4, 3 * lights
    sc = scenes.with_emission(scenes.fruit_bowl(n=n, L=1, nd=nd, nb=nb, n_lights=lights), seed=2)
    W = np.random.default_rng(1).normal(size=(n, 4, C))
    full = run_gpu(sc, W=W, geometry=True)
    d = api.upload(sc)
    pipe = api.Pipeline(checkpoint=-1)
    pipe.build(d)
    pipe.trace(d)
    info = rgs.rgs_transport_info_get(pipe.transport)
    A = 4 * n * C * 4
    need = (2 * nb + 1) * A + (nb + 2) * A + 12 * info["n_hits"] + 16 * n * nd
    rgs.rgs_set_memory_budget(pipe.transport, info["device_bytes"] + need + 8 * n * nd)
    B, _ = pipe.solve(d["E"], nb)
    out = pipe.adjoint_geometry(torch.as_tensor(W, dtype=torch.float32, device="cuda"))
    assert np.array_equal(B.double().cpu().numpy(), full["B"])
    for key, v in zip(("dE", "dad", "dop", "dp", "ds", "dtu", "dtv"), out):
        assert rel_l2(v.double().cpu().numpy(), full[key]) <= 1e-5, key  # (sums in another order)


# bytes a ray beside the index, index builds of the adjoint, whether by 12-column tiles: room for the
# larger records; for the smaller ones only; for neither
@pytest.mark.parametrize("lights,per_ray,builds,tiles", [
    (4, 72, 1, True), (4, 40, 1, False), (4, 8, 6, True), (10, 72, 1, True), (10, 40, 6, True), (10, 8, 6, True)])
def test_records_by_what_they_leave_to_the_index(lights, per_ray, builds, tiles):
    n, nd, nb, C = 2000, 64, 3, 3 * lights
    sc = scenes.with_emission(scenes.fruit_bowl(n=n, L=2, nd=nd, nb=nb, n_lights=lights), seed=2)
    W = np.random.default_rng(1).normal(size=(n, 9, C))
    full = run_gpu(sc, W=W)
    d = api.upload(sc)
    pipe = api.Pipeline()
    pipe.build(d)
    pipe.trace(d)
    pipe.solve(d["E"], nb)
    info = rgs.rgs_transport_info_get(pipe.transport)
    A, more = 4 * n * C * 9, 60 * n  # (more: the adjoint's own per-surfel buffers)
    room = (nb + 2) * A + 12 * info["n_hits"] + per_ray * n * nd
    rgs.rgs_set_memory_budget(pipe.transport, info["device_bytes"] + more + room)
    rgs.rgs_profile_reset()
    rgs.rgs_profile_enable(True)
    out = pipe.adjoint(torch.as_tensor(W, dtype=torch.float32, device="cuda"))
    torch.cuda.synchronize()
    rgs.rgs_profile_enable(False)
    rep = rgs.rgs_profile_report()
    assert rep["k_src_fill"][0] == builds and (rep.get("k_adj_src_tile", (0, 0))[0] > 0) == tiles
    for key, v in zip(("dE", "dad", "dop"), out):
        assert rel_l2(v.double().cpu().numpy(), full[key]) <= 1e-5, key
