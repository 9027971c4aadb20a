"""The pair adjoint's transmittances are the products the trace formed, not a quotient of rounded
values: dL/dlambda of one bounce, which does not depend on lambda, has the same bits for every lambda
(with up to three surfels a source has two receivers at most, whose sum has no order); and the
gradients are the same where memory keeps no transmittances."""
import numpy as np
import pytest
import torch

from paper_2509_18497_gb300 import api, rgs, scenes

from gpu_helpers import rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_18497_gb300 import build
    build.build()


def _dlam(sc, lam, W):
    d = api.upload(dict(sc, lam=np.full(sc["n"], lam)))
    pipe = api.Pipeline(pairs=True)
    pipe.build(d)
    pipe.trace(d)
    pipe.solve(d["E"], 1)
    return pipe.adjoint_pairs(torch.as_tensor(W, dtype=torch.float32, device="cuda"))[3].cpu().numpy()


@pytest.mark.parametrize("n", [2, 3])
def test_lambda_gradient_does_not_depend_on_lambda(n):
    for seed in range(30):
        sc = scenes.with_emission(scenes.random_cluster(n=n, seed=seed, L=1, nb=1, n_lights=1), seed=seed)
        sc["s"] = sc["s"] * 4.0  # (the third one stands in the way of the other two)
        W = np.random.default_rng(seed).normal(size=(n, 4, 3))
        want = _dlam(sc, 1.0, W)
        for lam in (0.7, 1.3, 3.1):
            assert np.array_equal(_dlam(sc, lam, W), want), (seed, lam)


def test_transmittances_kept_and_traced():
    sc = scenes.with_emission(scenes.random_cluster(n=300, seed=5, L=2, nb=2, n_lights=1), seed=5)
    W = torch.as_tensor(np.random.default_rng(1).normal(size=(300, 9, 3)), dtype=torch.float32, device="cuda")
    out = []
    for budget in (False, True):
        d = api.upload(sc)
        pipe = api.Pipeline(pairs=True)
        pipe.build(d)
        pipe.trace(d)
        held = rgs.rgs_transport_info_get(pipe.transport)
        if budget:  # a trace with no room beside the records gives the transmittances' memory back
            rgs.rgs_set_memory_budget(pipe.transport, 1)
            pipe.trace(d)
            now = rgs.rgs_transport_info_get(pipe.transport)["device_bytes"]
            assert now == held["device_bytes"] - 4 * held["n_hits"]
        pipe.solve(d["E"], d["nb"])
        out.append([x.double().cpu().numpy() for x in pipe.adjoint_pairs_geometry(W)])
    for a, b in zip(*out):
        assert rel_l2(b, a) <= 1e-6  # (atomic sums in another order)
