"""Both forms of the shooting solver (one cluster for many shots, two launches per shot) at the
edges of their row layout, against the FP64 oracle: fewer and more than 32 columns, rows
that do not fill a warp, every SH degree, more shots than there is radiance to shoot, and
rows of equal luminance (the lower caller index is shot first).

Tolerance: 1e-4 relative L2, the FP32 bar of the other solver tests (each receiver adds one
FP32 term of ~1e-7 relative rounding per shot; the picks are equal unless two luminances
agree to 1e-7)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2509_18497_gb300 import api, rgs, scenes

from gpu_helpers import rel_l2

pytestmark = pytest.mark.gpu

TOL = 1e-4


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_18497_gb300 import build
    build.build()


def _both(sc, shots):
    d = api.upload(sc)
    pipe = api.Pipeline(pairs=True)
    pipe.build(d)
    pipe.trace(d)
    Bh, dB = rgs.rgs_prog_refine(pipe.transport, shots, E=d["E"])
    Bho, dBo = O.Oracle(sc).pairs().prog_refine(shots, E=sc["E"])
    return Bh.double().cpu().numpy(), dB.double().cpu().numpy(), Bho, dBo


# rows updated per shot, about n / 2 x 3 lights (L + 1)^2: up to 160,000 by one cluster
@pytest.mark.parametrize("n, L, lights, shots", [
    (1, 2, 1, 3), (2, 0, 1, 5), (40, 3, 1, 60), (97, 1, 5, 40), (48, 2, 12, 30), (33, 3, 11, 20),
    (700, 2, 13, 12), (700, 3, 21, 8), (900, 2, 40, 6)])
def test_shots_against_the_oracle(n, L, lights, shots):
    sc = scenes.with_emission(scenes.random_cluster(n=n, seed=n, L=L, nb=2, n_lights=lights), seed=2)
    Bh, dB, Bho, dBo = _both(sc, shots)
    assert rel_l2(Bh, Bho) <= TOL, rel_l2(Bh, Bho)
    assert rel_l2(dB, dBo) <= TOL, rel_l2(dB, dBo)


@pytest.mark.parametrize("lights", [1, 40])
def test_nothing_left_to_shoot(lights):
    """Surfels that do not see each other: every one is shot once, then nothing is left."""
    sc = scenes.random_cluster(n=64, seed=3, L=2, nb=1, n_lights=lights)
    z = np.zeros((64, 3))
    z[:, 0] = np.arange(64) * 3.0
    sc["p"] = z
    sc["tu"], sc["tv"] = np.tile([1.0, 0, 0], (64, 1)), np.tile([0, 1.0, 0], (64, 1))
    sc = scenes.with_emission(sc, seed=5)
    Bh, dB, Bho, dBo = _both(sc, 200)
    assert float(np.abs(dB).max()) == 0.0 and float(np.abs(dBo).max()) == 0.0
    assert rel_l2(Bh, Bho) <= TOL


def test_equal_luminances_go_in_caller_order():
    """Emission only, the same on every surfel: the first shots are caller indices 0, 1, 2."""
    sc = scenes.random_cluster(n=50, seed=8, L=1, nb=1, n_lights=1)
    sc["light_I"] = np.zeros((1, 3))
    E = np.zeros((50, 4, 3))
    E[:, 0] = 0.5
    for i in range(50):  # no receivers: the rows stay equal while they are shot
        sc["p"][i] = (3.0 * i, 0.0, 0.0)
    sc["tu"], sc["tv"] = np.tile([1.0, 0, 0], (50, 1)), np.tile([0, 1.0, 0], (50, 1))
    sc["E"] = E
    _, dB, _, _ = _both(sc, 3)
    assert np.flatnonzero(np.abs(dB).max(axis=(1, 2)) == 0.0).tolist() == [0, 1, 2]
