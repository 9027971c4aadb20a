"""The shooting solver's pick between rows whose luminances differ by 3e-10 relative, in rows of
wide dynamic range: the brighter one is shot first, whichever has the lower caller index, as the
sums in 64 bits order them (both forms, one cluster and two launches per shot).

The surfels do not see each other; E and no light.  Row a: 1 and fifteen coefficients whose low
bits lie below 2^-31 of 1.  Row b: 1 and one coefficient, the sum at most 1e-9 below row a's."""
from fractions import Fraction

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


def _rows(x):
    a = np.zeros(16, np.float32)
    a[0], a[1:] = 1.0, np.float32(x)
    exact = lambda r: sum((Fraction(float(v)) for v in r), Fraction(0))
    b = np.zeros(16, np.float32)
    b[0] = 1.0
    b[1] = np.float32(float(15 * Fraction(float(np.float32(x)))))
    while exact(b) >= exact(a):
        b[1] = np.nextafter(b[1], np.float32(0))
    assert 0 < exact(a) - exact(b) < Fraction(1, 10 ** 9)
    return a, b


# rows updated per shot decide the form: one launch for all shots up to 160,000 values, here none
# are updated (no surfel sees another), so the many-launch form needs rows past a block's memory
@pytest.mark.parametrize("lights", [1, 900], ids=["cluster", "launches"])
@pytest.mark.parametrize("x", [3.337e-4, 4.7e-4])
@pytest.mark.parametrize("first", ["brighter", "darker"])
def test_the_brighter_row_is_shot(x, lights, first):
    n = 40
    sc = scenes.random_cluster(n=n, seed=3, L=3, nb=1, n_lights=lights)
    sc["p"] = np.stack([3.0 * np.arange(n), np.zeros(n), np.zeros(n)], 1)
    sc["tu"], sc["tv"] = np.tile([1.0, 0, 0], (n, 1)), np.tile([0, 1.0, 0], (n, 1))
    sc["light_I"] = np.zeros((lights, 3))
    a, b = _rows(x)
    i, j = (7, 23) if first == "brighter" else (23, 7)
    sc["E"] = np.zeros((n, 16, 3))
    sc["E"][i], sc["E"][j] = a[:, None], b[:, None]
    d = api.upload(sc)
    pipe = api.Pipeline(pairs=True)
    pipe.build(d)
    pipe.trace(d)
    rgs.rgs_profile_reset()
    rgs.rgs_profile_enable(True)
    _, dB = rgs.rgs_prog_refine(pipe.transport, 1, E=d["E"])
    torch.cuda.synchronize()
    rgs.rgs_profile_enable(False)
    assert (rgs.rgs_profile_report().get("k_pr_shoot", (0, 0.0))[0] > 0) == (lights == 1)
    left = np.flatnonzero(np.abs(dB.cpu().numpy()).max(axis=(1, 2)) > 0).tolist()
    assert left == [j]
