"""Rays with more hits than a list keeps, against the FP64 oracle's hits: the nearest 96 are kept
and an image composites all of them, whatever the depth at which the traversal stops.

A stack of wide, faint, axis-aligned surfels 2e-6 apart, all of them on every ray: the 96th
depth lies inside every subtree's range, closer to the subtrees' first planes than the rounding of
an 8-bit box test on a 30-unit node (8e-6 of its width), and no cutoff or depth order depends on
FP32 (depth gaps of 2e-6 and more at depths below 1 with errors below 1e-7, 1e-4 and 3e-4
at depths of 40 and 120 with errors below 3e-5; rays that leave an ellipse are not used).

Tolerance 2e-5: a weight is a product of up to 500 factors of relative error 2^-24 (random: 1.4e-6)
times a Gaussian of relative error 1e-6; one hit lost or exchanged moves a ray by 1e-3 and more."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2509_18497_gb300 import api, rgs

from gpu_helpers import rel_l2, run_gpu

pytestmark = pytest.mark.gpu

TOL = 2e-5
HMAX = 96
LAYERS, BELOW = 500, 12


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_18497_gb300 import build
    build.build()


def _stack(seed, L=0, gap=2e-6):
    """LAYERS layers `gap` apart from y = 0 on in the caller's shuffled order, then BELOW receivers 0.1 under them."""
    rng = np.random.default_rng(seed)
    n = LAYERS + BELOW
    p = rng.uniform(-0.3, 0.3, size=(n, 3))
    p[:LAYERS, 1] = gap * rng.permutation(LAYERS)
    p[LAYERS:, 1] = -0.1
    s = np.full((n, 2), 5.0)
    s[LAYERS:] = 1e-3
    o = rng.uniform(0.01, 0.03, size=n)
    o[LAYERS:] = 1.0
    rows = lambda *v: np.tile(np.array(v, np.float64), (n, 1))
    sc = dict(n=n, L=L, nd=128, nb=1, seed=seed, p=p, tu=rows(1, 0, 0), tv=rows(0, 0, -1), s=s, o=o, ad=rows(0.5, 0.5, 0.5),
              k=np.ones(n), as_=rows(0, 0, 0), shin=np.full(n, 1.0), light_pos=np.zeros((0, 3)), light_I=np.zeros((0, 3)),
              E=rng.uniform(0.0, 1.0, size=(n, (L + 1) ** 2, 3)))
    sc["E"][LAYERS:] = 0.0
    for key, v in sc.items():
        if isinstance(v, np.ndarray):
            sc[key] = v.astype(np.float32).astype(np.float64)
    return sc


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_the_nearest_hits_are_kept(seed):
    """One bounce (constant SH) of receivers under the stack: B = o 4 ad / (4 nd) sum over the rays' nearest 96 hits."""
    sc = _stack(seed)
    g = run_gpu(sc)
    assert g["info"]["n_full_rays"] > 0
    orc = O.Oracle(sc)
    used = 0
    for i in range(LAYERS, sc["n"]):
        x = np.zeros(3)
        whole = True
        for r in range(sc["nd"]):
            j, _, alpha, _ = orc.trace_ray(i, sc["p"][i], orc.ray_dir(i, sc["nd"], sc["seed"], r))
            whole &= len(j) == LAYERS
            a = alpha * np.concatenate([[1.0], np.cumprod(1.0 - alpha)[:-1]])
            x += (a[:HMAX, None] * sc["E"][j[:HMAX], 0]).sum(0)
        if whole:
            used += 1
            want = 4 * 0.5 / (4 * sc["nd"]) * x
            assert np.abs(g["B"][i, 0] / want - 1).max() <= TOL, (i, g["B"][i, 0] / want - 1)
    assert used >= BELOW // 2


@pytest.mark.parametrize("height,gap,fov", [(0.1, 2e-6, 0.5), (0.6, 2e-6, 0.5), (40.0, 1e-4, 0.02), (120.0, 3e-4, 0.006)])
def test_pixels_lose_no_hit(height, gap, fov):
    """An image from under the stack, whose pixels take six passes each, from within the scene's
    box, from outside and from far outside."""
    sc = _stack(5, L=1, gap=gap)
    pipe = api.Pipeline()
    d = api.upload(sc)
    pipe.build(d)
    pipe.trace(d)
    orc = O.Oracle(sc).transport()
    w, h = 33, 9
    rng = np.random.default_rng(1)
    B, G = rng.normal(size=(sc["n"], 4, 3)), rng.normal(size=(h, w, 3))
    B[:, 0] = np.abs(B[:, 0]) + 1.0
    B[LAYERS:] = 0.0
    cam = [0.0, -float(np.float32(height)), 0.0, 0.0, 1.0, 0.05, 1.0, 0.0, 0.0]
    up = lambda x: torch.as_tensor(x.astype(np.float32), device="cuda")
    img = rgs.rgs_render(pipe.transport, up(B), cam, w, h, fov).double().cpu().numpy()
    dB = rgs.rgs_render_adjoint(pipe.transport, up(G), cam, w, h, fov).double().cpu().numpy()
    want = orc.render(B, cam, w, h, fov)
    assert np.abs(want).min() > 0 and rel_l2(img, want) <= TOL
    assert rel_l2(dB[:LAYERS], orc.render_adjoint(G, cam, w, h, fov)[:LAYERS]) <= TOL
