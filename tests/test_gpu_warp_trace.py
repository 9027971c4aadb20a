"""The warp-cooperative tracer at the sizes where it can go wrong, against the FP64 oracle:
trees with fewer than four children per node, rays with more hits than a warp's list keeps
(the nearest are kept, in several rounds), pixels that take several compositing passes,
images and source counts that leave warps ragged, and boxes far from the origin (the nodes
hold them in 8 bits).

Tolerance: the FP32 bar of the parity tests, 1e-4 relative L2 (FP32 sums over at most
nd * hits terms, ~1e-6; a hit flipping at the cutoff changes one ray by ~1e-2 alpha, rarely)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2509_18497_gb300 import api, rgs, scenes

from gpu_helpers import rel_l2, run_gpu, run_oracle

pytestmark = pytest.mark.gpu

TOL = 1e-4


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_18497_gb300 import build
    build.build()
    rgs.load()


def _check(sc, pairs=False, alpha=(rgs.RGS_ALPHA_GAUSS, O.ALPHA_GAUSS)):
    sc = scenes.with_emission(sc, seed=3)
    W = np.random.default_rng(2).normal(size=(sc["n"], (sc["L"] + 1) ** 2, 3 * max(len(sc["light_pos"]), 1)))
    g = run_gpu(sc, W=W, alpha_model=alpha[0], pairs=pairs)
    o = run_oracle(sc, W=W, alpha_model=alpha[1], pairs=pairs)
    for key in ("B", "dE", "dad", "dop") + (("dlam",) if pairs else ()):
        assert rel_l2(g[key], o[key]) <= TOL, (key, rel_l2(g[key], o[key]))
    return g, o


@pytest.mark.parametrize("pairs", [False, True], ids=["hemisphere", "pairs"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6, 33, 257])
def test_small_trees(n, pairs):
    _check(scenes.random_cluster(n=n, seed=n, L=2, nd=32, nb=2, n_lights=2), pairs)


@pytest.mark.parametrize("n", [255, 256, 513])
def test_pairs_source_chunks(n):
    """Blocks of 256 sources, full and with one over."""
    _check(scenes.random_cluster(n=n, seed=n, L=1, nd=32, nb=1, n_lights=1), True)


@pytest.mark.parametrize("n", [2048, 2561])
def test_pairs_large_source_chunks(n):
    """Blocks of 512 sources: surfels of opacity 0 inside the cloud change nothing for the others."""
    m = 150
    sc = scenes.with_emission(scenes.random_cluster(n=m, seed=7, L=1, nd=32, nb=2, n_lights=1), seed=3)
    W = np.random.default_rng(2).normal(size=(m, 4, 3))
    o = run_oracle(sc, W=W, pairs=True)
    rng = np.random.default_rng(n)
    src = rng.integers(0, m, size=n - m)
    big = dict(sc, n=n)
    for key, v in sc.items():
        if isinstance(v, np.ndarray) and v.ndim and v.shape[0] == m:
            big[key] = np.concatenate([v, v[src]])
    lo, hi = sc["p"].min(0), sc["p"].max(0)
    big["p"][m:] = (lo + (hi - lo) * rng.uniform(0.3, 0.7, size=(n - m, 3))).astype(np.float32)
    big["s"][m:] *= 0.1
    big["o"][m:] = 0.0
    big["E"][m:] = 0.0
    at = rng.permutation(n)  # the caller's order mixes the two
    for key, v in big.items():
        if isinstance(v, np.ndarray) and v.ndim and v.shape[0] == n:
            big[key] = v[at]
    real = np.argsort(at)[:m]
    Wb = np.zeros((n, 4, 3))
    Wb[real] = W
    g = run_gpu(big, W=Wb, pairs=True)
    for key in ("B", "dE", "dad", "dop", "dlam"):
        assert rel_l2(g[key][real], o[key]) <= TOL, (key, rel_l2(g[key][real], o[key]))


def _overlapping(n, o_lo, o_hi, seed=5):
    """A cloud whose surfels all cover each other: about half of them on every ray."""
    sc = scenes.random_cluster(n=n, seed=seed, L=1, nd=32, nb=2, n_lights=1)
    sc["s"] = np.asarray(sc["s"] * 8.0, np.float32).astype(np.float64)
    sc["o"] = np.random.default_rng(seed).uniform(o_lo, o_hi, size=n).astype(np.float32).astype(np.float64)
    return sc


def test_more_hits_than_a_list_keeps():
    """Rays with up to ~400 hits whose nearest 96 leave less than the transmittance cut."""
    g, o = _check(_overlapping(500, 0.7, 0.95))
    assert np.diff(o["orc"].hits()["off"]).max() > 2 * 96
    assert g["info"]["n_full_rays"] == 0


@pytest.mark.parametrize("shape", [(7, 5), (33, 9), (8, 4)], ids=str)
@pytest.mark.parametrize("opacity", [(0.02, 0.05), (0.3, 0.9)], ids=["faint", "dense"])
def test_pixels_of_several_passes(opacity, shape):
    """Faint: every pixel composites hundreds of hits, in several passes of the kernel."""
    sc = _overlapping(500, *opacity, seed=7)
    pipe = api.Pipeline()
    d = api.upload(sc)
    pipe.build(d)
    pipe.trace(d)
    orc = O.Oracle(sc).transport()
    w, h = shape
    rng = np.random.default_rng(1)
    B, G = rng.normal(size=(sc["n"], 4, 3)), rng.normal(size=(h, w, 3))
    cam = [0.5, 0.6, 4.0, 0.0, 0.0, -1.0, 0.0, 1.0, 0.0]
    up = lambda x: torch.as_tensor(x.astype(np.float32), device="cuda")
    img = rgs.rgs_render(pipe.transport, up(B), cam, w, h, 0.5).double().cpu().numpy()
    dB = rgs.rgs_render_adjoint(pipe.transport, up(G), cam, w, h, 0.5).double().cpu().numpy()
    assert rel_l2(img, orc.render(B, cam, w, h, 0.5)) <= TOL
    assert rel_l2(dB, orc.render_adjoint(G, cam, w, h, 0.5)) <= TOL


@pytest.mark.parametrize("alpha", [(rgs.RGS_ALPHA_DISC, O.ALPHA_DISC), (rgs.RGS_ALPHA_GFSGS, O.ALPHA_GFSGS)],
                         ids=["disc", "gfsgs"])
def test_far_from_the_origin(alpha):
    """The cloud in a corner of a large scene: boxes of 8 bits on nodes of very different sizes."""
    sc = scenes.random_cluster(n=200, seed=11, L=2, nd=64, nb=2, n_lights=1)
    sc["p"][:100] = np.asarray(sc["p"][:100] + 8.0, np.float32).astype(np.float64)
    _check(sc, alpha=alpha)


@pytest.mark.parametrize("n", [1024, 1025, 4097, 8192, 8193])
def test_surfel_order_at_the_sort_sizes(n):
    """Scenes at the sizes where the Morton sort pads, fills its block, or goes over to the radix
    passes, with equal keys (pairs of surfels at one centre): sampled receivers against the oracle."""
    sc = scenes.random_cluster(n=n, seed=n, L=1, nd=32, nb=1, n_lights=1, extent=4.0)
    sc["s"] = sc["s"] * 0.3
    sc["p"][1::2] = sc["p"][0:n - n % 2:2]
    g = run_gpu(sc, iterates=True)
    orc = O.Oracle(sc)
    recv = np.random.default_rng(1).choice(n, size=12, replace=False)
    assert rel_l2(g["iters"][0][recv], orc.sample_direct(recv)) <= TOL
    assert rel_l2(g["iters"][1][recv], orc.sample_bounce1(recv)) <= TOL


@pytest.mark.parametrize("shape", [(999, 500), (1003, 499), (1001, 601), (1201, 1001)], ids=str)
def test_images_of_every_tile_height(shape):
    """8, 16 and 32 pixels to a warp (below 500,000 and 1,200,000 pixels, and beyond), with tiles
    that the image's edges cut.  Among a million pixels a few lie where rounding decides (a
    cutoff, the order of two near-equal depths): those whose value in 64 bits changes when the
    camera moves by 1e-6 are left out, at most one in 10,000."""
    sc = scenes.random_cluster(n=14, seed=4, L=1, nd=32, nb=1, n_lights=1)
    pipe = api.Pipeline()
    d = api.upload(sc)
    pipe.build(d)
    pipe.trace(d)
    orc = O.Oracle(sc).transport()
    w, h = shape
    rng = np.random.default_rng(1)
    B, G = rng.normal(size=(sc["n"], 4, 3)), rng.normal(size=(h, w, 3))
    cam = [0.5, 0.6, 3.0, 0.0, 0.0, -1.0, 0.0, 1.0, 0.0]
    want = orc.render(B, cam, w, h, 0.5)
    stable = np.ones((h, w), bool)
    for axis in range(3):
        for step in (-1e-6, 1e-6):
            moved = list(cam)
            moved[axis] += step
            stable &= np.abs(orc.render(B, moved, w, h, 0.5) - want).max(-1) < 1e-3
    assert stable.mean() > 1 - 1e-4
    G[~stable] = 0.0
    up = lambda x: torch.as_tensor(x.astype(np.float32), device="cuda")
    img = rgs.rgs_render(pipe.transport, up(B), cam, w, h, 0.5).double().cpu().numpy()
    dB = rgs.rgs_render_adjoint(pipe.transport, up(G), cam, w, h, 0.5).double().cpu().numpy()
    assert np.abs(want).max() > 0 and rel_l2(img[stable], want[stable]) <= TOL
    assert rel_l2(dB, orc.render_adjoint(G, cam, w, h, 0.5)) <= TOL
