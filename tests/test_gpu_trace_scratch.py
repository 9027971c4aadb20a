"""The pooled hit lists of a trace and an image under a memory budget: 40 MB (a block per SM) where the
budget leaves nothing, instead of up to 319 MB, with the same results."""
import numpy as np
import pytest
import torch

from paper_2509_18497_gb300 import api, rgs, scenes

from gpu_helpers import rel_l2

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_18497_gb300 import build
    build.build()


def _pooled(call):
    """call()'s result and the bytes by which the library's pool grew."""
    torch.cuda.synchronize()
    rgs.rgs_trim_workspace()
    before = torch.cuda.mem_get_info()[0]
    out = call()
    torch.cuda.synchronize()
    return out, before - torch.cuda.mem_get_info()[0]


def test_hit_lists_within_the_budget():
    sc = scenes.with_emission(scenes.fruit_bowl(n=6000, L=1, nd=64, nb=1), seed=1)
    d = api.upload(sc)
    pipe = api.Pipeline()
    pipe.build(d)
    pipe.trace(d)
    B = torch.empty((6000, 4, 3), device="cuda")
    B.normal_(generator=torch.Generator(device="cuda").manual_seed(1))
    cam, size, img = [0.0, 2.6, 4.4, 0.0, -0.43, -0.9, 0.0, 1.0, 0.0], (1300, 1000), torch.empty((1000, 1300, 3), device="cuda")

    def both():
        _, a = _pooled(lambda: pipe.trace(d))
        solved = pipe.solve(d["E"], 1)[0].double().cpu().numpy()
        _, b = _pooled(lambda: rgs.rgs_render(pipe.transport, B, cam, *size, 0.7, img_out=img))
        return a, b, solved, img.double().cpu().numpy()

    both()
    a, b, B1, img1 = both()
    assert a > 200 * MB and b > 200 * MB
    pipe.mem_budget = 1
    rgs.rgs_set_memory_budget(pipe.transport, 1)
    a, b, B2, img2 = both()
    assert a <= 80 * MB and b <= 80 * MB
    assert rel_l2(B2, B1) <= 1e-6 and rel_l2(img2, img1) <= 1e-6
