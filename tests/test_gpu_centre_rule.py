"""Beam centres by a thread and by a warp per pattern: bit-exact on both sides of the rule."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2111_07347_gb300 import tmgb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,radius,few,many", [
    (np.uint16, 1.0, 864, 865),                            # 9 pixels: up to 96 patterns a pixel
    (np.uint16, 3.0, 50, 4705),
    (np.float32, 1.0, 675, 676),                           # 150 x 9 / 2 steps
    (np.float32, 3.0, 2450, 2451),                         # 150 x 49 / 3
    (np.float32, 9.5, 10, 4000)])
def test_centres_are_exact_on_both_sides(dtype, radius, few, many):
    import torch
    rng = np.random.default_rng(int(10 * radius))
    H, W = 40, 36
    base = rng.poisson(4.0, (64, H, W)).astype(dtype)
    base[:, 17:21, 15:20] += np.asarray(60, dtype)
    if dtype == np.float32:
        base *= rng.uniform(0.3, 1.7, base.shape).astype(np.float32)
    ref = O.find_centres(base, ((W - 1) / 2.0, (H - 1) / 2.0), radius, 3)
    ctx = tmgb.Context(0)
    for n in (few, many):
        a = np.tile(base, ((n + 63) // 64, 1, 1))[:n]
        f = torch.from_numpy(a.view(np.int16)).cuda().view(torch.uint16) if dtype == np.uint16 else torch.from_numpy(a).cuda()
        c = ctx.find_centres(f, radius=radius, iterations=3).cpu().numpy()
        assert np.array_equal(c, np.tile(ref, ((n + 63) // 64, 1))[:n])
    ctx.close()
