"""The one-pass preprocessing kernel on frames that take it (at least 96 rows and five times the filters'
reach): the bits of the separate passes, which serve a result written over its input."""
import numpy as np
import pytest

from paper_2111_07347_gb300 import tmgb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,H,W,dog,blur", [
    (1, 100, 97, (1.0, 4.0), 1.0),                         # the least rows for a reach of 20
    (700, 101, 131, (1.0, 4.0), 1.0),                      # more frames than resident blocks
    (5, 144, 64, (0.3, 0.6), 0.5), (2, 257, 65, (2.0, 5.3), 0.0), (3, 112, 96, (1.0, 4.0), 0.0), (3, 250, 243, (0.7, 2.3), 2.0),
    (4, 200, 400, (1.5, 2.5), 4.0), (2, 512, 512, (0.5, 1.5), 0.5), (3, 250, 255, (2.0, 10.0), 2.0),
    (9, 144, 144, None, 1.0), (40, 300, 509, None, 0.2)])
def test_one_pass_equals_the_separate_passes_on_large_frames(n, H, W, dog, blur):
    import torch
    ctx = tmgb.Context(0)
    rng = np.random.default_rng(n * 1000 + H)
    frames = torch.from_numpy(rng.poisson(3.0, size=(n, H, W)).astype(np.float32)).cuda()
    apart = ctx.preprocess(frames, dog=dog, blur=blur)
    over = frames.clone()
    ctx.preprocess(over, dog=dog, blur=blur, out=over)
    assert torch.equal(apart, over)
    u16 = ctx.preprocess(torch.from_numpy(frames.cpu().numpy().astype(np.uint16)).cuda(), dog=dog, blur=blur)
    assert torch.equal(apart, u16)
    ctx.close()
