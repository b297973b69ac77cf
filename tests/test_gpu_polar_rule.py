"""The polar transform of float frames on both sides of the rule that transforms staged frames first, and
the scalar staging of frames whose rows are not whole 16-byte units."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2111_07347_gb300 import tmgb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,n_r,n_theta", [
    (128, 128, 16, 36), (128, 128, 60, 91), (128, 128, 60, 92),      # a third of 16384 samples: between 91 and 92
    (97, 131, 20, 40), (97, 131, 60, 180), (200, 224, 30, 90), (64, 64, 30, 90), (7, 5, 4, 8)])
@pytest.mark.parametrize("gamma,subtract,threshold", [(0.5, 0.0, 0.0), (1.0, 0.2, 1.5), (0.4, 0.1, 0.0)])
def test_polar_equals_the_oracle_and_the_u16_path(H, W, n_r, n_theta, gamma, subtract, threshold):
    """Both sides against the oracle, with and without a pixel mask; on u16-valued frames the float path
    gives the u16 path's samples."""
    import torch
    rng = np.random.default_rng(H * W + n_r)
    a = rng.poisson(3.0, (5, H, W)).astype(np.uint16)
    f = torch.from_numpy(a.astype(np.float32)).cuda()
    u = torch.from_numpy(a.view(np.int16)).cuda().view(torch.uint16)
    mask = torch.from_numpy((rng.random((H, W)) > 0.2).astype(np.uint8)).cuda()
    ctx = tmgb.Context(0)
    ref = O.polar(a.astype(np.float32), n_r, n_theta, gamma=gamma, subtract=subtract, threshold=threshold)
    kw = dict(gamma=gamma, subtract=subtract, threshold=threshold)
    got = ctx.polar_transform(f, n_r, n_theta, **kw)
    P = got[0].cpu().numpy().astype(np.float64)
    assert np.all(np.abs(P - ref) <= 1e-6 * (np.abs(ref).max() + abs(subtract)))
    for m in (None, mask):
        x = ctx.polar_transform(f, n_r, n_theta, mask=m, **kw)
        y = ctx.polar_transform(u, n_r, n_theta, mask=m, **kw)
        assert torch.equal(x[0], y[0])
    ctx.check()
    ctx.close()
