"""Frame sums on both sides of the rule that gives a thread four pixels, and where the partial sums of
all groups do not fit the context's budget."""
import numpy as np
import pytest

from paper_2111_07347_gb300 import tmgb

pytestmark = pytest.mark.gpu


def _frames(n, H, W):
    import torch
    a = np.random.default_rng(n + H).integers(0, 65536, (n, H, W), dtype=np.uint16)
    return a, torch.from_numpy(a.view(np.int16)).cuda().view(torch.uint16)


@pytest.mark.parametrize("n,H,W,shift", [(128, 512, 512, 0), (320, 256, 256, 0), (400, 256, 256, 0),
                                         (700, 64, 64, 0), (2100, 33, 31, 0), (1000, 128, 128, 1), (129, 300, 500, 0)])
def test_sums_are_exact(n, H, W, shift):
    """shift: frames that start on an odd pixel (four-pixel loads are not aligned)."""
    import torch
    a, f = _frames(n, H, W)
    if shift:
        flat = torch.empty(n * H * W + shift, dtype=torch.uint16, device="cuda")
        flat[shift:] = f.reshape(-1)
        f = flat[shift:].view(n, H, W)
    ctx = tmgb.Context(0)
    out = torch.full((H, W), 0.5, dtype=torch.float64, device="cuda")
    want = a.sum(axis=0, dtype=np.uint64).astype(np.float64)
    assert np.array_equal(ctx.frame_sum(f).cpu().numpy(), want)
    assert np.array_equal(ctx.frame_sum(f, out=out, accumulate=True).cpu().numpy(), want + 0.5)
    ctx.close()


@pytest.mark.parametrize("budget", [4 << 20, 2 << 20])
def test_a_small_budget_takes_fewer_groups(budget):
    """1300 frames: nineteen groups of 256 x 256 partial sums take 10 MB, four take 2 MB."""
    a, f = _frames(1300, 256, 256)
    ctx = tmgb.Context(0, budget)
    if budget == 2 << 20:
        with pytest.raises(tmgb.TmError) as e:
            ctx.frame_sum(f)
        assert e.value.code == tmgb.TM_ERR_OOM
    else:
        assert np.array_equal(ctx.frame_sum(f).cpu().numpy(), a.sum(axis=0, dtype=np.uint64).astype(np.float64))
    ctx.close()
