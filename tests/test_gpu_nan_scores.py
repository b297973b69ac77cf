"""Scores that are not numbers: an infinite pixel that one sample of the outermost ring touches makes the
pattern's norm infinite, so Q is 0 for the templates that miss that sample and not a number for the
others.  Every result row is written, numbers first, ties by index."""
import numpy as np
import pytest

from paper_2111_07347_gb300 import synth, tmgb
from tests.test_gpu_bounds import _topn

N_R, N_THETA, SIDE, COLUMN = 101, 360, 256, 359


def _pixel():
    """The pixel that is the lower right tap of the sample (row N_R - 1, column COLUMN) and no tap of any
    other sample."""
    th = 2.0 * np.pi * np.arange(N_THETA) / N_THETA
    r = np.arange(N_R)[:, None]
    x0 = np.floor((SIDE - 1) / 2.0 + r * np.cos(th)).astype(int)
    y0 = np.floor((SIDE - 1) / 2.0 + r * np.sin(th)).astype(int)
    px, py = x0[-1, COLUMN] + 1, y0[-1, COLUMN] + 1
    touch = (np.abs(2 * (px - x0) - 1) == 1) & (np.abs(2 * (py - y0) - 1) == 1)
    assert touch.sum() == 1 and touch[-1, COLUMN]
    return int(px), int(py)


def _templates(K):
    """Three spots each; two of three templates have one on the outermost ring."""
    rng = synth.make_rng(81)
    radii = np.array([20.0, 45.0, 70.0, 90.0])
    a, b = [], []
    for k in range(K):
        r = rng.choice(radii, 3, replace=False)
        if k % 3 != 2:
            r[0] = N_R - 1
        a.extend(r)
        b.extend(2.0 * np.pi * rng.integers(0, N_THETA, 3) / N_THETA)
    off = np.arange(K + 1, dtype=np.int64) * 3
    return synth.TemplateSet(off, np.array(a), np.array(b), rng.uniform(0.5, 2.0, 3 * K), coords="polar", mirror=False)


def test_the_pixel_touches_one_sample():
    _pixel()


@pytest.mark.gpu
@pytest.mark.parametrize("K,top_n", [(9, 7), (700, 5), (700, 64), (1500, 128)])
def test_scores_that_are_not_numbers_rank_last(K, top_n):
    import torch
    px, py = _pixel()
    rng = np.random.default_rng(K)
    frames = rng.poisson(3.0, (40, SIDE, SIDE)).astype(np.float32)
    frames[::2, py, px] = np.inf
    f = torch.from_numpy(frames).cuda()
    ctx = tmgb.Context(0)
    lid = ctx.load_library(_templates(K), N_R, N_THETA)
    polar, norm, _ = ctx.polar_transform(f, N_R, N_THETA, gamma=1.0)
    assert torch.isinf(norm[::2]).all() and torch.isfinite(norm[1::2]).all()
    q, s = (a.cpu().numpy() for a in ctx.correlate(lid, polar, norm))
    assert np.isnan(q[::2]).any(axis=1).all() and not np.isnan(q[1::2]).any()
    tk, tsh, tq = _topn(q, s, np.ones(q.shape, bool), top_n)
    for refine in (False, True):
        out = torch.full((1, len(frames), top_n, 5), -7, dtype=torch.int32, device="cuda")
        h = tmgb.hits_to_numpy(ctx.index(f, lid, top_n=top_n, gamma=1.0, refine=refine, out=out))[0]
        ctx.check()
        assert np.array_equal(h["template_index"], tk)
        assert np.array_equal(h["shift"], tsh)
        assert np.array_equal(h["score"], tq, equal_nan=True)
    ctx.close()
