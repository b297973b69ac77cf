"""Launch shapes of the score kernel: every size it claims to support can be launched, and such calls
return the top-N of the unpruned scores."""
import numpy as np
import pytest

from paper_2111_07347_gb300 import synth, tmgb
from tests.test_gpu_bounds import _topn

LIMIT = 227 * 1024 - 2560


def _wrapped_pitch(n_theta):
    """Row pitch of the wrapped layout: shift blocks of 32 rounded up to an unrolled kernel's."""
    nb = -(-n_theta // 32)
    nb = next(v for v in (1, 2, 3, 4, 6, 8, 12, 16, 24, 32) if nb <= v)
    return max(n_theta + 32, 32 * nb)


def test_supported_sizes_have_a_launch_shape():
    """Wherever the wrapped rows and the lists of the largest block (32 warps up to 384 angles, else
    16) fit shared memory there is a shape, with the smallest block among them."""
    refused = 0
    for n_theta in list(range(64, 400, 23)) + [384, 385, 400, 500, 512, 720, 768, 769, 1000, 1024]:
        warps = 32 if n_theta <= 384 else 16
        for top_n in (1, 2, 3, 5, 7, 10, 20, 32, 33, 64, 100, 128):
            for n_rad in range(1, 130):
                fits = n_rad * _wrapped_pitch(n_theta) * 4 + 8 + 8 * top_n + 12 * warps * top_n <= LIMIT
                shapes = tmgb.tm_score_shapes_host(n_rad, n_theta, top_n)
                if fits:
                    assert shapes[0] == 256 and shapes[-1] == 32 * warps, (n_rad, n_theta, top_n, shapes)
                refused += not shapes
    assert refused > 0                                    # the range reaches past what fits


@pytest.mark.parametrize("n_theta,top_n,n_rad", [(512, 10, 27), (512, 32, 25), (512, 32, 26), (400, 10, 30),
                                                 (400, 64, 25), (400, 64, 27), (720, 20, 18), (720, 128, 11),
                                                 (720, 128, 14), (1024, 20, 13)])
def test_sizes_at_the_layouts_border_have_a_shape(n_theta, top_n, n_rad):
    assert tmgb.tm_score_shapes_host(n_rad, n_theta, top_n)[:1] == [256]


@pytest.mark.gpu
@pytest.mark.parametrize("step", [3.0, 2.5])              # 428 templates (scored whole), 604 (bounded)
@pytest.mark.parametrize("n_theta,top_n", [(512, 32), (400, 64)])
def test_index_at_the_layouts_border(n_theta, top_n, step):
    import torch
    ts = synth.kinematic_library("hcp", step_deg=step)    # 25 radii
    scan = synth.render_scan(synth.make_rng(80), ts, 12, 256, 256, n_theta=n_theta)
    f = torch.from_numpy(scan.frames).cuda()
    ctx = tmgb.Context(0)
    lid = ctx.load_library(ts, 128, n_theta)
    hits = tmgb.hits_to_numpy(ctx.index(f, lid, top_n=top_n))[0]
    ctx.check()
    polar, norm, _ = ctx.polar_transform(f, 128, n_theta)
    q, s = (a.cpu().numpy() for a in ctx.correlate(lid, polar, norm))
    tk, tsh, tq = _topn(q, s, np.ones(q.shape, bool), top_n)
    assert np.array_equal(hits["template_index"], tk)
    assert np.array_equal(hits["shift"], tsh)
    assert np.array_equal(hits["score"], tq)
    ctx.close()
