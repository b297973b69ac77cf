"""The two routes of the FP32 top-N calls, each on libraries that take it: the bounds and the score kernel
(512 and more templates, up to 56 radii) over their shapes, and the sparse kernel (more radii) with its
tiles.  The launch counts say which route ran; results equal, bit for bit, the top-N of every
template's unpruned score.  And the bounded waits of both run out, are reported, and leave a context
that goes on."""
import time

import numpy as np
import pytest

from paper_2111_07347_gb300 import synth, tmgb
from tests.test_gpu_bounds import _topn

pytestmark = pytest.mark.gpu
BOUND_LAUNCHES, SPARSE_LAUNCHES = 4, 2                     # polar, windows, bounds, scores; polar, sparse


def _many_radii():
    """428 templates of 78 spots on 84 radii: more than the bounds' contraction takes."""
    return synth.kinematic_library("hcp", step_deg=3.0, **synth.MULTIPHASE_KINEMATICS)


def _frames(ts, n, n_theta, seed):
    import torch
    frames = synth.render_scan(synth.make_rng(seed), ts, n, 256, 256, n_theta=n_theta).frames
    if n > 2:
        frames[1] = 0
        frames[2, :, :128] = 0
    return torch.from_numpy(frames).cuda()


def _check(ctx, lid, f, hits, n_r, n_theta, top_n, subtract=0.0, prefilter=1.0):
    polar, norm, radial = ctx.polar_transform(f, n_r, n_theta, subtract=subtract)
    K = ctx.library_info(lid)["n_templates"]
    mask, active = None, np.ones((f.shape[0], K), bool)
    if prefilter < 1.0:
        mask, _ = ctx.prefilter(lid, radial, prefilter)
        bits = np.unpackbits(mask.cpu().numpy().view(np.uint8), bitorder="little").reshape(f.shape[0], -1)
        active = bits[:, :K].astype(bool)
    q, s = (a.cpu().numpy() for a in ctx.correlate(lid, polar, norm, mask=mask))
    tk, tsh, tq = _topn(q, s, active, top_n)
    assert np.array_equal(hits["template_index"], tk)
    assert np.array_equal(hits["shift"], tsh)
    assert np.array_equal(hits["score"], tq)


@pytest.mark.parametrize("which,step,n,n_r,n_theta,unit,subtract,prefilter,top_n", [
    ("fcc", 1.0, 33, 90, 77, False, 0.0, 1.0, 5),         # few angles, uneven pieces, no bulk staging
    ("hcp", 2.0, 21, 128, 64, True, 0.0, 1.0, 5),         # the fewest angles
    ("hcp", 2.0, 20, 128, 720, False, 0.3, 0.6, 7),
    ("hcp", 2.0, 20, 128, 720, True, 0.3, 1.0, 7),
    ("hcp", 2.0, 9, 128, 1024, False, 0.0, 1.0, 5),       # the most angles
    ("random", 1.0, 170, 62, 180, False, 0.0, 1.0, 5),    # 56 radii: nine chunks, the longest contraction
    ("random", 1.0, 170, 62, 360, True, 0.2, 1.0, 3)])
def test_bounds_over_their_shapes(which, step, n, n_r, n_theta, unit, subtract, prefilter, top_n):
    if which == "random":
        ts = synth.random_templates(synth.make_rng(7), 600, r_range=(6.0, 61.0))
    else:
        ts = synth.kinematic_library(which, step_deg=step)
    f = _frames(ts, n, n_theta, 84)
    ctx = tmgb.Context(0)
    lid = ctx.load_library(ts, n_r, n_theta, unit_intensity=unit)
    radii = len(np.unique(ctx.library_export(lid)["r"]))
    assert ctx.library_info(lid)["n_templates"] >= 512 and (radii == 56 if which == "random" else radii <= 25)
    hits = tmgb.hits_to_numpy(ctx.index(f, lid, top_n=top_n, subtract=subtract, prefilter=prefilter))[0]
    launches = ctx.last_stats["launches"]
    ctx.check()
    assert launches == BOUND_LAUNCHES if prefilter == 1.0 else launches > BOUND_LAUNCHES
    _check(ctx, lid, f, hits, n_r, n_theta, top_n, subtract, prefilter)
    ctx.close()


@pytest.mark.parametrize("tile", [1, 2, 4])
def test_sparse_kernel_tiles_are_exact(tile, tmp_path, monkeypatch):
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("TMGB_TUNE_CACHE", str(cache))
    ts = _many_radii()
    f = _frames(ts, 50, 360, 85)
    first = tmgb.Context(0)
    first.autotune(f, first.load_library(ts, 128, 360), top_n=5)
    first.close()
    key, threads, seeds = cache.read_text().split()[:3]
    cache.write_text(f"{key} {threads} {seeds} {tile} 0.0\n")
    ctx = tmgb.Context(0)
    lid = ctx.load_library(ts, 128, 360)
    hits = tmgb.hits_to_numpy(ctx.index(f, lid, top_n=5))[0]
    assert ctx.last_stats["launches"] == SPARSE_LAUNCHES
    ctx.check()
    _check(ctx, lid, f, hits, 128, 360, 5)
    ctx.close()


@pytest.mark.parametrize("which,launches,bits", [("sparse", SPARSE_LAUNCHES, 0x4), ("bounds", BOUND_LAUNCHES, 0x8)])
def test_waits_run_out_and_the_context_goes_on(which, launches, bits):
    """TM_INDEX_TEST_STALL: the staging expects bytes that never come, and the bounds' MMAs are never
    issued.  Every wait gives up after about a second and sets its bit of the error word."""
    import torch
    ts = _many_radii() if which == "sparse" else synth.kinematic_library("hcp", step_deg=2.0)
    f = _frames(ts, 8, 360, 86)
    ctx = tmgb.Context(0)
    lid = ctx.load_library(ts, 128, 360)
    want = ctx.index(f, lid, top_n=5)
    assert ctx.last_stats["launches"] == launches
    ctx.check()
    t0 = time.perf_counter()
    ctx.index(f, lid, top_n=5, test_stall=True)
    with pytest.raises(tmgb.TmError) as e:
        ctx.check()
    assert time.perf_counter() - t0 < 30.0
    assert e.value.code == tmgb.TM_ERR_TIMEOUT
    assert int(str(e.value).split("0x")[1].rstrip(")"), 16) & bits == bits
    assert torch.equal(ctx.index(f, lid, top_n=5), want)
    ctx.check()
    ctx.close()


def test_refinement_leaves_unwritten_rows_alone():
    """A scoring kernel that stopped on a wait leaves rows of the caller's buffer as they were; the angle
    refinement that follows reads no template through them."""
    import torch
    ts = synth.kinematic_library("hcp", step_deg=2.0)
    f = _frames(ts, 8, 360, 87)
    ctx = tmgb.Context(0)
    lid = ctx.load_library(ts, 128, 360)
    out = torch.full((1, 8, 5, 5), 0x7F7F7F7F, dtype=torch.int32, device="cuda")
    kept = out.clone()
    ctx.index(f, lid, top_n=5, refine=True, test_stall=True, out=out)
    with pytest.raises(tmgb.TmError):
        ctx.check()
    assert torch.equal(out, kept)
    ctx.index(f, lid, top_n=5, refine=True, out=out)
    ctx.check()
    assert (out[..., 0] >= 0).all()
    ctx.close()


@pytest.mark.parametrize("which,step,K,n,launches", [
    ("hcp", 4.0, 242, 413, 2), ("hcp", 4.0, 242, 414, BOUND_LAUNCHES),     # 100000 pattern-template pairs
    ("fcc+", 3.0, 216, 600, 2),                                            # 34 spots a template: always whole
    ("few", 4.0, 199, 1000, 2), ("few", 4.0, 200, 1000, BOUND_LAUNCHES)])
def test_small_libraries_on_both_sides_of_the_rule(which, step, K, n, launches):
    if which == "few":
        ts = synth.random_templates(synth.make_rng(8), K, spots=(4, 12))
    else:
        ts = synth.kinematic_library(which.rstrip("+"), step_deg=step,
                                     **(synth.MULTIPHASE_KINEMATICS if which.endswith("+") else {}))
    f = _frames(ts, 60, 180, 88).repeat(-(-n // 60), 1, 1)[:n].contiguous()
    ctx = tmgb.Context(0)
    lid = ctx.load_library(ts, 100, 180)
    assert ctx.library_info(lid)["n_templates"] == K
    hits = tmgb.hits_to_numpy(ctx.index(f, lid, top_n=5))[0]
    assert ctx.last_stats["launches"] == launches
    ctx.check()
    _check(ctx, lid, f, hits, 100, 180, 5)
    ctx.close()
