"""Templates left out by the tensor-core bounds: the fused top-N equals, bit for bit, the top-N
taken from every template's unpruned score (tm_correlate) over the forms the rule accepts."""
import numpy as np
import pytest

from paper_2111_07347_gb300 import synth, tmgb


def _topn(q, s, active, N):
    """Top-N by (Q desc, template asc) over the active templates of each pattern."""
    n = q.shape[0]
    tk, tsh = np.full((n, N), -1, np.int64), np.full((n, N), -1, np.int64)
    tq = np.full((n, N), -np.inf, np.float32)
    for p in range(n):
        idx = np.flatnonzero(active[p])
        order = idx[np.lexsort((idx, -q[p, idx].astype(np.float64)))][:N]
        tk[p, :len(order)], tsh[p, :len(order)], tq[p, :len(order)] = order, s[p, order], q[p, order]
    return tk, tsh, tq


def test_pieces_cover_every_visited_column():
    """CPU: for every angle count and shape of the bounds, the run of pieces taken for a (chunk,
    window) pair holds every column t + s with t in the chunk and s in the window."""
    for n_theta in list(range(72, 200)) + [240, 250, 300, 320, 359, 360, 361, 512, 720, 1023, 1024]:
        for nch in (24, 18, 12, 9):
            for nw in (6, 12):
                P = int(np.lcm(nch, nw))
                if P > n_theta:
                    continue
                start = np.array([i * n_theta // P for i in range(2 * P + 2)])
                piece_of = np.repeat(np.arange(2 * P + 1), np.diff(start))
                cl, wl = P // nch, P // nw
                before = 1 if n_theta % P else 0
                for j in range(nch):
                    for h in range(nw):
                        lo = start[j * cl] + start[h * wl]
                        hi = start[(j + 1) * cl] - 1 + start[(h + 1) * wl] - 1
                        first = j * cl + h * wl - before
                        run = cl + wl + before
                        assert piece_of[lo] >= first and piece_of[hi] < first + run, (n_theta, nch, nw, j, h)


FORMS = [
    # library, step, n, n_r, n_theta, unit, subtract, prefilter, top_n
    ("fcc", 1.0, 50, 128, 360, False, 0.0, 1.0, 5),
    ("hcp", 1.0, 41, 128, 360, False, 0.0, 1.0, 5),
    ("hcp", 1.0, 1, 128, 360, False, 0.0, 0.5, 5),
    ("hcp", 1.5, 500, 128, 360, True, 0.4, 1.0, 5),       # twelve windows, negative polar values
    ("fcc", 1.5, 7, 128, 360, True, 0.0, 0.3, 128),       # the longest result list
    ("tetragonal", 1.5, 80, 128, 360, False, 0.2, 1.0, 3),
    ("tetragonal", 2.0, 30, 120, 250, False, 0.0, 1.0, 5),   # uneven pieces
    ("fcc", 2.0, 33, 90, 77, False, 0.0, 1.0, 5),         # few angles: rows staged without bulk copies
    ("hcp", 2.0, 33, 128, 361, True, 0.0, 1.0, 1),
    ("hcp", 3.0, 20, 128, 720, False, 0.3, 0.6, 7),
    ("hcp", 3.0, 9, 128, 1024, False, 0.0, 1.0, 5),
    ("random", 1.0, 300, 60, 180, False, 0.0, 1.0, 5),    # 55 radii: the coarsest chunks
    ("few", 1.0, 3, 60, 180, False, 0.0, 1.0, 8),         # fewer templates than results
]


@pytest.mark.gpu
@pytest.mark.parametrize("which,step,n,n_r,n_theta,unit,subtract,prefilter,top_n", FORMS)
def test_bounded_top_n_is_exact(which, step, n, n_r, n_theta, unit, subtract, prefilter, top_n):
    import torch
    rng = synth.make_rng(77)
    if which in ("random", "few"):
        ts = synth.random_templates(rng, 300 if which == "random" else 6)
    else:
        ts = synth.kinematic_library(which, step_deg=step)
    scan = synth.render_scan(rng, ts, n, 256, 256, n_theta=n_theta)
    frames = scan.frames
    if n > 2:
        frames[1] = 0                                     # a blank frame: every Q is 0 (or its background's)
        frames[2, :, :128] = 0
    ctx = tmgb.Context(0)
    lid = ctx.load_library(ts, n_r, n_theta, unit_intensity=unit)
    K = ctx.library_info(lid)["n_templates"]
    f = torch.from_numpy(frames).cuda()
    hits = tmgb.hits_to_numpy(ctx.index(f, lid, top_n=top_n, subtract=subtract, prefilter=prefilter))[0]
    ctx.check()
    polar, norm, radial = ctx.polar_transform(f, n_r, n_theta, subtract=subtract)
    mask, active = None, np.ones((n, K), bool)
    if prefilter < 1.0:
        mask, _ = ctx.prefilter(lid, radial, prefilter)
        bits = np.unpackbits(mask.cpu().numpy().view(np.uint8), bitorder="little").reshape(n, -1)
        active = bits[:, :K].astype(bool)
    q, s = ctx.correlate(lid, polar, norm, mask=mask)
    tk, tsh, tq = _topn(q.cpu().numpy(), s.cpu().numpy(), active, top_n)
    assert np.array_equal(hits["template_index"], tk)
    assert np.array_equal(hits["shift"], tsh)
    assert np.array_equal(hits["score"], tq)
    ctx.close()


@pytest.mark.gpu
def test_bounds_leave_a_small_budget_to_the_general_path():
    """A context whose budget has no room for the bounds' templates indexes all the same, with the
    same result."""
    import torch
    ts = synth.kinematic_library("hcp", step_deg=3.0)
    scan = synth.render_scan(synth.make_rng(78), ts, 12, 256, 256, n_theta=360)
    f = torch.from_numpy(scan.frames).cuda()
    big = tmgb.Context(0)
    want = tmgb.hits_to_numpy(big.index(f, big.load_library(ts, 128, 360), top_n=5))
    budget = 400 << 20
    for b in (budget, 64 << 20, 32 << 20):
        ctx = tmgb.Context(0, b)
        lid = ctx.load_library(ts, 128, 360)
        assert np.array_equal(tmgb.hits_to_numpy(ctx.index(f, lid, top_n=5)), want)
        ctx.check()
        ctx.close()
    big.close()


@pytest.mark.gpu
def test_bounds_replay_in_a_graph_and_on_two_streams():
    """Calls that go through the bounds give the same hits replayed as a CUDA graph, and on two
    streams whose scratch is their own."""
    import torch
    ts = synth.kinematic_library("hcp", step_deg=1.5)
    scan = synth.render_scan(synth.make_rng(79), ts, 200, 256, 256, n_theta=360)
    f = torch.from_numpy(scan.frames).cuda()
    ctx = tmgb.Context(0)
    lid = ctx.load_library(ts, 128, 360)
    assert ctx.library_info(lid)["n_templates"] >= 512
    want = ctx.index(f, lid, top_n=5)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    outs = [torch.zeros_like(want) for _ in streams]
    for _ in range(4):
        for st, out in zip(streams, outs):
            out.zero_()
        torch.cuda.synchronize()
        for st, out in zip(streams, outs):
            ctx.index(f, lid, top_n=5, out=out, stream=st, graph=True)
        torch.cuda.synchronize()
        for out in outs:
            assert torch.equal(out, want)
    ctx.close()
