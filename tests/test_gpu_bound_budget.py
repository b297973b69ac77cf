"""Libraries whose bound templates do not fit the context's budget."""
import dataclasses
import time

import numpy as np
import pytest

from paper_2111_07347_gb300 import synth, tmgb

pytestmark = pytest.mark.gpu


def _enqueue_time(fn):
    """Best host time of a call that only enqueues, over five runs of eight."""
    import torch
    best = np.inf
    for _ in range(5):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(8):
            fn()
        best = min(best, (time.perf_counter() - t0) / 8)
    torch.cuda.synchronize()
    return best


def test_refused_bounds_cost_nothing_and_change_nothing():
    """The smallest budget in which a library without bounds (a negative intensity) and then this one
    can be indexed leaves no room for the bound templates: the calls go through the sparse kernel, whose
    scratch is there, give the same hits, and a refusal costs the host next to nothing."""
    import torch
    ts = synth.kinematic_library("hcp", step_deg=0.5)
    scan = synth.render_scan(synth.make_rng(82), ts, 1, 256, 256, n_theta=360)
    f = torch.from_numpy(scan.frames).cuda()
    negative = dataclasses.replace(ts, intensity=ts.intensity.copy())
    negative.intensity[0] *= -1.0

    def run(mb):
        ctx = tmgb.Context(0, mb << 20)
        try:
            ctx.index(f, ctx.load_library(negative, 128, 360), top_n=5)
            lid = ctx.load_library(ts, 128, 360)
            return ctx, lid, ctx.index(f, lid, top_n=5)
        except tmgb.TmError as e:
            assert e.code == tmgb.TM_ERR_OOM
            torch.cuda.synchronize()
            ctx.close()
            return None

    lo, hi = 8, 1024
    while hi - lo > 1:
        mid = (lo + hi) // 2
        got = run(mid)
        lo, hi = (mid, hi) if got is None else (lo, mid)
        if got:
            torch.cuda.synchronize()
            got[0].close()
    ctx, lid, hits = run(hi)
    launches = ctx.last_stats["launches"]
    big = tmgb.Context(0)
    lib = big.load_library(ts, 128, 360)
    want = big.index(f, lib, top_n=5)
    assert torch.equal(hits, want)
    assert launches < big.last_stats["launches"]           # polar and sparse kernels alone
    out = torch.empty_like(want)
    refused = _enqueue_time(lambda: ctx.index(f, lid, top_n=5, out=out))
    normal = _enqueue_time(lambda: big.index(f, lib, top_n=5, out=out))
    assert refused < 3.0 * normal + 2e-4, (refused, normal)
    ctx.check()
    ctx.close()
    big.close()
