"""tm_autotune times the sparse kernel, also for libraries whose calls go through the bounds."""
import pytest

from paper_2111_07347_gb300 import synth, tmgb

pytestmark = pytest.mark.gpu


def test_autotune_times_the_sparse_kernel(tmp_path, monkeypatch):
    """The recorded time is the sparse kernel's, at least 1.3 times that of the bounds and scores which
    serve the library's calls; a context without room for the sparse kernel's scratch records nothing."""
    import torch
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("TMGB_TUNE_CACHE", str(cache))
    ts = synth.kinematic_library("hcp", step_deg=0.5)
    scan = synth.render_scan(synth.make_rng(83), ts, 512, 256, 256, n_theta=360)
    f = torch.from_numpy(scan.frames).cuda().repeat(4, 1, 1)
    ctx = tmgb.Context(0)
    lid = ctx.load_library(ts, 128, 360)
    want = ctx.index(f, lid, top_n=5)
    ctx.profile_enable(True)
    for _ in range(3):
        ctx.index(f, lid, top_n=5)
    bounded = ctx.profile_read()["sparse"][0] / 3
    ctx.profile_enable(False)
    assert ctx.autotune(f, lid, top_n=5) in (128, 256, 512)
    ms = float(cache.read_text().split()[-1])
    assert ms > 1.3 * bounded, (ms, bounded)
    assert torch.equal(ctx.index(f, lid, top_n=5), want)
    ctx.check()
    ctx.close()
    cache.unlink()
    small = tmgb.Context(0, 64 << 20)
    lid = small.load_library(ts, 128, 360)
    with pytest.raises(tmgb.TmError) as e:
        small.autotune(f[:1], lid, top_n=5)
    assert e.value.code == tmgb.TM_ERR_OOM and not cache.exists()
    assert torch.equal(small.index(f[:1], lid, top_n=5), want[:, :1])
    small.check()
    small.close()
