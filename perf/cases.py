"""Performance cases of the indexing framework: the calls its users make, on synthetic scans.

Each case is one pass through the public entry points of ``paper_2111_07347_gb300.tmgb`` on
frames that are already in place (on the device, or in pinned host memory for the host-buffer
call).  Frames are rendered like the repository's synthetic scans (a library template rotated in
plane, a direct beam and a diffuse background under counting noise), the libraries are its
kinematic ones; sizes come from its workloads, tests and benchmark or are generic.

A program keeps a context with its template libraries loaded for as long as it indexes scans, so
contexts are kept between states; the frames of a state are its own.
"""
import functools
import math

import numpy as np
import torch

from paper_2111_07347_gb300 import synth, tmgb

DEV = torch.device("cuda", 0)
ELECTRONS = 2000


# ------------------------------------------------------------------------------- cases

def _case(kind, **kw):
    c = dict(kind=kind, phase="hcp", step=0.5, n=1024, H=256, W=256, dtype="u16", n_r=128, n_theta=360, dr=1.0,
             gamma=0.5, subtract=0.0, top_n=5, prefilter=1.0, rescore_k=64, unit=False, centres=False, refine=False,
             threshold=0.0)
    c.update(kw)
    return c


def listed():
    return [
        # one detector frame indexed as it arrives: launches and the latency of a single pattern
        _case("index", name="live_pattern", phase="fcc", n=1, prefilter=0.5),
        # one line of a scan from an on-line acquisition
        _case("index", name="scan_line", n=288),
        # the small workload: 16 x 16 scan of float frames, 300 random templates, 60 x 180 grid
        _case("index", name="tiny_scan", phase="random", n=256, H=128, W=128, dtype="f32", n_r=60, n_theta=180),
        # a large single-phase map against the full HCP library (the headline workload's shape)
        _case("index", name="hcp_map", n=32768),
        # a 128 x 128 scan with the radial pre-filter keeping half of the library
        _case("index", name="fcc_scan_prefilter", phase="fcc", n=16384, prefilter=0.5),
        # background-removed float frames with their own beam centres, refined angles, odd sizes
        _case("index", name="clean_frames", phase="fcc", n=1500, H=250, W=243, dtype="f32", n_r=120, centres=True,
              refine=True, threshold=0.4, top_n=3),
        # two-stage indexing: frame sums, matrix mask, masked frames against a unit-intensity library
        _case("two_stage", name="two_stage", n=8192, unit=True, subtract=0.4),
        # three phases of 24 to 244 spots a template through the tensor-core pre-score
        _case("index_bf16", name="three_phase_tensor", phase="multi", n=768),
        # every template's pre-score, as used to choose candidates
        _case("prescore", name="prescore_hcp", n=512),
        # the stage calls: polar transform, pre-filter, every survivor's best Q and shift
        _case("stages", name="stages_many_spots", phase="fcc+", n=200, prefilter=0.3),
        # preprocessing of raw frames: beam centres, difference of Gaussians and blur
        _case("preprocess", name="preprocess_scan", n=4096),
        # a scan in pinned host memory, results back in host memory
        _case("host", name="host_scan", n=8192),
    ]


def draw(rng):
    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    kind = rng.choice(["index", "index", "index", "index", "clean", "two_stage", "index_bf16", "prescore", "stages",
                       "preprocess", "host"])
    side = lambda: rng.choice([128, 144, 192, 200, 256, 256, 256, rng.randint(96, 256)])  # noqa: E731
    H, W = side(), side()
    n_theta = rng.choice([360, 360, 360, 180, 240, 300, 320, 336])
    n_r = rng.randint(max(40, min(H, W) // 2 - 20), min(128, min(H, W) // 2 + 8))
    step = rng.choice([0.5, 0.5, 0.75, 1.0])
    single = rng.choice(["fcc", "hcp", "hcp", "tetragonal"])
    if kind == "index":
        pre = rng.choice([1.0, 1.0, 1.0, round(rng.uniform(0.2, 0.8), 2)])
        return _case("index", phase=single, step=step, n=log_int(1, 16384), H=H, W=W, n_r=n_r, n_theta=n_theta,
                     prefilter=pre, top_n=rng.choice([1, 3, 5, 5, 10]), subtract=rng.choice([0.0, 0.0, 0.3]),
                     unit=rng.choice([False, False, True]), refine=rng.choice([False, False, True]),
                     gamma=rng.choice([0.5, 0.5, 1.0, 0.6]))
    if kind == "clean":
        return _case("index", phase=single, step=step, n=log_int(1, 2048), H=H, W=W, dtype="f32", n_r=n_r,
                     n_theta=n_theta, centres=True, refine=rng.choice([False, True]),
                     threshold=rng.choice([0.0, 0.4]), prefilter=rng.choice([1.0, 0.5]))
    if kind == "two_stage":
        return _case("two_stage", n=log_int(64, 8192), H=H, W=W, n_r=n_r, n_theta=n_theta, step=step, unit=True,
                     subtract=rng.choice([0.0, 0.4]))
    if kind == "index_bf16":
        return _case("index_bf16", phase=rng.choice(["multi", "hcp", "fcc+"]), n=log_int(4, 512), n_theta=n_theta,
                     rescore_k=rng.choice([64, 128]), prefilter=rng.choice([1.0, 1.0, 0.5]))
    if kind == "prescore":
        return _case("prescore", phase=rng.choice(["hcp", "fcc", "fcc+"]), step=step, n=log_int(4, 512), H=H, W=W,
                     n_r=n_r, n_theta=n_theta, prefilter=rng.choice([1.0, 0.5]))
    if kind == "stages":
        return _case("stages", phase=rng.choice(["fcc", "hcp", "fcc+"]), step=step, n=log_int(1, 200), H=H, W=W,
                     dtype=rng.choice(["u16", "f32"]), n_r=n_r, n_theta=n_theta,
                     prefilter=round(rng.uniform(0.1, 0.5), 2), gamma=rng.choice([0.5, 1.0, 0.4]),
                     subtract=rng.choice([0.0, 0.2]), centres=rng.choice([False, True]))
    if kind == "preprocess":
        return _case("preprocess", n=log_int(1, 4096), H=H, W=W, dtype=rng.choice(["u16", "u16", "f32"]))
    return _case("host", phase=single, step=step, n=log_int(256, 8192), H=H, W=W, n_r=n_r, n_theta=n_theta)


# ------------------------------------------------------------------------------- inputs

@functools.lru_cache(maxsize=16)
def _templates(phase, step):
    """The template sets of a phase: a kinematic library (fcc, hcp, tetragonal), the 300 random
    templates of the small workload, the many-spot settings ("fcc+"), or all three of those
    ("multi")."""
    if phase == "random":
        return (synth.random_templates(synth.make_rng(0), 300),)
    if phase == "multi":
        return tuple(synth.multiphase_libraries(step))
    if phase.endswith("+"):
        return (synth.kinematic_library(phase[:-1], step_deg=step, **synth.MULTIPHASE_KINEMATICS),)
    return (synth.kinematic_library(phase, step_deg=step),)


@functools.lru_cache(maxsize=3)
def _handle(phase, step, n_r, n_theta, dr, unit):
    """The context a program keeps, with the libraries of its phases loaded."""
    ctx = tmgb.Context(0)
    ids = [ctx.load_library(ts, n_r, n_theta, dr, unit_intensity=unit) for ts in _templates(phase, step)]
    return ctx, ids


def _render(gen, ts, n, H, W, electrons=ELECTRONS, shares=(0.4, 0.4, 0.2), fixed=None, centre=None):
    """int32 counts [n][H][W]: `electrons` per frame over template spots (sigma 1.5 px), direct
    beam (sigma 2 px) and an exponential background, each frame a random template and in-plane
    angle (or the `fixed` pair)."""
    f64 = dict(dtype=torch.float64, device=DEV)
    if ts.coords == "polar":
        sx, sy = ts.a * np.cos(ts.b), ts.a * np.sin(ts.b)
    else:
        sx, sy = ts.a * ts.px_per_unit, ts.b * ts.px_per_unit
    sx, sy = torch.tensor(sx, **f64), torch.tensor(sy, **f64)
    csum = torch.cat([torch.zeros(1, **f64), torch.tensor(ts.intensity, **f64).cumsum(0)])
    off = torch.tensor(np.asarray(ts.offsets), device=DEV)
    K0 = ts.n_templates
    out = torch.empty((n, H, W), dtype=torch.int32, device=DEV)
    rand = lambda *s: torch.rand(s, generator=gen, **f64)  # noqa: E731
    for c0 in range(0, n, 1024):
        m = min(1024, n - c0)
        if fixed is None:
            k = torch.randint(0, ts.n_expanded, (m, 1), generator=gen, device=DEV)
            phi = rand(m, 1) * (2 * math.pi)
        else:
            k = torch.full((m, 1), fixed[0], device=DEV, dtype=torch.int64)
            phi = torch.full((m, 1), fixed[1], **f64)
        b, flip = k % K0, torch.where(k >= K0, -1.0, 1.0)
        lo, hi = off[b], off[b + 1]
        part = rand(m, electrons)
        target = csum[lo] + rand(m, electrons) * (csum[hi] - csum[lo])
        i = torch.searchsorted(csum, target, right=True) - 1
        i = torch.minimum(torch.maximum(i, lo), (hi - 1).clamp_min(0)).clamp_max(max(0, sx.numel() - 1))
        px, py = sx[i], sy[i] * flip
        gx = torch.randn((m, electrons), generator=gen, **f64)
        gy = torch.randn((m, electrons), generator=gen, **f64)
        c, s = torch.cos(phi), torch.sin(phi)
        rho = -(W / 8.0) * (torch.log(1 - rand(m, electrons)) + torch.log(1 - rand(m, electrons)))
        ang = rand(m, electrons) * (2 * math.pi)
        spot, beam = part < shares[0], (part >= shares[0]) & (part < shares[0] + shares[1])
        x = torch.where(spot, c * px - s * py + 1.5 * gx, torch.where(beam, 2.0 * gx, rho * torch.cos(ang)))
        y = torch.where(spot, s * px + c * py + 1.5 * gy, torch.where(beam, 2.0 * gy, rho * torch.sin(ang)))
        ctr = torch.tensor([(W - 1) / 2.0, (H - 1) / 2.0], **f64) if centre is None else centre[c0:c0 + m].double()
        x, y = x + ctr[..., 0].reshape(-1, 1), y + ctr[..., 1].reshape(-1, 1)
        col, row = torch.floor(x + 0.5).long(), torch.floor(y + 0.5).long()
        ok = (col >= 0) & (col < W) & (row >= 0) & (row < H) & ~(spot & (hi <= lo))
        flat = (torch.arange(m, device=DEV).unsqueeze(1) * H + row) * W + col
        img = torch.zeros(m * H * W, dtype=torch.int32, device=DEV)
        img.scatter_add_(0, torch.where(ok, flat, 0).reshape(-1), ok.to(torch.int32).reshape(-1))
        out[c0:c0 + m] = img.view(m, H, W)
    return out


def _frames(case, seed):
    """The frames of a state, the beam centres they were drawn about (or None)."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    n, H, W = case["n"], case["H"], case["W"]
    sets = _templates(case["phase"], case["step"])
    if case["kind"] == "two_stage":
        # one matrix grain in every frame, a precipitate in half of them
        fcc = _templates("fcc", 0.5)[0]
        pick = np.random.default_rng(int(seed))
        img = _render(gen, fcc, n, H, W, shares=(0.5, 0.35, 0.15),
                      fixed=(int(pick.integers(0, fcc.n_expanded)), float(pick.uniform(0.0, 2.0 * math.pi))))
        add = _render(gen, sets[0], n, H, W, electrons=500, shares=(1.0, 0.0, 0.0))
        img += add * (torch.rand((n, 1, 1), generator=gen, device=DEV) < 0.5)
        return img.to(torch.uint16), None
    centre = None
    if case["centres"]:
        jitter = torch.rand((n, 2), generator=gen, device=DEV) * 4.0 - 2.0
        centre = (jitter + torch.tensor([(W - 1) / 2.0, (H - 1) / 2.0], device=DEV)).float().contiguous()
    if len(sets) == 1:
        img = _render(gen, sets[0], n, H, W, centre=centre)
    else:                                       # each frame shows one of the phases
        img = torch.empty((n, H, W), dtype=torch.int32, device=DEV)
        for i, ts in enumerate(sets):
            img[i::len(sets)] = _render(gen, ts, len(range(i, n, len(sets))), H, W)
    if case["dtype"] == "u16":
        return img.to(torch.uint16), centre
    f = img.float()
    if case["kind"] != "preprocess" and case["phase"] != "random":
        # smoothed, background-subtracted float frames (as preprocessing leaves them)
        f = torch.nn.functional.avg_pool2d(f.unsqueeze(1), 3, 1, 1, count_include_pad=False).squeeze(1)
        f = (f - f.mean(dim=(1, 2), keepdim=True)).clamp_min(0.0).contiguous()
    return f, centre


def prepare(case, seed):
    ctx, ids = _handle(case["phase"], case["step"], case["n_r"], case["n_theta"], case["dr"], case["unit"])
    frames, centres = _frames(case, seed)
    if case["kind"] == "host":
        frames = torch.empty(frames.shape, dtype=frames.dtype, pin_memory=True).copy_(frames)
        out = torch.empty((len(ids), case["n"], case["top_n"], 5), dtype=torch.int32, pin_memory=True)
        return dict(case=case, ctx=ctx, ids=ids, frames=frames, out=out)
    st = dict(case=case, ctx=ctx, ids=ids, frames=frames, centres=centres)
    if case["kind"] == "prescore":              # a pre-score is taken of polar images already made
        st["polar"] = ctx.polar_transform(frames, case["n_r"], case["n_theta"], case["dr"], gamma=case["gamma"])
    return st


# ------------------------------------------------------------------------------- one pass

def _fields(hits):
    """The columns of tm_hit rows, each as its own type (views of the result)."""
    return dict(template=hits[..., 0], shift=hits[..., 1], score=hits[..., 2].view(torch.float32),
                angle=hits[..., 3].view(torch.float32), mirror=hits[..., 4])


def run(state):
    c, ctx, ids, frames = state["case"], state["ctx"], state["ids"], state["frames"]
    kind = c["kind"]
    if kind in ("index", "index_bf16"):
        path = tmgb.TM_PATH_BF16_RESCORE if kind == "index_bf16" else tmgb.TM_PATH_FP32_SPARSE
        return _fields(ctx.index(frames, ids, top_n=c["top_n"], gamma=c["gamma"], subtract=c["subtract"],
                                 prefilter=c["prefilter"], path=path, rescore_k=c["rescore_k"],
                                 centres=state["centres"], threshold=c["threshold"], refine=c["refine"]))
    if kind == "two_stage":
        sums = ctx.frame_sum(frames)
        mask = ctx.matrix_mask(sums, c["n"], 0.3)
        out = _fields(ctx.index(frames, ids, top_n=c["top_n"], gamma=c["gamma"], subtract=c["subtract"], mask=mask))
        return dict(sums=sums, mask=mask, **out)
    if kind == "prescore":
        polar, norm, radial = state["polar"]
        return dict(score=ctx.prescore(ids[0], polar, norm, radial, c["prefilter"]))
    if kind == "stages":
        polar, norm, radial = ctx.polar_transform(frames, c["n_r"], c["n_theta"], c["dr"], gamma=c["gamma"],
                                                  subtract=c["subtract"], centres=state["centres"])
        mask, cosine = ctx.prefilter(ids[0], radial, c["prefilter"])
        q, s = ctx.correlate(ids[0], polar, norm, mask)
        return dict(polar=polar, norm=norm, radial=radial, cosine=cosine, mask=mask, q=q, shift=s)
    if kind == "preprocess":
        return dict(centres=ctx.find_centres(frames), clean=ctx.preprocess(frames, dog=(1.0, 4.0), blur=1.0))
    hits = ctx.index_host(frames, ids, top_n=c["top_n"], gamma=c["gamma"], subtract=c["subtract"], out=state["out"])
    return _fields(hits)


# ------------------------------------------------------------------------------- what a pass needs

def work(case):
    n, px, cells = case["n"], case["H"] * case["W"], case["n_r"] * case["n_theta"]
    sets = _templates(case["phase"], case["step"])
    K = [ts.n_expanded for ts in sets]
    spots = [int(ts.offsets[-1]) * (2 if ts.mirror else 1) for ts in sets]
    kind = case["kind"]
    frame = n * px * (2 if case["dtype"] == "u16" else 4)
    lib = sum(8 * s + 8 * k for s, k in zip(spots, K))
    hits = n * len(sets) * case["top_n"] * 20
    polar_flops = 9 * n * cells                     # one bilinear sample and its square per grid point
    if kind == "preprocess":                        # 9 + 33 taps along each axis, then 9 and 9
        return dict(bytes=frame + 4 * n * px + 8 * n, flops=2 * 102 * n * px)
    if kind == "prescore":                          # the rows the library has spots on
        radii = len(np.unique(np.floor(np.hypot(sets[0].a, sets[0].b) * sets[0].px_per_unit / case["dr"] + 0.5)))
        return dict(bytes=4 * n * min(radii, case["n_r"]) * case["n_theta"] + lib + 4 * n * K[0],
                    flops=2 * case["prefilter"] * n * case["n_theta"] * spots[0])
    if kind == "stages":
        return dict(bytes=frame + lib + n * (4 * cells + 4 * case["n_r"] + 4 + 12 * K[0] + K[0] // 8),
                    flops=polar_flops + 2 * n * case["prefilter"] * case["n_theta"] * spots[0])
    # the top N: the polar images, then at least the N returned templates at every shift
    least = sum(2 * n * case["top_n"] * case["n_theta"] * s // max(1, k) for s, k in zip(spots, K))
    if kind == "two_stage":
        return dict(bytes=2 * frame + 9 * px + lib + hits, flops=polar_flops + least + n * px)
    if kind == "index_bf16":                        # every template's correlation along the azimuth
        least = sum(2 * case["prefilter"] * n * case["n_theta"] * s for s in spots)
    return dict(bytes=frame + lib + hits, flops=polar_flops + least)


# ------------------------------------------------------------------------------- 64-bit values

def _polar64(case, frames, centres):
    """The polar images in float64, [n][n_r][n_theta]."""
    n, H, W = frames.shape
    f64 = dict(dtype=torch.float64, device=DEV)
    if frames.dtype == torch.uint16:
        v = frames.to(torch.int32).double()
    else:
        v = frames.double()
    if case["threshold"] > 0.0:
        v = torch.where(v < case["threshold"], 0.0, v)
    v = v.clamp_min(0.0) ** case["gamma"] - case["subtract"]
    r = torch.arange(case["n_r"], **f64) * case["dr"]
    th = torch.arange(case["n_theta"], **f64) * (2.0 * math.pi / case["n_theta"])
    dx, dy = r[:, None] * torch.cos(th), r[:, None] * torch.sin(th)
    out = torch.empty((n, case["n_r"], case["n_theta"]), **f64)
    for c0 in range(0, n, 256):
        m = min(256, n - c0)
        if centres is None:
            cx = torch.full((m, 1, 1), (W - 1) / 2.0, **f64)
            cy = torch.full((m, 1, 1), (H - 1) / 2.0, **f64)
        else:
            cx = centres[c0:c0 + m, 0].double().view(-1, 1, 1)
            cy = centres[c0:c0 + m, 1].double().view(-1, 1, 1)
        x, y = cx + dx, cy + dy
        x0, y0 = torch.floor(x), torch.floor(y)
        fx, fy = x - x0, y - y0
        acc = torch.zeros((m, case["n_r"], case["n_theta"]), **f64)
        img = v[c0:c0 + m].reshape(m, H * W)
        for ax, ay in ((0, 0), (1, 0), (0, 1), (1, 1)):
            xi, yi = (x0 + ax).long(), (y0 + ay).long()
            ok = (xi >= 0) & (xi < W) & (yi >= 0) & (yi < H)
            idx = torch.where(ok, yi * W + xi, 0).expand(m, -1, -1).reshape(m, -1)
            tap = torch.where(ok.expand(m, -1, -1), img.gather(1, idx).view(acc.shape), 0.0)
            acc += (fx if ax else 1 - fx) * (fy if ay else 1 - fy) * tap
        out[c0:c0 + m] = acc
    return out


def _images64(case, ts):
    """The rounded templates: the distinct radii, and per spot its template (mirror copies at
    k + K0), its position radius-row * n_theta + angle column, and its intensity."""
    nt = case["n_theta"]
    k = np.repeat(np.arange(ts.n_templates), np.diff(ts.offsets))
    if ts.coords == "polar":
        r, th = ts.a, ts.b
    else:
        x, y = ts.a * ts.px_per_unit, ts.b * ts.px_per_unit
        r, th = np.hypot(x, y), np.arctan2(y, x)
    inten = np.ones_like(ts.intensity) if case["unit"] else ts.intensity
    if ts.mirror:
        k, r = np.concatenate([k, k + ts.n_templates]), np.concatenate([r, r])
        th, inten = np.concatenate([th, -th]), np.concatenate([inten, inten])
    ri = np.floor(r / case["dr"] + 0.5).astype(np.int64)
    t = np.fmod(th, 2.0 * math.pi)
    t = np.where(t < 0.0, t + 2.0 * math.pi, t)
    ti = np.floor(t / (2.0 * math.pi / nt) + 0.5).astype(np.int64) % nt
    ok = ri < case["n_r"]
    k, ri, ti, inten = k[ok], ri[ok], ti[ok], inten[ok]
    radii, a = np.unique(ri, return_inverse=True)
    return radii, k, a * nt + ti, inten


def _best64(case, ts, polar):
    """Q of Eq. 1 in float64 at each template's best shift: [n][K]."""
    nt, n = case["n_theta"], polar.shape[0]
    radii, k, pos, inten = _images64(case, ts)
    K, R = ts.n_expanded, len(radii)
    norm = polar.square().sum(dim=(1, 2)).sqrt()
    ph = torch.fft.rfft(polar[:, torch.as_tensor(radii, device=DEV)], dim=2)              # [n][R][M]
    ph = ph / torch.where(norm > 0, norm, 1.0).view(-1, 1, 1)
    q = torch.empty((n, K), dtype=torch.float64, device=DEV)
    for k0 in range(0, K, 512):
        k1 = min(K, k0 + 512)
        sel = (k >= k0) & (k < k1)
        t = torch.zeros((k1 - k0, R * nt), dtype=torch.float64, device=DEV)
        t.index_put_((torch.as_tensor(k[sel] - k0, device=DEV), torch.as_tensor(pos[sel], device=DEV)),
                     torch.as_tensor(inten[sel], device=DEV), accumulate=True)
        tn = t.square().sum(dim=1).sqrt()
        th = torch.fft.rfft((t / torch.where(tn > 0, tn, 1.0)[:, None]).view(k1 - k0, R, nt), dim=2).conj()
        for p0 in range(0, n, 64):
            g = torch.einsum("krm,nrm->nkm", th, ph[p0:p0 + 64])
            best = torch.fft.irfft(g, n=nt, dim=2).amax(dim=2)
            q[p0:p0 + 64, k0:k1] = torch.where((norm[p0:p0 + 64, None] > 0) & (tn > 0), best, 0.0)
    return q


def _cosine64(case, ts, radial):
    """The pre-filter's scores in float64: [n][K]."""
    radii, k, pos, inten = _images64(case, ts)
    prof = torch.zeros((ts.n_expanded, case["n_r"]), dtype=torch.float64, device=DEV)
    prof.index_put_((torch.as_tensor(k, device=DEV), torch.as_tensor(radii[pos // case["n_theta"]], device=DEV)),
                    torch.as_tensor(inten, device=DEV), accumulate=True)
    d = radial.norm(dim=1)[:, None] * prof.norm(dim=1)[None]
    return torch.where(d > 0, radial @ prof.T / torch.where(d > 0, d, 1.0), 0.0)


def _gauss64(x, sigma, dim):
    r = int(math.floor(4.0 * sigma + 0.5))
    w = [math.exp(-0.5 * (i / sigma) ** 2) for i in range(-r, r + 1)]
    idx = torch.arange(x.shape[dim], device=DEV)
    acc = torch.zeros_like(x)
    for i, v in enumerate(w):
        acc += (v / sum(w)) * x.index_select(dim, (idx + i - r).clamp(0, x.shape[dim] - 1))
    return acc


def exact(case, seed):
    kind = case["kind"]
    n = case["n"]
    sets = _templates(case["phase"], case["step"])
    pairs = n * sum(ts.n_expanded for ts in sets)
    if kind == "preprocess":
        frames, _ = _frames(case, seed)
        out = torch.empty(frames.shape, dtype=torch.float64, device=DEV)
        for c0 in range(0, n, 256):
            f = frames[c0:c0 + 256]
            x = f.to(torch.int32).double() if f.dtype == torch.uint16 else f.double()
            d = (_gauss64(_gauss64(x, 1.0, 2), 1.0, 1) - _gauss64(_gauss64(x, 4.0, 2), 4.0, 1)).clamp_min(0.0)
            out[c0:c0 + 256] = _gauss64(_gauss64(d, 1.0, 2), 1.0, 1)
        return dict(centres=None, clean=out)
    if kind == "two_stage":
        frames, _ = _frames(case, seed)
        sums = torch.zeros(frames.shape[1:], dtype=torch.float64, device=DEV)
        for c0 in range(0, n, 256):
            sums += frames[c0:c0 + 256].to(torch.int32).sum(dim=0)
        return dict(sums=sums, mask=None, template=None, shift=None, score=None, angle=None, mirror=None)
    if pairs > 12_000_000:
        return None
    frames, centres = _frames(case, seed)
    if kind == "stages":
        polar = _polar64(case, frames, centres)
        radial = polar.sum(dim=2)
        return dict(polar=polar, norm=polar.square().sum(dim=(1, 2)).sqrt(), radial=radial,
                    cosine=_cosine64(case, sets[0], radial), mask=None, q=None, shift=None)
    if kind == "index_bf16" or (kind == "prescore" and case["prefilter"] < 1.0):
        return None
    polar = _polar64(case, frames, centres)
    if kind == "prescore":
        return dict(score=_best64(case, sets[0], polar))
    score = []
    for ts in sets:
        q = _best64(case, ts, polar)
        if case["prefilter"] < 1.0:
            kept = _cosine64(case, ts, polar.sum(dim=2)).topk(math.ceil(case["prefilter"] * ts.n_expanded), dim=1)
            q = torch.full_like(q, -math.inf).scatter(1, kept.indices, q.gather(1, kept.indices))
        score.append(q.topk(case["top_n"], dim=1).values)
    score = torch.stack(score)
    return dict(template=None, shift=None, score=score, angle=None, mirror=None)
