"""The workloads this library is timed on, through its public entry points.

Every case is one call pattern of a user's program:

  track    a queued stretch of a movie: per frame step, resample and an asynchronous estimate, then one
           read-out of the particles (the checkpoint a long run writes now and then).  The filter is already
           locked on its spot, and the next pass goes on where the last one stopped.
  live     one camera frame, closed loop: the frame comes from page-locked host memory and the caller waits for
           the estimate before the next one (the smallest call: latency and launches).
  restart  particles of unknown spread are set (a checkpoint, a lost object searched again over the whole
           frame) and stepped once, then read back.
  grad     the log marginal likelihood of a movie and its gradient, from a fresh prior draw.
  batch    a bank of independent filters of uneven sizes over a few frames, with every estimate.
  noalloc  the allocation-free systematic draw on log-weights the caller holds.

The movies are seeded Poisson counts of one Gaussian spot on a background of 10 counts.  The spot goes round a
small closed loop, so that a filter can follow it for as many passes as are asked for.
"""
import math

import numpy as np
import torch

import paper_1310_5045_gb300 as ppf
from paper_1310_5045_gb300._binding import systematic_resample_noalloc

BACKGROUND = 10.0
SIGMA_XI = math.sqrt(10.0)
LOOP = 32          # frames of a tracking movie, one turn of its loop
WARM_FRAMES = 4    # frames a tracking filter has seen before its first pass: it is locked on the spot
DTYPES = {"f32": (ppf.F32, torch.float32), "bf16": (ppf.BF16, torch.bfloat16), "f16": (ppf.F16, torch.float16)}
MOST_STEPS = 38_000_000 * 8  # particle steps of the largest listed case at an 11 x 11 patch


def listed():
    return [
        # closed-loop tracking of one spot in a small camera window, frame by frame
        {"name": "live_128_16k", "kind": "live", "n": 16384, "width": 128, "height": 128, "radius": 4, "sigma": 1.5,
         "snr": 6.0, "dtype": "f32", "scheme": "systematic", "group": 2048},
        # the 20-frame 128 x 128 movie in one go, the paper's distributed resampling with sorted greedy routing
        {"name": "movie_128_16k_rpa_sgs", "kind": "track", "n": 16384, "width": 128, "height": 128, "radius": 4,
         "sigma": 1.5, "snr": 6.0, "dtype": "f32", "scheme": "rpa_sgs", "alpha": 0.0, "group": 2048, "ess": 0.0,
         "cell": False, "frames": 20},
        # an ordinary single-spot run on an odd camera crop: ragged particle count, half-precision frames,
        # resampling only while N_eff is below half the particles
        {"name": "track_crop_1m_ess", "kind": "track", "n": 1_000_003, "width": 515, "height": 387, "radius": 5,
         "sigma": 1.6, "snr": 5.0, "dtype": "f16", "scheme": "systematic", "alpha": 0.0, "group": 4096, "ess": 0.5,
         "cell": False, "frames": 8},
        # the paper-scale run: 38 million particles on 512 x 512 frames, systematic resampling every frame
        {"name": "track_512_38m", "kind": "track", "n": 38_000_000, "width": 512, "height": 512, "radius": 5,
         "sigma": 1.6, "snr": 5.0, "dtype": "f32", "scheme": "systematic", "alpha": 0.0, "group": 4096, "ess": 0.0,
         "cell": False, "frames": 8},
        # proportional allocation with sorted greedy routing at a node's share of the particles, bfloat16 frames
        {"name": "track_512_8m_rpa_sgs", "kind": "track", "n": 8_000_000, "width": 512, "height": 512, "radius": 5,
         "sigma": 1.6, "snr": 5.0, "dtype": "bf16", "scheme": "rpa_sgs", "alpha": 0.0, "group": 4096, "ess": 0.0,
         "cell": False, "frames": 8},
        # local resampling with ring exchange, particles and groups of odd sizes
        {"name": "track_512_3m_rna", "kind": "track", "n": 3_141_593, "width": 512, "height": 512, "radius": 5,
         "sigma": 1.4, "snr": 5.0, "dtype": "f32", "scheme": "rna", "alpha": 0.1, "group": 4001, "ess": 0.0,
         "cell": False, "frames": 8},
        # adaptive ring exchange on a dim spot, small patches
        {"name": "track_256_2m_arna", "kind": "track", "n": 1 << 21, "width": 256, "height": 256, "radius": 4,
         "sigma": 1.5, "snr": 3.0, "dtype": "f32", "scheme": "arna", "alpha": 0.5, "group": 4096, "ess": 0.0,
         "cell": False, "frames": 8},
        # the piecewise constant likelihood (pcSIR)
        {"name": "track_512_8m_cell", "kind": "track", "n": 8_000_000, "width": 512, "height": 512, "radius": 5,
         "sigma": 1.6, "snr": 5.0, "dtype": "f32", "scheme": "systematic", "alpha": 0.0, "group": 4096, "ess": 0.0,
         "cell": True, "frames": 8},
        # a search over the whole frame: particles spread everywhere
        {"name": "restart_512_4m", "kind": "restart", "n": 4_000_000, "width": 512, "height": 512, "radius": 5,
         "sigma": 1.6, "snr": 5.0, "dtype": "f32", "group": 4096},
        # fitting the model's parameters: 50 frames of 256 x 256, 2^20 particles
        {"name": "grad_256_1m_k50", "kind": "grad", "n": 1 << 20, "width": 256, "height": 256, "radius": 4,
         "sigma": 1.5, "snr": 6.0, "dtype": "f32", "frames": 50},
        # many spots at once: a bank of filters with 256 to 65536 particles each on 64 x 64 windows
        {"name": "batch_1024_64", "kind": "batch", "filters": 1024, "width": 64, "height": 64, "radius": 5,
         "dtype": "f32", "ess": 0.0, "frames": 8},
        # the draw alone inside a host program that plans all device memory itself
        {"name": "noalloc_16m", "kind": "noalloc", "n": 1 << 24, "spread": 4.0},
    ]


def _between(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["track"] * 8 + ["live", "restart", "grad", "batch", "batch", "noalloc"])
    if kind == "noalloc":
        return {"kind": kind, "n": _between(rng, 1000, 1 << 24), "spread": round(rng.uniform(0.5, 12.0), 3)}
    if kind == "batch":
        return {"kind": kind, "filters": _between(rng, 4, 1536), "width": rng.randint(40, 80),
                "height": rng.randint(40, 80), "radius": rng.randint(2, 5), "dtype": rng.choice(list(DTYPES)),
                "ess": rng.choice([0.0, 0.0, 0.5]), "frames": rng.randint(2, 8)}
    c = {"kind": kind, "width": rng.randint(64, 700), "height": rng.randint(64, 700), "radius": rng.randint(2, 7),
         "sigma": round(rng.uniform(1.0, 2.0), 3), "snr": round(rng.uniform(2.0, 8.0), 3),
         "dtype": rng.choice(["f32", "f32", "bf16", "f16"])}
    pixels = (2 * c["radius"] + 1) ** 2
    if kind == "grad":
        c["frames"] = rng.randint(4, 50)
        c["n"] = _between(rng, 4096, 1 << 21)
        return c
    c["scheme"] = rng.choice(["systematic"] * 4 + ["rpa_gs", "rpa_sgs", "rpa_lgs", "rpa2_gs", "rpa2_sgs", "rpa2_lgs",
                                                   "rna", "rna", "arna"])
    if kind == "live":
        c["n"] = _between(rng, 1000, 500_000)
        c["group"] = min(c["n"], rng.choice([512, 2048, 4096]))
        return c
    if kind == "restart":
        del c["scheme"]
        c["n"] = _between(rng, 50_000, 8_000_000)
        c["group"] = 4096
        return c
    c["frames"] = rng.randint(4, 8)
    c["n"] = _between(rng, 2000, min(38_000_000, int(MOST_STEPS * 121 / max(121, pixels) / c["frames"])))
    # at most 16384 groups; odd group sizes too
    c["group"] = max(min(c["n"], rng.choice([1000, 2048, 4096, 4096, 8191])), -(-c["n"] // 16000))
    c["alpha"] = rng.choice([0.05, 0.1, 0.5]) if c["scheme"] in ("rna", "arna") else 0.0
    c["ess"] = rng.choice([0.0, 0.0, 0.5])
    c["cell"] = rng.random() < 0.15
    return c


# ------------------------------------------------------------------ inputs
def _amplitude(snr):
    """The peak count with I0 / sqrt(I0 + background) = snr."""
    return 0.5 * (snr * snr + math.sqrt(snr ** 4 + 4.0 * snr * snr * BACKGROUND))


def _loop_movie(gen, frames, width, height, sigma, amp, radius, dtype):
    """`frames` frames of a spot that goes once round a circle of `radius` pixels."""
    at = torch.rand(3, generator=gen, device="cuda", dtype=torch.float64).tolist()
    cx, cy = (0.35 + 0.3 * at[0]) * (width - 1), (0.35 + 0.3 * at[1]) * (height - 1)
    phase = 2.0 * math.pi * (at[2] + torch.arange(frames, device="cuda", dtype=torch.float64) / frames)
    x, y = cx + radius * torch.cos(phase), cy + radius * torch.sin(phase)
    return _poisson(gen, x, y, torch.full_like(x, sigma), torch.full_like(x, amp), width, height, dtype)


def _poisson(gen, x, y, sigma, amp, width, height, dtype):
    px = torch.arange(width, device="cuda", dtype=torch.float64)
    py = torch.arange(height, device="cuda", dtype=torch.float64)
    gx = torch.exp(-((px - x[:, None]) ** 2) / (2 * sigma * sigma)[:, None])
    gy = torch.exp(-((py - y[:, None]) ** 2) / (2 * sigma * sigma)[:, None])
    rate = BACKGROUND + amp[:, None, None] * gy[:, :, None] * gx[:, None, :]
    return torch.poisson(rate.float(), generator=gen).to(dtype).contiguous()


def _model(case, seed, **kw):
    return ppf.Model(width=case["width"], height=case["height"], patch_radius=case["radius"],
                     psf_sigma=case["sigma"], amplitude=_amplitude(case["snr"]), background=BACKGROUND,
                     sigma_xi=SIGMA_XI, sigma_m=0.5, sigma_v=0.1, sigma_I=1.0, v0_max=1.0, seed=seed, filter_id=0,
                     frame_dtype=DTYPES[case["dtype"]][0], **kw)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind == "noalloc":
        # log-weights of a tracking step: the chi-square like tail of a Gaussian posterior
        z = torch.randn(2, case["n"], generator=gen, device="cuda")
        lw = (-0.5 * case["spread"] * (z[0] * z[0] + z[1] * z[1])).contiguous()
        return {"kind": kind, "lw": lw, "seed": seed, "out": torch.empty(case["n"], dtype=torch.int32, device="cuda")}
    if kind == "batch":
        return _prepare_batch(case, seed, gen)
    dtype = DTYPES[case["dtype"]][1]
    amp = _amplitude(case["snr"])
    if kind == "grad":
        frames = _loop_movie(gen, case["frames"], case["width"], case["height"], case["sigma"], amp, 4.0, dtype)
        pf = ppf.ParticleFilter(_model(case, seed), case["n"], group_size=min(4096, case["n"]))
        return {"kind": kind, "pf": pf, "frames": frames}
    frames = _loop_movie(gen, LOOP, case["width"], case["height"], case["sigma"], amp, 4.0, dtype)
    if kind == "restart":
        particles = _spread_particles(case, gen)
        pf = ppf.ParticleFilter(_model(case, seed), case["n"], group_size=case["group"])
        return {"kind": kind, "pf": pf, "frames": frames, "particles": particles, "k": 0}
    pf = ppf.ParticleFilter(_model(case, seed, likelihood=1 if case.get("cell") else 0), case["n"],
                            group_size=case["group"])
    s = {"kind": kind, "pf": pf, "frames": frames, "scheme": ppf.SCHEMES[case["scheme"]],
         "alpha": case.get("alpha") or 0.1, "ess": case["ess"] * case["n"] if case.get("ess") else None, "k": 0}
    for _ in range(WARM_FRAMES):  # the filter finds its spot
        _frame(s)
    if kind == "live":
        s["host"] = [f.cpu().pin_memory() for f in frames]
    else:
        s["count"] = case["frames"]
        s["lw_prev"] = case["scheme"] in ("rna", "arna")
        s["slots"] = [torch.empty(ppf.Estimate.nbytes(), dtype=torch.uint8, pin_memory=True)
                      for _ in range(case["frames"])]
    torch.cuda.synchronize()
    return s


def _spread_particles(case, gen):
    """Particles over the whole frame, as a search for a lost spot starts."""
    u = torch.rand(5, case["n"], generator=gen, device="cuda")
    p = torch.zeros(6, case["n"], device="cuda")
    p[0] = u[0] * case["width"] - 0.5
    p[1] = u[1] * case["height"] - 0.5
    p[2] = 2.0 * u[2] - 1.0
    p[3] = 2.0 * u[3] - 1.0
    p[4] = _amplitude(case["snr"]) * (0.5 + u[4])
    return p


def _batch_plan(case, seed):
    """Per filter: spot width and amplitude (of the seed) and particle count (256 to 65536, log-uniform; the bank's
    own, whatever the seed)."""
    F = case["filters"]
    n = np.floor(np.exp(np.random.default_rng(F).uniform(math.log(256), math.log(65536), F))).astype(np.int64)
    rng = np.random.default_rng(seed)
    sigma = rng.uniform(1.0, 2.0, F)
    amp = np.array([_amplitude(v) for v in rng.uniform(2.0, 8.0, F)])
    return sigma, amp, n


def _prepare_batch(case, seed, gen):
    sigma, amp, n = _batch_plan(case, seed)
    F, K, W, H = case["filters"], case["frames"], case["width"], case["height"]
    code, dtype = DTYPES[case["dtype"]]
    models = [ppf.Model(width=W, height=H, patch_radius=case["radius"], psf_sigma=float(sigma[f]),
                        amplitude=float(amp[f]), background=BACKGROUND, sigma_xi=SIGMA_XI, sigma_m=0.5, sigma_v=0.1,
                        sigma_I=1.0, v0_max=1.0, seed=seed, filter_id=f, frame_dtype=code) for f in range(F)]
    at = torch.rand(3, F, generator=gen, device="cuda", dtype=torch.float64)
    s, a = torch.from_numpy(sigma).cuda(), torch.from_numpy(amp).cuda()
    frames = torch.empty((K, F, H, W), dtype=dtype, device="cuda")
    for k in range(K):  # slow spots: each goes round a circle of 0.75 pixels in K frames
        phase = 2.0 * math.pi * (at[2] + k / K)
        x = (0.35 + 0.3 * at[0]) * (W - 1) + 0.75 * torch.cos(phase)
        y = (0.35 + 0.3 * at[1]) * (H - 1) + 0.75 * torch.sin(phase)
        frames[k] = _poisson(gen, x, y, s, a, W, H, dtype)
    bank = ppf.BatchFilter(models, n)
    if case["ess"]:
        bank.set_ess_threshold(case["ess"])
    bank.run(frames, k0=1)  # the filters find their spots
    torch.cuda.synchronize()
    return {"kind": "batch", "bank": bank, "frames": frames, "k": K}


# --------------------------------------------------------------------- run
def _frame(s, slot=None):
    """The calls of one frame of a tracking loop."""
    s["k"] += 1
    pf = s["pf"]
    pf.step(s["frames"][(s["k"] - 1) % LOOP], s["k"])
    pf.resample(s["scheme"], s["alpha"], s["ess"])
    if slot is not None:
        pf.estimate_async(slot)


def _numbers(e):
    """A frame's estimate: its float64 values, and its counts."""
    return (np.array([*e.mean, e.log_evidence, e.ess, e.max_log_weight]),
            np.array([e.frame, e.status_flags, e.links, e.moved, e.max_group, e.min_group]))


def run(state):
    s, kind = state, state["kind"]
    if kind == "noalloc":
        return systematic_resample_noalloc(s["lw"], s["seed"], 0, 1, out=s["out"])
    if kind == "grad":
        value, gradient = s["pf"].loglik_grad(s["frames"])
        return {"loglik": value, "grad": gradient}
    if kind == "batch":
        est = s["bank"].run(s["frames"], k0=s["k"] + 1)
        s["k"] += int(s["frames"].shape[0])
        particles, ancestors = s["bank"].get_particles(state=True, anc=True)
        return {"estimates": {name: est[name] for name in est.dtype.names}, "particles": particles,
                "ancestors": ancestors}
    if kind == "live":
        s["k"] += 1
        pf = s["pf"]
        pf.step_host(s["host"][(s["k"] - 1) % LOOP], s["k"])
        pf.resample(s["scheme"], s["alpha"], s["ess"])
        return _numbers(pf.estimate())
    if kind == "restart":
        s["k"] += 1
        pf = s["pf"]
        pf.set_particles(s["particles"])
        pf.step(s["frames"][(s["k"] - 1) % LOOP], s["k"])
        est = pf.estimate()
        particles, _, _ = pf.get_particles()
        return [*_numbers(est), particles]
    for j in range(s["count"]):
        _frame(s, s["slots"][j])
    particles, ancestors, lw_prev = s["pf"].get_particles(state=True, anc=True, lw_prev=s["lw_prev"])
    est = [_numbers(ppf.Estimate.from_buffer(b)) for b in s["slots"]]  # get_particles has waited for the stream
    return {"estimates": np.stack([e[0] for e in est]), "counts": np.stack([e[1] for e in est]),
            "particles": particles, "ancestors": ancestors, "lw_prev": lw_prev}


def work(case):
    """Bytes and operations of one pass.  A particle's step reads its ancestor and the parent's five values and
    writes six; a draw reads its log-weight and writes an ancestor.  Operations: the separable patch sums of eq. 4
    (an FMA counts two), the squared sums, the propagation."""
    kind = case["kind"]
    if kind == "noalloc":
        return {"bytes": 8.0 * case["n"], "flops": 0.0}
    p = 2 * case["radius"] + 1
    flops = 2.0 * p * p + 6 * p + 16
    pixel = 4 if case["dtype"] == "f32" else 2
    frame = float(case["width"] * case["height"] * pixel)
    if kind == "batch":
        steps = float(_batch_plan(case, 0)[2].sum()) * case["frames"]
        return {"bytes": 56.0 * steps + case["filters"] * case["frames"] * frame + 56.0 * steps / case["frames"],
                "flops": flops * steps}
    n, k = float(case["n"]), case.get("frames", 1)
    if kind == "grad":  # the tangents too: two values read and written; twelve patch sums for the derivatives
        return {"bytes": (56.0 + 16.0) * n * k + k * frame, "flops": (3 * 2.0 * p * p + 30 * p) * n * k}
    if kind == "restart":  # the given particles are read, the stepped ones written
        return {"bytes": 48.0 * n + frame, "flops": flops * n}
    if kind == "live":
        return {"bytes": 56.0 * n + frame, "flops": flops * n}
    if case["cell"]:
        flops = 24.0
    # the read-out writes the particles and their ancestors once more
    return {"bytes": 56.0 * n * k + k * frame + 56.0 * n, "flops": flops * n * k}


# ------------------------------------------------------------------- exact
def _philox(index, frame, purpose, seed):
    """Philox4x32-10 blocks of the counters (index, frame, 0, purpose << 8) as four int64 tensors of 32-bit words."""
    m = 0xFFFFFFFF

    def mulhilo(const, v):  # 32 x 32 -> 64 bits in two int64 halves
        lo16, hi16 = v & 0xFFFF, v >> 16
        low = lo16 * const
        mid = hi16 * const + (low >> 16)
        return mid >> 16, ((mid & 0xFFFF) << 16) | (low & 0xFFFF)

    c = [index, torch.full_like(index, frame), torch.zeros_like(index), torch.full_like(index, purpose << 8)]
    k0, k1 = seed & m, (seed >> 32) & m
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
        hi0, lo0 = mulhilo(0xD2511F53, c[0])
        hi1, lo1 = mulhilo(0xCD9E8D57, c[2])
        c = [hi1 ^ c[1] ^ k0, lo1, hi0 ^ c[3] ^ k1, lo0]
    return c


def _normals(index, frame, seed):
    """The six propagation normals of every slot: 21-bit fields of one Philox block, Box-Muller in 64 bits."""
    r = _philox(index, frame, 1, seed)
    word = lambda bit: (r[bit // 32] >> (bit % 32)) | ((r[bit // 32 + 1] << (32 - bit % 32)) if bit < 96 else 0)  # noqa: E731
    u = [(2.0 * (word(21 * j) & 0x1FFFFF).double() + 1.0) * 2.0 ** -22 for j in range(6)]
    out = []
    for j in range(0, 6, 2):
        rho, theta = torch.sqrt(-2.0 * torch.log(u[j])), 2.0 * math.pi * u[j + 1]
        out += [rho * torch.cos(theta), rho * torch.sin(theta)]
    return out


def _f32(v):
    """A model parameter as the library holds it."""
    return float(np.float32(v))


def exact(case, seed):
    """The restarted step in 64 bits; the other cases draw ancestors from float32 weights, frame after frame, and
    have no value that plain arithmetic could give."""
    if case["kind"] != "restart":
        return None
    gen = torch.Generator(device="cuda").manual_seed(seed)
    amp = _amplitude(case["snr"])
    W, H, R, n = case["width"], case["height"], case["radius"], case["n"]
    frames = _loop_movie(gen, LOOP, W, H, case["sigma"], amp, 4.0, DTYPES[case["dtype"]][1])
    prior = _spread_particles(case, gen)
    z = frames[0].double() - BACKGROUND
    pad = 2 * R
    zp = torch.nn.functional.pad(z, (pad, pad, pad, pad))
    inv2s2 = 1.0 / (2.0 * _f32(case["sigma"]) ** 2)
    inv_sxi2 = 1.0 / _f32(SIGMA_XI) ** 2
    out = torch.empty(6, n, dtype=torch.float64, device="cuda")
    off = torch.arange(-R, R + 1, device="cuda")
    for lo in range(0, n, 1 << 18):
        hi = min(n, lo + (1 << 18))
        e = _normals(torch.arange(lo, hi, device="cuda", dtype=torch.int64), 1, seed)
        x, y, vx, vy, I0, _ = prior[:, lo:hi].double()
        x, y = x + vx + _f32(0.5) * e[0], y + vy + _f32(0.5) * e[1]
        vx, vy, I0 = vx + _f32(0.1) * e[2], vy + _f32(0.1) * e[3], I0 + e[4]
        cx, cy = torch.floor(x + 0.5).long(), torch.floor(y + 0.5).long()
        seen = (cx >= -R) & (cx <= W - 1 + R) & (cy >= -R) & (cy <= H - 1 + R)
        cxs, cys = torch.where(seen, cx, 0), torch.where(seen, cy, 0)
        px, py = cxs[:, None] + off, cys[:, None] + off
        gx = torch.exp(-inv2s2 * (px - x[:, None]) ** 2) * ((px >= 0) & (px < W))
        gy = torch.exp(-inv2s2 * (py - y[:, None]) ** 2) * ((py >= 0) & (py < H))
        patch = zp[(py + pad)[:, :, None], (px + pad)[:, None, :]]
        b = torch.einsum("nj,nji,ni->n", gy, patch, gx)
        c = (gx * gx).sum(1) * (gy * gy).sum(1)
        ll = I0 * (b - 0.5 * I0 * c) * inv_sxi2
        out[:, lo:hi] = torch.stack([x, y, vx, vy, I0, torch.where(seen, ll, 0.0)])
    lw = out[5]
    top = lw.max()
    w = torch.exp(lw - top)
    total = w.sum()
    mean = (out[:5] * w).sum(1) / total
    log_total = top + torch.log(total)
    est = torch.cat([mean, torch.stack([log_total - math.log(n), total * total / (w * w).sum(), top])])
    return [est.cpu().numpy(), None, out]
