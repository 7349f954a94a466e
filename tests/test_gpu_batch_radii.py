"""The batched step at every patch radius (packed FMAs up to 4, scalar above)
on frames that are not square and on all frame types: bit for bit the
single-filter contexts' particles and ancestors, over two frames."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["F32", "BF16", "F16"])
@pytest.mark.parametrize("radius", range(9))
def test_batch_equals_single_filters(radius, dtype):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1310_5045_gb300 as ppf
    W, H, ns = 53, 38, [1, 33, 1025, 4100]
    ttype = {"F32": torch.float32, "BF16": torch.bfloat16, "F16": torch.float16}[dtype]
    movies = [synth.make_movie(W=W, H=H, K=2, seed=10 * radius + f).frames for f in range(len(ns))]
    frames = torch.from_numpy(np.stack(movies, axis=1)).cuda().to(ttype).contiguous()  # (K, F, H, W)
    models = [ppf.Model(width=W, height=H, patch_radius=radius, psf_sigma=1.0 + 0.25 * f, amplitude=40.0 + 5 * f,
                        background=10.0, sigma_xi=4.0, sigma_m=0.5, sigma_v=0.1, sigma_I=1.0, v0_max=1.0, seed=radius,
                        filter_id=f, frame_dtype=getattr(ppf, dtype)) for f in range(len(ns))]
    bank = ppf.BatchFilter(models, ns)
    singles = [ppf.ParticleFilter(models[f], ns[f], group_size=ns[f]) for f in range(len(ns))]
    for k in (1, 2):
        bank.step(frames[k - 1], k)
        state, _ = bank.get_particles()
        bank.resample(k)
        _, anc = bank.get_particles(state=False, anc=True)
        for f, pf in enumerate(singles):
            lo, hi = bank.offsets[f], bank.offsets[f + 1]
            pf.step(frames[k - 1, f].contiguous(), k)
            assert torch.equal(state[:, lo:hi], pf.get_particles()[0]), (k, f)
            pf.resample(ppf.SYSTEMATIC)
            assert torch.equal(anc[lo:hi] - int(lo), pf.get_particles(state=False, anc=True)[1]), (k, f)
    for pf in singles:
        pf.close()
    bank.close()
