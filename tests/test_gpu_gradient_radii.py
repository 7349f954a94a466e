"""The gradient kernel at the patch radii the other gradient tests leave out:
the smallest, the two-block ones around them and those above 6, which run one
block per SM.  Against the FP64 oracle's reverse mode on the replayed path, with
the tolerances of tests/test_gpu_gradient.py (L 1e-5 relative, each derivative
1e-4 relative plus 1e-5 of the largest), on a frame that is not square and a
particle count that is no multiple of a block."""
import numpy as np
import pytest

import oracle as orc
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius", [0, 1, 3, 5, 6, 7, 8])
def test_gradient_matches_oracle_at_every_register_split(radius):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1310_5045_gb300 as ppf
    from gpu_common import paired_models
    mv = synth.make_movie(W=61, H=48, K=4, sigma=1.5, amplitude=30.0, background=10.0, seed=radius,
                          start_frac=(0.4, 0.6))
    gm, om = paired_models(ppf, width=61, height=48, patch_radius=radius, psf_sigma=1.5, amplitude=30.0,
                           background=10.0, sigma_m=0.5, sigma_I=0.0, seed=radius)
    N = 3001
    pf = ppf.ParticleFilter(gm, N, group_size=1000)
    theta = np.array([1.5, 30.0, 10.0, 0.5], dtype=np.float32).astype(np.float64)
    L, g, anc, anchors = pf.loglik_grad(torch.from_numpy(mv.frames).cuda(), theta, return_path=True)
    pf.close()
    rc, Lo, go, _, _ = orc.grad_run(om, N, mv.frames, theta, anc.cpu().numpy(), anchors.cpu().numpy())
    assert rc == 0
    assert L == pytest.approx(Lo, rel=1e-5)
    assert np.all(np.abs(g - go) <= 1e-4 * np.abs(go) + 1e-5 * np.max(np.abs(go))), (g, go)
