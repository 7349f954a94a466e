"""A frame whose prepared form has more than 2^31 pixel pairs: one column of
2^29 + 8 pixels (the row pitch, two pairs wide before it was spread over the
L1 banks, is four now).  Patch radius 0 and no noise, so that a particle's
log-weight is l = I0 (Zb - I0 / 2) / sigma_xi^2 of the pixel it stands on: two
roundings on exact values, 1e-6 relative to the larger term."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("likelihood", [0, 1])
def test_log_weights_all_over_a_frame_of_2_31_pairs(likelihood):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    free, _ = torch.cuda.mem_get_info()
    if free < 32 * 2**30:
        pytest.skip("needs ~32 GB of free device memory")
    import paper_1310_5045_gb300 as ppf
    H, n, I0, sxi = (1 << 29) + 8, 4096, 24.0, 4.0
    frame = (torch.arange(H, dtype=torch.int32, device="cuda") >> 6).remainder_(199).to(torch.float16).view(H, 1)
    model = ppf.Model(width=1, height=H, patch_radius=0, psf_sigma=1.0, amplitude=I0, background=10.0, sigma_xi=sxi,
                      sigma_m=0.0, sigma_v=0.0, sigma_I=0.0, v0_max=0.0, seed=0, filter_id=0, frame_dtype=ppf.F16,
                      likelihood=likelihood)
    pf = ppf.ParticleFilter(model, n, group_size=n)
    y = np.linspace(0, (1 << 29) // 64 - 1, n).astype(np.int64) * 64  # multiples of 64: exact in float32
    st = np.zeros((6, n), dtype=np.float32)
    st[1], st[4] = y, I0
    pf.set_particles(torch.from_numpy(st).cuda())
    pf.step(frame, 1)
    got = pf.get_particles()[0].cpu().numpy()
    pf.close()
    assert np.array_equal(got[1].astype(np.int64), y)
    zb = (y >> 6) % 199 - 10.0
    want = I0 * (zb - 0.5 * I0) / (sxi * sxi)
    assert np.all(np.abs(got[5] - want) <= 1e-6 * I0 * (np.abs(zb) + 0.5 * I0) / (sxi * sxi))
