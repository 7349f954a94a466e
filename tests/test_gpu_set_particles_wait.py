"""ppf_set_particles has copied the caller's buffers when it returns, whatever
likelihood the context uses: a C caller may overwrite them at once, from any
stream, while the context's own stream still has work queued."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("likelihood", [0, 1])
def test_buffers_may_be_reused_on_return(likelihood):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1310_5045_gb300 as ppf
    n = 5000
    model = ppf.Model(width=64, height=64, patch_radius=3, psf_sigma=1.5, amplitude=50.0, background=10.0,
                      sigma_xi=3.0, sigma_m=0.5, sigma_v=0.1, sigma_I=1.0, v0_max=1.0, seed=1, filter_id=0,
                      likelihood=likelihood)
    rng = np.random.default_rng(likelihood)
    state = torch.from_numpy(rng.uniform(1, 60, (6, n)).astype(np.float32)).cuda()
    anc = torch.from_numpy(rng.integers(0, n, n).astype(np.int32)).cuda()
    lwp = torch.from_numpy(rng.normal(0, 1, n).astype(np.float32)).cuda()
    want = [t.cpu() for t in (state, anc, lwp)]
    own, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    pf = ppf.ParticleFilter(model, n, group_size=n, stream=own)
    torch.cuda.synchronize()
    with torch.cuda.stream(own):
        torch.cuda._sleep(200_000_000)  # the context's stream is busy for a tenth of a second
    st = pf.L.ppf_set_particles(pf._ctx, C.c_void_p(state.data_ptr()), C.c_void_p(anc.data_ptr()),
                                C.c_void_p(lwp.data_ptr()))
    assert st == ppf.OK
    with torch.cuda.stream(other):
        for t in (state, anc, lwp):
            t.zero_()
    other.synchronize()
    got = pf.get_particles(state=True, anc=True, lw_prev=True)
    for g, w in zip(got, want):
        assert torch.equal(g.cpu(), w)
    pf.close()
