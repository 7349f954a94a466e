"""The binned likelihood path at the edges of its work: particle counts around
a work item's 1536 records, the scatter's chunk of 4096 slots and its 16-byte
vectors, all particles in one image tile or spread over the frame, and the
wider tiles of large frames.  The direct path is the reference: the two add the
same terms in the same order, so every output has the same bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _step(ppf, model, state, frame, path, carry):
    import torch
    n = state.shape[1]
    pf = ppf.ParticleFilter(model, n, group_size=n)
    pf.set_likelihood_path(path)
    lwp = None if carry else torch.from_numpy(np.linspace(-2, 0, n).astype(np.float32)).cuda()
    anc = None if carry else torch.from_numpy(np.arange(n, dtype=np.int32)[::-1].copy()).cuda()
    pf.set_particles(torch.from_numpy(state).cuda(), anc, lwp)
    anc0 = pf.get_particles(state=False, anc=True)[1].cpu().numpy()
    assert np.array_equal(anc0, np.arange(n)[::-1] if anc is not None else np.arange(n))
    pf.step(frame, 1)
    e = pf.estimate()
    st = pf.get_particles()[0].cpu().numpy()
    binned = pf.last_step_binned()
    pf.close()
    return st, np.array([*e.mean, e.log_evidence, e.ess, e.max_log_weight]), binned


@pytest.mark.parametrize("spread", [False, True])
@pytest.mark.parametrize("n", [1, 3, 1279, 1280, 1281, 1535, 1536, 1537, 2561, 3073, 4095, 4096, 4097, 4100, 40_003])
def test_binned_equals_direct(n, spread):
    _compare(n, spread, 200, 150, 5)


def test_wide_tiles_of_a_large_frame():
    _compare(30_001, True, 1920, 1900, 8)


def _compare(n, spread, width, height, r):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1310_5045_gb300 as ppf
    rng = np.random.default_rng(n)
    st = np.zeros((6, n), dtype=np.float32)
    st[0] = rng.uniform(-8, width + 8, n) if spread else rng.uniform(66, 90, n)
    st[1] = rng.uniform(-8, height + 8, n) if spread else rng.uniform(66, 90, n)
    st[2:4] = rng.normal(0.0, 0.5, (2, n))
    st[4] = rng.uniform(10, 70, n)
    st[5] = rng.normal(0.0, 1.0, n)
    frame = torch.from_numpy(rng.poisson(12.0, (height, width)).astype(np.float32)).cuda()
    model = ppf.Model(width=width, height=height, patch_radius=r, psf_sigma=1.5, amplitude=50.0, background=10.0,
                      sigma_xi=3.0, sigma_m=0.3, sigma_v=0.1, sigma_I=1.0, v0_max=1.0, seed=3, filter_id=0)
    for carry in (True, False):
        sd, ed, bd = _step(ppf, model, st, frame, ppf.PATH_DIRECT, carry)
        sb, eb, bb = _step(ppf, model, st, frame, ppf.PATH_BINNED, carry)
        assert bb and not bd
        assert np.array_equal(sd, sb) and np.array_equal(ed, eb)
