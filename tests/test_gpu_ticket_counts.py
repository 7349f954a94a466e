"""The fill's ticket counts (fixed-point quotients settled on the exact
thresholds) against the oracle's systematic draw: sizes around a thread's 16,
a warp's 512 and a tile's 4096 particles, log-weights that start on every
4-byte offset of a 16-byte vector, and weight shapes that put counts exactly on
whole tickets (equal weights), a tile's tickets into several runs (one heavy
particle, a steep decay) or leave most particles without any.  Ancestors are
integers: they must be equal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = ["equal", "pairs", "heavy", "steep", "gauss", "sparse"]


def _log_weights(shape, n, rng):
    if shape == "equal":
        return np.zeros(n, dtype=np.float32)
    if shape == "pairs":  # weights 1 and 2: every other count lands on a whole ticket
        return np.where(np.arange(n) % 2, 0.0, np.log(2.0)).astype(np.float32)
    if shape == "heavy":
        lw = np.full(n, -60.0, dtype=np.float32)
        lw[n // 3] = 0.0
        return lw
    if shape == "steep":
        return (-np.arange(n) * (40.0 / n)).astype(np.float32)
    if shape == "sparse":
        lw = np.full(n, -np.inf, dtype=np.float32)
        lw[rng.integers(0, n, max(1, n // 700))] = rng.normal(0, 2, max(1, n // 700)).astype(np.float32)
        return lw
    return (-rng.chisquare(2, n)).astype(np.float32)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n", [1, 2, 15, 17, 511, 513, 4095, 4097, 8185, 70_001])
def test_ancestors_equal_the_oracle(orc, n, shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1310_5045_gb300 as ppf
    rng = np.random.default_rng(n)
    lw = _log_weights(shape, n, rng)
    for shift in range(4):
        seed, frame = 17 * n + shift, 1 + shift
        buf = torch.full((n + 8,), 1e30, dtype=torch.float32, device="cuda")  # neighbours must never be weighed
        buf[shift:shift + n] = torch.from_numpy(lw)
        got = ppf._binding.systematic_resample_noalloc(buf[shift:shift + n], seed, 3, frame).cpu().numpy()
        rc, want, *_ = orc.resample(orc.Model(seed=seed, filter_id=3), orc.SYSTEMATIC, n, frame,
                                    np.array([0, n], dtype=np.int64), lw)
        assert rc == 0
        assert np.array_equal(got, want), (shape, n, shift, int(np.sum(got != want)))


@pytest.mark.parametrize("group", [511, 1024, 1025, 2048, 2049, 4097])
def test_rna_block_sizes(orc, group):
    """RNA's block follows the group size (16 particles per thread, 64 to 256
    threads): groups at the edges of each size, a ragged last group."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import synth
    import paper_1310_5045_gb300 as ppf
    from gpu_common import lockstep, paired_models
    mv = synth.make_movie(W=128, H=128, K=2, seed=3)
    gm, om = paired_models(ppf, seed=5)
    pf = ppf.ParticleFilter(gm, 3 * group + 7, group_size=group)
    lockstep(pf, gm, om, mv.frames, torch.from_numpy(mv.frames).cuda(), orc.RNA, K=2, alpha=0.25)
    pf.close()


@pytest.mark.parametrize("scheme", ["rpa_gs", "rpa_sgs", "rpa2_sgs"])
@pytest.mark.parametrize("groups", [1, 2, 33, 64, 65, 2048, 2049])
def test_schedule_group_counts(orc, groups, scheme):
    """The GS and SGS schedule in the fill's first block (up to 2048 groups)
    and on the side stream (above): counts at the edges of the sort's powers of
    two and of the rule, groups of 5 particles and one ragged."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import synth
    import paper_1310_5045_gb300 as ppf
    from gpu_common import lockstep, paired_models
    mv = synth.make_movie(W=64, H=64, K=2, seed=4)
    gm, om = paired_models(ppf, seed=groups, width=64, height=64, patch_radius=2)
    pf = ppf.ParticleFilter(gm, 5 * groups - (1 if groups > 1 else 0), group_size=5)
    assert len(pf.groups()) - 1 == groups
    lockstep(pf, gm, om, mv.frames, torch.from_numpy(mv.frames).cuda(), getattr(orc, scheme.upper()), K=2)
    pf.close()
