"""The caller's buffer of ParticleFilter.estimate_async: the kernel stores
8-byte words straight to a page-locked buffer, so only an aligned and wholly
mapped one may be handed to it; every other buffer gets the staged copy, and a
buffer that cannot hold the estimate is refused."""
import os
import subprocess
import types

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RULE = r"""
#include "ppf_mapped.h"
#include <cstdio>
#include <initializer_list>
// host bytes [64, end) of an imaginary address space are mapped `shift` bytes on; the pages that hold them are accessible
int main()
{
    const uintptr_t page = 4096;
    for (uintptr_t shift : {uintptr_t(0x10000), uintptr_t(0x10004)})
        for (uintptr_t end : {page - 200, page - 8, page, page + 1, page + 96, 2 * page})
            for (uintptr_t p = page - 240; p < page + 16; ++p) {
                auto map = [&](void *q) -> void * {
                    const uintptr_t a = (uintptr_t)q;
                    return a >= 64 && a < end ? (void *)(a + shift) : nullptr;
                };
                void *got = ppf::mapped_words((void *)p, 104, map);
                const bool aligned = p % 8 == 0 && shift % 8 == 0, reachable = p + 104 <= (end + page - 1) / page * page;
                if (got && (got != (void *)(p + shift) || !aligned || !reachable))
                    return std::printf("handed out: shift %zx p %zu end %zu\n", (size_t)shift, (size_t)p, (size_t)end), 1;
                if (!got && aligned && p + 104 <= end)
                    return std::printf("kept back: shift %zx p %zu end %zu\n", (size_t)shift, (size_t)p, (size_t)end), 1;
            }
    // the last byte on another page and in another mapping than the first
    auto split = [=](void *q) -> void * { return (void *)((uintptr_t)q + ((uintptr_t)q < page ? 0x10000 : 0x20000)); };
    return ppf::mapped_words((void *)(page - 48), 104, split) != nullptr;
}
"""


def test_direct_store_needs_an_aligned_and_wholly_mapped_buffer(tmp_path):
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(RULE)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_1310_5045_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_a_buffer_that_cannot_hold_the_estimate_is_refused():
    import torch

    import paper_1310_5045_gb300 as ppf
    pf = ppf.ParticleFilter.__new__(ppf.ParticleFilter)
    taken = []
    pf._torch, pf._ctx = torch, None
    pf.L = types.SimpleNamespace(ppf_estimate_async=lambda ctx, p: taken.append(p.value) or ppf.OK)
    n = ppf.Estimate.nbytes()
    for bad in (torch.empty(0, dtype=torch.uint8), torch.empty(n - 1, dtype=torch.uint8),
                torch.empty(2 * n, dtype=torch.uint8)[::2], torch.empty(n // 8 - 1, dtype=torch.float64)):
        with pytest.raises(ValueError):
            pf.estimate_async(bad)
    assert not taken
    buf = torch.empty(2 * n, dtype=torch.uint8)
    for out in (buf, buf[1:], buf[n:], torch.empty(n // 8, dtype=torch.float64)):
        assert pf.estimate_async(out) is out and taken[-1] == out.data_ptr()


@pytest.mark.gpu
@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("offset", [0, 1, 4, 8])
def test_estimate_at_any_address(pinned, offset):
    """The bytes of estimate() arrive at every offset, in page-locked and in
    pageable memory, and none around them changes."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import synth
    import paper_1310_5045_gb300 as ppf
    mv = synth.make_movie(W=64, H=64, K=3, seed=4)
    frames = torch.from_numpy(mv.frames).cuda()
    model = ppf.Model(width=64, height=64, patch_radius=4, psf_sigma=1.5, amplitude=50.0, background=10.0,
                      sigma_xi=3.0, sigma_m=0.5, sigma_v=0.1, sigma_I=1.0, v0_max=1.0, seed=4, filter_id=0)
    n = ppf.Estimate.nbytes()
    pf = ppf.ParticleFilter(model, 3000, group_size=1000)
    for k in range(1, 4):
        buf = torch.full((n + 32,), 0xA5, dtype=torch.uint8)
        buf = buf.pin_memory() if pinned else buf
        pf.step(frames[k - 1], k)
        pf.resample(ppf.RPA_SGS)
        pf.estimate_async(buf[offset:offset + n])
        pf.stream.synchronize()
        got, want = ppf.Estimate.from_buffer(buf[offset:offset + n]), pf.estimate()
        assert got == want and got.frame == k
        assert bool((buf[:offset] == 0xA5).all()) and bool((buf[offset + n:] == 0xA5).all())
    pf.close()
