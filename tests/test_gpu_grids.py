"""Every grid with passes specialised for its size against the run-time passes on the same grid.

The grids differ in the transform's plan (radices 2 to 18, eight to eighteen elements per thread), in the threads of a
sequence (not a multiple of a warp for most sizes with factors of 3) and in the column pass's tile boxes (the last one
reaching past the array).  Both paths compute in FP32 from the same state; one step's error against the FP64 oracle is
bounded by 2.5e-8 N past a coast (test_gpu_edges.py) and far less without one, so two steps of the two paths may differ
by 2 * 2 * 2.5e-8 N, and by no less than a few FP32 roundings.
"""
import numpy as np
import pytest

import synth as S

pytestmark = pytest.mark.gpu

qg = pytest.importorskip("paper_2508_06678_gb300")

WIDE = (64, 72, 96, 108, 128, 144, 162, 192, 216, 256, 288, 324)
FAST = (384, 432, 486, 512, 576, 648, 768, 864, 972, 1024, 1152, 1296, 1458, 1536, 1728, 1944, 2048, 2304, 2592, 2916,
        3072, 3456, 3888, 4096)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import os
    from paper_2508_06678_gb300._lib import LIB_PATH
    if not os.path.exists(LIB_PATH):
        from paper_2508_06678_gb300.build import build
        build()
    qg.load()


def _field(n, seed):
    """A random field with spectrum k^4 exp(-(16 k / n)^2), rms 4, on the GPU."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    f = torch.fft.rfft2(torch.randn(n, n, generator=g, device="cuda"))
    mx = torch.arange(n // 2 + 1, device="cuda")[None, :]
    my = torch.fft.fftfreq(n, 1.0 / n, device="cuda")[:, None]
    m2 = mx * mx + my * my
    w = torch.fft.irfft2(f * m2 * torch.exp(-0.5 * m2 * (16.0 / n) ** 2), s=(n, n))
    return (w * (4.0 / w.square().mean().sqrt())).contiguous()


def _run(n, kind, scheme, w, prec):
    import torch
    coast = S.island_mask(n, radius=0.6) if n <= 1024 else None
    sponge = S.sponge_mask(n) if n <= 1024 else None
    out = torch.empty((n, n), dtype=torch.float64, device="cuda")
    with qg.QGSolver(n, precision=prec, beta=5.0, U=0.5, mask=coast, sponge=sponge, kind=kind, c=0.2, dt=5e-4, eta=2e-3,
                     scheme=scheme) as s:
        s.set_state(w)
        s.step(2)
        s.get_state(out=out)
        s.sync()
    return out


@pytest.mark.parametrize("n", WIDE + FAST)
def test_specialised_grid_matches_run_time_passes(n, monkeypatch):
    w = _field(n, n)
    cases = [(S.SMAG, 0), (S.DLEITH, 0), (S.LEITH, 1)] if n <= 1024 else [(S.SMAG, 0), (S.DLEITH, 1)]
    for kind, scheme in cases:
        monkeypatch.delenv("QG_FORCE_GENERIC", raising=False)
        a = _run(n, kind, scheme, w, qg.QG_FP32)
        monkeypatch.setenv("QG_FORCE_GENERIC", "1")
        b = _run(n, kind, scheme, w, qg.QG_FP32)
        err = float((a - b).norm() / b.norm())
        assert err < max(1e-7 * n, 2e-6), (n, kind, scheme, err)


@pytest.mark.parametrize("n", (16, 18, 24, 32, 36, 48, 54, 64, 72, 108, 128, 162, 216, 256, 324, 486, 512, 648))
def test_fp64_grid_matches_fp32(n):
    """The FP64 passes (four elements per thread on 2^a, fused twiddles) against the FP32 ones on the same state."""
    w = _field(n, n + 1)
    for kind in (S.DSMAG, S.LEITH):
        a = _run(n, kind, 0, w, qg.QG_FP64)
        b = _run(n, kind, 0, w, qg.QG_FP32)
        err = float((a - b).norm() / a.norm())
        assert np.isfinite(err) and err < max(1e-7 * n, 2e-6), (n, kind, err)
