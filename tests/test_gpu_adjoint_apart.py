"""The gradient's passes with the pointwise products apart from the row passes.

FP64 Smagorinsky grids from 2916^2 and Leith grids from 3888^2 have too many physical rows for the row passes that form
a stage's products, so their gradients transform, multiply and transform back in separate launches.  QG_FORCE_GENERIC
takes those launches for the static closures on any grid; here on small ones, against the oracle's adjoint with the
tolerances of test_gpu_adjoint.py, and against the products formed in the row passes.
"""
import ctypes
import math

import numpy as np
import pytest

import oracle as O
import synth as S

pytestmark = pytest.mark.gpu

qg = pytest.importorskip("paper_2508_06678_gb300")
L = 2 * math.pi


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


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def gradient(n, kind, c, precision, mask, sponge, w, lam):
    """The gradient, its parameter derivatives, and the launches of its pointwise kernels."""
    with qg.QGSolver(n, precision=precision, beta=5.0, U=0.5, mask=S.island_mask(n, L, radius=0.9) if mask else None,
                     sponge=S.sponge_mask(n, L) if sponge else None, kind=kind, c=c, dt=5e-3, eta=2e-2,
                     sponge_rate=50.0) as s:
        got, g = s.step_vjp(w, lam)
        counts = (ctypes.c_int32 * 11)()
        ms = (ctypes.c_double * 11)()
        assert qg.load().qg_kernel_times(ctypes.c_void_p(s.h), counts, ms, 11) == 0
    return got, g, counts[10]


CASES = [(48, O.NONE, 0.0, True, True), (48, O.SMAG, 0.5, True, True), (54, O.LEITH, 0.6, True, True),
         (96, O.LEITH, 0.4, False, True), (96, O.SMAG, 0.4, True, False), (64, O.SMAG, 0.3, False, False)]


@pytest.mark.parametrize("precision", [qg.QG_FP64, qg.QG_FP32])
@pytest.mark.parametrize("n,kind,c,mask,sponge", CASES)
def test_products_apart_match_the_oracle(n, kind, c, mask, sponge, precision, monkeypatch):
    ops = O.Ops(n, L)
    w = S.init_field(3, n, L, k_peak=n / 6)
    lam = np.random.default_rng(n).standard_normal((n, n))
    ref, gr = O.full_step_vjp(ops, O.project(ops, w), lam, 5.0, 0.5, O.Closure(kind, c=c),
                              O.Params(dt=5e-3, eta=2e-2, sponge_rate=50.0),
                              S.island_mask(n, L, radius=0.9) if mask else None, S.sponge_mask(n, L) if sponge else None)
    dtype = np.float64 if precision == qg.QG_FP64 else np.float32
    w, lam = w.astype(dtype), lam.astype(dtype)
    _, _, fused = gradient(n, kind, c, precision, mask, sponge, w, lam)
    monkeypatch.setenv("QG_FORCE_GENERIC", "1")
    got, g, apart = gradient(n, kind, c, precision, mask, sponge, w, lam)
    # a product kernel per stage each way; past a coast its factor each way, and a combination in the curl's place
    assert apart == fused + 6 + (3 if mask else 0)
    assert rel(np.asarray(got, dtype=np.float64), ref) < (1e-10 if precision == qg.QG_FP64 else 1e-4)
    for key in ("C", "c", "sponge_rate"):
        if gr[key] != 0.0:
            assert g[key] == pytest.approx(gr[key], rel=1e-9 if precision == qg.QG_FP64 else 1e-3), key
