"""Every launch shape of the passes against something computed another way.

FP64 steps against the oracle, on grids of four, twelve and eighteen elements per thread, with two rows per CTA, with
columns shared out and rows on their own in the last round.  FP32 steps and gradients of every grid with passes of its
own against the FP64 passes, which share neither the transform's plan nor a kernel with them.

FP32 fields fill the 2/3 band evenly, to its last row and column.  Past a coast, with the default viscosity, the error
of a step is bounded by 2.5e-8 N (test_gpu_edges.py), of two steps by twice that.  The modes of the band's edge, which
carry about 1 / N of the field's square, are looked at on their own in runs without coast and viscosity (a coast's
curl puts its rounding there, the viscosity would damp them below it): a two-dimensional FP32 transform rounds to about
2e-7 of its field, a step holds the sponge's two and its stages' fifteen at a third of the weight, so two steps and the
state's way in and out come to 1e-6; the bounds are four times that for the band, and four times more for its edge.
(Not with the Leith closures: J shares a complex transform with g w_x, and over a field this rough g w_x is 1e4 times
J, whose rounding it then sets, whatever the coefficient.)
"""
import math

import numpy as np
import pytest

import oracle as O
import synth as S

pytestmark = pytest.mark.gpu

qg = pytest.importorskip("paper_2508_06678_gb300")

SIDE_BY_SIDE = (64, 72, 96, 108, 128, 144, 162, 192, 216, 256, 288, 324)
ONE_BY_ONE = (192, 216, 256, 288, 324, 384, 432, 486, 512, 576, 648, 768, 864, 972, 1024, 1152, 1296, 1458, 1536, 1728,
              1944, 2048, 2304, 2592, 2916, 3072, 3456, 3888, 4096)


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


FP64_CASES = [(n, kind) for n in (108, 162, 216, 256, 324, 384, 486) for kind in (S.SMAG, S.DLEITH, S.DSMAG)]
FP64_CASES += [(n, kind) for n in (512, 648, 768, 1024, 1296) for kind in (S.NONE, S.LEITH, S.SMAG)]


@pytest.mark.parametrize("n,kind", FP64_CASES)
def test_fp64_step_matches_the_oracle(n, kind):
    """Two steps: rounding only, 1e-12."""
    wl = S.Workload("t", n, "island", beta=5.0, U=0.5, closure=kind, c=0.2, radius=0.6, seed=n)
    w0 = S.init_field(n, n, k_peak=n / 16)
    ref = O.QGOracle(n, wl.L, wl.beta, wl.U, wl.mask(), wl.sponge_field(), O.Closure(kind, c=0.2), O.Params())
    ref.set_state(w0)
    ref.step(2)
    with qg.QGSolver.from_workload(wl, precision=qg.QG_FP64) as s:
        s.set_state(w0)
        s.step(2)
        got = s.get_state()
    w = ref.get_state()
    assert np.linalg.norm(got - w) / np.linalg.norm(w) < 1e-12


def even_field(n, seed):
    """A random field, rms 4, all modes of the 2/3 band but the mean equally strong on average; on the GPU, FP64."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    f = torch.fft.rfft2(torch.randn(n, n, dtype=torch.float64, generator=g, device="cuda"))
    K = (n - 1) // 3
    keep = (torch.arange(n // 2 + 1, device="cuda")[None, :] <= K) & \
        (torch.fft.fftfreq(n, 1.0 / n, device="cuda").abs()[:, None] <= K)
    f = f * keep
    f[0, 0] = 0
    w = torch.fft.irfft2(f, s=(n, n))
    return w * (4.0 / w.square().mean().sqrt())


def errors(a, b):
    """Relative L2 distance of a from b, over the whole band and over its outermost rows and columns."""
    import torch
    n = a.shape[0]
    K = (n - 1) // 3
    fa, fb = torch.fft.rfft2(a.double()), torch.fft.rfft2(b)

    def rel(pick):
        x, y = pick(fa), pick(fb)
        return float((x - y).norm() / y.norm())

    return rel(lambda f: f), max(rel(lambda f: f[:, K]), rel(lambda f: f[K, :K + 1]), rel(lambda f: f[n - K, :K + 1]))


_masks = {}


def masks(n):
    if n not in _masks:
        _masks.clear()
        _masks[n] = (S.island_mask(n, radius=0.6), S.sponge_mask(n))
    return _masks[n]


def two_steps(n, prec, kind, scheme, w, coast):
    import torch
    chi, chs = masks(n)
    out = torch.empty(n, n, dtype=torch.float64, device="cuda")
    with qg.QGSolver(n, precision=prec, beta=5.0, U=0.5, mask=chi if coast else None, sponge=chs, kind=kind, c=0.2,
                     dt=5e-4, nu=1.0 / 200.0 if coast else 0.0, eta=2e-3, scheme=scheme) as s:
        s.set_state(w)
        s.step(2)
        s.get_state(out=out)
        s.sync()
    return out


def fp64_takes(n, kind):
    """FP64 steps keep a row's physical fields in shared memory: six, four, twelve or eight."""
    return n <= {S.SMAG: 3456, S.DSMAG: 2048, S.DLEITH: 2592}.get(kind, 4096)


@pytest.mark.parametrize("n", sorted(set(SIDE_BY_SIDE + ONE_BY_ONE)))
def test_fp32_steps_match_the_fp64_passes(n):
    import torch
    w = even_field(n, n)
    for kind, scheme in ((S.SMAG, 0), (S.DSMAG, 0), (S.LEITH, 1)):
        if fp64_takes(n, kind):
            err, _ = errors(*(two_steps(n, prec, kind, scheme, w, True) for prec in (qg.QG_FP32, qg.QG_FP64)))
            assert err < max(5e-8 * n, 4e-6), (n, kind, scheme, err)
    for kind, scheme in ((S.NONE, 0), (S.SMAG, 0), (S.DSMAG, 0), (S.NONE, 1), (S.SMAG, 1)):
        if fp64_takes(n, kind):
            err, edge = errors(*(two_steps(n, prec, kind, scheme, w, False) for prec in (qg.QG_FP32, qg.QG_FP64)))
            assert err < 4e-6 and edge < 1.6e-5, (n, kind, scheme, err, edge)
    torch.cuda.empty_cache()


@pytest.mark.parametrize("n", (64, 108, 144, 162, 216, 324, 384, 486, 512, 648, 768))
def test_fp32_gradients_match_the_fp64_passes(n):
    """One step's gradient and its parameters' derivatives, within the bound of a step (the derivatives: ten times; they
    are inner products with lam, which shares half of w so that they are no sums of terms that cancel)."""
    import torch
    w = even_field(n, n)
    lam = 0.5 * (w + even_field(n, n + 1))
    chi, chs = masks(n)
    for kind in (S.NONE, S.SMAG, S.LEITH, S.DSMAG):
        got = []
        for prec, dtype in ((qg.QG_FP32, torch.float32), (qg.QG_FP64, torch.float64)):
            with qg.QGSolver(n, precision=prec, beta=5.0, U=0.5, mask=chi, sponge=chs, kind=kind, c=0.2, dt=5e-4,
                             eta=2e-3) as s:
                out, grads = s.step_vjp(w.to(dtype), lam.to(dtype))
                s.sync()
                got.append((out.clone(), grads))
        bound = max(2.5e-8 * n, 4e-6)
        err, edge = errors(got[0][0], got[1][0])
        assert err < bound and edge < 4 * bound, (n, kind, err, edge)
        for key, ref in got[1][1].items():
            if ref != 0.0 and math.isfinite(ref):
                assert got[0][1][key] == pytest.approx(ref, rel=10 * bound), (n, kind, key)
