"""The bounds-checked debug build on the launch shapes that small grids do not reach.

test_gpu_checked.py runs the passes with a run-time length on grids up to 54, where a column pass has one column per
CTA.  Here, with the same library in a child process: the side-by-side FP32 passes with the length fixed at compile
time (64 to 324), two columns per CTA (FP32 576 and 648 with a run-time length), row passes of two rows with products
(FP64 256), columns shared out over several CTAs and single rows in the last round (FP64 1024), and the gradient's
passes of each.  Every run must report no bad index and match the oracle.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import math, os, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
import paper_2508_06678_gb300 as qg
import oracle as O
import synth as S

def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, dtype=np.float64) - b) / np.linalg.norm(b))

F32, F64 = qg.QG_FP32, qg.QG_FP64
count = 0
steps = [(n, F32, kind, scheme, False) for n in (64, 72, 108, 162, 192, 216, 324) for kind in (S.DSMAG, S.DLEITH)
         for scheme in (O.RK3_EXACT, O.AB2CN)]
steps += [(n, F32, kind, scheme, False) for n in (64, 96, 144) for kind in (S.NONE, S.SMAG, S.LEITH)
          for scheme in (O.RK3_EXACT, O.AB2CN)]
steps += [(n, F32, kind, O.RK3_EXACT, True) for n in (576, 648) for kind in (S.SMAG, S.DLEITH)]
steps += [(256, F64, kind, O.RK3_EXACT, False) for kind in (S.NONE, S.LEITH, S.DSMAG)]
steps += [(1024, F64, kind, scheme, False) for kind in (S.NONE, S.LEITH) for scheme in (O.RK3_EXACT, O.AB2CN)]
for n, prec, kind, scheme, generic in steps:
    dt, eta = (2e-3, 1e-3) if scheme == O.RK3_EXACT else (5e-4, 2e-3)
    wl = S.Workload("chk", n, "island", beta=5.0, U=0.5, closure=kind, c=0.2, radius=0.6, seed=n + kind, dt=dt, eta=eta)
    w0 = S.init_field(n + kind, n, k_peak=n / 16)
    ref = O.QGOracle(n, wl.L, wl.beta, wl.U, wl.mask(), wl.sponge_field(), O.Closure(kind, c=0.2),
                     O.Params(dt=dt, eta=eta, scheme=scheme))
    ref.set_state(w0)
    ref.step(2)
    os.environ.pop("QG_FORCE_GENERIC", None)
    if generic:
        os.environ["QG_FORCE_GENERIC"] = "1"
    with qg.QGSolver.from_workload(wl, precision=prec, scheme=scheme) as s:
        s.set_state(w0)
        s.step(2)
        s.sync()  # raises QGError(QG_ERR_BOUNDS) if any checked access was out of range
        err = rel(s.get_state(), ref.get_state())
        s.diagnostics()
        s.sync()
    assert err < (1e-12 if prec == F64 else 1e-4), (n, kind, scheme, prec, err)
    count += 1
os.environ.pop("QG_FORCE_GENERIC", None)
for n, prec, kind, c in [(96, F64, S.SMAG, 0.4), (256, F64, S.LEITH, 0.3), (108, F32, S.LEITH, 0.4),
                         (216, F32, S.DSMAG, 0.0), (144, F32, S.DLEITH, 0.0), (128, F32, S.NONE, 0.0)]:
    L = 2 * math.pi
    chi, chs = S.island_mask(n, L, radius=0.9), S.sponge_mask(n, L)
    ops = O.Ops(n, L)
    w = S.init_field(3, n, L, k_peak=n / 6)
    lam = np.random.default_rng(n).standard_normal((n, n))
    ref, _ = O.full_step_vjp(ops, O.project(ops, w), lam, 5.0, 0.5, O.Closure(kind, c=c),
                             O.Params(dt=5e-3, eta=2e-2, sponge_rate=50.0), chi, chs)
    dtype = np.float64 if prec == F64 else np.float32
    with qg.QGSolver(n, precision=prec, beta=5.0, U=0.5, mask=chi, sponge=chs, kind=kind, c=c, dt=5e-3, eta=2e-2,
                     sponge_rate=50.0) as s:
        got, _ = s.step_vjp(w.astype(dtype), lam.astype(dtype))
        s.sync()
    err = rel(got, ref)
    assert err < (1e-10 if prec == F64 else 1e-4), (n, kind, prec, err)
    count += 1
print("checked runs", count, "of", len(steps) + 6)
"""


@pytest.fixture(scope="module")
def checked_lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_06678_gb300.build import CHECKED_DIR, build_checked
    path = os.path.join(CHECKED_DIR, "libqg.so")
    if not os.path.exists(path):
        build_checked()
    return path


def test_checked_build_wide_two_column_two_row_and_split_passes(checked_lib):
    env = dict(os.environ, QG_LIB=checked_lib)
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "checked runs 63 of 63" in r.stdout
