"""The bounded wait for a tile, in every column pass that has one.

test_gpu_failure.py lets the wait run out at 256^2, where the dynamic closures' column passes load their columns
without tiles.  Here the grids are large enough that the Germano reduction waits for tiles: in its register form
(384^2, 512^2) and in the form that keeps its sums in scratch (2048^2).  As there, one CTA of the first step's first
column pass arms its barrier for a tile it never requests, so nothing is in flight when it gives up.
"""
import numpy as np
import pytest

import synth as S

pytestmark = pytest.mark.gpu

qg = pytest.importorskip("paper_2508_06678_gb300")


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


@pytest.mark.parametrize("n,kind", [(384, S.DLEITH), (512, S.DSMAG), (512, S.LEITH), (2048, S.DLEITH)])
def test_wait_for_a_tile_times_out_and_set_state_recovers(n, kind, monkeypatch):
    wl = S.Workload("t", n, "island", beta=5.0, U=0.5, closure=kind, c=0.2, radius=0.6, seed=3)
    w0 = S.init_field(3, n, k_peak=20.0)
    monkeypatch.setenv("QG_INJECT_TMA_STALL", "5")
    s = qg.QGSolver.from_workload(wl, precision=qg.QG_FP32)
    monkeypatch.delenv("QG_INJECT_TMA_STALL")
    try:
        s.set_state(w0)
        s.step(1)
        with pytest.raises(qg.QGError) as ei:
            s.sync()
        assert ei.value.code == qg.QG_ERR_TIMEOUT
        s.set_state(w0)
        s.step(3)
        got = s.get_state()
    finally:
        s.close()
    with qg.QGSolver.from_workload(wl, precision=qg.QG_FP32) as clean:
        clean.set_state(w0)
        clean.step(3)
        ref = clean.get_state()
    assert np.array_equal(got, ref)
