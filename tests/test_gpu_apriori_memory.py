"""The a priori analysis asks for the device memory it uses: without a coast or a sponge, none for theirs.

A 2048^2 -> 256^2 call without either needs 300 MB (ten mixed arrays of 2048 x 683, two spectra of 683 x 1368, one
field, all FP64, and 12 MB of coarse ones); a coast's and a sponge's arrays would be 127 MB more.  With 360 MB free the
call runs, and gives what it gives with the whole device free.
"""
import math

import numpy as np
import pytest

import synth as S

pytestmark = pytest.mark.gpu

qg = pytest.importorskip("paper_2508_06678_gb300")


def test_apriori_without_a_coast_runs_in_the_memory_it_uses():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import os
    from paper_2508_06678_gb300._lib import LIB_PATH, qg_closure, qg_params
    if not os.path.exists(LIB_PATH):
        from paper_2508_06678_gb300.build import build
        build()
    qg.load()
    w = S.init_field(1, 2048, k_peak=40.0)

    def call():
        return qg.qg_sgs_apriori(w, 256, 2 * math.pi, None, None, qg_closure(S.SMAG, 0, 0.17, 2.0),
                                 qg_params(2e-3, 5e-3, 0.0, 1e-3, 50.0, 0, 0), 0.5, 5.0)

    ref = call()  # also loads the kernels
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    held = torch.empty(free - 360 * 1000 * 1000, dtype=torch.uint8, device="cuda")
    try:
        got = call()
    finally:
        del held
        torch.cuda.empty_cache()
    for a, b in zip(got[:3], ref[:3]):
        assert np.array_equal(np.asarray(a), np.asarray(b))
    assert got[3] == ref[3]
