"""Rounding of the FP64 transforms, on its own: steps whose exact result is their input.

With dt = 1e-300 the explicit terms vanish and the viscous, coast and sponge factors are exactly 1, but a step still
takes the state through every transform of those sub-steps: (u, v) to physical space and back into the curl, and the
vorticity to physical space and back.  What comes out differs from what went in by the transforms' rounding alone, and
errors that are the same in every step (of the twiddle tables, of 1 / N^2, of the small DFTs' constants) add up.

The bounds are 1.1 times (the spread from one set of fields to another) what plain Stockham transforms of radix 8 or 16,
4, 2 and 3 with the twiddles multiplied one by one gave in the same runs on a GB300: 7.37e-15 at 128^2, 1.18e-14 at
256^2, 2.07e-14 at 512^2, 4.48e-14 at 1024^2; 8.42e-15 at 72^2, 7.58e-15 at 96^2, 1.48e-14 at 108^2, 1.20e-14 at 144^2,
1.32e-14 at 192^2, 1.77e-14 at 216^2, 1.97e-14 at 384^2, 4.51e-14 at 768^2.
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


def round_trip_error(n, steps):
    """RMS over three fields of the relative L2 distance between the state before and after the steps."""
    errs = []
    with qg.QGSolver(n, precision=qg.QG_FP64, beta=5.0, U=0.5, mask=S.island_mask(n, radius=0.6),
                     sponge=S.sponge_mask(n), kind=S.NONE, dt=1e-300) as s:
        for seed in (1, 2, 3):
            w = S.init_field(seed, n, k_peak=n / 16)
            with qg.QGSolver(n, precision=qg.QG_FP64, kind=S.NONE, dt=1e-300) as plain:
                plain.set_state(w)  # the field's 2/3 band, without its mean
                w = plain.get_state()
            s.set_state(w)
            s.step(steps)
            errs.append(np.linalg.norm(s.get_state() - w) / np.linalg.norm(w))
    return float(np.sqrt(np.mean(np.square(errs))))


POWERS_OF_TWO = [(128, 20, 8.1e-15), (256, 20, 1.3e-14), (512, 10, 2.3e-14), (1024, 10, 4.9e-14)]


@pytest.mark.parametrize("n,steps,bound", POWERS_OF_TWO)
def test_round_trips_of_the_state_powers_of_two(n, steps, bound):
    assert round_trip_error(n, steps) < bound


FACTORS_OF_THREE = [(72, 20, 9.3e-15), (96, 20, 8.3e-15), (108, 20, 1.63e-14), (144, 20, 1.32e-14), (192, 20, 1.45e-14),
                    (216, 20, 1.95e-14), (384, 10, 2.17e-14), (768, 10, 4.96e-14)]


@pytest.mark.parametrize("n,steps,bound", FACTORS_OF_THREE)
def test_round_trips_of_the_state_factors_of_three(n, steps, bound):
    assert round_trip_error(n, steps) < bound
