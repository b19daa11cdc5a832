"""Dose and sigma with more batches than stay in registers: each read-out uses the batch sizes of its own call."""
import numpy as np
import pytest

import ocmc_inputs as I
import oracle as O

pytestmark = pytest.mark.gpu


# Tolerances: an exact integer sum and about 6 roundings for the dose; B squares summed in FP32 (B / 2 roundings of
# the sum at most, half of that in its root) and 1e-6 of the largest batch dose for sigma.
@pytest.mark.parametrize("B", [24, 25, 26, 999, 1000])
def test_read_outs_one_after_the_other(B):
    from paper_1503_01722_gb300 import build
    build.build()
    from paper_1503_01722_gb300 import ocmc
    ph = I.homogeneous((13, 11, 9), (0.3, 0.2, 0.4))
    t = np.random.default_rng(B).integers(0, 1 << 40, (B,) + ph.density.shape, dtype=np.int64)
    zero = np.zeros_like(t)
    with ocmc.Engine(0, n_batches=B) as e:
        e.create_phantom(ph)
        N = 0
        for add, n in ((t, B + 3), (zero, 7 * B + 1), (zero, 1000 * B)):     # batches of unequal, changing size
            e.add_raw_tally(add, N, n)
            N += n
            d, s = e.dose()
            D, S = O.finalize(t, ph, N)
            top = t.max(0) / 2.0 ** 28 / (0.3 * 0.2 * 0.4) / max(1, N // B)
            assert (np.abs(d - D) <= 1e-6 * D).all()
            assert (np.abs(s - S) <= (4e-6 + B * 2.0 ** -25) * S + 1e-6 * top).all()
