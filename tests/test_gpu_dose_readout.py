"""Dose and sigma of tallies that are given (no transport in between), for every number of batches at which the
read-out kernel changes its form, and tallies added to a cleared and to a filled one."""
import numpy as np
import pytest

import ocmc_inputs as I
import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ocmc():
    from paper_1503_01722_gb300 import build
    build.build()
    from paper_1503_01722_gb300 import ocmc as m
    return m


def phantom():
    ph = I.homogeneous((13, 11, 9), (0.3, 0.2, 0.4))
    ph.density[:] = np.random.default_rng(2).uniform(0.001, 2.0, ph.density.shape)
    ph.density[3, 4, 5] = 0.0
    return ph


def tally(B, shape, seed):
    r = np.random.default_rng(seed)
    t = r.integers(0, 1 << 40, (B,) + shape, dtype=np.int64)
    t[:, 0] = r.integers(0, 3, (B,) + shape[1:])          # almost nothing
    t[:, 1] = 1 << 52                                     # batches alike
    return t


def ready(ocmc, ph, B):
    e = ocmc.Engine(0, n_batches=B)
    e.create_phantom(ph)
    return e


# B <= 4, 12, 24 voxels' batches in registers, above that read twice. FP32 after an exact integer sum: about
# 6 roundings and a division of 2 units for the dose, 3 for the voxel sizes; a batch's difference from the mean carries 4 roundings
# of the batch's own dose.
@pytest.mark.parametrize("B", [1, 2, 4, 5, 12, 13, 24, 25, 40])
def test_dose_of_a_given_tally(ocmc, B):
    import torch
    ph = phantom()
    t = tally(B, ph.density.shape, B)
    N = 1000 * B + 7                                      # batches of unequal size
    with ready(ocmc, ph, B) as e:
        e.add_raw_tally(t, 0, N)
        d, s = e.dose()
        d_only, _ = e.dose(sigma=False)
        out = torch.full(ph.density.shape, -1.0, device="cuda"), torch.full(ph.density.shape, -1.0, device="cuda")
        e.dose(out=out)
    D, S = O.finalize(t, ph, N)
    rho = ph.density.astype(np.float64)
    top = t.max(0) / 2.0 ** 28 / np.where(rho > 0, rho, np.inf) / (0.3 * 0.2 * 0.4) / (N // B)
    assert (np.abs(d - D) <= 1e-6 * D).all()
    assert (np.abs(s - S) <= 4e-6 * S + 1e-6 * top).all()
    assert np.array_equal(d, d_only)
    assert np.array_equal(out[0].cpu().numpy(), d) and np.array_equal(out[1].cpu().numpy(), s)


@pytest.mark.parametrize("device", [False, True])
def test_adding_to_a_cleared_and_to_a_filled_tally(ocmc, device):
    import torch
    ph = phantom()
    a, b = tally(3, ph.density.shape, 1), tally(3, ph.density.shape, 2)
    put = (lambda t: torch.from_numpy(t).cuda()) if device else (lambda t: t)
    with ready(ocmc, ph, 3) as e:
        e.set_source(I.beam_on(ph, 1, I.mono(6.0), (1.0, 1.0), 100.0))
        for _ in range(2):                                # fresh, then after a reset
            e.add_raw_tally(put(a), 0, 10)                # onto a cleared one
            assert np.array_equal(e.raw_tally(), a)
            e.add_raw_tally(put(b), 10, 10)
            assert np.array_equal(e.raw_tally(), a + b)
            e.reset()
            assert not e.raw_tally().any()
        e.run_range(0, 500, 1000, seed=3)                 # onto a run's
        r = e.raw_tally()
        assert r.any()
        e.add_raw_tally(put(a), 500, 500)
        assert np.array_equal(e.raw_tally(), r + a)
        e.reset()
        e.run_range(0, 500, 1000, seed=3)                 # a run onto an added one gives the same as the other order
        e.reset()
        e.add_raw_tally(put(a), 500, 500)
        e.run_range(0, 500, 1000, seed=3)
        assert np.array_equal(e.raw_tally(), r + a)
        e.create_phantom(ph)                              # the same grid again clears it
        assert not e.raw_tally().any()
        e.add_raw_tally(put(b), 0, 10)
        assert np.array_equal(e.raw_tally(), b)
