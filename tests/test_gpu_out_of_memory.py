"""Allocations that cannot succeed (more than the GPU has, so nothing is taken): an error of that call, and the context
goes on."""
import numpy as np
import pytest

import ocmc_inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ocmc():
    from paper_1503_01722_gb300 import build
    build.build()
    from paper_1503_01722_gb300 import ocmc as m
    return m


def out_of_memory(ocmc, call):
    with pytest.raises(ocmc.OcmcError) as x:
        call()
    assert x.value.status == ocmc.ERR_OOM


def test_tally(ocmc):
    ph = I.homogeneous((400, 400, 400), (0.1, 0.1, 0.1))           # 1000 batches: 512 GB
    beam = I.beam_on(ph, 0, I.mono(6.0), (5.0, 5.0), 100.0)
    small = I.homogeneous((20, 20, 20), (1.0, 1.0, 1.0))

    def result(e):
        e.run(20_000, seed=1)
        return e.raw_tally()

    with ocmc.Engine(0) as f:
        f.create_phantom(small)
        f.set_source(beam)
        ref = result(f)
    with ocmc.Engine(0, n_batches=1000) as e:
        e.set_source(beam)
        for first in (None, small):                                # without a phantom, over one
            if first:
                e.create_phantom(first)
            out_of_memory(ocmc, lambda: e.create_phantom(ph))
            for call in (lambda: e.run(1000), e.dose, e.raw_tally):
                with pytest.raises(ocmc.OcmcError) as x:
                    call()
                assert x.value.status == ocmc.ERR_STATE
        e.set_params(n_batches=10)
        e.create_phantom(small)
        assert np.array_equal(result(e), ref)
        with pytest.raises(ocmc.OcmcError):                        # refused: the phantom stays
            e.create_phantom(density=-np.ones((2, 2, 2), np.float32), material=np.zeros((2, 2, 2), np.uint8), voxel=(1, 1, 1))
        e.reset()
        assert np.array_equal(result(e), ref)


def test_beamlet_tables(ocmc):
    ph = I.ct_like()
    n = 8000                                                       # tables for every voxel: over 500 GB
    bl = [dict(b, n_histories=4) for b in I.beamlets(ph, n_beamlets=n, seed=1)]
    spec = I.spectrum_6mv()
    with ocmc.Engine(0, beamlet_capacity_scale=1.0) as f:
        f.create_phantom(ph)
        f.set_beamlets(0, *spec, bl)
        f.run_beamlets(seed=2)
        ref = [f.beamlet_dose(b) for b in range(0, n, 500)]
    with ocmc.Engine(0, beamlet_capacity_scale=1.0) as e:
        e.create_phantom(ph)
        e.set_beamlets(0, *spec, bl[:50])
        e.run_beamlets(seed=2)                                     # tables that are there already
        e.set_params(beamlet_capacity_scale=1e6)
        e.set_beamlets(0, *spec, bl)
        out_of_memory(ocmc, lambda: e.run_beamlets(seed=2))
        with pytest.raises(ocmc.OcmcError) as x:
            e.beamlet_dose(0)
        assert x.value.status == ocmc.ERR_STATE
        e.set_params(beamlet_capacity_scale=1.0)
        e.run_beamlets(seed=2)
        got = [e.beamlet_dose(b) for b in range(0, n, 500)]
    for a, b in zip(got, ref):
        assert all(np.array_equal(x, y) for x, y in zip(a, b))
