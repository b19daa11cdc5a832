"""Fields wider than the phantom: most particles miss it, and their energy is summed like that of those that hit."""
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


@pytest.mark.parametrize("particle,N", [(0, 1_000_003), (1, 50_001)])
def test_energy_of_missed_particles(ocmc, particle, N):
    ph = I.homogeneous((20, 20, 20), (0.25, 0.25, 0.25))
    beam = I.beam_on(ph, particle, I.mono(6.0), (20.0, 20.0), 100.0)
    ref = None
    for kw in ({}, dict(block_threads=32, blocks_per_sm=1), dict(block_threads=256, max_registers=80)):
        with ocmc.Engine(0, n_batches=2, **kw) as e:
            e.create_phantom(ph)
            e.set_source(beam)
            e.run(N, seed=2)
            t, st = e.raw_tally(), e.stats()
        assert st["histories"] == N and 0.9 * N < st["missed"] < N
        assert st["e_miss"] == 6.0 * st["missed"]              # 6 MeV is a whole number of the sums' units
        assert st["e_in"] == 6.0 * (N - st["missed"])
        ref = (t, st["missed"], st["e_esc"]) if ref is None else ref
        assert np.array_equal(t, ref[0]) and (st["missed"], st["e_esc"]) == ref[1:]
