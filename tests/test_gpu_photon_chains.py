"""Long chains of fictitious photon events (k_chains): low-energy photons in air beside dense bone fly
hundreds of Woodcock steps between real events. Which of them a warp leaves to k_chains depends on the
launch shape and on how many histories run together, so the tally must not."""
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


def air_and_bone(n):
    ph = I.homogeneous(n, (0.5, 0.5, 0.5), density=0.0012)
    ph.material[-2:] = I.BONE
    ph.density[-2:] = 1.9
    return ph


def run(ocmc, ph, beam, calls, **kw):
    with ocmc.Engine(0, n_batches=2, **kw) as e:
        e.create_phantom(ph)
        e.set_source(beam)
        for first, count, total in calls:
            e.run_range(first, count, total, seed=5)
        return e.raw_tally(), e.stats()


@pytest.mark.parametrize("n,keV", [((40, 36, 44), 15.0), ((31, 33, 40), 40.0), ((40, 40, 40), 1500.0)])
def test_tally_does_not_depend_on_who_flies_the_chains(ocmc, n, keV):
    ph = air_and_bone(n)
    beam = I.beam_on(ph, 0, I.mono(keV * 1e-3), (8.0, 8.0), 100.0)
    N = 1500
    ref, st = run(ocmc, ph, beam, [(0, N, N)], block_threads=32, blocks_per_sm=1)
    if keV < 20:
        assert st["photon_flights"] > 100 * N       # chains are what this case is about
    assert st["dropped"] == 0 and st["majorant_violations"] == 0
    for kw in ({}, {"block_threads": 256, "blocks_per_sm": 2, "max_registers": 80}, {"e_class_split": 0.0}):
        t, s = run(ocmc, ph, beam, [(0, N, N)], **kw)
        assert np.array_equal(t, ref)
        for k in ("photon_flights", "fictitious", "compton", "photo", "escaped", "lane_steps", "e_esc"):
            assert s[k] == st[k], (kw, k)
    # every history alone (its chains always end in k_chains), then all of them in one range
    few = 24
    one, s1 = run(ocmc, ph, beam, [(h, 1, N) for h in range(few)])
    all_, s2 = run(ocmc, ph, beam, [(0, few, N)])
    assert np.array_equal(one, all_) and s1["photon_flights"] == s2["photon_flights"]
