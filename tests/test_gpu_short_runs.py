"""Runs around the sizes at which the launch changes how many warps of a block draw histories and how many
each draws at once, and parameters that change which stacks a warp refills from: the tally must not change."""
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


KEYS = ("histories", "missed", "compton", "moller", "escaped", "lane_steps", "e_in", "e_esc", "dropped")


# on 152 blocks: one history, one block's first, whole draws of 28 on 4 warps and one more, all 32 warps
# at 28 and one more, and more than a draw of 32 each
@pytest.mark.parametrize("particle,keV,N", [(1, 15000.0, n) for n in (1, 27, 152 * 28 * 4, 152 * 28 * 4 + 1, 152 * 28 * 32, 152 * 28 * 32 + 1)] +
                         [(0, 6000.0, n) for n in (1, 152 * 28 * 4 + 1, 152 * 28 * 32 + 1, 200001)] + [(1, 3000.0, 200001)])
def test_tally_does_not_depend_on_the_draw(ocmc, particle, keV, N):
    ph = I.ct_like((32, 32, 32), (0.75, 0.75, 0.75))
    beam = I.beam_on(ph, particle, I.mono(keV * 1e-3), (8.0, 8.0), 100.0)
    ref = None
    for kw in (dict(block_threads=256, max_registers=80, e_class_split=0.0, refill_min=1), {}, dict(refill_min=32),
               dict(e_class_split=6.0, block_threads=32, blocks_per_sm=2), dict(switch_low=0, e_class_split=1.0)):
        with ocmc.Engine(0, n_batches=3, **kw) as e:
            e.create_phantom(ph)
            e.set_source(beam)
            e.run(N, seed=9)
            t, s = e.raw_tally(), e.stats()
        assert s["histories"] == N and s["dropped"] == 0
        if ref is None:
            ref = t, s
        assert np.array_equal(t, ref[0]), kw
        for k in KEYS:
            assert s[k] == ref[1][k], (kw, k)
