"""Electron runs long enough to hold their hard events until several lanes of a warp have one: the tally and
the counts are those of a run that does not (the same histories on more warps)."""
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


KEYS = ("histories", "missed", "compton", "pair", "moller", "brems", "hard_fictitious", "annihilations", "escaped",
        "geo_crossings", "lane_steps", "e_in", "e_esc", "dropped")
# 152 blocks of one warp: from 64 histories a warp events wait
HELD = dict(block_threads=32, blocks_per_sm=1)
LINE = 152 * 64


@pytest.mark.parametrize("N,keV,params", [
    (LINE - 1, 6000.0, {}), (LINE, 6000.0, {}), (LINE + 1, 6000.0, {}), (30011, 25000.0, {}), (20000, 400.0, {}),
    (20000, 9000.0, {"flags": 1}), (20000, 9000.0, {"flags": 2}), (20000, 9000.0, {"flags": 8}),
    (20000, 12000.0, {"e_abs_g": 0.6, "w_cb": 0.6}), (20000, 12000.0, {"w_cc": 0.02, "e_abs_e": 0.02})])
def test_held_events_change_nothing(ocmc, N, keV, params):
    ph = I.ct_like((24, 24, 24), (1.0, 1.0, 1.0))
    beam = I.beam_on(ph, 1, I.mono(keV * 1e-3), (8.0, 8.0), 100.0)

    def run(**kw):
        with ocmc.Engine(0, n_batches=2, **params, **kw) as e:
            e.create_phantom(ph)
            e.set_source(beam)
            e.run(N, seed=4)
            return e.raw_tally(), e.stats()
    ref, st = run()                                        # 4864 warps: at most 7 histories each
    assert st["histories"] == N and st["dropped"] == 0
    for kw in (HELD, dict(HELD, stack_capacity=256), dict(HELD, stack_capacity=512, switch_high=40, switch_low=31),
               dict(HELD, refill_min=1, e_class_split=0.0), dict(HELD, refill_min=32), dict(HELD, max_registers=80),
               dict(HELD, max_registers=56)):
        t, s = run(**kw)
        assert np.array_equal(t, ref), kw
        for k in KEYS:
            assert s[k] == st[k], (kw, k)
