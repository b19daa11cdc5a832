"""Calls of one context on different streams (torch's do not wait for the default one): every order of runs, resets
and uploads gives, bit for bit, what the same calls give one after the other on the default stream."""
import numpy as np
import pytest

import ocmc_inputs as I

pytestmark = pytest.mark.gpu

LONG, SHORT = 3_000_000, 200_000       # photons: the first are still in flight when the next calls are made


@pytest.fixture(scope="module")
def ocmc():
    from paper_1503_01722_gb300 import build
    build.build()
    from paper_1503_01722_gb300 import ocmc as m
    return m


@pytest.fixture(scope="module")
def streams():
    import torch
    return None, torch.cuda.Stream(), torch.cuda.Stream()


def engine(ocmc, ph, **kw):
    e = ocmc.Engine(0, **dict({"n_batches": 20}, **kw))
    e.create_phantom(ph)
    e.set_source(I.beam_on(ph, 0, I.spectrum_6mv(), (6.0, 6.0), 100.0))
    return e


@pytest.fixture(scope="module")
def ph():
    return I.ct_like(n=(96, 96, 96), voxel=(0.25, 0.25, 0.25), seed=3)


@pytest.fixture(scope="module")
def ref(ocmc, ph):
    """Tallies and statistics of a long run, a short one and both."""
    out = []
    for runs in ((LONG,), (SHORT,), (LONG, SHORT)):
        with engine(ocmc, ph) as e:
            for k, n in enumerate(runs):
                e.run(n, seed=11 + (n == SHORT))
            out.append((e.raw_tally(), e.stats()))
    return out


PAIRS = [(0, 1), (1, 0), (1, 2), (1, 1), (0, 0)]


@pytest.mark.parametrize("a,b", PAIRS)
def test_run_reset_run(ocmc, ph, ref, streams, a, b):
    with engine(ocmc, ph) as e:
        for _ in range(3):
            e.run(LONG, seed=11, stream=streams[a])
            e.reset()
            e.run(SHORT, seed=12, stream=streams[b])
            assert np.array_equal(e.raw_tally(), ref[1][0])
            s = e.stats()
            assert s["histories"] == SHORT and s["e_dep"] == ref[1][1]["e_dep"] and s["compton"] == ref[1][1]["compton"]
            e.reset()


@pytest.mark.parametrize("a,b", PAIRS)
def test_run_after_run(ocmc, ph, ref, streams, a, b):
    with engine(ocmc, ph) as e:
        e.run(LONG, seed=11, stream=streams[a])
        e.run(SHORT, seed=12, stream=streams[b])
        s = e.stats()
        assert np.array_equal(e.raw_tally(), ref[2][0])
        assert s["histories"] == LONG + SHORT and s["e_dep"] == ref[2][1]["e_dep"]


@pytest.mark.parametrize("a,b", [(0, 1), (1, 2), (2, 0)])
def test_new_batches_tables_source_and_phantom_behind_a_run(ocmc, ph, streams, a, b):
    import torch
    rec = np.zeros(5000, I.PS_DTYPE)
    rec["x"], rec["y"], rec["z"], rec["w"], rec["E"] = 12.0, 12.0, -1.0, 1.0, np.linspace(1.0, 6.0, len(rec))
    small = I.ct_like(n=(64, 64, 64), voxel=(0.25, 0.25, 0.25), seed=4)
    got = []
    for on in ((None, None), (streams[a], streams[b])):
        with engine(ocmc, ph) as e:
            r = []
            e.run(LONG, seed=1, stream=on[0])
            e.set_params(n_batches=8, e_abs_g=0.02)           # another tally and other tables
            e.run(SHORT, seed=2, stream=on[1])
            r.append(e.raw_tally())
            e.set_phase_space(rec)
            e.run(LONG, seed=3, stream=on[0])
            e.set_phase_space(np.roll(rec, 1)[:4000])         # over the records that the run still reads
            e.run(SHORT, seed=4, stream=on[1])
            r.append(e.raw_tally())
            e.run(LONG, seed=5, stream=on[0])
            e.create_phantom(small)
            e.run(SHORT, seed=6, stream=on[1])
            r += [e.raw_tally(), *e.dose()]
            out = torch.empty(small.density.shape, device="cuda"), torch.empty(small.density.shape, device="cuda")
            e.dose(out=out)
            r += [t.cpu().numpy() for t in out]
            got.append(r)
    for x, y in zip(*got):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("scale", [0.0, 1.0])             # dense tallies, hash tables
def test_beamlets_behind_and_before_a_run(ocmc, ph, streams, scale):
    bl = I.beamlets(ph, n_beamlets=9, seed=2, log10_mean=4.0, log10_sd=0.3, lo=1000, hi=50_000, offset=2.0)
    got = []
    for on in ((None, None), streams[1:]):
        with engine(ocmc, ph, beamlet_capacity_scale=scale) as e:
            e.set_beamlets(0, *I.spectrum_6mv(), bl)
            e.run(LONG, seed=1, stream=on[0])
            e.run_beamlets(seed=7, stream=on[1])
            e.run(SHORT, seed=2, stream=on[0])
            r = [x for item in e.beamlet_doses(raw=True) for x in item] + [e.raw_tally()]
            r += [x for item in [e.beamlet_dose(b) for b in range(9)] for x in item]
            got.append(r)
    for x, y in zip(*got):
        assert np.array_equal(x, y)


def test_a_captured_run(ocmc, ph, ref):
    import torch
    with engine(ocmc, ph) as e:
        e.run(SHORT, seed=12)                              # tables and stacks are there
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            e.run(SHORT, seed=12, stream=torch.cuda.current_stream())
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(e.raw_tally(), 2 * ref[1][0])
        e.run(SHORT, seed=12)                              # plain calls go on as before
        assert np.array_equal(e.raw_tally(), 3 * ref[1][0])


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("a,b", [(1, 1), (1, 0), (0, 1), (1, 2)])
def test_tally_added_behind_a_clear(ocmc, ph, ref, streams, a, b, device):
    """run, reset, add, run, add: the clear runs before the first addition, the runs before the additions."""
    import torch
    t = np.random.default_rng(5).integers(1, 1 << 40, (20,) + ph.density.shape, dtype=np.int64)
    put = torch.from_numpy(t).cuda() if device else t
    torch.cuda.synchronize()
    with engine(ocmc, ph) as e:
        for k in range(3):
            e.run(LONG, seed=11, stream=streams[a])
            if k == 1:
                e.create_phantom(ph)                       # clears as well
            else:
                e.reset()
            e.add_raw_tally(put, 0, 1000)
            if k == 2:
                assert np.array_equal(e.raw_tally(), t)
            e.run(SHORT, seed=12, stream=streams[b])
            e.add_raw_tally(put, 0, 1000)
            assert np.array_equal(e.raw_tally(), 2 * t + ref[1][0])
