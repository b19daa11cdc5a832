"""Every beamlet's sparse list at once (ocmc_get_beamlet_sizes / _entries): dense tallies against hash
tables and against the one-beamlet call, on grids that do not fill their last chunk, and a context whose
phantom changes between runs."""
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


def plan(n, seed, count):
    ph = I.ct_like(n=n, voxel=tuple(24.0 / k for k in n), seed=seed)
    return ph, I.beamlets(ph, n_beamlets=count, seed=seed, log10_mean=3.2, log10_sd=0.4, lo=1, hi=20_000, offset=2.0)


@pytest.mark.parametrize("n,count", [((32, 32, 32), 5), ((33, 31, 29), 7), ((8, 8, 16), 3), ((5, 7, 11), 2), ((61, 40, 23), 40)])
def test_lists_of_dense_tallies_and_tables(ocmc, n, count):
    ph, bl = plan(n, 4, count)
    bl[-1]["iso"] = (-500.0, -500.0, -500.0)      # a beamlet that misses the phantom: an empty list
    spec = I.spectrum_6mv()
    res = []
    for scale in (0.0, 1.0):                      # dense tallies; hash tables
        with ocmc.Engine(0, beamlet_capacity_scale=scale) as e:
            e.create_phantom(ph)
            e.set_beamlets(0, *spec, bl)
            e.run_beamlets(seed=8)
            lists, plain = e.beamlet_doses(raw=True), e.beamlet_doses()
            one = [e.beamlet_dose(b) for b in range(count)]
        for (i, d, r), (pi, pd), (oi, od, orw) in zip(lists, plain, one):
            assert np.array_equal(i, oi) and np.array_equal(d, od) and np.array_equal(r, orw)
            assert np.array_equal(i, pi) and np.array_equal(d, pd)
        res.append(lists)
    assert len(res[0][-1][0]) == 0 and sum(len(x[0]) for x in res[0]) > 0
    for a, b in zip(*res):
        assert all(np.array_equal(x, y) for x, y in zip(a, b))


def test_a_new_phantom_gets_its_own_tallies(ocmc):
    spec = I.spectrum_6mv()
    with ocmc.Engine(0) as e:
        for n in ((16, 16, 16), (40, 30, 20), (30, 40, 20), (9, 9, 9)):
            ph, bl = plan(n, 2, 4)
            bl = [dict(b, iso=(12.0, 12.0, 12.0)) for b in bl]
            e.create_phantom(ph)
            if n == (16, 16, 16):
                e.set_beamlets(0, *spec, bl)
                first = bl
            e.run_beamlets(seed=3)
            got = e.beamlet_doses(raw=True)
            with ocmc.Engine(0, beamlet_capacity_scale=1.0) as f:
                f.create_phantom(ph)
                f.set_beamlets(0, *spec, first)
                f.run_beamlets(seed=3)
                ref = f.beamlet_doses(raw=True)
            for a, b in zip(got, ref):
                assert all(np.array_equal(x, y) for x, y in zip(a, b))


def test_entries_need_sizes_and_room(ocmc):
    import ctypes as C
    ph, bl = plan((16, 16, 16), 2, 3)
    with ocmc.Engine(0) as e:
        e.create_phantom(ph)
        e.set_beamlets(0, *I.spectrum_6mv(), bl)
        ptr = np.zeros(4, np.int64)
        p = C.c_void_p(ptr.ctypes.data)
        assert ocmc.lib.ocmc_get_beamlet_sizes(e._c, p) == ocmc.ERR_STATE
        e.run_beamlets(seed=1)
        assert ocmc.lib.ocmc_get_beamlet_entries(e._c, None, None, None, 0) == ocmc.ERR_STATE
        assert ocmc.lib.ocmc_get_beamlet_sizes(e._c, p) == ocmc.OK and ptr[3] > 0
        assert ocmc.lib.ocmc_get_beamlet_entries(e._c, None, None, None, int(ptr[3]) - 1) == ocmc.ERR_ARG
        assert ocmc.lib.ocmc_get_beamlet_entries(e._c, None, None, None, int(ptr[3])) == ocmc.OK
