"""A beamlet plan that stays while the context changes around it: parameters, phantoms, kinds of tally."""
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


def phantom(seed=4, n=(32, 30, 28)):
    return I.ct_like(n=n, voxel=tuple(24.0 / k for k in n), seed=seed)


def plan(ph, count=6):
    return I.beamlets(ph, n_beamlets=count, seed=5, log10_mean=3.3, log10_sd=0.3, lo=100, hi=20_000, offset=2.0)


def lists(e):
    return [a for item in e.beamlet_doses(raw=True) for a in item]


def same(a, b):
    return len(a) == len(b) and all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("scale", [0.0, 1.0])             # dense tallies, hash tables
@pytest.mark.parametrize("change", [{"e_abs_g": 0.05}, {"e_abs_e": 0.5}, {"w_cb": 0.05}, {"w_cc": 0.4}, {"d_maxs": 0.05},
                                    {"f_maxe": 0.2}, {"flags": 8}, {"beamlet_capacity_scale": 2.0},
                                    {"beamlet_capacity_scale": 0.0}, {"block_threads": 256, "refill_min": 20}])
def test_changed_parameters_hold_for_the_next_run(ocmc, scale, change):
    ph = phantom()
    bl = plan(ph)
    with ocmc.Engine(0, beamlet_capacity_scale=scale) as e:
        e.create_phantom(ph)
        e.set_beamlets(0, *I.spectrum_6mv(), bl)
        e.run_beamlets(seed=3)
        before = lists(e)
        e.set_params(**change)
        assert same(lists(e), before)                      # the last run's results stay
        e.run_beamlets(seed=3)
        got = lists(e)
        now = e.params
    with ocmc.Engine(0, params=now) as f:
        f.create_phantom(ph)
        f.set_beamlets(0, *I.spectrum_6mv(), bl)
        f.run_beamlets(seed=3)
        assert same(got, lists(f))
    physics = not set(change) & {"beamlet_capacity_scale", "block_threads"}
    assert same(got, before) != physics


@pytest.mark.parametrize("scale", [0.0, 1.0])
@pytest.mark.parametrize("n", [(32, 30, 28), (30, 28, 32), (20, 21, 22)])    # the same grid, as many voxels, another number
def test_a_new_phantom_drops_the_old_lists(ocmc, scale, n):
    first, second = phantom(), phantom(seed=9, n=n)
    bl = plan(first)
    spec = I.spectrum_6mv()
    with ocmc.Engine(0, beamlet_capacity_scale=scale) as e:
        e.create_phantom(first)
        e.set_beamlets(0, *spec, bl)
        e.run_beamlets(seed=3)
        before = lists(e)
        with pytest.raises(ocmc.OcmcError):                # refused: nothing changes
            e.create_phantom(density=second.density - 40.0, material=second.material, voxel=second.voxel)
        assert same(lists(e), before)
        e.create_phantom(second)
        for call in (lambda: e.beamlet_doses(), lambda: e.beamlet_doses(raw=True), lambda: e.beamlet_dose(0)):
            with pytest.raises(ocmc.OcmcError) as x:
                call()
            assert x.value.status == ocmc.ERR_STATE
        assert ocmc.lib.ocmc_get_beamlet_entries(e._c, None, None, None, 1 << 40) == ocmc.ERR_STATE
        e.run_beamlets(seed=3)
        got = lists(e)
    with ocmc.Engine(0, beamlet_capacity_scale=scale) as f:
        f.create_phantom(second)
        f.set_beamlets(0, *spec, bl)
        f.run_beamlets(seed=3)
        assert same(got, lists(f))


@pytest.mark.parametrize("scale", [0.0, 1.0])
def test_errors_belong_to_the_run_that_made_them(ocmc, scale):
    """Stacks of 64 records that are not switched on size overflow: reported by the dose of a dose run, or by a
    beamlet run, and by nothing after it."""
    ph = I.homogeneous((24, 24, 24), (0.5, 0.5, 0.5))
    bl = plan(ph, 40)
    narrow, wide = {"stack_capacity": 64, "switch_high": 1 << 20}, {"stack_capacity": 0, "switch_high": 0}

    def overflows(call):
        with pytest.raises(ocmc.OcmcError) as x:
            call()
        assert x.value.status == ocmc.ERR_OVERFLOW

    with ocmc.Engine(0, beamlet_capacity_scale=scale, e_abs_e=0.02, e_abs_g=0.01) as e:
        e.create_phantom(ph)
        e.set_source(I.beam_on(ph, 0, I.mono(18.0), (4.0, 4.0), 100.0))
        e.set_beamlets(0, *I.mono(18.0), bl)
        e.set_params(**narrow)
        e.run(400_000, seed=1)
        overflows(e.dose)
        e.set_params(**wide)
        for seed in (3, 3, 4):                             # sized, replayed, another seed
            e.run_beamlets(seed=seed)
            assert e.stats()["dropped"] == 0
        overflows(e.dose)                                  # the dose's error is still there
        e.reset()
        e.run(400_000, seed=1)
        e.set_params(**narrow)
        e.set_beamlets(0, *I.mono(18.0), [dict(b, n_histories=10_000) for b in bl])
        overflows(lambda: e.run_beamlets(seed=3))
        e.dose()


def test_memory_of_the_other_kind_is_given_back(ocmc):
    import torch
    ph = phantom(n=(128, 128, 96))
    bl = I.beamlets(ph, n_beamlets=64, seed=5, log10_mean=3.3, log10_sd=0.3, lo=100, hi=20_000, offset=2.0)
    dense = 8 * 64 * ph.density.size                       # 805 MB
    spec = I.spectrum_6mv()

    def used(e, scale):
        e.set_params(beamlet_capacity_scale=scale)
        e.set_beamlets(0, *spec, bl)
        e.run_beamlets(seed=1)
        r = lists(e)
        return torch.cuda.mem_get_info()[0], r

    with ocmc.Engine(0) as e:
        e.create_phantom(ph)
        free_dense, a = used(e, 0.0)
        free_tables, b = used(e, 1.0)                      # tables of some 50 MB
        free_again, c = used(e, 0.0)
    assert same(a, b) and same(a, c)
    assert free_tables - free_dense > 0.6 * dense
    assert abs(free_again - free_dense) < 0.1 * dense


@pytest.mark.parametrize("raw", [False, True])
def test_lists_where_the_host_does_not_pin(ocmc, monkeypatch, raw):
    import torch
    ph = phantom()
    with ocmc.Engine(0) as e:
        e.create_phantom(ph)
        e.set_beamlets(0, *I.spectrum_6mv(), plan(ph))
        e.run_beamlets(seed=1)
        ref = [a for item in e.beamlet_doses(raw=raw) for a in item]
        empty = torch.empty

        def refuse(*a, **k):
            if k.get("pin_memory"):
                raise RuntimeError("CUDA error: out of memory")
            return empty(*a, **k)

        monkeypatch.setattr(torch, "empty", refuse)
        assert same([a for item in e.beamlet_doses(raw=raw) for a in item], ref)
