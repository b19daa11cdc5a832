"""Phantom values at the edges of what is accepted, wherever in the grid they are."""
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


@pytest.mark.parametrize("value,ok", [(0.0, True), (-0.0, True), (1e-45, True), (30.0, True), (np.nextafter(np.float32(30), np.float32(31)), False),
                                      (-1e-45, False), (-1.0, False), (np.nan, False), (-np.nan, False), (np.inf, False), (-np.inf, False)])
def test_density_edges(ocmc, value, ok):
    n = (41, 40, 43)                          # more than one block of the check, the last one partial
    with ocmc.Engine(0) as e:
        for at in (0, 65535, 65536, 41 * 40 * 43 - 1):
            ph = I.homogeneous(n, (0.5, 0.5, 0.5))
            ph.density.ravel()[at] = value
            if ok:
                e.create_phantom(ph)
            else:
                with pytest.raises(ocmc.OcmcError, match="density") as x:
                    e.create_phantom(ph)
                assert x.value.status == ocmc.ERR_ARG


@pytest.mark.parametrize("material,ok", [(2, True), (3, False), (255, False)])
def test_material_edges(ocmc, material, ok):
    with ocmc.Engine(0) as e:
        for at in (0, 65535, 65536, 41 * 40 * 43 - 1):
            ph = I.homogeneous((41, 40, 43), (0.5, 0.5, 0.5))
            ph.material.ravel()[at] = material
            if ok:
                e.create_phantom(ph)
            else:
                with pytest.raises(ocmc.OcmcError, match="material"):
                    e.create_phantom(ph)
