"""The table build's split work: compositions of 1 to 16 elements (the lanes take them eight at a time)
against the oracle's closed forms, the inverse range as the inverse of the range, and the screening
table against the oracle's solver over its whole range of path lengths."""
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


@pytest.fixture(autouse=True)
def _restore():
    yield
    O.reset_materials()


def composition(n):
    Z = [1, 6, 7, 8, 11, 12, 13, 14, 15, 16, 17, 19, 20, 26, 29, 30][:n]
    w = [1.0 / (k + 2) for k in range(n)]
    return {"Z": Z, "A": [2.05 * z + 0.1 for z in Z], "w": w, "I": 60.0 + 6.0 * n, "density": 1.0 + 0.1 * n}


@pytest.mark.parametrize("counts", [(1,), (7, 8, 9), (16, 15, 2)])
def test_tables_of_any_number_of_elements(ocmc, counts):
    defs = [composition(n) for n in counts]
    O.set_materials(defs)
    E = np.geomspace(0.0105, 29.0, 301).astype(np.float32)
    Ed = E.astype(np.float64)
    ph = I.homogeneous((8, 8, 8), (0.5, 0.5, 0.5))
    ph.material[:] = np.arange(512).reshape(8, 8, 8) % len(defs)
    with ocmc.Engine(0) as e:
        e.set_materials(defs)
        e.create_phantom(ph)
        for m in range(len(defs)):
            t = e.test_tables(m, E).astype(np.float64)
            # interpolation errors of 512 nodes: the bounds of the material tests
            for col, ch in ((0, 0), (1, 1), (2, 2)):
                assert np.max(np.abs(t[:, col] / O.mu(m, Ed, ch) - 1)) < 1e-3, (m, col)
            sel = Ed > 0.05
            assert np.max(np.abs(t[sel, 4] / O.lambda1_inv(m, Ed[sel]) - 1)) < 1e-3, m
            sb = O.sigma_brems(m, Ed)
            assert np.max(np.abs(t[:, 6] / sb - 1)) < 2e-3, m
            # inverse range: slowing down by the range difference of two energies ends at the lower one
            # (linear interpolation of the two tables between nodes 2 % apart: below 1e-3 in energy)
            R = t[:, 3].astype(np.float32)
            hi, lo = np.arange(60, 301), np.arange(40, 281)
            end = e.test_csda(m, E[hi], R[hi] - R[lo])
            assert np.max(np.abs(end / E[lo] - 1)) < 2e-3, m


def test_screening_table(ocmc):
    """cos theta = 1 - 2 A q / (1 + A - q), q = 1 - xi, with the oracle's A at each path length and the
    sample's own draw. The table is linear in ln A between nodes 0.059 apart in ln G1, where ln A bends by
    at most about 2 / (1 + A) of what 1 - cos theta feels: below 2e-3; FP32 near cos theta = 1: 3e-7."""
    n, seed = 6, 3
    x = np.array([ocmc.test_philox((seed, 0), j, 0, 0x5A5A + ocmc.SAMPLE_MS, 0, 1)[0, 0] for j in range(n)])
    q = 1.0 - ((x >> 8) + 1.0) * 2.0 ** -24
    ph = I.homogeneous((8, 8, 8), (0.5, 0.5, 0.5))
    with ocmc.Engine(0) as e:
        e.create_phantom(ph)
        for G1 in np.geomspace(1.01e-12, 14.99, 211):
            c = e.test_sample(ocmc.SAMPLE_MS, 1.0, n, seed=seed, aux=float(G1)).astype(np.float64)
            A = O.ms_solve_A(float(np.float32(G1)))
            ref = 2.0 * A * q / (1.0 + A - q)
            assert np.all(np.abs((1.0 - c) - ref) <= 2e-3 * ref + 3e-7), G1
