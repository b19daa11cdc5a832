"""A tally that the GPU can address is added from wherever it lies: device memory or pinned host memory;
onto a cleared tally (a copy) as onto a filled one (a kernel)."""
import ctypes as C

import numpy as np
import pytest

import ocmc_inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("where", ["device", "pinned", "host"])
def test_memory_of_an_added_tally(where):
    import torch

    from paper_1503_01722_gb300 import build
    build.build()
    from paper_1503_01722_gb300 import ocmc
    ph = I.homogeneous((13, 11, 9), (0.3, 0.2, 0.4))
    t = np.random.default_rng(1).integers(0, 1 << 40, (3,) + ph.density.shape, dtype=np.int64)
    m = torch.from_numpy(t.copy())
    m = m.cuda() if where == "device" else m.pin_memory() if where == "pinned" else m
    torch.cuda.synchronize()
    with ocmc.Engine(0, n_batches=3) as e:
        e.create_phantom(ph)
        for k in (1, 2):
            st = ocmc.lib.ocmc_add_raw_tally(e._c, C.c_void_p(m.data_ptr()), int(where != "host"), 0, 10)
            assert st == ocmc.OK
            assert np.array_equal(e.raw_tally(), k * t)
