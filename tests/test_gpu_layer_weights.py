"""Single layers through the test entry, each call with other weights: the first convolution behind the packing of the
weights reads the packed ones, and so does the data gradient behind it."""
import numpy as np
import pytest

from oracle import unet as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,cin,cout", [(2, 32, 16), (2, 64, 32), (1, 16, 32), (0, 16, 16), (0, 32, 16)])
def test_new_weights_in_every_call(mode, cin, cout):
    from paper_1503_01722_gb300 import build
    build.build()
    from paper_1503_01722_gb300 import ocmc
    rng = np.random.default_rng(cin + cout + mode)
    taps, fine, coarse = (27 if mode == 0 else 8), (16, 16, 16), (8, 8, 8)
    gin, gout = (coarse if mode == 2 else fine), (coarse if mode == 1 else fine)
    fwd, back = {0: (U.conv3, U.conv3_dx), 1: (U.down, lambda d, w: U.down_dx(d, w, x.shape)), 2: (U.up, U.up_dx)}[mode]
    for _ in range(10):
        x = U.bf16(rng.standard_normal(gin + (cin,)))
        W = U.bf16(rng.standard_normal((taps, cin, cout)) / np.sqrt(taps * cin))
        dy = U.bf16(rng.standard_normal(gout + (cout,)))
        y, dx, _ = ocmc.unet_test_layer(mode, fine, cin, cout, x, W, dy)
        # stored in BF16: relative rounding 2^-9, and an absolute one where sums cancel
        for got, ref in ((y, fwd(x, W)), (dx, back(dy, W))):
            assert np.allclose(got, ref, rtol=8e-3, atol=1e-2 * np.abs(ref).max())
