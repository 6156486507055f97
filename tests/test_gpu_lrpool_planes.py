"""The learning-pool routing kernel that takes whole windows and writes delta's
limb planes: odd maps the pools cut off, windows of one row or column, several
row shares, split and unsplit weight gradients, one to four limbs of delta."""
import numpy as np
import pytest

from paper_2407_11698_gb300 import binding as nb
from paper_2407_11698_gb300 import synth

from netpair import NetPair

pytestmark = pytest.mark.gpu
C = nb.NITRO_CONV3X3


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# (cin, cout, h, w, 2x2 pool, d_lr, batch)
SHAPES = [(32, 32, 11, 13, 1, 128, 5), (32, 40, 9, 8, 0, 200, 3), (3, 16, 17, 9, 1, 16, 2),
          (32, 36, 8, 31, 0, 500, 4), (1, 20, 5, 7, 0, 50, 3), (32, 64, 16, 16, 1, 64, 1)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("wlr_max,fused", [(2, False), (3000, True), (2**20, False), (2**31 - 1, False)])
def test_matches_oracle(shape, wlr_max, fused):
    cin, cout, h, w, pool, d_lr, batch = shape
    pair = NetPair([{"layers": [(C, cin, cout, h, w, pool)], "in_features": h * w * cin}], batch,
                   fused_update=fused, d_lr=d_lr)
    try:
        o = pair.ob[0]
        o.Wlr = np.random.default_rng(3).integers(-wlr_max, wlr_max + 1, o.Wlr.shape)
        pair.gb[0].set(nb.NITRO_T_WLR, 0, o.Wlr.reshape(-1))
        for s in range(2):
            pair.step(synth.images(8, s, batch, (h, w, cin)), synth.labels(8, s, batch))
            pair.compare("step %d" % s)
    finally:
        pair.close()


# maps wider than 65536 columns, with several rows a window: (cin, cout, h, w, 2x2 pool, d_lr)
@pytest.mark.parametrize("shape", [(1, 4, 2, 70000, 0, 8192), (1, 4, 4, 70001, 1, 8192)])
def test_wide_map_matches_oracle(shape):
    cin, cout, h, w, pool, d_lr = shape
    pair = NetPair([{"layers": [(C, cin, cout, h, w, pool)], "in_features": h * w * cin}], 2, d_lr=d_lr)
    try:
        pair.step(synth.images(8, 0, 2, (h, w, cin)), synth.labels(8, 0, 2))
        assert np.any(pair.ob[0].delta[0][:, :, 65536:])     # gradients land past the column in question
        pair.compare("step 0")
    finally:
        pair.close()
