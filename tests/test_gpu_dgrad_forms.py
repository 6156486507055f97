"""The fused input gradient's three ways to keep its sums: 32 bits with an fp32 sum
that decides OVERFLOW, 32 bits once OVERFLOW is latched, 64 bits for many limbs;
results around the int32 edge, both tile widths, with and without the
lower layer's pool, channel counts a tile cuts."""
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


# (channels of the lower layer, of the upper, h, w, lower layer pools, batch)
SHAPES = [(64, 64, 9, 10, 0, 3), (128, 72, 8, 8, 0, 3), (48, 320, 12, 9, 1, 2), (256, 64, 10, 16, 1, 2),
          (16, 24, 17, 5, 1, 4)]


@pytest.mark.parametrize("shape", SHAPES)
# largest |W_lr| and |W| of the upper layer: sums far inside int32, around its edge, over
# it with few limbs, over it with many
@pytest.mark.parametrize("wlr_max,w_max", [(60, 100), (3000, 20000), (30000, 30000), (3000000, 100),
                                           (2000000, 9000000), (20000000, 2**31 - 1)])
def test_matches_oracle(shape, wlr_max, w_max):
    c1, c2, h, w, pool, batch = shape
    h1, w1 = (h // 2, w // 2) if pool else (h, w)
    pair = NetPair([{"layers": [(C, 3, c1, h, w, pool), (C, c1, c2, h1, w1, 0)], "in_features": h * w * 3}],
                   batch, gamma_inv_lr=2**40)
    try:
        rng = np.random.default_rng(c1 + w_max % 1000)
        o, g = pair.ob[0], pair.gb[0]
        o.W[0] = rng.integers(-4000, 4001, o.W[0].shape)
        o.W[1] = rng.integers(-w_max, w_max + 1, o.W[1].shape)
        o.Wlr = rng.integers(-wlr_max, wlr_max + 1, o.Wlr.shape)
        for i in range(2):
            g.set(nb.NITRO_T_W, i, o.W[i].reshape(-1))
        g.set(nb.NITRO_T_WLR, 0, o.Wlr.reshape(-1))
        for s in range(2):       # the second step finds OVERFLOW latched where the first overflowed
            pair.step(synth.images(8, s, batch, (h, w, 3)), synth.labels(8, s, batch))
            pair.compare("step %d" % s)
    finally:
        pair.close()

