"""The learning layer's backward launch: quads of channels and single channels,
class counts around its passes, batches around its sample tiles and slabs, odd maps
a pool cuts off, W_lr from one limb to an int32 overflow of delta_fw."""
import numpy as np
import pytest

from paper_2407_11698_gb300 import binding as nb
from paper_2407_11698_gb300 import synth

from netpair import NetPair

pytestmark = pytest.mark.gpu
C, L = nb.NITRO_CONV3X3, nb.NITRO_LINEAR


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# (layer, classes, batch)
SHAPES = [((L, 7, 1, 1, 1, 0), 1, 1), ((L, 33, 68, 1, 1, 0), 11, 65), ((L, 64, 63, 1, 1, 0), 16, 17),
          ((C, 3, 5, 7, 9, 1), 17, 16), ((C, 32, 36, 5, 11, 1), 64, 3), ((C, 8, 6, 3, 4, 0), 10, 15),
          ((C, 32, 24, 8, 8, 0), 2, 130), ((C, 16, 4, 2, 2, 1), 33, 64)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("wlr_max,fused", [(2, False), (3000, True), (2**20, False), (2**31 - 1, False)])
def test_matches_oracle(shape, wlr_max, fused):
    layer, G, batch = shape
    in_f = layer[1] * (layer[3] * layer[4] if layer[0] == C else 1)
    pair = NetPair([{"layers": [layer], "in_features": in_f}], batch, fused_update=fused, num_classes=G)
    try:
        o = pair.ob[0]
        o.Wlr = np.random.default_rng(3).integers(-wlr_max, wlr_max + 1, o.Wlr.shape)
        pair.gb[0].set(nb.NITRO_T_WLR, 0, o.Wlr.reshape(-1))
        shp = (layer[3], layer[4], layer[1]) if layer[0] == C else (layer[1],)
        for s in range(2):
            pair.step(synth.images(8, s, batch, shp), synth.labels(8, s, batch, G))
            pair.compare("step %d" % s)
    finally:
        pair.close()
