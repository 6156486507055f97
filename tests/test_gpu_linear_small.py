"""Linear layers on the one-launch CUDA-core kernels and across the line to the
tensor cores: widths around the tiles (256 inputs, 16 outputs, 64 x 16 of the
weight gradient), odd widths, batches around a group of eight and a slab of 32,
one to four limbs of W, dropout, the fused update."""
import numpy as np
import pytest

from paper_2407_11698_gb300 import binding as nb
from paper_2407_11698_gb300 import synth

from netpair import NetPair

pytestmark = pytest.mark.gpu
L = nb.NITRO_LINEAR


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# (in, out, batch); 1024 x 1024 at batch 33 and 49 straddle the two lines (32 M, 48 M products)
SHAPES = [(1, 1, 1), (63, 17, 9), (64, 16, 8), (257, 15, 7), (784, 100, 64), (100, 50, 33), (2049, 40, 3),
          (512, 64, 65), (1024, 1024, 33), (1024, 1024, 49)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("w_max", [100, 30000, 2**23 - 70000, 2**31 - 1])
@pytest.mark.parametrize("fused,drop", [(False, 0), (True, 9830)])
def test_matches_oracle(shape, w_max, fused, drop):
    din, out, batch = shape
    pair = NetPair([{"layers": [(L, din, out, 1, 1, 0)], "in_features": din}], batch, fused_update=fused,
                   dropout_p16=drop)
    try:
        w = np.random.default_rng(1).integers(-w_max, w_max + 1, pair.ob[0].W[0].shape)
        pair.ob[0].W[0] = w
        pair.gb[0].set(nb.NITRO_T_W, 0, w.reshape(-1))
        for s in range(2):
            pair.step(synth.images(8, s, batch, (din,)), synth.labels(8, s, batch))
            pair.compare("step %d" % s)
    finally:
        pair.close()
