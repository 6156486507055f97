"""Large batches: samples shared out over CTAs in the linear weight gradient and in
dW_lr, the general GEMM above its line and in the forward of many small CTAs, and the
forwards' lines between one launch, the tensor cores and the GEMM."""
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


def run(layers, in_f, shape, batch, w_max=600, wlr_max=60, classes=10, batch0=None, **hyper):
    pair = NetPair([{"layers": layers, "in_features": in_f}], batch, num_classes=classes, **hyper)
    rng = np.random.default_rng(2)
    try:
        o, g = pair.ob[0], pair.gb[0]
        for i in range(len(layers)):
            o.W[i] = rng.integers(-w_max, w_max + 1, o.W[i].shape)
            g.set(nb.NITRO_T_W, i, o.W[i].reshape(-1))
        o.Wlr = rng.integers(-wlr_max, wlr_max + 1, o.Wlr.shape)
        g.set(nb.NITRO_T_WLR, 0, o.Wlr.reshape(-1))
        # the smaller batch follows the larger one: sums start from zero again
        for s, b in enumerate((batch, batch0 or batch)):
            pair.step(synth.images(8, s, b, shape), synth.labels(8, s, b, classes))
            pair.compare("step %d" % s)
    finally:
        pair.close()


# (in, out, batch, batch of the second step): four slabs of 32 and on are shared out; 500 x 520 at
# 1600 is above the line to the GEMM; 64 x 64 at 1793 and 128 x 100 at 1025 are past the forward's
# line to the tensor cores, 16 x 24 at 1540 and 13 x 7 at 2600 past the line to the GEMM
@pytest.mark.parametrize("din,out,batch,batch0", [(13, 7, 97, 96), (13, 7, 2600, 129), (64, 16, 128, 1), (65, 17, 1000, 31),
                                                  (64, 64, 1793, 300), (128, 100, 1025, 200), (16, 24, 1540, 33),
                                                  (500, 520, 1600, 100), (257, 33, 1056, 1055)])
@pytest.mark.parametrize("w_max,drop", [(600, 0), (2**31 - 1, 9830)])
def test_linear_matches_oracle(din, out, batch, batch0, w_max, drop):
    run([(L, din, out, 1, 1, 0)], din, (din,), batch, w_max=w_max, batch0=batch0, dropout_p16=drop)


# (features, classes, batch): dW_lr of an output block, shared out from four slabs of 128 on (six
# where the features are no quads); 20000 features from 32 slabs on
@pytest.mark.parametrize("d,classes,batch", [(16, 10, 385), (16, 10, 513), (50, 47, 641), (50, 10, 900), (1024, 64, 1027),
                                             (20000, 2, 4097)])
@pytest.mark.parametrize("wlr_max", [60, 2**31 - 1])
def test_output_block_matches_oracle(d, classes, batch, wlr_max):
    run([], d, (d,), batch, wlr_max=wlr_max, classes=classes, batch0=17)


# dW_lr shared out beside the delta of a conv, with and without a learning pool
@pytest.mark.parametrize("layer,d_lr", [((C, 3, 16, 4, 4, 1), 0), ((C, 8, 12, 6, 6, 0), 60), ((C, 2, 5, 3, 3, 0), 0)])
@pytest.mark.parametrize("wlr_max", [60, 2**31 - 1])
def test_conv_block_matches_oracle(layer, d_lr, wlr_max):
    run([layer], layer[1] * layer[3] * layer[4], (layer[3], layer[4], layer[1]), 900, wlr_max=wlr_max,
        classes=26, batch0=40, d_lr=d_lr)
