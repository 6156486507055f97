"""The fused forward with its K range shared out over a cluster: two, four and eight
CTAs a tile, K-blocks that do not divide, empty last parts, both tile widths, one
to four limbs with cancelling sums, pools; against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2407_11698_gb300 import binding as nb
from paper_2407_11698_gb300 import synth

pytestmark = pytest.mark.gpu
C = nb.NITRO_CONV3X3


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# (cin, cout, h, w, pool, batch)
SHAPES = [(128, 64, 8, 8, 0, 1), (128, 256, 8, 8, 1, 1), (512, 128, 4, 4, 1, 2), (192, 40, 9, 7, 1, 3),
          (256, 256, 16, 16, 0, 1), (320, 72, 5, 6, 0, 4), (896, 512, 4, 4, 1, 9), (128, 1024, 8, 16, 0, 3),
          (128, 128, 30, 31, 1, 1)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind", ["limb1", "limb2", "limb3", "limb4", "cancel"])
def test_matches_oracle(shape, kind):
    import torch
    cin, cout, h, w, pool, batch = shape
    rng = np.random.default_rng(cin + cout)
    top = {"limb1": 127, "limb2": 32639, "limb3": 8355711, "limb4": 2**31 - 1, "cancel": 2**30}[kind]
    wt = rng.integers(-top, top + 1, (cout, 3, 3, cin))
    x = synth.images(5, 0, batch, (h, w, cin))
    if kind == "cancel":
        wt[..., 1::2] = -wt[..., ::2] + rng.integers(-4000, 4000, wt[..., ::2].shape)
        x[..., 1::2] = x[..., ::2]
    blk = nb.Block([(C, cin, cout, h, w, pool)], h * w * cin, max_batch=batch)
    ob = O.OracleBlock([O.LayerDesc(C, cin, cout, h, w, pool)])
    blk.set(nb.NITRO_T_W, 0, wt.reshape(-1))
    ob.W[0] = wt.astype(np.int64)
    out = torch.empty((batch, blk.out_features), dtype=torch.int8, device="cuda")
    xs = torch.from_numpy(x).cuda().reshape(batch, -1)
    for _ in range(3):
        blk.forward(xs, out)
    ob.forward(x.astype(np.int64))
    assert np.array_equal(out.cpu().numpy().reshape(-1), ob.act[0].reshape(-1))
    assert np.array_equal(blk.get(nb.NITRO_T_REGION, 0), ob.region[0].reshape(-1))
    if pool:
        assert np.array_equal(blk.get(nb.NITRO_T_ARGMAX, 0), ob.argmax[0].reshape(-1))
    assert blk.status() == nb.NITRO_OK
    blk.close()
