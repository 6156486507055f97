"""Linear forwards large enough for the tensor cores, whose epilogue is fused: input
widths that end inside a K-block and at the limit of the error bound (and the general
route just above it), output widths inside a tile, batches around a tile, with and
without a K split, one to four limbs, sums near zero, two layers in a row, dropout at a later step."""
import numpy as np
import pytest

import oracle as O
from paper_2407_11698_gb300 import binding as nb
from paper_2407_11698_gb300 import synth

pytestmark = pytest.mark.gpu
L = nb.NITRO_LINEAR


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


SHAPES = [(129, [648, 640]), (64, [8192, 264]), (64, [8192, 104]), (70, [8200, 328]), (64, [3000, 328]), (1, [8000, 6024]),
          (200, [768, 768, 400]), (1000, [200, 328, 200])]


@pytest.mark.parametrize("batch,widths", SHAPES)
@pytest.mark.parametrize("kind", ["limb1", "limb2", "limb3", "limb4", "cancel"])
@pytest.mark.parametrize("p16", [0, 9830])
def test_matches_oracle(batch, widths, kind, p16):
    import torch
    descs = [(L, a, b, 1, 1, 0) for a, b in zip(widths, widths[1:])]
    rng = np.random.default_rng(batch)
    top = {"limb1": 127, "limb2": 32639, "limb3": 8355711, "limb4": 2**31 - 1, "cancel": 2**30}[kind]
    x = synth.images(5, 0, batch, (widths[0],))
    blk = nb.Block(descs, widths[0], max_batch=batch, seed=21, dropout_p16=p16)
    ob = O.OracleBlock([O.LayerDesc(*d) for d in descs], seed=21, dropout_p16=p16)
    try:
        for i, (a, b) in enumerate(zip(widths, widths[1:])):
            w = rng.integers(-top, top + 1, (b, a))
            if kind == "cancel":
                w[:, 1::2] = -w[:, ::2] + rng.integers(-4000, 4000, w[:, ::2].shape)
            blk.set(nb.NITRO_T_W, i, w.reshape(-1))
            ob.W[i] = w.astype(np.int64)
        if p16:
            blk.set(nb.NITRO_T_STEP, 0, np.array([5], dtype=np.uint32))
            ob.t = 5
        if kind == "cancel":
            x[:, 1::2] = x[:, ::2]
        out = torch.empty((batch, widths[-1]), dtype=torch.int8, device="cuda")
        xs = torch.from_numpy(x).cuda()
        for _ in range(2):
            blk.forward(xs, out)
        ob.forward(x.astype(np.int64))
        assert np.array_equal(out.cpu().numpy().reshape(-1), ob.act[-1].reshape(-1))
        for i in range(len(descs)):
            assert np.array_equal(blk.get(nb.NITRO_T_REGION, i), ob.region[i].reshape(-1))
        assert blk.status() == nb.NITRO_OK
    finally:
        blk.close()
