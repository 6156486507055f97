"""The learning layer's cluster kernel and the loss the next kernel forms: feature
counts around the tile and the cluster split, odd rows, one to four limbs of
W_lr, class counts around a pass, batches around a group and above one loss CTA."""
import numpy as np
import pytest

import oracle as O
from paper_2407_11698_gb300 import binding as nb
from paper_2407_11698_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("d,G,B", [(1, 1, 1), (7, 3, 9), (255, 10, 8), (256, 10, 7), (257, 11, 16), (1000, 16, 33),
                                   (2048, 17, 5), (2051, 64, 3), (4096, 10, 64), (70000, 2, 3), (16, 64, 300),
                                   (600000, 10, 2), (40, 10, 2000)])
@pytest.mark.parametrize("top", [127, 32639, 8355711, 2**31 - 1, "edge"])
@pytest.mark.parametrize("offset", [0, 1])
def test_matches_oracle(d, G, B, top, offset):
    import torch
    if d == 600000 and top == 127:
        top = "edge3"        # every digit at -128 over many tiles: the 32-bit sums' limit
    blk = nb.Block([], d, max_batch=B, num_classes=G)
    ob = O.OracleBlock([], in_features=d, num_classes=G)
    rng = np.random.default_rng(d + G)
    if top in ("edge", "edge3"):
        w = np.full((G, d), -(128 + 128 * 256 + (128 * 65536 if top == "edge" else 127 * 65536)))
    else:
        w = rng.integers(-top, top + 1, (G, d))
    blk.set(nb.NITRO_T_WLR, 0, w.reshape(-1))
    ob.Wlr = w.astype(np.int64)
    x = synth.images(9, 0, B, (d,))
    if isinstance(top, str):
        x[:] = -128
    y = synth.labels(9, 0, B, G)
    buf = torch.zeros(B * d + 8, dtype=torch.int8, device="cuda")      # rows at an odd address
    xs = buf[offset:offset + B * d].view(B, d)
    xs.copy_(torch.from_numpy(x))
    loss = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    try:
        for _ in range(2):          # the second call meets the words the first one left
            blk.forward(xs)
            blk.backward(xs, torch.from_numpy(y).cuda(), loss)
            ob.forward(x.astype(np.int64))
            want = ob.backward(x.astype(np.int64), y.astype(np.int64))
            assert np.array_equal(blk.get(nb.NITRO_T_GRAD_L, 0, check=False), ob.grad_l.reshape(-1))
            assert int(blk.get(nb.NITRO_T_SSE, 0, check=False)[0]) == ob.sse
            assert int(loss.item()) == ob.sse // 2
            assert np.array_equal(blk.get(nb.NITRO_T_DWLR, 0, check=False), ob.dWlr.reshape(-1))
            assert blk.status_bits() == ob.status
    finally:
        blk.close()
