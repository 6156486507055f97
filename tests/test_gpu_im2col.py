"""The im2col pack of narrow inputs: every channel count it takes, rows that are and are
not whole words, inputs at odd addresses, several rows a CTA and a partial last
group, maps of one row or column, the widest row that shared memory holds."""
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


# (cin, h, w, batch)
@pytest.mark.parametrize("cin,h,w,batch", [(1, 28, 28, 90), (2, 13, 1, 200), (3, 33, 32, 70), (3, 1, 31, 3),
                                           (4, 37, 5, 300), (5, 6, 7, 400), (6, 9, 10, 150), (7, 11, 12, 900),
                                           (4, 2, 4094, 1), (1, 3, 16382, 1), (7, 2, 2338, 1)])
@pytest.mark.parametrize("offset", [0, 1])
def test_forward_matches_oracle(cin, h, w, batch, offset):
    import torch
    blk = nb.Block([(C, cin, 8, h, w, 0)], h * w * cin, max_batch=batch)
    ob = O.OracleBlock([O.LayerDesc(C, cin, 8, h, w, 0)])
    try:
        wt = np.random.default_rng(h).integers(-3000, 3001, (8, 3, 3, cin))
        blk.set(nb.NITRO_T_W, 0, wt.reshape(-1))
        ob.W[0] = wt.astype(np.int64)
        x = synth.images(5, 0, batch, (h, w, cin))
        buf = torch.zeros(x.size + 4, dtype=torch.int8, device="cuda")
        xs = buf[offset:offset + x.size].view(batch, -1)
        xs.copy_(torch.from_numpy(x).reshape(batch, -1))
        out = torch.empty((batch, blk.out_features), dtype=torch.int8, device="cuda")
        blk.forward(xs, out)
        ob.forward(x.astype(np.int64))
        assert np.array_equal(out.cpu().numpy().reshape(-1), ob.act[0].reshape(-1))
    finally:
        blk.close()
