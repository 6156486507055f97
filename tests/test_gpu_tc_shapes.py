"""Tensor-core conv layers at the shapes that padding and overhanging tiles bring in:
maps smaller than a tile side, channel counts below a K-block, output rows of
8-byte multiples; and the allocation-free forward on both of its routes."""
import numpy as np
import pytest

import oracle as O
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


# (cin, cmid, cout, h, w, pools, batch): two layers, so the second one's input gradient runs too
SHAPES = [(8, 16, 24, 5, 7, (0, 1), 9), (9, 24, 40, 3, 4, (0, 0), 5), (31, 8, 72, 7, 7, (1, 0), 3),
          (33, 40, 8, 2, 30, (0, 0), 2), (1, 8, 16, 1, 1, (0, 0), 17), (20, 56, 136, 6, 3, (0, 1), 8),
          (7, 12, 20, 4, 9, (0, 0), 3), (64, 64, 64, 4, 4, (0, 0), 11), (16, 104, 24, 9, 2, (1, 0), 6)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("scale", [1, 900, 70001])
def test_block_matches_oracle(shape, scale):
    cin, cmid, cout, h, w, (p0, p1), batch = shape
    h1, w1 = (h // 2, w // 2) if p0 else (h, w)
    pair = NetPair([{"layers": [(C, cin, cmid, h, w, p0), (C, cmid, cout, h1, w1, p1)],
                     "in_features": h * w * cin}], batch)
    try:
        for g, o in zip(pair.gb, pair.ob):
            for i in range(2):
                o.W[i] = np.clip(o.W[i] * scale, -2**31, 2**31 - 1)
                g.set(nb.NITRO_T_W, i, o.W[i].reshape(-1))
        for s in range(2):
            pair.step(synth.images(8, s, batch, (h, w, cin)), synth.labels(8, s, batch))
            pair.compare("step %d" % s)
    finally:
        pair.close()


# (batch, h, w, cin, cout, pool, offset of the outputs): below and above the line for
# narrow inputs, operands that fit the array and that do not, outputs that 8-byte
# stores cannot reach
NOALLOC = [(1, 10, 10, 3, 8, 1, 0), (16, 28, 28, 3, 64, 1, 0), (3, 9, 13, 32, 24, 1, 8), (2, 5, 7, 16, 40, 0, 0),
           (3, 9, 13, 32, 24, 1, 4), (2, 8, 8, 12, 20, 1, 0), (2, 4, 4, 256, 512, 0, 16), (1, 8, 8, 904, 16, 0, 0)]


@pytest.mark.parametrize("shape", NOALLOC)
def test_noalloc_matches_oracle(shape):
    import torch
    B, h, w, cin, cout, pool, off = shape
    for call, top in enumerate((100, 2**31 - 1, 30000)):
        x = synth.images(4, call, B, (h, w, cin))
        wt = np.random.default_rng(call).integers(-top, top + 1, (cout, 3, 3, cin)).astype(np.int32)
        n, m = B * h * w * cout, B * (h // 2) * (w // 2) * cout if pool else B * h * w * cout
        out, region, am = (torch.full((k + 32,), 99, dtype=torch.int8, device="cuda") for k in (m, n, m))
        xd, wd = torch.from_numpy(x).cuda(), torch.from_numpy(wt).cuda()
        st = nb.nitro_conv3x3_forward_noalloc(xd.data_ptr(), wd.data_ptr(), B, h, w, cin, cout, pool, 10,
                                              out.data_ptr() + off, region.data_ptr() + off,
                                              am.data_ptr() + off if pool else None,
                                              torch.cuda.current_stream().cuda_stream)
        assert st == nb.NITRO_OK
        z = O.conv3x3_fwd(x.astype(np.int64), wt.astype(np.int64))
        _, reg, act = O.scale_relu(z, 256 * 9 * cin, 10)
        arg = None
        if pool:
            act, arg = O.maxpool_fwd(act)
        for got, want, k in ((out, act, m), (region, reg, n), (am, arg, m)):
            if want is None:
                continue
            got = got.cpu().numpy()
            assert np.array_equal(got[off:off + k], want.reshape(-1))
            assert (got[:off] == 99).all() and (got[off + k:] == 99).all()


# lines of pixels below and at 16 channels, few channels above the earlier line for narrow inputs
@pytest.mark.parametrize("shape", [(3, 1, 62, 12, 40, 0, 0), (3, 1, 62, 16, 40, 0, 0), (2, 9, 1, 8, 16, 0, 0),
                                   (121, 12, 4, 2, 24, 0, 0)])
def test_noalloc_lines_match_oracle(shape):
    test_noalloc_matches_oracle(shape)
