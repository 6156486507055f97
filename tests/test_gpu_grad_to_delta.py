"""The input gradient that goes through int64 (k_grad_to_delta) on odd maps: the row
and the column that the pool cuts off get a zero delta from the kernel, nothing
clears delta before it.  Each block is made in memory that was filled before."""
import ctypes

import numpy as np
import pytest

from paper_2407_11698_gb300 import binding as nb
from paper_2407_11698_gb300 import synth

from netpair import NetPair

pytestmark = pytest.mark.gpu
C, L = nb.NITRO_CONV3X3, nb.NITRO_LINEAR


def _fill_free_memory(torch):
    """Leaves the driver's small-allocation chunks full of ones; the returned addresses
    stay allocated, so that the chunks are kept."""
    torch.cuda.current_stream().synchronize()
    cu, held = ctypes.CDLL("libcuda.so.1"), []
    for size in (1 << 12, 1 << 14, 1 << 16, 1 << 18):
        ptrs = [ctypes.c_uint64() for _ in range((8 << 20) // size)]
        for p in ptrs:
            assert cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(size)) == 0
            assert cu.cuMemsetD8_v2(p, ctypes.c_ubyte(255), ctypes.c_size_t(size)) == 0
        torch.cuda.synchronize()
        for i, p in enumerate(ptrs):
            if i % 16 == 0:
                held.append(p)
            else:
                assert cu.cuMemFree_v2(p) == 0
    return cu, held


@pytest.mark.parametrize("cin,cout,h,w,tail", [(4, 6, 7, 9, (L, 72, 20, 1, 1, 0)), (3, 5, 9, 5, (C, 5, 7, 4, 2, 0)),
                                               (3, 8, 6, 7, (L, 72, 16, 1, 1, 0))])
def test_matches_oracle(cin, cout, h, w, tail):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    layers = [(C, cin, cout, h, w, 1), tail]
    batch = 50
    held = _fill_free_memory(torch)
    pair = NetPair([{"layers": layers, "in_features": h * w * cin}], batch)
    try:
        x = synth.images(8, 0, batch, (h, w, cin))
        pair.gb[0].forward(torch.from_numpy(x).cuda().reshape(batch, -1), None)
        before = pair.gb[0].get(nb.NITRO_T_DELTA, 0).reshape(batch, h, w, cout)
        cut = np.concatenate([before[:, 2 * (h // 2):].ravel(), before[:, :, 2 * (w // 2):].ravel()])
        if not cut.all():
            pytest.skip("delta's memory was clean: the test could not fail")
        for s in range(2):
            pair.step(synth.images(8, s, batch, (h, w, cin)), synth.labels(8, s, batch))
            pair.compare("step %d" % s)
    finally:
        pair.close()
        for p in held[1]:
            held[0].cuMemFree_v2(p)
