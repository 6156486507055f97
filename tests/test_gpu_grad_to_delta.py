"""The input gradient that goes through int64: rows and columns an odd map's pool cuts
off get a zero delta.  Each pooled block is made right after one without the pool,
whose deltas fill the same sizes of memory, was freed."""
import pytest

from paper_2407_11698_gb300 import binding as nb
from paper_2407_11698_gb300 import synth

from netpair import NetPair

pytestmark = pytest.mark.gpu
C, L = nb.NITRO_CONV3X3, nb.NITRO_LINEAR


@pytest.mark.parametrize("cin,cout,h,w,tail", [(4, 6, 7, 9, (L, 72, 20, 1, 1, 0)), (3, 5, 9, 5, (C, 5, 7, 4, 2, 0)),
                                               (3, 8, 6, 7, (L, 72, 16, 1, 1, 0))])
def test_matches_oracle(cin, cout, h, w, tail):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    for layers in ([(C, cin, cout, h, w, 0)], [(C, cin, cout, h, w, 1), tail]):
        pair = NetPair([{"layers": layers, "in_features": h * w * cin}], 50)
        try:
            for s in range(2):
                pair.step(synth.images(8, s, 50, (h, w, cin)), synth.labels(8, s, 50))
                pair.compare("step %d" % s)
        finally:
            pair.close()
