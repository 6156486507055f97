"""int64 outputs of the kernel-level contractions in stores of four, two or one value:
channel counts of every remainder by four at full and partial tiles, outputs at every
offset by 8 bytes; and small maps of eight channels on either side of the line to
the tensor cores."""
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


def check(B, h, w, cin, cout, off):
    import torch
    a = synth.int_tensor(1, (B, h, w, cin), -128, 127, dtype=np.int8)
    W = synth.int_tensor(2, (cout, 3, 3, cin), -30000, 30000, dtype=np.int32)
    d = synth.int_tensor(3, (B, h, w, cout), -2**20, 2**20, dtype=np.int32)
    a64, W64, d64 = (t.astype(np.int64) for t in (a, W, d))
    ad, Wd, dd = (torch.from_numpy(t).cuda() for t in (a, W, d))
    conv = nb.Conv3x3(B, h, w, cin, cout)
    try:
        for mode, x, y, want in ((nb.NITRO_CONTRACT_FWD, ad, Wd, O.conv3x3_fwd(a64, W64)),
                                 (nb.NITRO_CONTRACT_DGRAD, dd, Wd, O.conv3x3_dgrad(d64, W64))):
            out = torch.full((want.size + 8,), -77, dtype=torch.int64, device="cuda")
            conv.contract(mode, x, y, out[off:off + want.size])
            got = out.cpu().numpy()
            assert np.array_equal(got[off:off + want.size], want.reshape(-1)), mode
            assert (got[:off] == -77).all() and (got[off + want.size:] == -77).all()
        assert conv.status() == nb.NITRO_OK
    finally:
        conv.close()


@pytest.mark.parametrize("cin,cout", [(66, 24), (40, 34), (65, 130), (67, 64), (130, 72), (12, 6), (3, 38)])
@pytest.mark.parametrize("off", [0, 1, 2, 4])
def test_contractions_match_oracle(cin, cout, off):
    check(2, 9, 10, cin, cout, off)


@pytest.mark.parametrize("B,h,w,cin,cout", [(5, 3, 7, 8, 16), (3, 20, 1, 16, 8), (400, 7, 8, 8, 520), (2, 8, 8, 8, 8)])
def test_small_maps_of_eight_channels(B, h, w, cin, cout):
    check(B, h, w, cin, cout, 0)
