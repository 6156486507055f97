"""Handles made while the default stream is busy, and used at once on another stream:
what their kernels sum into must be clean then, not when the default stream gets to
it; and a handle whose first call is captured."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O
from paper_2407_11698_gb300 import binding as nb
from paper_2407_11698_gb300 import synth

C = nb.NITRO_CONV3X3


@pytest.fixture
def side():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nb.lib()
    return torch.cuda.Stream()


def busy():
    torch.cuda.synchronize()
    torch.cuda._sleep(1 << 30)            # half a second, on the default stream


def still_busy():
    if torch.cuda.default_stream().query():
        pytest.skip("making the handle waited for the default stream: the test could not fail")


def test_prep(side):
    n = 100003
    with torch.cuda.stream(side):
        x = torch.randint(0, 256, (n,), dtype=torch.uint8, device="cuda")
    want = O.prep_stats(x.cpu().numpy())
    p = nb.IntPrep()                      # loads the kernels: that waits for the device
    p.fit(x, stream=side)
    p.close()
    busy()
    p = nb.IntPrep()
    try:
        p.fit(x, stream=side)
        still_busy()
        side.synchronize()
        assert p.stats() == want          # after the default stream's work too
    finally:
        p.close()


def test_block(side):
    cin, cout, h, w, batch = 20, 16, 9, 9, 3
    ob = O.OracleBlock([O.LayerDesc(C, cin, cout, h, w, 0)], in_features=h * w * cin, seed=5)
    x = synth.images(3, 0, batch, (h, w, cin))
    ob.forward(x.astype(np.int64))
    with torch.cuda.stream(side):
        xd = torch.from_numpy(x).cuda().reshape(batch, -1)
        out = torch.empty((batch, h * w * cout), dtype=torch.int8, device="cuda")
    blk = nb.Block([(C, cin, cout, h, w, 0)], h * w * cin, seed=5, max_batch=batch, stream=side)
    blk.forward(xd, out, stream=side)
    blk.close()
    busy()
    blk = nb.Block([(C, cin, cout, h, w, 0)], h * w * cin, seed=5, max_batch=batch, stream=side)
    try:
        still_busy()
        for _ in range(2):                # while the default stream is busy, and after
            blk.forward(xd, out, stream=side)
            side.synchronize()
            with torch.cuda.stream(side):
                got = out.cpu().numpy().reshape(-1)
            assert np.array_equal(got, ob.act[0].reshape(-1))
            torch.cuda.synchronize()
    finally:
        blk.close()


def test_gemm(side):
    m, n, k = 70, 72, 64
    a = synth.int_tensor(1, (m, k), -128, 127, dtype=np.int8)
    b = synth.int_tensor(2, (n, k), -30000, 30000, dtype=np.int32)
    with torch.cuda.stream(side):
        ad, bd = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
        c = torch.empty((m, n), dtype=torch.int64, device="cuda")
    g = nb.IntGemm(m, n, k)
    g.run(ad, bd, c, stream=side)
    g.close()
    busy()
    g = nb.IntGemm(m, n, k)
    try:
        still_busy()
        g.run(ad, bd, c, stream=side)
        side.synchronize()
        want = a.astype(np.int64) @ b.astype(np.int64).T
        with torch.cuda.stream(side):
            got = c.cpu().numpy()
        assert np.array_equal(got, want)
    finally:
        torch.cuda.synchronize()
        g.close()


def test_first_call_captured(side):
    # a graph captured before any eager call, launched after one: both start from clean sums
    x = torch.randint(0, 256, (100003,), dtype=torch.uint8, device="cuda")
    y = torch.randint(0, 40, (5000,), dtype=torch.uint8, device="cuda")
    p = nb.IntPrep()
    try:
        side.wait_stream(torch.cuda.current_stream())
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(side):
            with torch.cuda.graph(graph, stream=side):
                p.fit(x, stream=side)
        p.fit(y)
        assert p.stats() == O.prep_stats(y.cpu().numpy())
        for _ in range(2):
            graph.replay()
            assert p.stats() == O.prep_stats(x.cpu().numpy())
        p.fit(y)
        assert p.stats() == O.prep_stats(y.cpu().numpy())
    finally:
        p.close()
