"""The one-pass fit of large datasets: sizes at its threshold, odd starts, the ends of
the byte range where the guesses are clamped, and data whose sampled mean misses mu,
so that the second pass runs, on one object in turn."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O
from paper_2407_11698_gb300 import binding as nb

THRESHOLD = 96 << 20
SAMPLES = 1 << 16


def sampled(n, off):
    """Start of every sampled 16-byte word (relative to x, which starts off bytes past a boundary)."""
    k = np.arange(SAMPLES, dtype=np.uint64)
    h = (k * np.uint64(2654435761)) & np.uint64(0xffffffff)
    h ^= h >> np.uint64(15)
    h = (h * np.uint64(0x85ebca6b)) & np.uint64(0xffffffff)
    share = np.uint64(((n - 15) >> 4) // SAMPLES)
    return (k * share + ((h * share) >> np.uint64(32))).astype(np.int64) * 16 + (-off) % 16


def data(kind, n, off):
    rng = np.random.default_rng(n + off)
    if isinstance(kind, int):
        return np.full(n, kind, dtype=np.uint8)
    x = np.clip(rng.normal(120, 60, n), 0, 255).astype(np.uint8)
    if kind == "miss":
        x[sampled(n, off)[:, None] + np.arange(16)] = 255
    elif kind == "low":
        x = (x > 250).astype(np.uint8)
    elif kind == "high":
        x = 255 - (x > 250).astype(np.uint8)
    return x


@pytest.mark.parametrize("n,off,kinds", [(THRESHOLD - 1, 0, ["natural", "miss"]),
                                         (THRESHOLD, 0, ["natural", "miss", 254, "miss", "high"]),
                                         (THRESHOLD + 37, 3, ["miss", 0, 255, "low", "natural"])])
def test_fit_matches_oracle(n, off, kinds):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = nb.IntPrep()
    try:
        for kind in kinds:
            x = data(kind, n, off)
            buf = torch.zeros(n + 64, dtype=torch.uint8, device="cuda")
            xd = buf[off:off + n]
            xd.copy_(torch.from_numpy(x))
            p.fit(xd)
            mu, om = O.prep_stats(x)
            assert p.stats() == (mu, om), kind
            out = torch.empty(n, dtype=torch.int8, device="cuda")
            p.apply(xd, out)
            lut = O.prep_apply(np.arange(256, dtype=np.uint8), mu, om)
            assert np.array_equal(out.cpu().numpy(), lut.astype(np.int8)[x]), kind
    finally:
        p.close()


# byte by byte where the offsets differ, and in two rounds of CTAs from 128 MB on
@pytest.mark.parametrize("n,xoff,ooff", [(3000001, 0, 3), (3000001, 5, 0), (200000, 1, 2), ((1 << 27) + 19, 0, 0),
                                         ((1 << 27) + 19, 7, 7)])
def test_map_matches_table(n, xoff, ooff):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = nb.IntPrep()
    try:
        x = data("natural", n, xoff)
        buf = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")
        xd = buf[xoff:xoff + n]
        xd.copy_(torch.from_numpy(x))
        out = torch.full((n + 16,), 99, dtype=torch.int8, device="cuda")
        p.fit(xd)
        p.apply(xd, out[ooff:ooff + n])
        lut = O.prep_apply(np.arange(256, dtype=np.uint8), *O.prep_stats(x)).astype(np.int8)
        got = out.cpu().numpy()
        assert np.array_equal(got[ooff:ooff + n], lut[x])
        assert (got[:ooff] == 99).all() and (got[ooff + n:] == 99).all()
    finally:
        p.close()


def test_profile_counts_the_bytes_that_a_fit_reads():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lib, p = nb.lib(), nb.IntPrep()
    names = [lib.nitro_profile_kernel_name(k) for k in range(lib.nitro_profile_kernel_count())]
    try:
        for n, want in ((THRESHOLD - 1, [THRESHOLD - 1] * 2), (THRESHOLD, [THRESHOLD + 16 * SAMPLES, 0])):
            x = torch.from_numpy(data("natural", n, 0)).cuda()
            lib.nitro_profile_reset()
            lib.nitro_profile_enable(1)
            p.fit(x)
            lib.nitro_profile_enable(0)
            got = []
            for name in (b"prep_sum", b"prep_mad"):
                c, ms, ops, by = ctypes.c_uint64(), ctypes.c_double(), ctypes.c_double(), ctypes.c_double()
                assert lib.nitro_profile_read(names.index(name), ctypes.byref(c), ctypes.byref(ms),
                                              ctypes.byref(ops), ctypes.byref(by)) == nb.NITRO_OK
                got.append(by.value)
            assert got == want
    finally:
        lib.nitro_profile_reset()
        p.close()
