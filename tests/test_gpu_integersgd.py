"""IntegerSGD's 32-bit divide and the limb planes it keeps: gradients on both
sides of 2^31, divisors around 2^31, weights that change limb count in both
directions or not at all.  The forward after each update reads the planes."""
import ctypes

import numpy as np
import pytest

import oracle as O
from oracle.nitro import integersgd, store32
from paper_2407_11698_gb300 import binding as nb
from paper_2407_11698_gb300 import synth

pytestmark = pytest.mark.gpu
C, L = nb.NITRO_CONV3X3, nb.NITRO_LINEAR

LAYERS = [(L, 64, 72, 1, 1, 0), (C, 64, 16, 8, 8, 0), (C, 36, 16, 8, 8, 0), (C, 3, 16, 8, 8, 0),
          (L, 13, 7, 1, 1, 0)]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("layer", LAYERS)
@pytest.mark.parametrize("trunc", [0, 1])
@pytest.mark.parametrize("gamma_lr,eta", [(1, 0), (512, 25000), (3355443, 2**31), (3355444, 2**31 + 7),
                                          (2**40, 2**45)])
def test_updates_and_planes(layer, trunc, gamma_lr, eta):
    import torch
    kind, cin, cout, h, w, pool = layer
    feat, n = h * w * cin, cout * cin * (9 if kind == C else 1)
    gamma = 640 * gamma_lr
    rng = np.random.default_rng(gamma_lr % 1000 + trunc)
    blk = nb.Block([layer], feat, max_batch=2, gamma_inv_lr=gamma_lr, eta_inv_fw=eta, sgd_round=trunc)
    ob = O.OracleBlock([O.LayerDesc(*layer)])
    x = synth.images(3, 0, 2, (h, w, cin) if kind == C else (cin,))
    out = torch.empty((2, blk.out_features), dtype=torch.int8, device="cuda")
    try:
        wt = rng.integers(-2**31, 2**31, n)
        wt[:n // 3] = rng.integers(-130, 131, n // 3)
        blk.set(nb.NITRO_T_W, 0, wt)
        for target in (100, 2**31 - 1, 30000, 127, 128, 0):
            # a step towards weights below `target`, then one that leaves most as they are
            goal = rng.integers(-target, target + 1, n)
            near = rng.integers(-2, 3, n) * (rng.random(n) < 0.1) * gamma
            for dw in ((wt - goal) * gamma + rng.integers(0, gamma, n), near,
                       rng.choice([-2**31 - 1, -2**31, 2**31 - 1, 2**31, -1, 0, 1], n)):
                dw = np.clip(dw.astype(object), -2**62, 2**62).astype(np.int64)
                blk.set(nb.NITRO_T_DW, 0, dw)
                blk.sgd()
                wt, _ = store32(integersgd(wt, dw, gamma, eta, trunc))
                assert np.array_equal(blk.get(nb.NITRO_T_W, 0, check=False), wt)
                ob.W[0] = wt.reshape(ob.W[0].shape)
                blk.forward(torch.from_numpy(x).cuda().reshape(2, -1), out)
                ob.forward(x.astype(np.int64))
                assert np.array_equal(out.cpu().numpy().reshape(-1), ob.act[0].reshape(-1))
    finally:
        blk.close()


def test_profile_counts_the_bytes_that_every_update_moves():
    # 12 bytes a weight are read (W, dW); stores depend on what changes
    lib = nb.lib()
    blk = nb.Block([(L, 64, 72, 1, 1, 0)], 64, max_batch=2)
    n, ms, ops, byts = ctypes.c_uint64(), ctypes.c_double(), ctypes.c_double(), ctypes.c_double()
    names = [lib.nitro_profile_kernel_name(k) for k in range(lib.nitro_profile_kernel_count())]
    try:
        lib.nitro_profile_reset()
        lib.nitro_profile_enable(1)
        blk.sgd()
        lib.nitro_profile_enable(0)
        assert lib.nitro_profile_read(names.index(b"integersgd"), ctypes.byref(n), ctypes.byref(ms),
                                      ctypes.byref(ops), ctypes.byref(byts)) == nb.NITRO_OK
        assert (n.value, byts.value) == (1, 12.0 * (64 * 72 + 72 * 10))
    finally:
        lib.nitro_profile_reset()
        blk.close()
