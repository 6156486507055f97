"""NITRO-Scaling in the fused forward epilogue: z* = floor(z / SF) from z modulo
2^32 and an fp32 sum.  The rule is restated in numpy and compared with integer
division over limb sums at the edges of its error bound, then the kernel with
the oracle on weights of one to four limbs, with sums that cancel, at the
channel counts where the chunk count changes and where the rule stops."""
import numpy as np
import pytest

import oracle as O
from paper_2407_11698_gb300 import binding as nb
from paper_2407_11698_gb300 import synth

C = nb.NITRO_CONV3X3
MAX_BLOCKS = 128      # K-blocks of 64 the fused epilogue takes


def f32(x):
    return np.asarray(x, np.float64).astype(np.float32)


def quotient(v, sf, kb_total, pair_first):
    """z* clamped to [-200, 200] of limb sums v [limb][chunk][n], as the kernel
    computes it: limb pairs of a chunk together (pair_first) or limb by limb."""
    limbs, cpp = v.shape[0], v.shape[1]
    lo, zf = np.zeros(v.shape[2], np.int64), np.zeros(v.shape[2], np.float32)
    groups = [range(l, min(l + 2, limbs)) for l in range(0, limbs, 2)] if pair_first \
        else [[l] for l in range(limbs)]
    for g in groups:
        for c in range(cpp):
            t = f32(v[g[0], c])
            if len(g) == 2:
                t = f32(v[g[1], c] * 256.0 + t.astype(np.float64))
            zf = f32(t.astype(np.float64) * 2.0 ** (8 * g[0]) + zf)
            for l in g:
                lo += v[l, c] << (8 * l)
    wrap = lambda t: ((t + 2**31) & 0xffffffff) - 2**31      # noqa: E731
    rint = lambda t: np.clip(np.rint(t.astype(np.float64)), -2**31, 2**31 - 1).astype(np.int64)  # noqa: E731
    inv = np.float32(1.0) / np.float32(sf)
    csz = -(-kb_total // cpp)
    err = 2.0 ** (8 * (limbs - 1)) * 1.02 / 16 * csz * cpp * (cpp + 4.2)
    if err <= 0.25 * sf:
        q = np.clip(rint(zf * inv), -200, 200)
        return q + (wrap(lo - q * sf) < 0) * -1
    q1 = rint(zf * inv)
    r1 = wrap(lo - q1 * sf)
    q2 = rint(f32(r1) * inv)
    q = np.clip(q1 + q2 - (wrap(r1 - q2 * sf) < 0), -200, 200)
    return np.where(np.abs(zf) > err + 400.0 * sf, np.where(zf < 0, -200, 200), q)


@pytest.mark.parametrize("kb_total,cin", [(1, 1), (1, 3), (1, 7), (9, 32), (9, 64), (18, 128), (27, 160),
                                          (36, 256), (72, 512), (126, 896), (128, 896)])
@pytest.mark.parametrize("limbs", [1, 2, 3, 4])
@pytest.mark.parametrize("pair_first", [True, False])
def test_rule_matches_integer_division(kb_total, cin, limbs, pair_first):
    rng = np.random.default_rng(kb_total * 100 + limbs)
    cpp = -(-kb_total // 16)
    top = -(-kb_total // cpp) * 2**20      # |limb sum| of one chunk
    sf, n = 256 * 9 * cin, 60000
    sums = [rng.integers(-top, top + 1, (limbs, cpp, n)),
            rng.choice([-top, top], (limbs, cpp, n)),
            rng.integers(-3 * sf, 3 * sf, (limbs, cpp, n)).clip(-top, top)]
    # sums that cancel: the top limb's chunks add up to almost nothing
    c = rng.integers(-top, top + 1, (limbs, cpp, n))
    c[-1, -1] = (-c[-1, :-1].sum(0) + rng.integers(-2, 3, n)).clip(-top, top)
    sums.append(c)
    # sums next to a multiple of SF, where floor turns
    e = np.zeros((limbs, cpp, n), np.int64)
    e[0, 0] = (rng.integers(-130, 131, n) * sf + rng.integers(-1, 2, n)).clip(-top, top)
    sums.append(e)
    for v in sums:
        z = sum((v[l].sum(0) << (8 * l)) for l in range(limbs))
        got, want = quotient(v, sf, kb_total, pair_first), z // sf
        assert np.array_equal(np.clip(got, -128, 128), np.clip(want, -128, 128))


def _weights(kind, cout, cin, rng):
    top = {"limb1": 127, "limb2": 32639, "limb3": 8355711, "limb4": 2**31 - 1}
    if kind in top:
        return rng.integers(-top[kind], top[kind] + 1, (cout, 3, 3, cin))
    if kind == "edge":      # every digit of the split at -128
        return np.full((cout, 3, 3, cin), -(128 + 128 * 256 + 128 * 65536 + 127 * 2**24))
    w = rng.integers(-(2**30), 2**30, (cout, 3, 3, cin))      # neighbours cancel
    w[..., 1::2] = -w[..., ::2][..., :w[..., 1::2].shape[-1]] + rng.integers(-4000, 4000, w[..., 1::2].shape)
    return w


@pytest.mark.gpu
@pytest.mark.parametrize("cin,cout,hw,pool", [(3, 32, 9, 1), (1, 64, 8, 0), (64, 64, 10, 1), (128, 128, 8, 0),
                                              (160, 48, 8, 1), (512, 128, 4, 1), (896, 32, 8, 0),
                                              (904, 32, 8, 1)])
@pytest.mark.parametrize("kind", ["limb1", "limb2", "limb3", "limb4", "edge", "cancel"])
def test_kernel_matches_oracle(cin, cout, hw, pool, kind):
    import torch
    B, rng = 3, np.random.default_rng(cin + hw)
    w = _weights(kind, cout, cin, rng)
    x = synth.images(5, 0, B, (hw, hw, cin))
    if kind == "cancel":
        x[..., 1::2] = x[..., ::2][..., :x[..., 1::2].shape[-1]]
    blk = nb.Block([(C, cin, cout, hw, hw, pool)], hw * hw * cin, max_batch=B)
    ob = O.OracleBlock([O.LayerDesc(C, cin, cout, hw, hw, pool)])
    blk.set(nb.NITRO_T_W, 0, w.reshape(-1))
    ob.W[0] = w.astype(np.int64)
    out = torch.empty((B, blk.out_features), dtype=torch.int8, device="cuda")
    blk.forward(torch.from_numpy(x).cuda().reshape(B, -1), out)
    ob.forward(x.astype(np.int64))
    assert np.array_equal(out.cpu().numpy().reshape(-1), ob.act[0].reshape(-1))
    assert np.array_equal(blk.get(nb.NITRO_T_REGION, 0), ob.region[0].reshape(-1))
    if pool:
        assert np.array_equal(blk.get(nb.NITRO_T_ARGMAX, 0), ob.argmax[0].reshape(-1))
    blk.close()
