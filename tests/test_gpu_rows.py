"""The kernels with one query head per warp at the edges of their tiles and units: contexts
around 16, 32 and 64 keys and around a unit's most tiles, every width alone and mixed, pages
of every size, wide query groups, more than 32 query heads with a mode each, calls with more
units than warps, scales from the smallest binary16 up, infinite 16-bit values."""
import numpy as np
import pytest
import torch

from paper_2607_06601_gb300 import workloads as wl
from tests._parity import Pair, dev

pytestmark = pytest.mark.gpu

LOCAL, FULL = 1, 2
LAYOUTS = [  # d, G, P, Hq, Hkv: all read by the one-head-per-warp kernels
    (64, 32, 32, 3, 3), (64, 64, 16, 2, 2), (64, 32, 64, 16, 1), (128, 128, 32, 2, 2), (128, 64, 64, 3, 3),
    (128, 32, 16, 10, 2),
]


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    torch.cuda.set_device(0)


def _fill(pair, rng, ctxs, Hkv, d, bits, scale=1.0, modes=None):
    for s, n in enumerate(ctxs):
        for p0 in range(0, n, 1024):
            m = min(n, p0 + 1024) - p0
            kv = [wl.bf16_bits(scale * rng.standard_normal((m, Hkv, d), dtype=np.float32)) for _ in range(2)]
            md = np.full(m, FULL) if modes is None else modes(m)
            pair.append(0, np.full(m, s), np.arange(p0, p0 + m), kv[0], kv[1], rng.choice(bits, size=m), md)


@pytest.mark.parametrize("bits", [(2,), (4,), (8,), (16,), (2, 4, 8, 16)])
@pytest.mark.parametrize("d,G,P,Hq,Hkv", LAYOUTS)
def test_tile_edges(d, G, P, Hq, Hkv, bits):
    rng = np.random.default_rng(d + G + P + sum(bits))
    ctxs = [1, 15, 16, 17, 31, 32, 33, 63, 64, 65, 700, 1025]
    pair = Pair(1, len(ctxs), Hq, Hkv, d, G, P, max(ctxs) + 1, [sum(ctxs) // P + 2 * len(ctxs)] * 4)
    _fill(pair, rng, ctxs, Hkv, d, bits)
    for modes, win in ((FULL, 0), (LOCAL, 1), (LOCAL, 33), (LOCAL, 300)):
        q = wl.bf16_bits(rng.standard_normal((len(ctxs), Hq, d), dtype=np.float32))
        ts = [n - 1 if win != 33 else max(0, n - 20) for n in ctxs]  # also with keys after the query
        pair.attend(0, np.arange(len(ctxs)), ts, q, [modes] * len(ctxs), window_scalar=win)


@pytest.mark.parametrize("n", [300, 1030])
def test_more_units_than_warps(n):
    """Queries of every kind in one call: units are handed out, and queries above 256 are
    ordered in rounds (above 1024 in two launches)."""
    rng = np.random.default_rng(n)
    d, G, P, H, S, ctx = 64, 32, 32, 8, 4, 1500
    pair = Pair(1, S, H, H, d, G, P, ctx, [S * (ctx // P + 2)] * 4, max_queries=n)
    _fill(pair, rng, [ctx] * S, H, d, (2, 4, 8, 16), modes=lambda m: rng.choice(3, size=m))
    q = wl.bf16_bits(rng.standard_normal((n, H, d), dtype=np.float32))
    pair.attend(0, rng.integers(0, S, n), rng.integers(0, ctx, n), q, rng.choice(3, size=n),
                windows=rng.integers(1, 600, n))


@pytest.mark.parametrize("d,G,P,Hq,Hkv", [(64, 32, 32, 40, 40), (128, 64, 16, 36, 12)])
def test_many_heads_each_its_mode(d, G, P, Hq, Hkv):
    rng = np.random.default_rng(Hq)
    S, ctx = 3, 900
    pair = Pair(1, S, Hq, Hkv, d, G, P, ctx, [S * (ctx // P + 2)] * 4, head_modes=1)
    for s in range(S):
        kv = [wl.bf16_bits(rng.standard_normal((ctx, Hkv, d), dtype=np.float32)) for _ in range(2)]
        pair.append(0, np.full(ctx, s), np.arange(ctx), kv[0], kv[1], rng.choice((2, 4, 8, 16), size=ctx),
                    rng.choice(3, size=(ctx, Hq)))
    q = wl.bf16_bits(rng.standard_normal((S, Hq, d), dtype=np.float32))
    pair.attend(0, np.arange(S), [ctx - 1, 500, 40], q, rng.choice(3, size=(S, Hq)), window_scalar=70)


@pytest.mark.parametrize("scale,qscale", [(2.0 ** -20, 1.0), (2.0 ** -9, 2.0 ** 9), (3000.0, 2.0 ** -12), (1.0, 2.0 ** -30)])
def test_value_ranges(scale, qscale):
    """Scales near binary16's ends and queries far from 1: the f16 operands are rescaled by
    powers of two, so rows stay within the stated bar."""
    rng = np.random.default_rng(3)
    d, G, P, H, ctx = 64, 32, 32, 4, 500
    pair = Pair(1, 1, H, H, d, G, P, ctx, [ctx // P + 2] * 4)
    _fill(pair, rng, [ctx], H, d, (2, 4, 8, 16), scale)
    q = wl.bf16_bits(qscale * rng.standard_normal((1, H, d), dtype=np.float32))
    pair.attend(0, [0], [ctx - 1], q, [FULL])


def test_infinite_values_stay_in_their_rows():
    """A 16-bit token with an infinite value in one dimension: that dimension is infinite, the
    others and the queries before it are as without it."""
    rng = np.random.default_rng(8)
    d, G, P, H, ctx = 64, 32, 32, 2, 200
    pair = Pair(1, 1, H, H, d, G, P, ctx, [ctx // P + 2] * 4)
    k = wl.bf16_bits(rng.standard_normal((ctx, H, d), dtype=np.float32))
    v = rng.standard_normal((ctx, H, d), dtype=np.float32)
    bits = rng.choice((2, 4, 8), size=ctx)
    bits[::5] = 16
    v[100, 1, 7] = np.inf
    pair.append(0, np.zeros(ctx), np.arange(ctx), k, wl.bf16_bits(v), bits, np.full(ctx, FULL))
    q = wl.bf16_bits(rng.standard_normal((2, H, d), dtype=np.float32))
    out = pair.gpu.decode_attn(0, dev(np.zeros(2, np.int32), torch.int32), dev(np.array([99, ctx - 1], np.int32), torch.int32),
                               dev(q, torch.bfloat16), dev(np.full(2, FULL, np.uint8), torch.uint8)).float().cpu().numpy()
    assert pair.gpu.status() == 0
    want = np.isinf(np.zeros_like(out))
    want[1, 1, 7] = True
    assert np.array_equal(np.isinf(out), want) and not np.isnan(out).any() and out[1, 1, 7] > 0


GROUPS = [  # d, G, P, Hq, Hkv: read by the kernels with a KV head and its query group per warp
    (64, 32, 32, 4, 2), (64, 64, 16, 8, 1), (64, 64, 64, 12, 4), (128, 128, 32, 10, 2), (128, 64, 64, 8, 2),
    (128, 32, 16, 4, 2),
]


@pytest.mark.parametrize("bits", [(2,), (4,), (8,), (16,), (2, 4, 8, 16)])
@pytest.mark.parametrize("d,G,P,Hq,Hkv", GROUPS)
def test_group_tile_edges(d, G, P, Hq, Hkv, bits):
    test_tile_edges(d, G, P, Hq, Hkv, bits)


@pytest.mark.parametrize("n", [2, 50, 100, 200])
def test_rows_of_several_splits(n):
    """Calls of 64 to 6400 (query, head) rows with up to a dozen splits each: the kernel that
    merges them gives a row 8, 4, 2 and 1 warps."""
    rng = np.random.default_rng(n)
    d, G, P, Hq, Hkv, S, ctx = 64, 64, 16, 32, 8, 2, 3000
    pair = Pair(1, S, Hq, Hkv, d, G, P, ctx, [S * (ctx // P + 2)] * 4, max_queries=n)
    _fill(pair, rng, [ctx] * S, Hkv, d, (2, 4, 8, 16), modes=lambda m: rng.choice(3, size=m))
    q = wl.bf16_bits(rng.standard_normal((n, Hq, d), dtype=np.float32))
    pair.attend(0, rng.integers(0, S, n), np.r_[ctx - 1, rng.integers(0, ctx, n - 1)], q, rng.choice(3, size=n),
                windows=rng.integers(1, 900, n))
