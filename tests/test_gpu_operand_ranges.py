"""What the tensor cores' operands and sums keep of the attention's binary32 arithmetic: sums
whose codes cancel against the zero points, scores far below zero,
scales of very different sizes in one row."""
import numpy as np
import pytest
import torch

from paper_2607_06601_gb300 import workloads as wl
from tests._parity import Pair, dev

pytestmark = pytest.mark.gpu

SKIP, LOCAL, FULL = 0, 1, 2


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    torch.cuda.set_device(0)


def _ratio(got, ref):
    """The error of rows over that of rounding the exact rows to bf16 (1: nothing but the rounding)."""
    rounded = torch.from_numpy(ref).bfloat16().double().numpy()
    return np.sqrt(((got - ref) ** 2).mean() / ((rounded - ref) ** 2).mean())


@pytest.mark.parametrize("bits,outliers", [(2, True), (4, True), (8, False)])
@pytest.mark.parametrize("d,G,P,H,g", [(64, 32, 32, 16, 1), (128, 128, 32, 8, 1), (64, 64, 32, 2, 10), (128, 64, 32, 2, 8)])
def test_sums_add_nothing_to_the_rounding(d, G, P, H, g, bits, outliers):
    """Rows of 2000 keys in few splits, whose sums of p * s * c and of p * z are a hundred times
    the row and cancel: the error is that of rounding the exact row to bf16.  An error of 2^-23 of
    sums 100 times as large is under 1/30 of that rounding's (about 2^-9.2 of the row): in
    quadrature 1.0006 of it, and over 16384 elements the two correlate by less than 3 / 128 of
    2 / 30."""
    rng = np.random.default_rng(100 * bits + d)
    S, ctx = 1024 // d, 2000
    # (a cache of long contexts: a wide group's calls of these sizes take the units of several heads)
    pair = Pair(1, S, H * g, H, d, G, P, ctx if g == 1 else 8192, [S * (ctx // P + 2)] * 4, split_bytes=100000)
    chan = np.ones(H * d, dtype=np.float32)
    if outliers:
        chan[rng.permutation(H * d)[:max(1, H * d // 100)]] = 8
    for s in range(S):
        for p0 in range(0, ctx, 1000):
            kv = [wl.bf16_bits(rng.standard_normal((1000, H, d), dtype=np.float32) * chan.reshape(H, d))
                  for _ in range(2)]
            pair.append(0, np.full(1000, s), np.arange(p0, p0 + 1000), kv[0], kv[1], np.full(1000, bits),
                        np.full(1000, FULL))
    seqs = np.tile(np.arange(S), 1 if g == 1 else 4)  # (four times: rows enough for a wide group's units)
    q = wl.bf16_bits(rng.standard_normal((len(seqs), H * g, d), dtype=np.float32))
    got, ref = pair.attend(0, seqs, [ctx - 1] * len(seqs), q, [FULL] * len(seqs))
    ratio = _ratio(got, ref)
    assert ratio <= 1.0006 + 0.0016, f"{ratio:.5f} times the error of rounding the exact rows"


@pytest.mark.parametrize("d,G,P,Hq,Hkv", [(64, 32, 32, 4, 4), (64, 64, 16, 10, 1), (128, 64, 32, 8, 2)])
@pytest.mark.parametrize("bits", [8, 16])
@pytest.mark.parametrize("step", [False, True])
def test_every_score_far_below_zero(d, G, P, Hq, Hkv, bits, step):
    """Finite inputs whose scores all lie between -1e30 and -3.4e38: the largest one decides.
    (16-bit keys of 2^55 and queries of 2^55; 8-bit keys of 2^10 and queries of 2^98.)  Different
    keys' scores differ by 2^-8 of themselves at least, far above binary32's rounding and far
    beyond the softmax's reach, and the largest is one key's."""
    rng = np.random.default_rng(bits + d)
    ctx = 100
    pair = Pair(1, 2, Hq, Hkv, d, G, P, ctx + 8, [2 * ctx // P + 8] * 4)
    size = 2.0 ** 55 if bits == 16 else 2.0 ** 10
    qsize = 2.0 ** 55 if bits == 16 else 2.0 ** 98

    def rows(frac):  # every value of a key the same and negative: a constant group, scale 0
        k = np.broadcast_to((-size * (1 + frac)).astype(np.float32)[:, None, None], (len(frac), Hkv, d))
        return wl.bf16_bits(np.ascontiguousarray(k)), wl.bf16_bits(rng.standard_normal((len(frac), Hkv, d), dtype=np.float32))

    frac = (np.arange(ctx) + 20) * 37 % 101 / 101.0
    for s in range(2):
        pair.append(0, np.full(ctx, s), np.arange(ctx), *rows(frac), np.full(ctx, bits), np.full(ctx, FULL))
    q = wl.bf16_bits(np.full((2, Hq, d), qsize, dtype=np.float32))
    if step:
        # sequence 0's own token is above every key, sequence 1's below most
        _, ref = pair.step(0, [0, 1], [ctx, ctx + 1], *rows(np.array([-0.1, 0.9])), [bits, bits], [FULL, FULL], q)
    else:
        _, ref = pair.attend(0, [0, 1], [ctx - 1, 50], q, [FULL, FULL])
    assert (np.abs(ref).max(axis=-1) > 0).all()


# Rows whose parts differ in size: the weights and the query are kept with about as many bits as
# binary32 has, so that an error stays under 1/16 of the rounding to bf16 (2^-9): in quadrature
# 1.002 of it, and over 4096 elements the two correlate by less than 3 / 64 of 2 / 16.
MIXED = 1.002 + 0.006


def _rows(pair, seqs, ts, q):
    """Full queries' rows and the oracle's.  (Not Pair.attend: its absolute bound of 2e-2 beyond the
    rounding is for values of order 1; of rows of 2^13 it is 2^-18.6, which only the binary32 sums of
    a few keys would meet.)"""
    seqs, ts, modes = np.asarray(seqs, np.int32), np.asarray(ts, np.int32), np.full(len(seqs), FULL, np.uint8)
    out = pair.gpu.decode_attn(0, dev(seqs, torch.int32), dev(ts, torch.int32), dev(q, torch.bfloat16),
                               dev(modes, torch.uint8))
    st, ref = pair.orc.decode_attn(0, seqs, ts, q, modes)
    assert st == 0 and pair.gpu.status() == 0
    return out.double().cpu().numpy(), ref


def _mixed(pair, rng, ctx, Hkv, d, bits, kscale=1.0, vscale=1.0):
    """ctx tokens of one sequence; bits, kscale and vscale per token (the scales per dimension too)."""
    k, v = (rng.standard_normal((ctx, Hkv, d)) * x for x in (kscale, vscale))
    pair.append(0, np.zeros(ctx), np.arange(ctx), wl.bf16_bits(k), wl.bf16_bits(v), bits, np.full(ctx, FULL))


def test_constant_groups_then_tiny_scales():
    """Every 8-bit token's V groups are constant (scale 0), the 4- and 2-bit tokens that follow them
    have the smallest scales: the weights' power of two is chosen by the first scale that is not 0."""
    rng = np.random.default_rng(21)
    d, G, H, ctx = 64, 32, 64, 800
    pair = Pair(1, 1, H, H, d, G, 32, ctx, [ctx // 32 + 2] * 4, split_bytes=100000)
    bits = rng.choice((2, 4, 8), size=ctx)
    k = rng.standard_normal((ctx, H, d))
    v = np.where((bits == 8)[:, None, None], 2.0 ** -21, 2.0 ** -21 * rng.standard_normal((ctx, H, d)))
    pair.append(0, np.zeros(ctx), np.arange(ctx), wl.bf16_bits(k), wl.bf16_bits(v), bits, np.full(ctx, FULL))
    q = wl.bf16_bits(3 * rng.standard_normal((1, H, d)))
    got, ref = pair.attend(0, [0], [ctx - 1], q, [FULL])
    assert _ratio(got, ref) <= MIXED, _ratio(got, ref)


@pytest.mark.parametrize("d,G,H", [(64, 32, 64), (128, 32, 32)])
def test_groups_with_scales_far_apart(d, G, H):
    """V's first quantiser group is 2^26 times as large as the others."""
    rng = np.random.default_rng(22)
    ctx = 800
    pair = Pair(1, 1, H, H, d, G, 32, ctx, [ctx // 32 + 2] * 4, split_bytes=100000)
    size = np.where(np.arange(d) < G, 2.0 ** 12, 2.0 ** -14)
    _mixed(pair, rng, ctx, H, d, rng.choice((2, 4, 8), size=ctx), vscale=size)
    q = wl.bf16_bits(3 * rng.standard_normal((1, H, d)))
    got, ref = _rows(pair, [0], [ctx - 1], q)
    for part in (slice(0, G), slice(G, d)):
        assert _ratio(got[..., part], ref[..., part]) <= MIXED, _ratio(got[..., part], ref[..., part])


def test_large_scales_of_keys_without_weight():
    """Every 16th token has V scales 2^26 times as large as the others' and scores some 100 below
    theirs (e^-100 of the weight)."""
    rng = np.random.default_rng(23)
    d, G, H, ctx = 64, 32, 64, 800
    pair = Pair(1, 1, H, H, d, G, 32, ctx, [ctx // 32 + 2] * 4, split_bytes=100000)
    odd = np.arange(ctx) % 16 == 3
    q = np.abs(rng.standard_normal((1, H, d))) + 0.5
    k = rng.standard_normal((ctx, H, d)) + np.where(odd, -16.0, 0.0)[:, None, None]
    v = rng.standard_normal((ctx, H, d)) * np.where(odd, 2.0 ** 12, 2.0 ** -14)[:, None, None]
    pair.append(0, np.zeros(ctx), np.arange(ctx), wl.bf16_bits(k), wl.bf16_bits(v), rng.choice((2, 4, 8), size=ctx),
                np.full(ctx, FULL))
    got, ref = pair.attend(0, [0], [ctx - 1], wl.bf16_bits(q), [FULL])
    assert _ratio(got, ref) <= MIXED, _ratio(got, ref)


@pytest.mark.parametrize("bits", [(2,), (4,), (8,)])
def test_query_groups_far_apart(bits):
    """The query's first quantiser group is 2^28 times as large as its second, whose keys are as many
    times larger: both decide the scores."""
    rng = np.random.default_rng(24)
    d, G, H, ctx = 64, 32, 64, 800
    pair = Pair(1, 1, H, H, d, G, 32, ctx, [ctx // 32 + 2] * 4, split_bytes=100000)
    first = np.arange(d) < G
    _mixed(pair, rng, ctx, H, d, rng.choice(bits, size=ctx), kscale=np.where(first, 2.0 ** -14, 2.0 ** 13))
    q = wl.bf16_bits(rng.standard_normal((1, H, d)) * np.where(first, 2.0 ** 14, 2.0 ** -14))
    got, ref = pair.attend(0, [0], [ctx - 1], q, [FULL])
    assert _ratio(got, ref) <= MIXED, _ratio(got, ref)


@pytest.mark.parametrize("bits", [(2,), (4,), (8,)])
@pytest.mark.parametrize("d,G", [(64, 64), (64, 32), (128, 64)])
def test_query_group_with_parts_far_apart(d, G, bits):
    """A query group: each head's quantiser groups are 2^27 apart in the query, for which the keys make
    up, and one of the two heads is 2^28 times the other (its rows are one key's values)."""
    rng = np.random.default_rng(25)
    Hkv, ctx = 2048 // d, 800
    pair = Pair(1, 1, 2 * Hkv, Hkv, d, G, 32, ctx, [ctx // 32 + 2] * 4, split_bytes=100000)
    first = np.arange(d) < G
    kscale = np.where(first, 2.0 ** -14, 2.0 ** 13)
    _mixed(pair, rng, ctx, Hkv, d, rng.choice(bits, size=ctx), kscale=kscale)
    q = rng.standard_normal((1, 2 * Hkv, d)) / kscale
    q[:, 1::2] *= 2.0 ** 28
    got, ref = pair.attend(0, [0], [ctx - 1], wl.bf16_bits(q), [FULL])
    for h in (0, 1):
        assert _ratio(got[:, h::2], ref[:, h::2]) <= MIXED, _ratio(got[:, h::2], ref[:, h::2])


@pytest.mark.parametrize("d,G,P,Hq,Hkv", [(64, 32, 32, 64, 32), (64, 64, 16, 64, 16), (128, 64, 64, 32, 8), (128, 32, 32, 32, 16)])
@pytest.mark.parametrize("size", [2.0 ** -4, 2.0 ** -8, 2.0 ** -10, 2.0 ** -14, 2.0 ** -20])
def test_query_group_small_values(d, G, P, Hq, Hkv, size):
    """Query groups with small V: the low part of a weight is far above f16's end."""
    rng = np.random.default_rng(26)
    ctx = 800
    pair = Pair(1, 1, Hq, Hkv, d, G, P, ctx, [ctx // P + 2] * 4, split_bytes=100000)
    _mixed(pair, rng, ctx, Hkv, d, rng.choice((2, 4, 8), size=ctx), vscale=size)
    got, ref = pair.attend(0, [0], [ctx - 1], wl.bf16_bits(3 * rng.standard_normal((1, Hq, d))), [FULL])
    assert _ratio(got, ref) <= MIXED, _ratio(got, ref)


@pytest.mark.parametrize("d,G,Hq,Hkv", [(64, 32, 60, 10), (128, 64, 40, 8), (128, 32, 24, 8)])
def test_wide_group_scales_far_apart(d, G, Hq, Hkv):
    """Groups wider than 8 / (d / G) heads: V's first quantiser group is 2^26 times as large as the others, and large scales of keys
    without weight."""
    rng = np.random.default_rng(27)
    ctx = 800
    pair = Pair(1, 2, Hq, Hkv, d, G, 32, 8192, [2 * (ctx // 32 + 2)] * 4, split_bytes=100000)
    _mixed(pair, rng, ctx, Hkv, d, rng.choice((2, 4, 8), size=ctx), vscale=np.where(np.arange(d) < G, 2.0 ** 12, 2.0 ** -14))
    odd = (np.arange(ctx) % 16 == 3)[:, None, None]
    k = rng.standard_normal((ctx, Hkv, d)) - 16.0 * odd
    v = rng.standard_normal((ctx, Hkv, d)) * np.where(odd, 2.0 ** 12, 2.0 ** -14)
    pair.append(0, np.ones(ctx), np.arange(ctx), wl.bf16_bits(k), wl.bf16_bits(v), rng.choice((2, 4, 8), size=ctx),
                np.full(ctx, FULL))
    n = 32768 // (Hq * d) + 1  # of each sequence: rows enough for a wide group's units
    q = np.abs(3 * rng.standard_normal((2 * n, Hq, d))) + 0.5
    q[:n] = rng.standard_normal((n, Hq, d))
    got, ref = _rows(pair, [0] * n + [1] * n, [ctx - 1] * 2 * n, wl.bf16_bits(q))
    first = slice(0, n), slice(None)
    for part in ((*first, slice(0, G)), (*first, slice(G, d)), (slice(n, 2 * n),)):
        assert _ratio(got[part], ref[part]) <= MIXED, _ratio(got[part], ref[part])


@pytest.mark.parametrize("d,G,Hq,Hkv", [(64, 32, 4, 2), (128, 64, 8, 2), (64, 64, 16, 2)])
@pytest.mark.parametrize("sign", [1, -1])
def test_infinite_values_of_a_query_group(d, G, Hq, Hkv, sign):
    """A 16-bit token with an infinite value in one dimension of one KV head, also as the only key of
    a query (weight 1, whose low part is 0): infinite there, for the heads that read it, alone."""
    rng = np.random.default_rng(28)
    ctx, g = 200, Hq // Hkv
    pair = Pair(1, 1, Hq, Hkv, d, G, 32, ctx, [ctx // 32 + 2] * 4)
    k, v = (rng.standard_normal((ctx, Hkv, d)) for _ in range(2))
    bits = np.where(np.arange(ctx) % 5 == 0, 16, rng.choice((2, 4, 8), size=ctx))
    v[100, 1, 7] = sign * np.inf
    pair.append(0, np.zeros(ctx), np.arange(ctx), wl.bf16_bits(k), wl.bf16_bits(v), bits, np.full(ctx, FULL))
    q = wl.bf16_bits(rng.standard_normal((3, Hq, d)))
    i32 = lambda x: dev(np.array(x, np.int32), torch.int32)
    out = pair.gpu.decode_attn(0, i32([0, 0, 0]), i32([99, 100, ctx - 1]), dev(q, torch.bfloat16),
                               dev(np.array([FULL, LOCAL, FULL], np.uint8), torch.uint8), window_scalar=1)
    assert pair.gpu.status() == 0
    out = out.float().cpu().numpy()
    want = np.zeros(out.shape, dtype=bool)
    want[1:, g:2 * g, 7] = True
    assert np.array_equal(np.isinf(out), want) and not np.isnan(out).any() and (out[want] * sign > 0).all()
