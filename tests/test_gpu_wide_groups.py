"""Query groups wider than 8 / (d / G) heads, whose units take that many heads of a group at a time (the
last of a group fewer), or one head in calls of few rows: decode steps, rows of several splits, calls with more units than warps,
skip tokens that store KV, failing queries."""
import numpy as np
import pytest
import torch

from paper_2607_06601_gb300 import workloads as wl
from tests._parity import Pair, dev
from tests.test_gpu_rows import _fill
from tests.test_gpu_step import _prefill, _steps

pytestmark = pytest.mark.gpu

SKIP, LOCAL, FULL = 0, 1, 2
LONG = 8192  # calls of 2^15 row elements and more take the wide units in a cache of that context
LAYOUTS = [  # d, G, P, Hq, Hkv
    (64, 32, 32, 12, 2), (64, 64, 16, 20, 2), (128, 128, 32, 9, 1), (128, 64, 32, 20, 4), (128, 32, 16, 6, 2), (128, 64, 64, 16, 2),
]


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("d,G,P,Hq,Hkv", LAYOUTS)
def test_steps_and_splits(d, G, P, Hq, Hkv):
    swk = LAYOUTS.index((d, G, P, Hq, Hkv)) % 2
    rng = np.random.default_rng(d + G + P + Hq + swk)
    ctxs = ([0, 1, 17, 100, 611, 31, 2500] * 13)[:90]
    ctxs = [c if c < 2500 or i == 6 else 200 for i, c in enumerate(ctxs)]
    maxctx = LONG
    pair = Pair(1, len(ctxs), Hq, Hkv, d, G, P, maxctx, [len(ctxs) * (260 // P + 2) + 2500 // P] * 4, skip_writes_kv=swk)
    _prefill(pair, rng, ctxs, Hkv, d)
    pos = _steps(pair, rng, ctxs, Hq, Hkv, d, 12)
    pair.check_regions()
    for win in (1, 40, 1200):
        q = wl.bf16_bits(rng.standard_normal((2 * len(ctxs), Hq, d), dtype=np.float32))
        pair.attend(0, list(range(len(ctxs))) * 2, [p - 1 for p in pos] + [p // 2 for p in pos], q,
                    rng.choice(3, size=2 * len(ctxs)), window_scalar=win)


@pytest.mark.parametrize("d,G,P,Hq,Hkv", LAYOUTS)
def test_more_units_than_warps(d, G, P, Hq, Hkv):
    """Two launches' worth of queries, some of them failing (the lowest one's error is reported), and
    calls of one head per unit before and after on the same cache."""
    rng = np.random.default_rng(Hq)
    S, ctx, n = 3, 400, 700
    pair = Pair(1, S, Hq, Hkv, d, G, P, ctx, [S * (ctx // P + 2)] * 4, max_queries=n)
    _prefill(pair, rng, [ctx] * S, Hkv, d)
    q = wl.bf16_bits(rng.standard_normal((n, Hq, d), dtype=np.float32))
    seqs, ts = rng.integers(0, S, n), rng.integers(0, ctx, n)
    modes, win = rng.choice(3, size=n), rng.integers(1, 400, n)
    few = slice(0, 2)  # its splits' arrivals are counted from zero
    for part in (few, slice(0, n), few, few):
        pair.attend(0, seqs[part], ts[part], q[part], modes[part], windows=win[part])
    ts[600], seqs[650] = ctx, S
    pair.attend(0, seqs, ts, q, modes, windows=win, expect=4)


@pytest.mark.parametrize("bits", [(2,), (4,), (8,), (16,), (2, 4, 8, 16)])
@pytest.mark.parametrize("d,G,P,Hq,Hkv", LAYOUTS)
def test_tile_edges(d, G, P, Hq, Hkv, bits):
    rng = np.random.default_rng(d + G + P + sum(bits))
    ctxs = [1, 15, 16, 17, 31, 32, 33, 63, 64, 65, 700, 1025]
    pair = Pair(1, len(ctxs), Hq, Hkv, d, G, P, LONG, [sum(ctxs) // P + 2 * len(ctxs)] * 4)
    _fill(pair, rng, ctxs, Hkv, d, bits)
    rep = -(-65536 // (len(ctxs) * Hq * d))
    seqs = np.tile(np.arange(len(ctxs)), rep)
    for modes, win in ((FULL, 0), (LOCAL, 1), (LOCAL, 33), (LOCAL, 300)):
        q = wl.bf16_bits(rng.standard_normal((len(seqs), Hq, d), dtype=np.float32))
        ts = [ctxs[s] - 1 if win != 33 else max(0, ctxs[s] - 20) for s in seqs]  # also with keys after the query
        pair.attend(0, seqs, ts, q, [modes] * len(seqs), window_scalar=win)
