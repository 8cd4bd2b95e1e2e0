"""Splits of more tiles than a warp plans at once: a large split_bytes leaves a row fewer splits than
its tiles ask for, and a unit takes them in runs.  The cache's scratch and the static call's need stay
those of the splits."""
import numpy as np
import pytest
import torch

from paper_2607_06601_gb300 import trr, workloads as wl
from tests._parity import Pair, check_attention, dev

SKIP, LOCAL, FULL = 0, 1, 2
LAYOUTS = [  # d, G, P, Hq, Hkv, head_modes
    (128, 64, 64, 2, 2, 0), (128, 128, 32, 2, 2, 0), (128, 32, 16, 2, 2, 0), (64, 32, 16, 3, 3, 0), (64, 64, 64, 2, 2, 0),
    (128, 64, 64, 8, 2, 0), (64, 32, 16, 4, 1, 0), (128, 64, 64, 8, 1, 0), (128, 64, 64, 4, 2, 1), (64, 32, 16, 2, 2, 1),
]


def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    torch.cuda.set_device(0)


def _fill(pair, rng, ctxs, Hq, Hkv, d, bits, hm):
    for s, n in enumerate(ctxs):
        for p0 in range(0, n, 1024):
            m = min(n, p0 + 1024) - p0
            kv = [wl.bf16_bits(rng.standard_normal((m, Hkv, d), dtype=np.float32)) for _ in range(2)]
            pair.append(0, np.full(m, s), np.arange(p0, p0 + m), kv[0], kv[1], rng.choice(bits, size=m),
                        rng.choice(3, size=(m, Hq) if hm else m, p=[0.1, 0.3, 0.6]))


@pytest.mark.gpu
@pytest.mark.parametrize("bits", [(16,), (2, 4, 8, 16)])
@pytest.mark.parametrize("d,G,P,Hq,Hkv,hm", LAYOUTS)
def test_units_of_several_runs(d, G, P, Hq, Hkv, hm, bits):
    _cuda()
    rng = np.random.default_rng(d + P + Hq + len(bits))
    ctxs = [3000, 1500, 33, 0]
    pair = Pair(1, len(ctxs), Hq, Hkv, d, G, P, 3200, [sum(ctxs) // P + 30] * 4, split_bytes=1 << 20, head_modes=hm)
    _fill(pair, rng, ctxs, Hq, Hkv, d, bits, hm)
    n = len(ctxs)
    for t, win in (([2999, 1499, 32, 0], 900), ([2500, 700, 20, 0], 1800)):
        q = wl.bf16_bits(rng.standard_normal((2 * n, Hq, d), dtype=np.float32))
        modes = [[FULL] * n + [LOCAL] * n, rng.choice(3, size=(2 * n, Hq))][hm]
        pair.attend(0, list(range(n)) * 2, t * 2, q, modes, window_scalar=win)
    if not hm:
        for i in range(3):
            kv = [wl.bf16_bits(rng.standard_normal((n, Hkv, d), dtype=np.float32)) for _ in range(2)]
            pair.step(0, list(range(n)), [c + i for c in ctxs], kv[0], kv[1], rng.choice(bits, size=n), [FULL] * n,
                      wl.bf16_bits(rng.standard_normal((n, Hq, d), dtype=np.float32)))
    pair.check_regions()


@pytest.mark.gpu
def test_units_of_several_runs_give_up_a_wait():
    """The bounded waits hold in every run of tiles."""
    _cuda()
    rng = np.random.default_rng(6)
    S, ctx = 8, 1500
    pair = Pair(1, S, 8, 8, 128, 64, 64, ctx, [S * 26] * 4, split_bytes=1 << 20)
    _fill(pair, rng, [ctx] * S, 8, 8, 128, (2, 4, 8, 16), 0)
    q = wl.bf16_bits(rng.standard_normal((S, 8, 128), dtype=np.float32))
    args = [dev(x.astype(np.int32), torch.int32) for x in (np.arange(S), np.full(S, ctx - 1))]
    pair.gpu.set_wait_limit(1)
    pair.gpu.decode_attn(0, *args, dev(q, torch.bfloat16), dev(np.full(S, FULL, np.uint8), torch.uint8))
    assert pair.gpu.status() == 8
    pair.gpu.set_wait_limit(0)
    pair.attend(0, np.arange(S), [ctx - 1] * S, q, [FULL] * S)


@pytest.mark.parametrize("d,G,P,split_bytes,splits", [(128, 64, 64, 1 << 20, 19), (128, 64, 32, 1 << 20, 37),
                                                      (64, 32, 16, 1 << 20, 74), (128, 64, 64, 0, 365)])
def test_scratch_of_large_splits(d, G, P, split_bytes, splits):
    """A cache's scratch: two caches that differ in max_queries alone differ by their partials and
    arrival counters, which follow the splits of 32768 positions: one per split_bytes of 8-bit tokens, or
    per 28 pages."""
    Hq, n = 8, 1024
    need = [trr.trr_cache_required_bytes(trr.make_config(1, 1, Hq, Hq, d, G, P, 32768, [4] * 4, 1, q, split_bytes, 0, 0))
            for q in (n, 2 * n)]
    assert need[1] - need[0] == n * Hq * (4 * splits * (d + 4) + 4 * (1 + -(-splits // 32)))


@pytest.mark.gpu
def test_static_call_with_large_splits():
    """300 queries of 8 heads at 19 splits each need 25 of the static array's 32 MiB."""
    _cuda()
    rng = np.random.default_rng(7)
    d, G, P, H, ctx, n = 128, 64, 64, 8, 1200, 300
    pair = Pair(1, 1, H, H, d, G, P, 32768, [ctx // P + 2] * 4, max_queries=16, split_bytes=1 << 20)
    _fill(pair, rng, [ctx], H, H, d, (2, 4, 8, 16), 0)
    seqs, ts = np.zeros(n, np.int32), rng.integers(0, ctx, n).astype(np.int32)
    modes = np.where(np.arange(n) < 20, FULL, LOCAL).astype(np.uint8)
    q = wl.bf16_bits(rng.standard_normal((n, H, d), dtype=np.float32))
    out = torch.empty((n, H, d), dtype=torch.bfloat16, device="cuda")
    trr.trr_decode_attn_static(pair.gpu.handle, 0, dev(seqs, torch.int32), dev(ts, torch.int32), dev(q, torch.bfloat16),
                               dev(modes, torch.uint8), None, 40, 0.0, out)
    st, ref = pair.orc.decode_attn(0, seqs, ts, q, modes, None, 40)
    assert st == 0 and pair.gpu.status() == 0
    check_attention(out.float().cpu().numpy().astype(np.float64), ref, modes)
