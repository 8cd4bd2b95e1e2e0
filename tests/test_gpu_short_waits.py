"""A wait limit far below a copy's latency runs out in every call that waits, also in calls of a unit
or two: the first copies' limit counts from before they are issued."""
import numpy as np
import pytest
import torch

from paper_2607_06601_gb300 import workloads as wl
from tests._parity import Pair, dev

pytestmark = pytest.mark.gpu

FULL, TIMEOUT = 2, 8


@pytest.mark.parametrize("step", [False, True])
@pytest.mark.parametrize("d,G,P,Hq,Hkv", [(64, 64, 16, 16, 1), (64, 32, 32, 1, 1), (128, 64, 64, 2, 2)])
def test_small_calls_run_out(d, G, P, Hq, Hkv, step):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    torch.cuda.set_device(0)
    rng = np.random.default_rng(9)
    ctx = 300
    pair = Pair(1, 1, Hq, Hkv, d, G, P, ctx + 8, [ctx // P + 3] * 4)
    kv = [wl.bf16_bits(rng.standard_normal((ctx, Hkv, d), dtype=np.float32)) for _ in range(2)]
    pair.append(0, np.zeros(ctx), np.arange(ctx), kv[0], kv[1], rng.choice((2, 4, 8, 16), size=ctx), np.full(ctx, FULL))
    new = [wl.bf16_bits(rng.standard_normal((1, Hkv, d), dtype=np.float32)) for _ in range(2)]
    q = wl.bf16_bits(rng.standard_normal((1, Hq, d), dtype=np.float32))
    seq, at = (dev(np.array([x], np.int32), torch.int32) for x in (0, ctx if step else ctx - 1))
    mode, bits = (dev(np.array([x], np.uint8), torch.uint8) for x in (FULL, 4))
    k, v, qd = (dev(x, torch.bfloat16) for x in (*new, q))
    for i in range(20):  # with the code of the call in the instruction caches, and without
        pair.gpu.set_wait_limit(1)
        if step:
            pair.gpu.decode_step(0, seq, at, k, v, bits, mode, qd)
        else:
            pair.gpu.decode_attn(0, seq, at, qd, mode)
        assert pair.gpu.status() == TIMEOUT, i
        pair.gpu.set_wait_limit(0)
        if not step and i % 2:
            pair.attend(0, [0], [ctx - 1], q, [FULL])
    if step:
        pair.step(0, [0], [ctx], new[0], new[1], [4], [FULL], q)
    pair.check_regions()
