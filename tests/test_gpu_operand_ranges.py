"""What the tensor cores' operands and sums keep of the attention's binary32 arithmetic: sums
whose codes cancel against the zero points."""
import numpy as np
import pytest
import torch

from paper_2607_06601_gb300 import workloads as wl
from tests._parity import Pair

pytestmark = pytest.mark.gpu

SKIP, LOCAL, FULL = 0, 1, 2


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("bits,outliers", [(2, True), (4, True), (8, False), (2, False)])
@pytest.mark.parametrize("d,G,P,H", [(64, 32, 32, 16), (128, 128, 32, 8)])
def test_sums_add_nothing_to_the_rounding(d, G, P, H, bits, outliers):
    """Rows of 2000 keys in few splits, whose sums of p * s * c and of p * z are a hundred times
    the row and cancel: the error is that of rounding the exact row to bf16.  An error of 2^-23 of
    sums 100 times as large is under 1/30 of that rounding's (about 2^-9.2 of the row): in
    quadrature 1.0006 of it, and over 16384 elements the two correlate by less than 3 / 128 of
    2 / 30."""
    rng = np.random.default_rng(100 * bits + d)
    S, ctx = 1024 // d, 2000
    pair = Pair(1, S, H, H, d, G, P, ctx, [S * (ctx // P + 2)] * 4, split_bytes=100000)
    chan = np.ones(H * d, dtype=np.float32)
    if outliers:
        chan[rng.permutation(H * d)[:H * d // 100]] = 8
    for s in range(S):
        for p0 in range(0, ctx, 1000):
            kv = [wl.bf16_bits(rng.standard_normal((1000, H, d), dtype=np.float32) * chan.reshape(H, d))
                  for _ in range(2)]
            pair.append(0, np.full(1000, s), np.arange(p0, p0 + 1000), kv[0], kv[1], np.full(1000, bits),
                        np.full(1000, FULL))
    q = wl.bf16_bits(rng.standard_normal((S, H, d), dtype=np.float32))
    got, ref = pair.attend(0, np.arange(S), [ctx - 1] * S, q, [FULL] * S)
    rounded = torch.from_numpy(ref).bfloat16().double().numpy()
    ratio = np.sqrt(((got - ref) ** 2).mean() / ((rounded - ref) ** 2).mean())
    assert ratio <= 1.0006 + 0.0016, f"{ratio:.5f} times the error of rounding the exact rows"
