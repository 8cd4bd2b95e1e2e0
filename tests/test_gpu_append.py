"""trr_kv_append at the edges of its kernel: entry counts around the small and the large
instance (and their partly filled warps), entries that come sequence after sequence,
interleaved and in no order at all, one sequence and as many as entries, pages opened and
filled inside the call.  Bytes and metadata are those of the oracle."""
import numpy as np
import pytest
import torch

from paper_2607_06601_gb300 import workloads as wl
from tests._parity import Pair

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("order", ["sorted", "interleaved", "shuffled"])
@pytest.mark.parametrize("n,S", [(1, 1), (33, 5), (255, 3), (256, 256), (257, 7), (1023, 2), (1024, 1024), (1024, 1)])
def test_append_edges(n, S, order):
    rng = np.random.default_rng(n + S)
    d, G, P, Hkv = ((64, 32, 16, 3), (128, 64, 32, 1), (64, 64, 64, 2))[(n + S) % 3]
    maxctx = 2 * (n // S + 1) + 40
    pair = Pair(1, S, Hkv, Hkv, d, G, P, maxctx, [2 * S + 2 * n // P + 8] * 4)
    at = np.zeros(S, dtype=np.int64)
    for _ in range(2):  # the second call continues partly filled pages
        seqs = np.sort(np.concatenate([np.arange(S), rng.integers(0, S, n - S)])) if n >= S else np.arange(n)
        if order == "interleaved":
            seqs = seqs[np.argsort(np.arange(n) % max(1, n // S), kind="stable")]
        elif order == "shuffled":
            rng.shuffle(seqs)
        pos = np.empty(n, dtype=np.int64)
        for i, s in enumerate(seqs):
            pos[i] = at[s]
            at[s] += 1 + (at[s] < 8 and int(rng.integers(0, 2)))
        keep = pos < maxctx
        seqs, pos = seqs[keep], pos[keep]
        m = len(seqs)
        kv = [wl.bf16_bits(rng.standard_normal((m, Hkv, d), dtype=np.float32)) for _ in range(2)]
        pair.append(0, seqs, pos, kv[0], kv[1], rng.choice((2, 4, 8, 16), size=m), rng.choice(3, size=m))
        pair.check_regions()


@pytest.mark.parametrize("n", [200, 900])
def test_append_lowest_failing_entry(n):
    """Unsorted calls with two failing entries change nothing and report the lower one."""
    rng = np.random.default_rng(n)
    d, G, P, Hkv, S = 64, 32, 16, 2, 8
    pair = Pair(1, S, Hkv, Hkv, d, G, P, 4 * n, [4 * n] * 4)
    seqs = rng.integers(0, S, n)
    pos = np.arange(n)  # above every earlier position of the entry's sequence
    kv = wl.bf16_bits(rng.standard_normal((n, Hkv, d), dtype=np.float32))
    bits, modes = rng.choice((2, 4, 8, 16), size=n), np.full(n, 2)
    for lo, hi, want in ((n // 3, n // 2, 1), (n // 2, n // 3, 4)):
        p, b = pos.copy(), bits.copy()
        b[lo] = 3   # INVALID_ARG
        p[hi] = -1  # BAD_POSITION
        pair.append(0, seqs, p, kv, kv, b, modes, expect=want)
        pair.check_regions()
    pair.append(0, seqs, pos, kv, kv, bits, modes)
    pair.check_regions()
