"""The tensor-core attention where its softmax references and its chunk merge can go wrong, against the
fp64 oracle (GPU only).

The reference of a row is the maximum over its item's first 128 keys.  bf16 outputs: 2e-2 absolute, as
everywhere for bf16 KV (P and the output are rounded to 8 bits; |V| is about 1 to 4 here).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2601_11652_gb300 import workload as wl  # noqa: E402
from paper_2601_11652_gb300.device_batch import DeviceBatch  # noqa: E402


def _check(b):
    db = DeviceBatch.from_host(b)
    db.attention()
    torch.cuda.synchronize()
    assert db.device_status() == (0, -1)
    err = np.max(np.abs(db.results()["out"] - oracle.attention(b)))
    assert err <= 2e-2, err


def _scale_keys(b, r, t0, t1, s):
    """Keys t0 .. t1 of request r times s (bf16 bits)."""
    for t in range(t0, t1):
        page = b.block_tables[r, t // 16]
        x = wl.bf16_bits_to_f32(b.k_cache[page, :, t % 16]) * np.float32(s)
        b.k_cache[page, :, t % 16] = wl.f32_to_bf16_bits(x)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("split", [False, True])  # one item per head, or chunks whose partials are merged
def test_scores_far_above_the_first_tile(D, split):
    """Keys past the first tile scaled so that scores exceed the first tile's maximum by well over 2^64
    for most rows (score sd 40 x log2 e), in the last rows' causal range too."""
    ctx, B = (3000, 2) if split else (700, 40)
    b = wl.make_batch_from_lengths("peaks", draft_lens=[5] * B, context_lens=[ctx + 7 * i for i in range(B)], Hq=32, Hkv=8,
                                   D=D, V=64, dtype="bf16", sigma=0.5, key=(170 + D, int(split)), shuffle_blocks=True)
    for r in range(0, B, 2):  # every other request: its neighbours stay ordinary
        n = int(b.context_lens[r]) + 6
        _scale_keys(b, r, 300, 340, 40.0)
        _scale_keys(b, r, n - 3, n, 40.0)
    _check(b)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("k, Hq, Hkv", [(0, 4, 4), (0, 32, 8), (4, 8, 2), (7, 32, 8), (8, 32, 8), (12, 28, 4), (15, 32, 8), (16, 32, 8)])
def test_rows_and_chunks(D, k, Hq, Hkv):
    """1 to 91 query rows per KV head (both softmax halves, one and two row groups, odd row counts in the
    merge), chunk ends on and next to tile and causal edges."""
    ctx = [0, 1, 127 - k, 128, 255, 256 + 128 - k, 2047, 2300]
    b = wl.make_batch_from_lengths("rows", draft_lens=[k] * len(ctx), context_lens=ctx, Hq=Hq, Hkv=Hkv, D=D, V=64,
                                   dtype="bf16", sigma=0.5, key=(180 + k, D), shuffle_blocks=True)
    _check(b)


def test_many_chunks():
    """One request and one KV head: over 32 chunks to merge."""
    b = wl.make_batch_from_lengths("chunks", draft_lens=[6], context_lens=[20001], Hq=4, Hkv=1, D=128, V=64, dtype="bf16",
                                   sigma=0.5, key=(190, 0))
    _check(b)
