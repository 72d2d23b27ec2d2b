"""A step that shares the SMs between its two kernels, against the fp64 oracle (GPU only): as many (request, head)
pairs as between the smallest share and all the SMs, a share for long contexts beside little vocabulary and the
reverse, and an fp32 cache with and without a share of its own for the acceptance.  Tolerances as everywhere: 2e-2
(bf16 KV), 1e-4 (fp32).  Its attention outputs are those of the attention entry point to the bit: where a
sequence is cut follows from the attention's inputs alone."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2601_11652_gb300 import workload as wl  # noqa: E402
from paper_2601_11652_gb300.device_batch import DeviceBatch  # noqa: E402


@pytest.mark.parametrize("dtype, B, Hq, Hkv, D, k, ctx, V", [
    ("bf16", 1, 8, 2, 128, (8, 8), (20000, 20000), 64),      # one request cut into its chunks, a share of about 40 of 152 SMs
    ("bf16", 40, 4, 1, 128, (0, 8), (0, 300), 60000),        # 40 pairs, the smallest share
    ("bf16", 6, 8, 8, 64, (0, 8), (20000, 30000), 64),       # 48 pairs, a share of about 110
    ("bf16", 16, 8, 8, 64, (0, 8), (5000, 9000), 300),       # 128 pairs, a share of about 100
    ("f32", 12, 4, 4, 64, (0, 8), (200, 900), 5000),         # 48 pairs, a share of about 50
    ("f32", 1, 32, 4, 64, (15, 15), (52000, 52000), 10),     # 13000 tile passes: every SM with the attention
])
def test_step_split(dtype, B, Hq, Hkv, D, k, ctx, V):
    rng = np.random.default_rng([B, D, V])
    b = wl.make_batch_from_lengths("split", draft_lens=rng.integers(k[0], k[1] + 1, B),
                                   context_lens=rng.integers(ctx[0], ctx[1] + 1, B), Hq=Hq, Hkv=Hkv, D=D, V=V, dtype=dtype,
                                   sigma=0.5, key=(310, B, V), shuffle_blocks=True)
    db = DeviceBatch.from_host(b)
    db.step()
    torch.cuda.synchronize()
    assert db.device_status() == (0, -1)
    got, ref = db.results(), oracle.accept(b)
    assert np.max(np.abs(got["out"] - oracle.attention(b))) <= (2e-2 if dtype == "bf16" else 1e-4)
    near = (ref["accept_margin"] < 1e-6) | (ref["sample_margin"] < 1e-9)
    assert np.all(near | ((got["accepted_len"] == ref["accepted_len"]) & (got["next_token"] == ref["next_token"])))


@pytest.mark.parametrize("V", [64, 30000])
@pytest.mark.parametrize("dtype, B, Hq, Hkv, D, k, ctx", [
    ("bf16", 1, 8, 2, 128, (8, 8), (20000, 20000)),      # fewer pairs than SMs
    ("bf16", 40, 28, 4, 128, (0, 8), (0, 6000)),         # 160 pairs of ragged lengths, the longest ones cut
    ("bf16", 20, 8, 4, 64, (0, 8), (5000, 9000)),        # 80 pairs: fewer than SMs, more than the attention's share
    ("f32", 40, 4, 4, 64, (0, 4), (0, 900)),
])
def test_step_attention_is_the_entry_points(dtype, B, Hq, Hkv, D, k, ctx, V):
    rng = np.random.default_rng([B, D, 3])
    b = wl.make_batch_from_lengths("bits", draft_lens=rng.integers(k[0], k[1] + 1, B),
                                   context_lens=rng.integers(ctx[0], ctx[1] + 1, B), Hq=Hq, Hkv=Hkv, D=D, V=V, dtype=dtype,
                                   sigma=0.5, key=(320, B, D), shuffle_blocks=True)
    db = DeviceBatch.from_host(b)
    bits = torch.int16 if dtype == "bf16" else torch.int32
    db.attention()
    alone = db.t["out"].view(bits).clone()
    db.t["out"].zero_()
    db.step()
    torch.cuda.synchronize()
    assert db.device_status() == (0, -1)
    assert torch.equal(db.t["out"].view(bits), alone)
