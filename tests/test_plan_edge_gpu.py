"""The planner past one request per thread (1024), and with lengths it refuses but has to count, against the
fp64 oracle (GPU only).  Tolerances as everywhere: 2e-2 (bf16 KV), 1e-4 (fp32)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from gpu_util import ATTN_TOL, compare_accept  # noqa: E402
from paper_2601_11652_gb300 import workload as wl  # noqa: E402
from paper_2601_11652_gb300.device_batch import DeviceBatch  # noqa: E402


def _batch(B, dtype, k_hi, ctx_hi, V=64, long=None):
    rng = np.random.default_rng([B, ctx_hi])
    ctx = rng.integers(0, ctx_hi + 1, B)
    if long is not None:  # a few sequences long enough to be cut, on both sides of request 1024
        ctx[long] = 9000
    return wl.make_batch_from_lengths("many", draft_lens=rng.integers(0, k_hi + 1, B), context_lens=ctx, Hq=4, Hkv=2, D=64,
                                      V=V, dtype=dtype, sigma=0.5, key=(330, B, ctx_hi), shuffle_blocks=True)


@pytest.mark.parametrize("dtype, k_hi", [("bf16", 3), ("bf16", 40), ("f32", 3), ("f32", 40)])  # one row group, and several
@pytest.mark.parametrize("B", [1024, 1025, 2500])
def test_many_requests(B, dtype, k_hi):
    b = _batch(B, dtype, k_hi, 60, long=[3, 1000, min(1023, B - 1), B - 1])
    db = DeviceBatch.from_host(b)
    db.step()
    torch.cuda.synchronize()
    assert db.device_status() == (0, -1)
    got = db.results()
    assert np.max(np.abs(got["out"] - oracle.attention(b))) <= ATTN_TOL[dtype]
    compare_accept(b, got["accepted_len"], got["next_token"], oracle.accept(b))


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_refused_among_many(dtype):
    """Requests with a context past their table in both halves: flagged and skipped, the others as if alone."""
    b = _batch(2100, dtype, 3, 60)
    ref = oracle.attention(b)
    bad = [0, 700, 1023, 1024, 1500, 2099]
    b.context_lens[bad] = 16 * b.max_blocks_per_seq
    db = DeviceBatch.from_host(b)
    db.attention()
    torch.cuda.synchronize()
    code, rid = db.device_status()
    assert code == 1 and rid in b.request_ids[bad]
    qs, out = b.q_row_start(), db.results()["out"]
    for r in set(range(b.B)) - set(bad):
        assert np.max(np.abs(out[qs[r]:qs[r + 1]] - ref[qs[r]:qs[r + 1]])) <= ATTN_TOL[dtype]


@pytest.mark.parametrize("length", [(1 << 20) + 1, 1 << 30, 2**31 - 1])
@pytest.mark.parametrize("at", [5, 40, 1030])
def test_long_refused_lengths(at, length):
    """A draft length that is refused but counted in the offsets of the requests after it: those no longer fit the
    caller's buffers and are refused too, those before it are served."""
    b = _batch(1100, "bf16", 3, 60)
    ref, acc = oracle.attention(b), oracle.accept(b)
    qs = b.q_row_start()
    b.draft_lens = b.draft_lens.copy()
    b.draft_lens[at] = length
    b.draft_lens[at + 2] = 70000  # refused as well, below the length from which the sums are taken in two parts
    db = DeviceBatch.from_host(b)
    db.t["out"].zero_()
    db.step()
    torch.cuda.synchronize()
    assert db.device_status()[0] != 0
    got = db.results()
    assert np.max(np.abs(got["out"][:qs[at]] - ref[:qs[at]])) <= ATTN_TOL["bf16"]
    assert not got["out"][qs[at]:].any()
    near = (acc["accept_margin"][:at] < 1e-6) | (acc["sample_margin"][:at] < 1e-9)
    same = (got["accepted_len"][:at] == acc["accepted_len"][:at]) & (got["next_token"][:at] == acc["next_token"][:at])
    assert np.all(near | same)
    assert np.all(got["accepted_len"][at:] == -1) and np.all(got["next_token"][at:] == -1)
